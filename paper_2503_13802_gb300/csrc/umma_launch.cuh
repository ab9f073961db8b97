// Definitions of umma_launch.h's launches, instantiated for UMMA_C8P and
// UMMA_NP by the including file.
#pragma once

#include "umma_conv.cuh"
#include "umma_launch.h"

namespace mh3d {
namespace unet {
namespace {

// The warp-specialised form (umma_conv.cuh: producer, MMA and epilogue
// warps, one persistent CTA per SM, NS halo slots): MH3D_UMMA_WS=1.
bool umma_ws()
{
    const char* e = std::getenv("MH3D_UMMA_WS");
    return e && e[0] == '1';
}

// Output rows per tile of the tcgen05 kernel (MH3D_UMMA_ROWS = 1, 2 or 4).
int umma_rows()
{
    const char* e = std::getenv("MH3D_UMMA_ROWS");
    if (e && (e[0] == '1' || e[0] == '2' || e[0] == '4')) return e[0] - '0';
    return 2;
}

template <int C8P, int NP, int NB, int R, class OutT>
cudaError_t launch_umma_t(const ConvSrc& s, const __nv_bfloat16* Wu, int N, const float* bias, int relu,
                          const float* oscale, OutT* out, int* status, cudaStream_t st,
                          const __nv_bfloat16* Wpair = nullptr)
{
    using G = umma::Geom<C8P, NP, NB, R>;
    auto* fn = umma::k_conv_umma<C8P, NP, NB, R, OutT>;
    const size_t smem = G::smem();
    if (smem > (size_t)smem_optin()) return cudaErrorInvalidValue;
    // resident CTAs per SM, with the attributes set, once per device (the
    // attributes belong to the current device)
    constexpr int kDevs = 64;
    static int occ_dev[kDevs] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kDevs) return cudaErrorInvalidDevice;
    int& occ = occ_dev[dev];
    if (occ == 0) {
        cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        // the whole carveout to shared memory, so that several CTAs fit
        if (e == cudaSuccess) e = cudaFuncSetAttribute(fn, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
        if (e != cudaSuccess) return e;
        // resident CTAs per SM from the shared memory (each CTA also reserves
        // 1 KB), the registers and the threads; every resident CTA holds
        // G::kCols of the SM's 512 TMEM columns
        int smem_sm = 0, regs_sm = 0;
        cudaFuncAttributes fa{};
        if (cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&regs_sm, cudaDevAttrMaxRegistersPerMultiprocessor, dev) != cudaSuccess ||
            cudaFuncGetAttributes(&fa, fn) != cudaSuccess)
            return cudaErrorInvalidValue;
        const int by_smem = smem_sm / (int)(smem + fa.sharedSizeBytes + 1024);
        const int by_regs = regs_sm / std::max(1, fa.numRegs * umma::kT);
        occ = std::max(1, std::min(std::min(by_smem, by_regs), std::min(2048 / umma::kT, 512 / G::kCols)));
    }
    const long long tiles = (long long)((s.W + umma::kM - 1) / umma::kM) * ((s.H + R - 1) / R) * s.D;
    if (tiles > (1LL << 30)) return cudaErrorInvalidValue;
    const int grid = (int)std::min<long long>(tiles, (long long)num_sms() * occ);
    fn<<<grid, umma::kT, smem, st>>>(s, Wu, N, bias, relu, oscale, out, (int)tiles, status, Wpair);
    return cudaGetLastError();
}

template <int C8P, int NP, int NS, class OutT>
cudaError_t launch_umma_ws_t(const ConvSrc& s, const __nv_bfloat16* Wu, int N, const float* bias, int relu,
                             const float* oscale, OutT* out, int* status, cudaStream_t st)
{
    using G = umma::GeomWs<C8P, NP, NS>;
    auto* fn = umma::k_conv_umma_ws<C8P, NP, NS, OutT>;
    const size_t smem = G::smem();
    constexpr int kDevs = 64;
    static bool attr_dev[kDevs] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kDevs) return cudaErrorInvalidDevice;
    if (!attr_dev[dev]) {
        cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        attr_dev[dev] = true;
    }
    const long long tiles = (long long)((s.W + umma::kM - 1) / umma::kM) * s.H * s.D;
    if (tiles > (1LL << 30)) return cudaErrorInvalidValue;
    const int grid = (int)std::min<long long>(tiles, (long long)num_sms());   // one CTA per SM
    fn<<<grid, umma::kWsT, smem, st>>>(s, Wu, N, bias, relu, oscale, out, (int)tiles, status);
    return cudaGetLastError();
}

// The deepest halo ring that fits (4, 3 or 2 slots); false if none does.
template <int C8P, int NP, class OutT>
bool launch_umma_ws(const ConvSrc& s, const __nv_bfloat16* Wu, int N, const float* bias, int relu,
                    const float* oscale, OutT* out, int* status, cudaStream_t st, cudaError_t* err)
{
    const size_t lim = (size_t)smem_optin();
    if (umma::GeomWs<C8P, NP, 4>::smem() <= lim)
        *err = launch_umma_ws_t<C8P, NP, 4>(s, Wu, N, bias, relu, oscale, out, status, st);
    else if (umma::GeomWs<C8P, NP, 3>::smem() <= lim)
        *err = launch_umma_ws_t<C8P, NP, 3>(s, Wu, N, bias, relu, oscale, out, status, st);
    else if (umma::GeomWs<C8P, NP, 2>::smem() <= lim)
        *err = launch_umma_ws_t<C8P, NP, 2>(s, Wu, N, bias, relu, oscale, out, status, st);
    else
        return false;
    return true;
}

}  // namespace

// One halo buffer and accumulator per CTA, several CTAs per SM (the
// default), or two per CTA with the next tile staged during this tile's
// MMAs (MH3D_UMMA_NB=2, where it fits).  Measured at 128x128x64 (network
// forward, channels (8, 16, 32)): 0.576 ms with one, 0.847 ms with two
// (half the resident CTAs).
template <int C8P, int NP, class OutT>
cudaError_t launch_umma_nb(const ConvSrc& s, const UmmaW& u, int N, const float* bias, int relu, const float* oscale,
                           OutT* out, int* status, cudaStream_t st)
{
    if (umma_ws()) {
        cudaError_t err = cudaSuccess;
        if (launch_umma_ws<C8P, NP>(s, u.w, N, bias, relu, oscale, out, status, st, &err)) return err;
    }
    const char* e = std::getenv("MH3D_UMMA_NB");
    const bool two = e && e[0] == '2';
    if (two && umma::Geom<C8P, NP, 2>::smem() <= (size_t)smem_optin())
        return launch_umma_t<C8P, NP, 2, 1>(s, u.w, N, bias, relu, oscale, out, status, st);
    // two rows a tile where two such CTAs fit an SM, one where only one does
    // (32 source channels: 131 KB with two rows, four warps an SM; upsampled
    // 32 -> 16 at 128x128x64 took 242 us)
    const char* er = std::getenv("MH3D_UMMA_ROWS");
    int R = umma_rows();
    if (!(er && er[0]) && umma::Geom<C8P, NP, 1, 2>::smem() > (size_t)smem_optin() / 2) R = 1;
    const __nv_bfloat16* wp = umma_pair() ? u.wp : nullptr;
    if (R == 4 && umma::Geom<C8P, NP, 1, 4>::smem() <= (size_t)smem_optin())
        return launch_umma_t<C8P, NP, 1, 4>(s, u.w, N, bias, relu, oscale, out, status, st, wp);
    if (R >= 2 && umma::Geom<C8P, NP, 1, 2>::smem() <= (size_t)smem_optin())
        return launch_umma_t<C8P, NP, 1, 2>(s, u.w, N, bias, relu, oscale, out, status, st, wp);
    return launch_umma_t<C8P, NP, 1, 1>(s, u.w, N, bias, relu, oscale, out, status, st, wp);
}

template cudaError_t launch_umma_nb<UMMA_C8P, UMMA_NP, float>(const ConvSrc&, const UmmaW&, int, const float*, int,
                                                              const float*, float*, int*, cudaStream_t);
template cudaError_t launch_umma_nb<UMMA_C8P, UMMA_NP, __nv_bfloat16>(const ConvSrc&, const UmmaW&, int, const float*,
                                                                      int, const float*, __nv_bfloat16*, int*,
                                                                      cudaStream_t);

}  // namespace unet
}  // namespace mh3d
