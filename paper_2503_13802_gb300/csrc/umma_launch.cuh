// Definitions of umma_launch.h's launches, instantiated for UMMA_C8P and
// UMMA_NP by the including file.
#pragma once

#include "umma_conv.cuh"
#include "umma_launch.h"

namespace mh3d {
namespace unet {

template <int C8P, int NP, class OutT>
cudaError_t launch_umma_nb(const ConvSrc& s, const UmmaW& u, int N, const float* bias, int relu, const float* oscale,
                           OutT* out, int* status, cudaStream_t st)
{
    using G = umma::Geom<C8P, NP>;
    auto* fn = umma::k_conv_umma<C8P, NP, OutT>;
    constexpr size_t smem = G::smem();
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
    const int ntx = (s.W + umma::kX - 1) / umma::kX, nty = (s.H + umma::kY - 1) / umma::kY;
    // as many CTAs as fit: they hide each other's staging and epilogues (a
    // forward at 128x128x64 takes 833, 661, 599, 583 and 559 us with 1, 2, 3, 4
    // and 6 an SM), although shorter runs multiply more planes twice
    const int grid = (int)std::min<long long>((long long)ntx * nty * s.D, (long long)num_sms() * occ);
    fn<<<grid, umma::kT, smem, st>>>(s, u.w, N, bias, relu, oscale, out, ntx, nty, status,
                                     umma_pair() ? u.wp : nullptr);
    return cudaGetLastError();
}

template cudaError_t launch_umma_nb<UMMA_C8P, UMMA_NP, float>(const ConvSrc&, const UmmaW&, int, const float*, int,
                                                              const float*, float*, int*, cudaStream_t);
template cudaError_t launch_umma_nb<UMMA_C8P, UMMA_NP, __nv_bfloat16>(const ConvSrc&, const UmmaW&, int, const float*,
                                                                      int, const float*, __nv_bfloat16*, int*,
                                                                      cudaStream_t);

}  // namespace unet
}  // namespace mh3d
