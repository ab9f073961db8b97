// Pencil kernels of the MH3D operator on sm_103a.
//
// The separable PSF h_k = c_k X_k (x) Y (x) Z (drive axis x) turns the 3D
// circular convolution of Eq. portz into one 1D circular convolution per
// axis; every axis is applied by a kernel that owns whole pencils of that
// axis in shared memory, transforms them (Stockham, fft_smem.cuh),
// multiplies in the Fourier domain and transforms back.  No 3D spectrum is
// ever stored.
//
//   T pass (y or z): tiles of `cols` consecutive x columns at one position of
//     the other transverse axis; column pairs are packed as one complex
//     pencil (both kernels are real, so real and imaginary parts convolve
//     independently).  Optional fusions: input or output times b (B of
//     Eq. dN), the CG direction update p = r + beta p in the loader, and the
//     CG epilogue q = b w + lambda R p with the partial p^T q in the storer.
//   X forward: row pairs packed as complex pencils; one forward FFT of
//     length nx, then per harmonic the product with the drive-axis spectrum
//     folded over the s aliases (the row selector P of Eq. dN is exactly a
//     spectral fold), an inverse FFT of length nx/s and the phase
//     e^{i theta_k} (Sec. 4.4) on the store.
//   X adjoint: per harmonic the projection Re(e^{-i theta_k} y_k), a forward
//     FFT of length nx/s, the periodised spectrum (zero insertion P^T) times
//     conj of the drive spectrum, summed over k on chip, one inverse FFT.
//   X normal: the drive-axis part of A^T A, sum_k X_k^T P^T P X_k, which in
//     the Fourier domain couples only the s aliases of each frequency:
//     an s x s block per alias class, precomputed in FP64.
#include <algorithm>
#include <cstdint>
#include <cstdio>

#include "ops_kernels.cuh"
#include "ops_functors.cuh"
#include "ops_xrt.cuh"

namespace mh3d {

// The T pass of any length.  What bounds it: latency -- a CTA's load,
// transform and store run in turn -- so the first stage reads its operands
// from global memory straight into registers (its radix in flight per
// thread), the last stage writes from registers, the spectral product sits
// between the last forward and first inverse stage, and a length of two
// radices (up to 144, most up to 256) crosses shared memory twice, with two
// barriers and one butterfly per thread and stage.  Against the former
// kernel (radices 2, 3, 4, 8; up to ten stages and barriers, run-time
// divisions per butterfly): 162 x 108 x 81, a y pass 29 us before.
template <int MODE, bool EPI>
__global__ void __launch_bounds__(256, 2) k_tpass(const __grid_constant__ TArgs a)
{
    extern __shared__ float2 sm[];
    __shared__ double red[34];
    __shared__ float cgs[3];
    float beta = 0.f, alpha = 0.f;
    if (a.cg.flags && !cg_enter_cta(a.cg, a.pupdate != 0, &beta, &alpha, cgs)) return;
    const int n = a.n, P = a.cols / 2, lgP = 31 - __clz(P), nst = a.rp.nst;
    float2* tw = sm;
    float2* mu = tw + n;
    float2* s0 = mu + n;
    float2* s1 = s0 + n * P;
    cp_table(tw, a.tw, n);
    cp_table(mu, a.mult, n);
    const int x0 = blockIdx.x * a.cols;
    const int base = (int)((long long)blockIdx.y * a.os);
    DotAcc acc, acc2;
    const TLoad ld{&a, base, x0};
    const TStore st{&a, base, x0};
    float2* src = s0;
    float2* dst = s1;
    auto flip = [&]() {
        float2* t = src;
        src = dst;
        dst = t;
    };
    if constexpr (MODE != 0) {
        t_update<MODE>(a, base, x0, lgP, beta, alpha, s1);
        cp_table_wait();
        __syncthreads();
    }
    if (nst < 2) {
        // one butterfly is the whole convolution (length 1: a product)
        if constexpr (MODE == 0) {
            cp_table_wait();
            __syncthreads();
        }
        if (nst == 0) {
            for (int p = threadIdx.x; p < P; p += blockDim.x) {
                const float2 v = c_mul(MODE != 0 ? s1[p] : ld.at(p)(0), mu[0]);
                if constexpr (EPI) s0[p] = v;
                else st.at(p)(0, v);
            }
        } else if constexpr (EPI) {
            rt_conv_any(ld, BufSt{s0, P}, mu, stage_fwd(a.rp, 0), lgP, tw);
        } else if constexpr (MODE != 0) {
            rt_conv_any(BufLd{s1, P}, st, mu, stage_fwd(a.rp, 0), lgP, tw);
        } else {
            rt_conv_any(ld, st, mu, stage_fwd(a.rp, 0), lgP, tw);
        }
    } else {
        if constexpr (MODE != 0) {
            rt_stage_buf<false>(s1, s0, P, stage_fwd(a.rp, 0), lgP, tw);
        } else {
            rt_stage_any<false, true>(ld, BufSt{s0, P}, stage_fwd(a.rp, 0), lgP, tw);
            cp_table_wait();
        }
        __syncthreads();
        for (int s = 1; s < nst - 1; ++s, flip()) {
            rt_stage_buf<false>(src, dst, P, stage_fwd(a.rp, s), lgP, tw);
            __syncthreads();
        }
        rt_conv_any(BufLd{src, P}, BufSt{dst, P}, mu, stage_fwd(a.rp, nst - 1), lgP, tw);
        __syncthreads();
        for (int s = 1; s < nst - 1; ++s) {
            flip();
            rt_stage_buf<true>(src, dst, P, stage_rev(a.rp, s), lgP, tw);
            __syncthreads();
        }
        flip();
        if constexpr (EPI) rt_stage_buf<true>(src, dst, P, stage_rev(a.rp, nst - 1), lgP, tw);
        else rt_stage_any<true, true>(BufLd{src, P}, st, stage_rev(a.rp, nst - 1), lgP, tw);
    }
    if constexpr (EPI) {
        __syncthreads();
        t_epilogue(a, base, x0, lgP, nst < 2 ? s0 : dst, &acc, a.part2 ? &acc2 : nullptr);
    }
    if (EPI && a.part) {
        const int bid = blockIdx.y * gridDim.x + blockIdx.x, nb = gridDim.x * gridDim.y;
        float2 t, t2;
        block_pair_acc2(acc, a.part2 ? &acc2 : nullptr, reinterpret_cast<float*>(red), &t, &t2);
        if (a.part2) grid_sum_finalize2(t, t2, a.part, a.part2, bid, nb, a.ticket, a.sum_out, a.sum_out2);
        else grid_sum_finalize(t, a.part, bid, nb, a.ticket, a.sum_out);
    }
    if (a.count_iter) cg_count_iteration(a.cg);
}

int tpass_blocks(int nx, int cols, int nouter) { return ((nx + cols - 1) / cols) * nouter; }

cudaError_t run_tpass(const TArgs& a, int nouter, cudaStream_t st)
{
    if (ct_tpass_available(a)) return run_tpass_ct(a, nouter, st);
    dim3 grid((a.nx + a.cols - 1) / a.cols, nouter);
    const int P = a.cols / 2;
    const size_t smem = sizeof(float2) * (size_t)(2 * a.n + 2 * a.n * P);
    const int T = std::min(256, std::max(64, round32(max_nb(a.rp) * P)));
    if (a.epilogue) k_tpass<0, true><<<grid, T, smem, st>>>(a);
    else if (a.pupdate == 2) k_tpass<2, false><<<grid, T, smem, st>>>(a);
    else if (a.pupdate) k_tpass<1, false><<<grid, T, smem, st>>>(a);
    else k_tpass<0, false><<<grid, T, smem, st>>>(a);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// X pass kernels (s = 1..4: ops_xrt.cuh)
// ---------------------------------------------------------------------------
// Any s and any length (one included), rounds of KG harmonics whose pencils
// are transformed together; the aliases folded, or the harmonics summed, in
// shared memory.  They serve s >= 5 and the adjoint of portrait rows below 108
// samples (kXAdjStaged), where a transform has few butterflies: what bounds
// them is the latency of a round's stages, so a round takes up to eight
// harmonics.  Measured, us a call: forward 96 x 96 x 96, s = 6, K = 8: 27.9
// (79.6 with one harmonic a round); adjoint 24 x 128 x 128, s = 1, K = 12: 43.6
// (74.3 on k_xadj_rt).
// The pencils of a round of kn harmonics: P times the power of two from kn on.
__device__ __forceinline__ int round_pencils(int kn, int P) { return P << (32 - __clz(kn - 1)); }

__global__ void __launch_bounds__(256, 3) k_xfwd(const __grid_constant__ XArgs a)
{
    extern __shared__ float2 sm[];
    const int nx = a.nx, mx = a.mx, P = 1 << a.lgP, ld = P + 1, KG = 1 << a.lgK, ldq = KG * P + 1;
    float2* twx = sm;
    float2* twm = twx + nx;
    float2* A0 = twm + mx;
    float2* A1 = A0 + nx * ld;
    float2* B0 = A1 + nx * ld;
    float2* B1 = B0 + mx * ldq;
    for (int i = threadIdx.x; i < nx; i += blockDim.x) twx[i] = a.twx[i];
    for (int i = threadIdx.x; i < mx; i += blockDim.x) twm[i] = a.twm[i];
    __syncthreads();
    const int row0 = blockIdx.x * 2 * P;
    const int res = fft_result_index(a.rpx.nst);
    float2* Ar = res ? A1 : A0;
    fft_run<false, false, true>(a.rpx, RowPairLd{a.vin, nx, row0, a.rows}, BufSt{Ar, ld}, A0, A1, ld, P, twx);
    const PortraitRows pr{row0, a.rows, mx, a.win};
    for (int k0 = 0; k0 < a.K; k0 += KG)
        fft_run<true, true, false>(a.rpm, FoldLd{Ar, ld, a.Xhat + (long long)k0 * nx, nx, mx, a.s, a.lgP, a.K - k0},
                                   RoundSt{a, pr, k0}, B0, B1, ldq, round_pencils(min(KG, a.K - k0), P), twm);
}

// OCC: CTAs an SM holds by registers (4 spills where a radix is above 8).
template <int OCC>
__global__ void __launch_bounds__(256, OCC) k_xadj(const __grid_constant__ XArgs a)
{
    extern __shared__ float2 sm[];
    const int nx = a.nx, mx = a.mx, P = 1 << a.lgP, ld = P + 1, KG = 1 << a.lgK, ldq = KG * P + 1;
    float2* twx = sm;
    float2* twm = twx + nx;
    float2* acc = twm + mx;            // [nx][ld]
    float2* S0 = acc + nx * ld;        // the inverse's buffers [nx][ld] or a round's [mx][ldq]
    float2 *S1 = S0 + nx * ld, *B1 = S0 + mx * ldq;
    for (int i = threadIdx.x; i < nx; i += blockDim.x) twx[i] = a.twx[i];
    for (int i = threadIdx.x; i < mx; i += blockDim.x) twm[i] = a.twm[i];
    __syncthreads();
    const int row0 = blockIdx.x * 2 * P;
    float2* Fr = fft_result_index(a.rpm.nst) ? B1 : S0;
    const PortraitRows pr{row0, a.rows, mx, a.win};
    for (int k0 = 0; k0 < a.K; k0 += KG) {
        const int kn = min(KG, a.K - k0);
        fft_run<false, false, true>(a.rpm, RoundKLd{a, pr, k0}, BufSt{Fr, ldq}, S0, B1, ldq, round_pencils(kn, P), twm);
        // acc[w][p] (+)= sum_kk conj(Xhat_k0+kk[w]) F_kk[w mod mx][p]
        for (int idx = threadIdx.x; idx < nx * P; idx += blockDim.x) {
            const int p = idx & (P - 1), w = idx >> a.lgP;
            const int m = w - (int)a.dmx.div((uint32_t)w) * mx;
            const float2 *x = a.Xhat + (long long)k0 * nx + w, *f = Fr + m * ldq + p;
            float2 t[4];   // four short sums (at most 8 harmonics) round less than one
#pragma unroll
            for (int i = 0; i < 4; ++i)
                t[i] = i < kn ? c_mulc(f[i << a.lgP], __ldg(x + i * nx)) : make_float2(0.f, 0.f);
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (4 + i < kn) t[i] = c_add(t[i], c_mulc(f[(4 + i) << a.lgP], __ldg(x + (4 + i) * nx)));
            const float2 v = c_add(c_add(t[0], t[1]), c_add(t[2], t[3]));
            acc[w * ld + p] = k0 == 0 ? v : c_add(acc[w * ld + p], v);
        }
        __syncthreads();
    }
    fft_run<true, true, false>(a.rpx, BufLd{acc, ld}, RowPairSt{a.vout, nx, row0, a.rows}, S0, S1, ld, P, twx);
}

__global__ void __launch_bounds__(256) k_xnrm(const __grid_constant__ XArgs a)
{
    extern __shared__ float2 sm[];
    __shared__ double red[34];
    float dummy;
    if (a.cg_active && !cg_enter(a.cg, false, &dummy, red)) return;
    const int nx = a.nx, lgP = a.lgP, P = 1 << lgP, ld = P + 1, nst = a.rpx.nst;
    float2* twx = sm;
    float2* A0 = twx + nx;
    float2* A1 = A0 + nx * ld;
    cp_table(twx, a.twx, nx);
    const int row0 = blockIdx.x * 2 * P;
    DotAcc dacc, dacc2;
    const RowPairLd rows{a.vin, nx, row0, a.rows};
    float2* src = A0;
    float2* dst = A1;
    auto flip = [&]() {
        float2* t = src;
        src = dst;
        dst = t;
    };
    if (nst == 0) {
        for (int p = threadIdx.x; p < P; p += blockDim.x) A0[p] = rows.at(p)(0);
        __syncthreads();
        for (int p = threadIdx.x; p < P; p += blockDim.x) A1[p] = QLd{A0, ld, a.Q, a.mx, a.s, a.dmx}.at(p)(0);
        cp_table_wait();
    } else {
        rt_stage_any<false, false>(rows, BufSt{A0, ld}, stage_fwd(a.rpx, 0), lgP, twx);
        cp_table_wait();
        __syncthreads();
        for (int s = 1; s < nst; ++s, flip()) {
            rt_stage_buf<false>(src, dst, ld, stage_fwd(a.rpx, s), lgP, twx);
            __syncthreads();
        }
        // the alias blocks on the first inverse stage's loads
        rt_stage_any<true, true>(QLd{src, ld, a.Q, a.mx, a.s, a.dmx}, BufSt{dst, ld}, stage_rev(a.rpx, 0), lgP, twx);
        for (int s = 1; s < nst; ++s) {
            __syncthreads();
            flip();
            rt_stage_buf<true>(src, dst, ld, stage_rev(a.rpx, s), lgP, twx);
        }
    }
    __syncthreads();
    nrm_epilogue_rt(a, row0, P, dst, ld, &dacc, a.part2 ? &dacc2 : nullptr);
    if (a.part) {
        float2 t, t2;
        block_pair_acc2(dacc, a.part2 ? &dacc2 : nullptr, reinterpret_cast<float*>(red), &t, &t2);
        if (a.part2) grid_sum_finalize2(t, t2, a.part, a.part2, blockIdx.x, gridDim.x, a.ticket, a.sum_out, a.sum_out2);
        else grid_sum_finalize(t, a.part, blockIdx.x, gridDim.x, a.ticket, a.sum_out);
    }
    if (a.count_iter) cg_count_iteration(a.cg);
}

int num_sms()
{
    static const int n = [] {
        int dev = 0, v = 0;
        if (cudaGetDevice(&dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || v < 1)
            v = 1;
        return v;
    }();
    return n;
}

int xpass_blocks(int rows, int pairs) { return (rows + 2 * pairs - 1) / (2 * pairs); }

namespace {

constexpr size_t kXSmemMax = 200 * 1024;

// Launch shape of the run-time forward and adjoint: 8 row pairs (16 left
// 144 x 144 x 72 with 324 CTAs, two an SM: a second wave nearly empty), fewer
// where they leave SMs without a CTA; then as many harmonics a round (1, 2
// or 4: the adjoint adds their sums one after another) as 256 threads hold, one thread per (harmonic, butterfly,
// pair), while two CTAs fit an SM's shared memory.
struct XShape {
    int lgP = 3, lgK = 0, threads = 0, pitch = 0;
    size_t smem = 0;
    bool ok = false, lean = false;
};
enum XKind { kXFwd, kXAdj, kXWin };
XShape x_rt_shape(const RadixPlan& rpx, const RadixPlan& rpm, int s, int K, int rows, XKind kind)
{
    const bool adj = kind == kXAdj;
    XShape h;
    if (s < 1 || s > 4 || rpx.nst < 1 || rpm.nst < 1 || rpm.nst > 3) return h;
    const int nx = rpx.n, mx = rpm.n, R = rpm.radix[rpm.nst - 1], NB = mx / R;
    if (s * R > kXRegs) return h;
    // the adjoint's staged rows: an odd pitch spreads a half-warp's rows over the banks
    h.pitch = mx | 1;
    auto smem = [&](int lgP, int lgK) {
        const size_t P = (size_t)1 << lgP, KG = (size_t)1 << lgK, a = 2 * (size_t)nx * (P + 1);
        const size_t b = 2 * (size_t)mx * (KG * P + 1) + (adj ? 2 * KG * 2 * P * h.pitch : 0);
        if (kind == kXWin) return sizeof(float2) * (nx + mx + 3 * KG * nx + a / 2 + std::max(a / 2, b));
        return sizeof(float2) * (nx + mx + (adj ? 2 : 3) * KG * nx + std::max(a, b));
    };
    while (h.lgP > 1 && xpass_blocks(rows, 1 << h.lgP) < num_sms()) --h.lgP;
    while (h.lgP > 0 && ((NB << h.lgP) > 256 || smem(h.lgP, 0) > kXSmemMax)) --h.lgP;
    if ((NB << h.lgP) > 256 || smem(h.lgP, 0) > kXSmemMax) return h;
    while (h.lgK < 2 && (1 << h.lgK) < K && (NB << (h.lgP + h.lgK + 1)) <= 256 && smem(h.lgP, h.lgK + 1) <= kXSmemMax / 2) ++h.lgK;
    const int want = std::max(std::max(max_nb(rpx) << h.lgP, max_nb(rpm) << (h.lgP + h.lgK)), NB << (h.lgP + h.lgK));
    h.threads = std::min(256, std::max(64, round32(want)));
    h.smem = smem(h.lgP, h.lgK);
    h.ok = true;
    return h;
}

// Launch shape of the any-s kernels: up to 8 harmonics a round while two CTAs
// fit an SM's shared memory; 16 row pairs a CTA, or 8 where that shortens the
// SM's queue -- the row pairs of its CTAs, in whole turns of as many as it
// holds at a time (three by their 80 registers) -- and every stage of a round
// still has a butterfly for each thread (192 x 192 x 64, s = 6, K = 16, adjoint:
// 101 us with 16, 81 with 8; 128 x 128 x 64, s = 8, K = 8: 31 and 37); fewer where
// they leave SMs without a CTA.
// The adjoint of short rows in more than one turn of CTAs is bound by its
// throughput: the lean form holds four CTAs an SM, cuts 8, 9 and 12 samples
// into two stages and takes 32 row pairs where that costs no harmonics (us a
// call with three CTAs and 16 pairs, and so: 16 x 256 x 128, s = 2, K = 3 31.2 and
// 27.2; 16 x 72 x 256, s = 1, K = 9 42 and 35; in one turn, 16 x 64 x 64, s = 2, K = 10,
// 18 and 21).
XShape x_any_shape(const XArgs& a, XKind kind)
{
    constexpr int kLgK = 3, kLeanRow = 24;   // (k_xadj sums at most 8 harmonics a round)
    const int nx = a.nx, mx = a.mx, K = a.K, sms = num_sms();
    XShape h;
    auto ctas = [&](int lgP) { return (xpass_blocks(a.rows, 1 << lgP) + sms - 1) / sms; };
    h.lean = kind == kXAdj && mx <= kLeanRow && ctas(4) > 3;
    const int resident = h.lean ? 4 : 3;
    auto smem = [&](int lgP, int lgK) {
        const size_t x = (size_t)nx * ((1 << lgP) + 1), q = (size_t)mx * ((1 << (lgP + lgK)) + 1);
        return sizeof(float2) * (nx + mx + (kind == kXAdj ? x + 2 * std::max(x, q) : 2 * x + 2 * q));
    };
    auto lg_harmonics = [&](int lgP) {
        int k = 0;
        while (k < kLgK && (1 << k) < K && smem(lgP, k + 1) <= std::max(kXSmemMax / 2, smem(lgP, k))) ++k;
        return k;
    };
    auto queue = [&](int lgP) {
        const int n = ctas(lgP);
        const int r = std::max(1, std::min(resident, (int)(228 * 1024 / (smem(lgP, lg_harmonics(lgP)) + 1024))));
        return (n <= r ? n : (n + r - 1) / r * r) << lgP;
    };
    const RadixPlan& rp = kind == kXAdj ? a.rpa[h.lean] : a.rpm;
    int nb = mx;   // butterflies of the smallest stage
    for (int s = 0; s < rp.nst; ++s) nb = std::min(nb, mx / rp.radix[s]);
    h.lgP = 4;
    if (h.lean) {
        if (lg_harmonics(5) == lg_harmonics(4) && queue(5) <= queue(4)) h.lgP = 5;
    } else if ((nb << (3 + lg_harmonics(3))) >= 256 && queue(3) < queue(4)) {
        h.lgP = 3;
    }
    while (h.lgP > 1 && xpass_blocks(a.rows, 1 << h.lgP) < sms) --h.lgP;
    while (h.lgP > 0 && smem(h.lgP, 0) > kXSmemMax) --h.lgP;
    h.lgK = lg_harmonics(h.lgP);
    h.threads = 256;
    h.smem = smem(h.lgP, h.lgK);
    h.ok = true;
    return h;
}

// Portrait rows from which the adjoint stages them and keeps its sums in
// registers (k_xadj_rt).  Shorter ones have too few butterflies a harmonic for
// its 128 registers and a round of four harmonics.  Us a call on it and on
// k_xadj: 24 samples (24 x 128 x 128, s = 1, K = 12) 74 and 44, 48 (48 x 216 x 64,
// s = 1, K = 14) 84 and 57, 64 (256 x 128 x 64, s = 4, K = 8) 60 and 56, 96 (96 x 96 x
// 64, s = 1, K = 6) 43 and 30; 108 (216 x 216 x 72, s = 2, K = 13) 210 and 270,
// 192 (192 x 128 x 54, s = 1, K = 13) 130 and 172.
constexpr int kXAdjStaged = 108;

}  // namespace

bool xpass_windowed(int nx, int s, int pairs) { return !ct_xpass_available(nx, s, pairs); }

int xnrm_rt_pairs(const RadixPlan& rpx)
{
    int lgP = 4;
    while (lgP > 0 && ((rpx.n / (rpx.nst ? rpx.radix[0] : 1)) << lgP > 256 ||
                       sizeof(float2) * (size_t)(rpx.n + 2 * rpx.n * ((1 << lgP) + 1)) > kXSmemMax))
        --lgP;
    return 1 << lgP;
}

cudaError_t run_xfwd(const XArgs& a0, cudaStream_t st)
{
    if (!a0.win.on && ct_xpass_available(a0.nx, a0.s, a0.pairs)) return run_xfwd_ct(a0, st);
    XArgs a = a0;
    const XShape h = x_rt_shape(a.rpx, a.rpm, a.s, a.K, a.rows, kXFwd);
    if (h.ok) {
        a.lgP = h.lgP;
        a.lgK = h.lgK;
        const int grid = xpass_blocks(a.rows, 1 << h.lgP);
        if (a.s == 1) return XRt<1>::fwd(a, grid, h.threads, h.smem, st);
        if (a.s == 2) return XRt<2>::fwd(a, grid, h.threads, h.smem, st);
        if (a.s == 3) return XRt<3>::fwd(a, grid, h.threads, h.smem, st);
        return XRt<4>::fwd(a, grid, h.threads, h.smem, st);
    }
    const XShape g = x_any_shape(a, kXFwd);
    a.lgP = g.lgP;
    a.lgK = g.lgK;
    k_xfwd<<<xpass_blocks(a.rows, 1 << g.lgP), g.threads, g.smem, st>>>(a);
    return cudaGetLastError();
}
cudaError_t run_xadj(const XArgs& a0, cudaStream_t st)
{
    if (!a0.win.on && ct_xpass_available(a0.nx, a0.s, a0.pairs)) return run_xadj_ct(a0, st);
    XArgs a = a0;
    const XShape h = a.mx >= kXAdjStaged ? x_rt_shape(a.rpx, a.rpm, a.s, a.K, a.rows, kXAdj) : XShape();
    if (h.ok) {
        a.pitch = h.pitch;
        a.lgP = h.lgP;
        a.lgK = h.lgK;
        const int grid = xpass_blocks(a.rows, 1 << h.lgP);
        if (a.s == 1) return XRt<1>::adj(a, grid, h.threads, h.smem, st);
        if (a.s == 2) return XRt<2>::adj(a, grid, h.threads, h.smem, st);
        if (a.s == 3) return XRt<3>::adj(a, grid, h.threads, h.smem, st);
        return XRt<4>::adj(a, grid, h.threads, h.smem, st);
    }
    const XShape g = x_any_shape(a, kXAdj);
    a.rpm = a.rpa[g.lean];
    a.lgP = g.lgP;
    a.lgK = g.lgK;
    a.dmx = FastDiv(a.mx);
    const int grid = xpass_blocks(a.rows, 1 << g.lgP);
    if (g.lean) k_xadj<4><<<grid, g.threads, g.smem, st>>>(a);
    else k_xadj<3><<<grid, g.threads, g.smem, st>>>(a);
    return cudaGetLastError();
}
// Both passes in one where the portrait length has two radices (other lengths
// take them one after the other).
bool xwin_available(const XArgs& a)
{
    return a.win.on && a.rpm.nst == 2 && x_rt_shape(a.rpx, a.rpm, a.s, a.K, a.rows, kXWin).ok;
}
cudaError_t run_xwin(const XArgs& a0, cudaStream_t st)
{
    XArgs a = a0;
    const XShape h = x_rt_shape(a.rpx, a.rpm, a.s, a.K, a.rows, kXWin);
    a.lgP = h.lgP;
    a.lgK = h.lgK;
    const int grid = xpass_blocks(a.rows, 1 << h.lgP);
    if (a.s == 1) return XRt<1>::win(a, grid, h.threads, h.smem, st);
    if (a.s == 2) return XRt<2>::win(a, grid, h.threads, h.smem, st);
    if (a.s == 3) return XRt<3>::win(a, grid, h.threads, h.smem, st);
    return XRt<4>::win(a, grid, h.threads, h.smem, st);
}
cudaError_t run_xnrm(const XArgs& a0, cudaStream_t st)
{
    if (ct_xpass_available(a0.nx, a0.s, a0.pairs)) return run_xnrm_ct(a0, st);
    XArgs a = a0;
    a.dmx = FastDiv(a.mx);
    const int P = xnrm_rt_pairs(a.rpx);
    a.lgP = 0;
    while ((1 << a.lgP) < P) ++a.lgP;
    const size_t smem = sizeof(float2) * (size_t)(a.nx + 2 * a.nx * (P + 1));
    k_xnrm<<<xpass_blocks(a.rows, P), std::min(256, std::max(64, round32(max_nb(a.rpx) * P))), smem, st>>>(a);
    return cudaGetLastError();
}

// Opt every pencil kernel into the device's full shared-memory carve-out
// (the opt-in limit minus the kernel's static shared memory).
template <class F>
static cudaError_t opt_in_smem(F* f, int optin)
{
    cudaFuncAttributes fa;
    cudaError_t e = cudaFuncGetAttributes(&fa, f);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - (int)fa.sharedSizeBytes);
}

cudaError_t ops_set_attributes()
{
    int dev = 0, optin = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e != cudaSuccess) return e;
    if ((e = opt_in_smem(k_tpass<0, false>, optin)) != cudaSuccess) return e;
    if ((e = opt_in_smem(k_tpass<0, true>, optin)) != cudaSuccess) return e;
    if ((e = opt_in_smem(k_tpass<1, false>, optin)) != cudaSuccess) return e;
    if ((e = opt_in_smem(k_tpass<2, false>, optin)) != cudaSuccess) return e;
    if ((e = opt_in_smem(k_xfwd, optin)) != cudaSuccess) return e;
    if ((e = XRt<1>::set_attributes(optin)) != cudaSuccess) return e;
    if ((e = XRt<2>::set_attributes(optin)) != cudaSuccess) return e;
    if ((e = XRt<3>::set_attributes(optin)) != cudaSuccess) return e;
    if ((e = XRt<4>::set_attributes(optin)) != cudaSuccess) return e;
    if ((e = opt_in_smem(k_xadj<3>, optin)) != cudaSuccess) return e;
    if ((e = opt_in_smem(k_xadj<4>, optin)) != cudaSuccess) return e;
    if ((e = opt_in_smem(k_xnrm, optin)) != cudaSuccess) return e;
    if ((e = xw_set_attributes()) != cudaSuccess) return e;
    return ct_set_attributes(optin);
}

}  // namespace mh3d
