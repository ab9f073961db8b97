// Run-time drive-axis passes for s = 1..4 (any length 2^a 3^b; the adjoint from
// portrait rows of kXAdjStaged samples on), and helpers
// shared with the other run-time kernels (ops.cu).  Each S is compiled in a
// file of its own (ops_x1.cu .. ops_x4.cu).
#pragma once

#include <algorithm>
#include <cstdint>
#include <type_traits>

#include "ops_functors.cuh"
#include "ops_kernels.cuh"

namespace mh3d {

// 8-byte asynchronous copies of the spectral tables: in flight under the
// first stage's loads, waited for before the first barrier.
__device__ __forceinline__ void cp_table(float2* dst, const float2* __restrict__ src, int n)
{
    for (int i = threadIdx.x; i < n; i += blockDim.x)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((uint32_t)__cvta_generic_to_shared(dst + i)),
                     "l"(src + i)
                     : "memory");
}
__device__ __forceinline__ void cp_table_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

inline int round32(int v) { return (v + 31) / 32 * 32; }

// Butterflies of the largest stage of a schedule, per pencil.
inline int max_nb(const RadixPlan& pl)
{
    int m = 1;
    for (int s = 0; s < pl.nst; ++s) m = std::max(m, pl.n / pl.radix[s]);
    return m;
}

constexpr int kXRegs = 24;   // alias values of one butterfly, s R

// The launches of one s.
template <int S>
struct XRt {
    static cudaError_t set_attributes(int optin);
    static cudaError_t fwd(const XArgs& a, int grid, int threads, size_t smem, cudaStream_t st);
    static cudaError_t adj(const XArgs& a, int grid, int threads, size_t smem, cudaStream_t st);
    static cudaError_t win(const XArgs& a, int grid, int threads, size_t smem, cudaStream_t st);
};

}  // namespace mh3d

#ifdef MH3D_XRT_S   // the kernels, in the file that compiles them

namespace mh3d {

// s = 1..4 (S): the CTA takes 2 P rows and rounds of KG harmonics; thread
// (kk, j, p) owns butterfly j (radix R, s R <= 24) of pencil p of the
// portrait-length transform's fused stage for the round's harmonic kk, and
// keeps its s aliases -- the drive-axis spectrum (forward) or its sum over
// its harmonics (adjoint) at j + r NB + a mx -- in registers.  A round is one
// pass through shared memory and, for portrait lengths of two radices, one
// barrier (two buffers, alternated); the drive spectra (and the adjoint's
// rows) are copied a round or two ahead.  What bounds them: the latency of a
// round, so the rounds are few and several CTAs an SM overlap them.  (One
// harmonic a round: 48 x 27 x 24, K = 6, 21 us an adjoint pass; the former
// kernels took five to nine barriers per four harmonics and staged the fold
// and the sum through shared memory.)
namespace {

// acc / fold helpers of one butterfly (j, p) of radix R.
template <int S, int R>
__device__ __forceinline__ void x_fold(const float2* F, const float2* xk, int j, int NB, int mx, float2* G)
{
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int m = j + r * NB;
        float2 g = c_mul(F[r], xk[m]);
#pragma unroll
        for (int al = 1; al < S; ++al) g = c_add(g, c_mul(F[al * R + r], xk[m + al * mx]));
        G[r] = g;
    }
}

// f(R) with the radix as a compile-time constant (those with S R <= kXRegs).
template <int S, class F>
__device__ __forceinline__ void x_radix(int radix, F&& f)
{
    switch (radix) {
        case 16: if constexpr (S * 16 <= kXRegs) f(std::integral_constant<int, 16>{}); break;
        case 12: if constexpr (S * 12 <= kXRegs) f(std::integral_constant<int, 12>{}); break;
        case 9: if constexpr (S * 9 <= kXRegs) f(std::integral_constant<int, 9>{}); break;
        case 8: if constexpr (S * 8 <= kXRegs) f(std::integral_constant<int, 8>{}); break;
        case 6: if constexpr (S * 6 <= kXRegs) f(std::integral_constant<int, 6>{}); break;
        case 4: if constexpr (S * 4 <= kXRegs) f(std::integral_constant<int, 4>{}); break;
        case 3: if constexpr (S * 3 <= kXRegs) f(std::integral_constant<int, 3>{}); break;
        case 2: if constexpr (S * 2 <= kXRegs) f(std::integral_constant<int, 2>{}); break;
        default: break;
    }
}

}  // namespace

// Thread (kk, j, p) of a round.
struct XThread {
    int kk, j, p;
    bool act;
    __device__ __forceinline__ XThread(const XArgs& a)
    {
        p = (int)threadIdx.x & ((1 << a.lgP) - 1);
        const int q = (int)threadIdx.x >> a.lgP;
        const FastDiv& d = a.rpm.dnb[a.rpm.nst - 1];
        kk = (int)d.div((uint32_t)q);
        j = q - kk * (int)d.d;
        act = kk < (1 << a.lgK);
    }
};

// The drive spectra of harmonics k0 .. k0 + n - 1 into shared memory.
__device__ __forceinline__ void stage_spectra(float2* dst, const XArgs& a, int k0, int n)
{
    const float2* src = a.Xhat + (long long)k0 * a.nx;
    for (int i = threadIdx.x; i < n * a.nx; i += blockDim.x)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((uint32_t)__cvta_generic_to_shared(dst + i)),
                     "l"(src + i)
                     : "memory");
}

struct RoundLd {   // from the staged rows [kk][2 P][pitch]
    const XArgs& a;
    const float2* raw;
    int k0;
    __device__ __forceinline__ RawRowsLd::At at(int q) const
    {
        const int kk = q >> a.lgP, p = q & ((1 << a.lgP) - 1), k = k0 + kk;
        // a harmonic past the last reads the round's first rows with phase 0
        const bool in = k < a.K;
        return RawRowsLd::At{raw + ((in ? kk << a.lgP : 0) + p) * 2 * a.pitch,
                             in ? __ldg(a.phase + k) : make_float2(0.f, 0.f), a.pitch};
    }
};

template <int S>
__global__ void __launch_bounds__(256, 2) k_xfwd_rt(const __grid_constant__ XArgs a)
{
    extern __shared__ float2 sm[];
    const int nx = a.nx, mx = a.mx, lgP = a.lgP, P = 1 << lgP, ld = P + 1;
    const int lgQ = lgP + a.lgK, KG = 1 << a.lgK, ldq = (1 << lgQ) + 1;
    float2* twx = sm;
    float2* twm = twx + nx;
    float2* xs = twm + mx;               // three rounds' spectra [KG][nx]
    float2* s0 = xs + 3 * KG * nx;
    float2* s1 = s0 + nx * ld;
    cp_table(twx, a.twx, nx);
    cp_table(twm, a.twm, mx);
    stage_spectra(xs, a, 0, min(2 * KG, a.K));   // rounds 0 and 1
    const int row0 = blockIdx.x * 2 * P;
    const int nstx = a.rpx.nst, nstm = a.rpm.nst;
    // the rows' spectrum, in s0 or s1
    float2* sp = s0;
    rt_stage_any<false, false>(RowPairLd{a.vin, nx, row0, a.rows}, BufSt{s0, ld}, stage_fwd(a.rpx, 0), lgP, twx);
    cp_table_wait();
    __syncthreads();
    for (int s = 1; s < nstx; ++s) {
        float2* dst = sp == s0 ? s1 : s0;
        rt_stage_buf<false>(sp, dst, ld, stage_fwd(a.rpx, s), lgP, twx);
        __syncthreads();
        sp = dst;
    }
    const int RM = a.rpm.radix[nstm - 1], NB = (int)a.rpm.dnb[nstm - 1].d;
    const XThread t(a);
    float2 F[kXRegs];
    if (t.act) {
        x_radix<S>(RM, [&](auto rc) {
            constexpr int R = decltype(rc)::value;
#pragma unroll
            for (int al = 0; al < S; ++al)
#pragma unroll
                for (int r = 0; r < R; ++r) F[al * R + r] = sp[(t.j + r * NB + al * mx) * ld + t.p];
        });
    }
    __syncthreads();   // the spectrum is in registers; its buffers become the rounds'
    float2* bb[2] = {s0, s0 + mx * ldq};
    const PortraitRows pr{row0, a.rows, mx, a.win};
    const StageGeom gl = stage_rev(a.rpm, nstm - 1);
    for (int k0 = 0, rd = 0; k0 < a.K; k0 += KG, ++rd) {
        // the spectra two rounds on, over those read a round ago
        if (k0 + 2 * KG < a.K) stage_spectra(xs + (rd + 2) % 3 * KG * nx, a, k0 + 2 * KG, min(KG, a.K - k0 - 2 * KG));
        asm volatile("cp.async.commit_group;" ::: "memory");
        float2* b = bb[nstm == 2 ? (rd & 1) : 0];
        const RoundSt pst{a, pr, k0};
        if (t.act && k0 + t.kk < a.K) {
            const float2* xk = xs + (rd % 3 * KG + t.kk) * nx;
            const int q = (t.kk << lgP) + t.p;
            x_radix<S>(RM, [&](auto rc) {
                constexpr int R = decltype(rc)::value;
                float2 G[R];
                x_fold<S, R>(F, xk, t.j, NB, mx, G);
                dft<R, true>(G);
                if (nstm == 1) {
                    const auto pp = pst.at(q);
#pragma unroll
                    for (int r = 0; r < R; ++r) pp(t.j * R + r, G[r]);
                } else {
#pragma unroll
                    for (int r = 0; r < R; ++r) b[(t.j * R + r) * ldq + q] = G[r];
                }
            });
        }
        asm volatile("cp.async.wait_group 1;" ::: "memory");   // the next round's spectra
        __syncthreads();
        if (nstm == 1) continue;
        for (int s = 1; s < nstm - 1; ++s) {   // three radices at most: bb[0] -> bb[1]
            rt_stage_buf<true>(bb[0], bb[1], ldq, stage_rev(a.rpm, s), lgQ, twm);
            __syncthreads();
            b = bb[1];
        }
        rt_stage_any<true, false>(BufLd{b, ldq}, pst, gl, lgQ, twm);
    }
}

template <int S>
__global__ void __launch_bounds__(256, 2) k_xadj_rt(const __grid_constant__ XArgs a)
{
    extern __shared__ float2 sm[];
    const int nx = a.nx, mx = a.mx, lgP = a.lgP, P = 1 << lgP, ld = P + 1;
    const int lgQ = lgP + a.lgK, KG = 1 << a.lgK, ldq = (1 << lgQ) + 1;
    float2* twx = sm;
    float2* twm = twx + nx;
    float2* xs = twm + mx;               // two rounds' spectra [KG][nx]
    float2* s0 = xs + 2 * KG * nx;       // the inverse's buffers, and before it:
    float2* s1 = s0 + nx * ld;
    float2* bb[2] = {s0, s0 + mx * ldq};  // the rounds' transform buffers
    float2* raw = bb[1] + mx * ldq;       // and two rounds' rows [KG][2 P][pitch]
    const int rawn = KG * 2 * P * a.pitch;
    const int row0 = blockIdx.x * 2 * P;
    const int nstx = a.rpx.nst, nstm = a.rpm.nst;
    const int RM = a.rpm.radix[nstm - 1], NB = (int)a.rpm.dnb[nstm - 1].d;
    const PortraitRows pr{row0, a.rows, mx, a.win};
    auto stage_round = [&](int rd) {
        const int k0 = rd * KG, n = min(KG, a.K - k0);
        if (n <= 0) return;
        stage_spectra(xs + (rd & 1) * KG * nx, a, k0, n);
        float2* d = raw + (rd & 1) * rawn;
        for (int kk = 0; kk < n; ++kk)
            stage_portraits(d + kk * 2 * P * a.pitch, a.pitch, a.din + (long long)(k0 + kk) * a.M, pr, P);
    };
    cp_table(twx, a.twx, nx);
    cp_table(twm, a.twm, mx);
    if (a.win.on || row0 + 2 * P > a.rows) {   // samples no copy writes read as zero
        for (int i = threadIdx.x; i < 2 * rawn; i += blockDim.x) raw[i] = make_float2(0.f, 0.f);
        __syncthreads();   // the zeros land before the copies
    }
    stage_round(0);
    cp_table_wait();
    __syncthreads();
    stage_round(1);
    const XThread t(a);
    float2 V[kXRegs];
#pragma unroll
    for (int i = 0; i < kXRegs; ++i) V[i] = make_float2(0.f, 0.f);
    const StageGeom g0 = stage_fwd(a.rpm, 0);
    for (int k0 = 0, rd = 0; k0 < a.K; k0 += KG, ++rd) {
        float2* b = bb[nstm == 2 ? (rd & 1) : 0];
        const RoundLd rows{a, raw + (rd & 1) * rawn, k0};
        const int q = (t.kk << lgP) + t.p;
        float2 v1[16];
        if (nstm > 1) {
            rt_stage_any<false, true>(rows, BufSt{b, ldq}, g0, lgQ, twm);   // (the rows are staged: no coalescing to keep)
        } else if (t.act) {   // one butterfly is the whole transform
            x_radix<1>(RM, [&](auto rc) {
                constexpr int R = decltype(rc)::value;
                const auto pl = rows.at(q);
#pragma unroll
                for (int r = 0; r < R; ++r) v1[r] = pl(r);
            });
        }
        __syncthreads();
        for (int s = 1; s < nstm - 1; ++s) {   // three radices at most: bb[0] -> bb[1]
            rt_stage_buf<false>(bb[0], bb[1], ldq, stage_fwd(a.rpm, s), lgQ, twm);
            __syncthreads();
            b = bb[1];
        }
        if (t.act && k0 + t.kk < a.K) {
            const float2* xk = xs + ((rd & 1) * KG + t.kk) * nx;
            x_radix<S>(RM, [&](auto rc) {
                constexpr int R = decltype(rc)::value;
                float2 v[R];
                if (nstm > 1) {
#pragma unroll
                    for (int r = 0; r < R; ++r) v[r] = b[(t.j + r * NB) * ldq + q];
#pragma unroll
                    for (int r = 1; r < R; ++r) v[r] = c_mul(v[r], twm[r * t.j]);
                } else {
#pragma unroll
                    for (int r = 0; r < R; ++r) v[r] = v1[r];
                }
                dft<R, false>(v);
#pragma unroll
                for (int al = 0; al < S; ++al)
#pragma unroll
                    for (int r = 0; r < R; ++r)
                        V[al * R + r] = c_add(V[al * R + r], c_mulc(v[r], xk[t.j + r * NB + al * mx]));
            });
        }
        if (k0 + KG < a.K) {
            // the next round's copies (issued a round ago) have landed, and
            // this round's have been read: their buffers take round rd + 2
            cp_table_wait();
            __syncthreads();
            stage_round(rd + 2);
        }
    }
    __syncthreads();   // the last round's buffers have been read
    for (int g = 0; g < KG; ++g) {   // the KG threads' sums, in order
        if (t.act && t.kk == g) {
            x_radix<S>(RM, [&](auto rc) {
                constexpr int R = decltype(rc)::value;
#pragma unroll
                for (int al = 0; al < S; ++al)
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        float2* d = s0 + (t.j + r * NB + al * mx) * ld + t.p;
                        *d = g == 0 ? V[al * R + r] : c_add(*d, V[al * R + r]);
                    }
            });
        }
        __syncthreads();
    }
    const RowPairSt out{a.vout, nx, row0, a.rows};
    float2* src = s0;
    for (int s = 0; s + 1 < nstx; ++s) {
        float2* dst = src == s0 ? s1 : s0;
        rt_stage_buf<true>(src, dst, ld, stage_rev(a.rpx, s), lgP, twx);
        __syncthreads();
        src = dst;
    }
    rt_stage_any<true, false>(BufLd{src, ld}, out, stage_rev(a.rpx, nstx - 1), lgP, twx);
}

// The end of the inverse transform, the window and the start of the forward
// one on a butterfly: radix[0] at j + r NB1 on both sides.
template <int R>
__device__ __forceinline__ void x_window(const float2* b0, float2* b1, int ldq, int lgP, int lgQ, int NB1, int m0, int len,
                                         uint32_t rowmask, const float2* twm)
{
    for (int idx = threadIdx.x; idx < NB1 << lgQ; idx += blockDim.x) {
        const int q = idx & ((1 << lgQ) - 1), j = idx >> lgQ, p = q & ((1 << lgP) - 1);
        const bool h0 = (rowmask >> (2 * p)) & 1u, h1 = (rowmask >> (2 * p + 1)) & 1u;
        float2 v[R];
#pragma unroll
        for (int r = 0; r < R; ++r) v[r] = b0[(j + r * NB1) * ldq + q];
#pragma unroll
        for (int r = 1; r < R; ++r) v[r] = c_mulc(v[r], twm[r * j]);
        dft<R, true>(v);
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const bool in = (unsigned)(j + r * NB1 - m0) < (unsigned)len;
            v[r] = make_float2(in && h0 ? v[r].x : 0.f, in && h1 ? v[r].y : 0.f);
        }
        dft<R, false>(v);
#pragma unroll
        for (int r = 0; r < R; ++r) b1[(j * R + r) * ldq + q] = v[r];
    }
}

// The drive-axis part of A^T M A on a padded plan (M: the field of view) in
// one pass, for portrait lengths of two radices: every harmonic's portrait
// rows exist in shared memory only, real as they are before their phase
// (which cancels), so that no portraits go through memory.  Rounds of KG
// harmonics as in the two passes above, two barriers a round: fold and first
// inverse radix; last inverse radix, window and first forward radix; last
// forward radix and sum.  CTAs whose rows all lie outside the window write
// zeros.
// Measured, 144 x 144 x 72 of a 128 x 128 x 64 window, s = 2, K = 8: a normal
// operator takes 43 us less than with the two passes (28 and 47 us with 33 MB of
// portraits written and read between them).
template <int S>
__global__ void __launch_bounds__(256, 2) k_xwin_rt(const __grid_constant__ XArgs a)
{
    extern __shared__ float2 sm[];
    const int nx = a.nx, mx = a.mx, lgP = a.lgP, P = 1 << lgP, ld = P + 1;
    const int lgQ = lgP + a.lgK, KG = 1 << a.lgK, ldq = (1 << lgQ) + 1;
    float2* twx = sm;
    float2* twm = twx + nx;
    float2* xs = twm + mx;                // three rounds' spectra [KG][nx]
    float2* s0 = xs + 3 * KG * nx;        // the rows' spectrum; later the sum
    float2* s1 = s0 + nx * ld;            // the transforms' other buffer, the rounds' buffers
    float2 *b0 = s1, *b1 = s1 + mx * ldq;
    const int row0 = blockIdx.x * 2 * P, nstx = a.rpx.nst;
    const PortraitRows pr{row0, a.rows, mx, a.win};
    uint32_t rowmask = 0;
    for (int r = 0; r < 2 * P; ++r) rowmask |= (uint32_t)(pr.row(row0 + r) >= 0) << r;
    if (!rowmask) {
        const int n = min(2 * P, a.rows - row0) * nx;
        for (int i = threadIdx.x; i < n; i += blockDim.x) a.vout[(long long)row0 * nx + i] = 0.f;
        return;
    }
    cp_table(twx, a.twx, nx);
    cp_table(twm, a.twm, mx);
    stage_spectra(xs, a, 0, min(2 * KG, a.K));   // rounds 0 and 1
    {
        float2* sp = (nstx & 1) ? s0 : s1;       // the last stage writes s0
        rt_stage_any<false, false>(RowPairLd{a.vin, nx, row0, a.rows}, BufSt{sp, ld}, stage_fwd(a.rpx, 0), lgP, twx);
        cp_table_wait();
        __syncthreads();
        for (int s = 1; s < nstx; ++s) {
            float2* dst = sp == s0 ? s1 : s0;
            rt_stage_buf<false>(sp, dst, ld, stage_fwd(a.rpx, s), lgP, twx);
            __syncthreads();
            sp = dst;
        }
    }
    const int RM = a.rpm.radix[1], NB = (int)a.rpm.dnb[1].d, R1 = a.rpm.radix[0], NB1 = (int)a.rpm.dnb[0].d;
    const int m0 = pr.m0(), len = pr.len();
    const XThread t(a);
    const int q = (t.kk << lgP) + t.p;
    float2 V[kXRegs];
#pragma unroll
    for (int i = 0; i < kXRegs; ++i) V[i] = make_float2(0.f, 0.f);
    for (int k0 = 0, rd = 0; k0 < a.K; k0 += KG, ++rd) {
        const bool act = t.act && k0 + t.kk < a.K;
        const float2* xk = xs + (rd % 3 * KG + t.kk) * nx;
        if (act) {
            x_radix<S>(RM, [&](auto rc) {
                constexpr int R = decltype(rc)::value;
                float2 G[R];
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const int m = t.j + r * NB;
                    float2 g = c_mul(s0[m * ld + t.p], xk[m]);
#pragma unroll
                    for (int al = 1; al < S; ++al) g = c_add(g, c_mul(s0[(m + al * mx) * ld + t.p], xk[m + al * mx]));
                    G[r] = g;
                }
                dft<R, true>(G);
#pragma unroll
                for (int r = 0; r < R; ++r) b0[(t.j * R + r) * ldq + q] = G[r];
            });
        }
        __syncthreads();
        // the spectra two rounds on, over those read a round ago
        if (k0 + 2 * KG < a.K) stage_spectra(xs + (rd + 2) % 3 * KG * nx, a, k0 + 2 * KG, min(KG, a.K - k0 - 2 * KG));
        asm volatile("cp.async.commit_group;" ::: "memory");
        x_radix<1>(R1, [&](auto rc) {
            x_window<decltype(rc)::value>(b0, b1, ldq, lgP, lgQ, NB1, m0, len, rowmask, twm);
        });
        asm volatile("cp.async.wait_group 1;" ::: "memory");   // the next round's spectra
        __syncthreads();
        if (act) {
            x_radix<S>(RM, [&](auto rc) {
                constexpr int R = decltype(rc)::value;
                float2 v[R];
#pragma unroll
                for (int r = 0; r < R; ++r) v[r] = b1[(t.j + r * NB) * ldq + q];
#pragma unroll
                for (int r = 1; r < R; ++r) v[r] = c_mul(v[r], twm[r * t.j]);
                dft<R, false>(v);
#pragma unroll
                for (int al = 0; al < S; ++al)
#pragma unroll
                    for (int r = 0; r < R; ++r)
                        V[al * R + r] = c_add(V[al * R + r], c_mulc(v[r], xk[t.j + r * NB + al * mx]));
            });
        }
    }
    __syncthreads();   // the spectrum and the last round's buffers have been read
    for (int g = 0; g < KG; ++g) {   // the KG threads' sums, in order
        if (t.act && t.kk == g) {
            x_radix<S>(RM, [&](auto rc) {
                constexpr int R = decltype(rc)::value;
#pragma unroll
                for (int al = 0; al < S; ++al)
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        float2* d = s0 + (t.j + r * NB + al * mx) * ld + t.p;
                        *d = g == 0 ? V[al * R + r] : c_add(*d, V[al * R + r]);
                    }
            });
        }
        __syncthreads();
    }
    const RowPairSt out{a.vout, nx, row0, a.rows};
    float2* src = s0;
    for (int s = 0; s + 1 < nstx; ++s) {
        float2* dst = src == s0 ? s1 : s0;
        rt_stage_buf<true>(src, dst, ld, stage_rev(a.rpx, s), lgP, twx);
        __syncthreads();
        src = dst;
    }
    rt_stage_any<true, false>(BufLd{src, ld}, out, stage_rev(a.rpx, nstx - 1), lgP, twx);
}

template <class F>
static cudaError_t xrt_opt_in(F* f, int optin)
{
    cudaFuncAttributes fa;
    const cudaError_t e = cudaFuncGetAttributes(&fa, f);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - (int)fa.sharedSizeBytes);
}
template <int S>
cudaError_t XRt<S>::set_attributes(int optin)
{
    cudaError_t e = xrt_opt_in(k_xfwd_rt<S>, optin);
    if (e == cudaSuccess) e = xrt_opt_in(k_xadj_rt<S>, optin);
    return e != cudaSuccess ? e : xrt_opt_in(k_xwin_rt<S>, optin);
}
template <int S>
cudaError_t XRt<S>::fwd(const XArgs& a, int grid, int threads, size_t smem, cudaStream_t st)
{
    k_xfwd_rt<S><<<grid, threads, smem, st>>>(a);
    return cudaGetLastError();
}
template <int S>
cudaError_t XRt<S>::adj(const XArgs& a, int grid, int threads, size_t smem, cudaStream_t st)
{
    k_xadj_rt<S><<<grid, threads, smem, st>>>(a);
    return cudaGetLastError();
}
template <int S>
cudaError_t XRt<S>::win(const XArgs& a, int grid, int threads, size_t smem, cudaStream_t st)
{
    k_xwin_rt<S><<<grid, threads, smem, st>>>(a);
    return cudaGetLastError();
}
template struct XRt<MH3D_XRT_S>;

}  // namespace mh3d

#endif   // MH3D_XRT_S
