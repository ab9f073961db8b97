// Shared-memory Stockham FFT engine for batches of short pencils (sm_103a).
//
// A batch is P pencils of one length n (2^a 3^b, n <= 1024; P a power of
// two).  Element e of
// pencil p lives at buf[e * ld + p] (pencil index fastest), so consecutive
// threads touch consecutive float2 words: a half warp covers 128 contiguous
// bytes, which is bank-conflict free for 64-bit accesses.  ld = P + 1 keeps
// column walks (j-fast mapping, below) at most two-way conflicted.
//
// Each radix-R stage is the self-sorting (Stockham) step: butterfly j reads
// elements j + r n/R (r < R), multiplies by the twiddles W_{Ns R}^{r (j mod Ns)},
// applies the length-R DFT in registers and writes elements
// (j - j mod Ns) R + j mod Ns + r Ns.  Stages alternate between two scratch
// buffers; the first stage reads through a loader functor and the last
// writes through a storer functor, so global loads, spectral multiplies,
// folds and epilogues fuse into the first or last stage.  Every stage ends
// with __syncthreads().
//
// Thread mappings: PFAST puts the pencil index fastest (butterfly idx ->
// p = idx % P, j = idx / P); !PFAST puts the butterfly index fastest, which
// makes the first stage read and the last stage write consecutive elements
// of one pencil -- the mapping used where a pencil is a contiguous row in
// global memory.
//
// Twiddle tables (W_n^t, t < n) come from the host, computed in FP64 and
// rounded once; the DFT kernels' constants are the sines and cosines of
// multiples of pi / 8, pi / 9 and pi / 6.
#pragma once

#include <cuda_runtime.h>

#include "mh3d_internal.h"

namespace mh3d {

__device__ __forceinline__ float2 c_add(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 c_sub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ float2 c_mul(float2 a, float2 b)
{
    return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}
// a * conj(b)
__device__ __forceinline__ float2 c_mulc(float2 a, float2 b)
{
    return make_float2(fmaf(a.x, b.x, a.y * b.y), fmaf(a.y, b.x, -a.x * b.y));
}
__device__ __forceinline__ float2 c_scale(float2 a, float s) { return make_float2(a.x * s, a.y * s); }
// Multiply by -i (forward transform) or +i (inverse transform).
template <bool INV>
__device__ __forceinline__ float2 c_rot(float2 a)
{
    return INV ? make_float2(-a.y, a.x) : make_float2(a.y, -a.x);
}

// In-register DFT of length R with sign -1 (forward) or +1 (INV).
template <int R, bool INV>
__device__ __forceinline__ void dft(float2* v);

template <>
__device__ __forceinline__ void dft<2, false>(float2* v)
{
    const float2 a = v[0], b = v[1];
    v[0] = c_add(a, b);
    v[1] = c_sub(a, b);
}
template <>
__device__ __forceinline__ void dft<2, true>(float2* v) { dft<2, false>(v); }

template <bool INV>
__device__ __forceinline__ void dft3(float2* v)
{
    constexpr float kS = 0.86602540378443864676f;   // sqrt(3)/2
    const float2 t1 = c_add(v[1], v[2]);
    const float2 t2 = make_float2(v[0].x - 0.5f * t1.x, v[0].y - 0.5f * t1.y);
    const float2 d = c_scale(c_sub(v[1], v[2]), kS);
    const float2 md = c_rot<INV>(d);
    v[0] = c_add(v[0], t1);
    v[1] = c_add(t2, md);
    v[2] = c_sub(t2, md);
}
template <>
__device__ __forceinline__ void dft<3, false>(float2* v) { dft3<false>(v); }
template <>
__device__ __forceinline__ void dft<3, true>(float2* v) { dft3<true>(v); }

template <bool INV>
__device__ __forceinline__ void dft4(float2* v)
{
    const float2 a = c_add(v[0], v[2]), b = c_sub(v[0], v[2]);
    const float2 c = c_add(v[1], v[3]), d = c_rot<INV>(c_sub(v[1], v[3]));
    v[0] = c_add(a, c);
    v[2] = c_sub(a, c);
    v[1] = c_add(b, d);
    v[3] = c_sub(b, d);
}
template <>
__device__ __forceinline__ void dft<4, false>(float2* v) { dft4<false>(v); }
template <>
__device__ __forceinline__ void dft<4, true>(float2* v) { dft4<true>(v); }

template <bool INV>
__device__ __forceinline__ void dft8(float2* v)
{
    constexpr float kH = 0.70710678118654752440f;   // sqrt(1/2)
    // y_{2q} = DFT4(v_m + v_{m+4}),  y_{2q+1} = DFT4((v_m - v_{m+4}) W8^m)
    float2 a[4], b[4];
#pragma unroll
    for (int m = 0; m < 4; ++m) {
        a[m] = c_add(v[m], v[m + 4]);
        b[m] = c_sub(v[m], v[m + 4]);
    }
    // W8^1 = (1 -+ i)/sqrt2, W8^2 = -+i, W8^3 = (-1 -+ i)/sqrt2  (upper sign forward)
    {
        const float2 t = b[1];
        const float2 r = c_rot<INV>(t);                    // -+ i t
        b[1] = make_float2(kH * (t.x + r.x), kH * (t.y + r.y));
    }
    b[2] = c_rot<INV>(b[2]);
    {
        const float2 t = b[3];
        const float2 r = c_rot<INV>(t);
        b[3] = make_float2(kH * (r.x - t.x), kH * (r.y - t.y));
    }
    dft4<INV>(a);
    dft4<INV>(b);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        v[2 * q] = a[q];
        v[2 * q + 1] = b[q];
    }
}
template <>
__device__ __forceinline__ void dft<8, false>(float2* v) { dft8<false>(v); }
template <>
__device__ __forceinline__ void dft<8, true>(float2* v) { dft8<true>(v); }

// Radix 9 as 3 x 3: y_{q1 + 3 q2} = sum_{m2} W3^{q2 m2} [W9^{q1 m2} sum_{m1} W3^{q1 m1} v_{3 m1 + m2}].
template <bool INV>
__device__ __forceinline__ void dft9(float2* v)
{
    constexpr float kC1 = 0.76604444311897803520f, kS1 = 0.64278760968653932632f;   // 2 pi / 9
    constexpr float kC2 = 0.17364817766693034885f, kS2 = 0.98480775301220805937f;   // 4 pi / 9
    constexpr float kC4 = -0.93969262078590838405f, kS4 = 0.34202014332566873304f;  // 8 pi / 9
    const float sg = INV ? 1.f : -1.f;
    float2 a[3][3];
#pragma unroll
    for (int m2 = 0; m2 < 3; ++m2) {
        float2 t[3] = {v[m2], v[3 + m2], v[6 + m2]};
        dft3<INV>(t);
#pragma unroll
        for (int q1 = 0; q1 < 3; ++q1) a[q1][m2] = t[q1];
    }
    a[1][1] = c_mul(a[1][1], make_float2(kC1, sg * kS1));
    a[1][2] = c_mul(a[1][2], make_float2(kC2, sg * kS2));
    a[2][1] = c_mul(a[2][1], make_float2(kC2, sg * kS2));
    a[2][2] = c_mul(a[2][2], make_float2(kC4, sg * kS4));
#pragma unroll
    for (int q1 = 0; q1 < 3; ++q1) {
        dft3<INV>(a[q1]);
#pragma unroll
        for (int q2 = 0; q2 < 3; ++q2) v[q1 + 3 * q2] = a[q1][q2];
    }
}
template <>
__device__ __forceinline__ void dft<9, false>(float2* v) { dft9<false>(v); }
template <>
__device__ __forceinline__ void dft<9, true>(float2* v) { dft9<true>(v); }

// Radix A B for coprime A, B by the prime-factor map (Good 1958): with
// n = B n1 + A n2 (mod A B) and k = k1 e1 + k2 e2 (mod A B), e1 = 1 (mod A),
// 0 (mod B) and e2 the other way round, W^{n k} = W_A^{n1 k1} W_B^{n2 k2}:
// no twiddles.  2 x 3 (e = 3, 4) and 3 x 4 (e = 4, 9).
template <int A, int B, int E1, int E2, bool INV>
__device__ __forceinline__ void dft_pf(float2* v)
{
    float2 t[A][B];
#pragma unroll
    for (int n1 = 0; n1 < A; ++n1) {
#pragma unroll
        for (int n2 = 0; n2 < B; ++n2) t[n1][n2] = v[(B * n1 + A * n2) % (A * B)];
        dft<B, INV>(t[n1]);
    }
#pragma unroll
    for (int k2 = 0; k2 < B; ++k2) {
        float2 u[A];
#pragma unroll
        for (int n1 = 0; n1 < A; ++n1) u[n1] = t[n1][k2];
        dft<A, INV>(u);
#pragma unroll
        for (int k1 = 0; k1 < A; ++k1) v[(k1 * E1 + k2 * E2) % (A * B)] = u[k1];
    }
}
template <>
__device__ __forceinline__ void dft<6, false>(float2* v) { dft_pf<2, 3, 3, 4, false>(v); }
template <>
__device__ __forceinline__ void dft<6, true>(float2* v) { dft_pf<2, 3, 3, 4, true>(v); }
template <>
__device__ __forceinline__ void dft<12, false>(float2* v) { dft_pf<3, 4, 4, 9, false>(v); }
template <>
__device__ __forceinline__ void dft<12, true>(float2* v) { dft_pf<3, 4, 4, 9, true>(v); }

// Radix 16 as 4 x 4: y_{q1 + 4 q2} = sum_{m2} W4^{q2 m2} [W16^{q1 m2} sum_{m1} W4^{q1 m1} v_{4 m1 + m2}].
template <bool INV>
__device__ __forceinline__ void dft16(float2* v)
{
    constexpr float kH = 0.70710678118654752440f;   // cos(pi/4)
    constexpr float kC = 0.92387953251128675613f;   // cos(pi/8)
    constexpr float kS = 0.38268343236508977173f;   // sin(pi/8)
    float2 a[4][4];
#pragma unroll
    for (int m2 = 0; m2 < 4; ++m2) {
        float2 t[4] = {v[m2], v[4 + m2], v[8 + m2], v[12 + m2]};
        dft4<INV>(t);
#pragma unroll
        for (int q1 = 0; q1 < 4; ++q1) a[q1][m2] = t[q1];
    }
    // twiddles W16^{q1 m2} (forward e^{-2 pi i q1 m2 / 16})
    const float sg = INV ? 1.f : -1.f;
    // q1 = 1: m2 = 1, 2, 3 -> angles pi/8, pi/4, 3pi/8
    a[1][1] = c_mul(a[1][1], make_float2(kC, sg * kS));
    a[1][2] = c_mul(a[1][2], make_float2(kH, sg * kH));
    a[1][3] = c_mul(a[1][3], make_float2(kS, sg * kC));
    // q1 = 2: angles pi/4, pi/2, 3pi/4
    a[2][1] = c_mul(a[2][1], make_float2(kH, sg * kH));
    a[2][2] = c_rot<INV>(a[2][2]);
    a[2][3] = c_mul(a[2][3], make_float2(-kH, sg * kH));
    // q1 = 3: angles 3pi/8, 3pi/4, 9pi/8
    a[3][1] = c_mul(a[3][1], make_float2(kS, sg * kC));
    a[3][2] = c_mul(a[3][2], make_float2(-kH, sg * kH));
    a[3][3] = c_mul(a[3][3], make_float2(-kC, -sg * kS));
#pragma unroll
    for (int q1 = 0; q1 < 4; ++q1) {
        dft4<INV>(a[q1]);
#pragma unroll
        for (int q2 = 0; q2 < 4; ++q2) v[q1 + 4 * q2] = a[q1][q2];
    }
}
template <>
__device__ __forceinline__ void dft<16, false>(float2* v) { dft16<false>(v); }
template <>
__device__ __forceinline__ void dft<16, true>(float2* v) { dft16<true>(v); }

// Plain shared-memory buffer access.  Loaders and storers of the run-time
// stages give at(p), the access to one pencil's elements, so that what
// depends on the pencil only is formed once per butterfly.
struct BufLd {
    const float2* b;
    int ld;
    __device__ __forceinline__ float2 operator()(int e, int p) const { return b[e * ld + p]; }
    struct At {
        const float2* b;
        int ld;
        __device__ __forceinline__ float2 operator()(int e) const { return b[e * ld]; }
    };
    __device__ __forceinline__ At at(int p) const { return At{b + p, ld}; }
};
struct BufSt {
    float2* b;
    int ld;
    __device__ __forceinline__ void operator()(int e, int p, float2 v) const { b[e * ld + p] = v; }
    struct At {
        float2* b;
        int ld;
        __device__ __forceinline__ void operator()(int e, float2 v) const { b[e * ld] = v; }
    };
    __device__ __forceinline__ At at(int p) const { return At{b + p, ld}; }
};

// ---------------------------------------------------------------------------
// Run-time schedules.  A stage's radix is a template parameter (one switch
// per stage), its length, strides and divisions are uniform values; the
// pencil count is a power of two, 1 << lgP.
// ---------------------------------------------------------------------------
// Geometry of stage s of a schedule: butterflies nb = n / R, Ns = product
// of the earlier radices, and the divisions by both.
struct StageGeom {
    int n, nb, Ns, R;
    FastDiv dnb, dns;
};
__device__ __forceinline__ StageGeom stage_fwd(const RadixPlan& pl, int s)
{
    return StageGeom{pl.n, (int)pl.dnb[s].d, pl.ns[s], pl.radix[s], pl.dnb[s], pl.dns[s]};
}
// Stage i of the reversed schedule (the inverse transforms).
__device__ __forceinline__ StageGeom stage_rev(const RadixPlan& pl, int i)
{
    const int s = pl.nst - 1 - i;
    return StageGeom{pl.n, (int)pl.dnb[s].d, pl.nsr[s], pl.radix[s], pl.dnb[s], pl.dnsr[s]};
}

// Butterfly idx of a stage: pencil and butterfly number, pencils fastest
// (PFAST) or butterflies fastest.
template <bool PFAST>
__device__ __forceinline__ void stage_index(int idx, const StageGeom& g, int lgP, int& p, int& j)
{
    if (PFAST) {
        p = idx & ((1 << lgP) - 1);
        j = idx >> lgP;
    } else {
        p = (int)g.dnb.div((uint32_t)idx);
        j = idx - p * g.nb;
    }
}

// The twiddles W_{Ns R}^{r k} of a butterfly (k = j mod Ns) applied to v.
template <int R, bool INV>
__device__ __forceinline__ void stage_twiddle(float2* v, int k, const StageGeom& g, const float2* __restrict__ tw)
{
    // table step n / (Ns R) = nb / Ns; a stage past the first has k < Ns
    const int step = k * (g.Ns == g.nb ? 1 : (int)g.dns.div((uint32_t)g.nb));
#pragma unroll
    for (int r = 1; r < R; ++r) {
        float2 w = tw[r * step];
        if (INV) w.y = -w.y;
        v[r] = c_mul(v[r], w);
    }
}

// One radix-R Stockham stage over 1 << lgP pencils.
template <int R, bool INV, bool PFAST, class LD, class ST>
__device__ __forceinline__ void rt_stage(const LD& ld, const ST& st, const StageGeom& g, int lgP,
                                         const float2* __restrict__ tw)
{
    const int total = g.nb << lgP;
    for (int idx = threadIdx.x; idx < total; idx += blockDim.x) {
        int p, j;
        stage_index<PFAST>(idx, g, lgP, p, j);
        float2 v[R];
        const auto lp = ld.at(p);
#pragma unroll
        for (int r = 0; r < R; ++r) v[r] = lp(j + r * g.nb);
        int dst;
        if (g.Ns == 1) {
            dst = j * R;
        } else if (g.Ns == g.nb) {
            dst = j;
            stage_twiddle<R, INV>(v, j, g, tw);
        } else {
            const int q = (int)g.dns.div((uint32_t)j), k = j - q * g.Ns;
            dst = q * g.Ns * R + k;
            stage_twiddle<R, INV>(v, k, g, tw);
        }
        dft<R, INV>(v);
        const auto sp = st.at(p);
#pragma unroll
        for (int r = 0; r < R; ++r) sp(dst + r * g.Ns, v[r]);
    }
}

template <bool INV, bool PFAST, class LD, class ST>
__device__ __forceinline__ void rt_stage_any(const LD& ld, const ST& st, const StageGeom& g, int lgP,
                                             const float2* __restrict__ tw)
{
    switch (g.R) {
        case 16: rt_stage<16, INV, PFAST>(ld, st, g, lgP, tw); break;
        case 12: rt_stage<12, INV, PFAST>(ld, st, g, lgP, tw); break;
        case 9: rt_stage<9, INV, PFAST>(ld, st, g, lgP, tw); break;
        case 8: rt_stage<8, INV, PFAST>(ld, st, g, lgP, tw); break;
        case 6: rt_stage<6, INV, PFAST>(ld, st, g, lgP, tw); break;
        case 4: rt_stage<4, INV, PFAST>(ld, st, g, lgP, tw); break;
        case 3: rt_stage<3, INV, PFAST>(ld, st, g, lgP, tw); break;
        case 2: rt_stage<2, INV, PFAST>(ld, st, g, lgP, tw); break;
        default: break;
    }
}

// A stage between shared-memory buffers, pencils fastest: one copy of the
// code per kernel file (the stages between a transform's first and last).
template <bool INV>
__device__ __noinline__ void rt_stage_buf(const float2* src, float2* dst, int lds, const StageGeom& g, int lgP,
                                          const float2* __restrict__ tw)
{
    rt_stage_any<INV, true>(BufLd{src, lds}, BufSt{dst, lds}, g, lgP, tw);
}

// The last forward stage, a multiplication by mu (element e by mu[e]) and the
// first inverse stage on the same butterflies, in registers.
template <int R, class LD, class ST>
__device__ __forceinline__ void rt_conv(const LD& ld, const ST& st, const float2* __restrict__ mu, const StageGeom& g, int lgP,
                                        const float2* __restrict__ tw)
{
    const int total = g.nb << lgP;
    for (int idx = threadIdx.x; idx < total; idx += blockDim.x) {
        const int p = idx & ((1 << lgP) - 1), j = idx >> lgP;
        float2 v[R];
        const auto lp = ld.at(p);
#pragma unroll
        for (int r = 0; r < R; ++r) v[r] = lp(j + r * g.nb);
        if (g.Ns > 1) {
#pragma unroll
            for (int r = 1; r < R; ++r) v[r] = c_mul(v[r], tw[r * j]);
        }
        dft<R, false>(v);
#pragma unroll
        for (int r = 0; r < R; ++r) v[r] = c_mul(v[r], mu[j + r * g.nb]);
        dft<R, true>(v);
        const auto sp = st.at(p);
#pragma unroll
        for (int r = 0; r < R; ++r) sp(j * R + r, v[r]);
    }
}
template <class LD, class ST>
__device__ __forceinline__ void rt_conv_any(const LD& ld, const ST& st, const float2* __restrict__ mu,
                                            const StageGeom& g, int lgP, const float2* __restrict__ tw)
{
    switch (g.R) {
        case 16: rt_conv<16>(ld, st, mu, g, lgP, tw); break;
        case 12: rt_conv<12>(ld, st, mu, g, lgP, tw); break;
        case 9: rt_conv<9>(ld, st, mu, g, lgP, tw); break;
        case 8: rt_conv<8>(ld, st, mu, g, lgP, tw); break;
        case 6: rt_conv<6>(ld, st, mu, g, lgP, tw); break;
        case 4: rt_conv<4>(ld, st, mu, g, lgP, tw); break;
        case 3: rt_conv<3>(ld, st, mu, g, lgP, tw); break;
        case 2: rt_conv<2>(ld, st, mu, g, lgP, tw); break;
        default: break;
    }
}

// Full transform of P (a power of two) pencils: first stage reads `first`,
// last stage writes `last`, intermediate stages use scratch buffers s0
// (written by stage 0, 2, ...) and s1 (stage 1, 3, ...), both with leading
// dimension lds >= P.  `last` may target either scratch buffer only if that
// buffer is not read by the last stage: the caller guarantees it (see
// fft_result_index).  FIRST_PFAST / LAST_PFAST choose the mapping of the
// first / last stage (a single-stage transform uses LAST_PFAST).  The
// inverse runs the schedule reversed.  Length 1 copies.
template <bool INV, bool FIRST_PFAST, bool LAST_PFAST, class LD, class ST>
__device__ __forceinline__ void fft_run(const RadixPlan& pl, const LD& first, const ST& last, float2* s0,
                                        float2* s1, int lds, int P, const float2* tw)
{
    const int lgP = 31 - __clz(P);
    if (pl.nst == 0) {
        for (int p = threadIdx.x; p < P; p += blockDim.x) last.at(p)(0, first.at(p)(0));
        __syncthreads();
        return;
    }
    for (int s = 0; s < pl.nst; ++s) {
        const StageGeom g = INV ? stage_rev(pl, s) : stage_fwd(pl, s);
        const bool isFirst = (s == 0), isLast = (s == pl.nst - 1);
        float2* dstb = (s & 1) ? s1 : s0;
        const float2* srcb = (s & 1) ? s0 : s1;   // buffer written by stage s-1
        if (isFirst && isLast) {
            rt_stage_any<INV, LAST_PFAST>(first, last, g, lgP, tw);
        } else if (isFirst) {
            rt_stage_any<INV, FIRST_PFAST>(first, BufSt{dstb, lds}, g, lgP, tw);
        } else if (isLast) {
            rt_stage_any<INV, LAST_PFAST>(BufLd{srcb, lds}, last, g, lgP, tw);
        } else {
            // inlined: a call gives the kernel a stack, and its launch behind
            // another one then takes 1 us longer (general model at 16 x 16 x 16,
            // K = 3: a forward of nine launches 45 us with it, 38 so)
            rt_stage_any<INV, true>(BufLd{srcb, lds}, BufSt{dstb, lds}, g, lgP, tw);
        }
        __syncthreads();
    }
}

// Index (0 -> s0, 1 -> s1) of the scratch buffer a transform of `nst`
// stages should write its last stage into when the result is to stay in
// scratch: stage s writes s_(s & 1), so the last stage (nst - 1) reads
// s_(nst & 1) and may write s_((nst + 1) & 1).  A transform that then reads
// this result must run with its scratch pair swapped: (s0', s1') =
// (s_(res ^ 1), s_res), so that its stage 0 does not overwrite its input.
__host__ __device__ __forceinline__ int fft_result_index(int nst) { return (nst + 1) & 1; }

// ----------------------------------------------------------------------------
// FP64-grade dot-product accumulation with FP32 arithmetic.
// GB300's FP64 pipe is narrow, so each thread accumulates its products as an
// unevaluated float pair (Dekker's exact product via fma, Knuth's TwoSum);
// the block and grid trees below add such pairs in FP32 too, and only a
// final total becomes a double.
// ----------------------------------------------------------------------------
struct DotAcc {
    float hi = 0.f, lo = 0.f;
    __device__ __forceinline__ void add(float a, float b)
    {
        const float p = a * b;
        const float pe = fmaf(a, b, -p);          // exact: a*b = p + pe
        const float s = hi + p;                   // TwoSum(hi, p)
        const float bb = s - hi;
        const float e = (hi - (s - bb)) + (p - bb);
        hi = s;
        lo += e + pe;
    }
    __device__ __forceinline__ double value() const { return (double)hi + (double)lo; }
};

// Block-wide FP64 sum (all threads participate; result valid in thread 0).
__device__ __forceinline__ double block_sum_f64(double v, double* sh /* >= 32 doubles */)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) sh[wid] = v;
    __syncthreads();
    double t = 0.0;
    if (threadIdx.x < 32) {
        const int nw = (blockDim.x + 31) >> 5;
        t = (threadIdx.x < nw) ? sh[threadIdx.x] : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    }
    return t;
}

// x = m 2^e for a positive normal double x: m in [1, 2) as a float (the
// leading 24 significand bits), e the unbiased exponent.  Integer operations
// only.  Returns false for zero, negative, subnormal, infinite or NaN x.
__device__ __forceinline__ bool dsplit(double x, float* m, int* e)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const int ef = (int)((b >> 52) & 0x7ffu);
    *e = ef - 1023;
    *m = __uint_as_float(0x3f800000u | (unsigned int)((b >> 29) & 0x7fffffu));
    return (b >> 63) == 0 && ef != 0 && ef != 0x7ff;
}

// x / y as a float for doubles x, y: the leading significand bits are
// divided in FP32 and the exponents subtracted.  Truncating each operand to
// 24 bits and rounding the quotient leave a relative error below 3e-7; the
// loop applies the quotient as a float anyway.  Falls back to the FP64
// division when either operand is not a positive normal number.
__device__ __forceinline__ float ddiv_to_float(double x, double y)
{
    float mx, my;
    int ex, ey;
    if (dsplit(x, &mx, &ex) && dsplit(y, &my, &ey)) return ldexpf(mx / my, ex - ey);
    return (float)(x / y);
}

__device__ __forceinline__ bool dbits_finite(double x)
{
    return ((((unsigned long long)__double_as_longlong(x)) >> 52) & 0x7ffu) != 0x7ffu;
}

__device__ __forceinline__ bool dbits_zero(double x)
{
    return (((unsigned long long)__double_as_longlong(x)) << 1) == 0ull;
}

// Sums of compensated FP32 accumulators.  The FP64 pipe is narrow on this
// part (one FP64 warp instruction holds it for many cycles, whatever its
// active lanes), so the whole reduction tree adds (hi, lo) pairs in FP32:
// the high words by TwoSum (Knuth), whose exact rounding error joins the
// low words.  A pair carries about 48 bits, as each thread's accumulator
// did, and only the final total is converted to FP64.  The trees are fixed
// (xor butterflies, lane order), so results do not depend on timing.
__device__ __forceinline__ void pair_add(float& hi, float& lo, float h2, float l2)
{
    const float s = hi + h2;
    const float bb = s - hi;
    const float e = (hi - (s - bb)) + (h2 - bb);
    hi = s;
    lo = (lo + l2) + e;
}

__device__ __forceinline__ void warp_sum_acc(float& hi, float& lo)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float h2 = __shfl_xor_sync(0xffffffffu, hi, o);
        const float l2 = __shfl_xor_sync(0xffffffffu, lo, o);
        pair_add(hi, lo, h2, l2);
    }
}

// Block-wide pair sums of one or two accumulators (all threads participate;
// results valid in thread 0).  sh: at least 4 floats per warp of the block.
__device__ __forceinline__ void block_pair_acc2(const DotAcc& a, const DotAcc* b, float* sh, float2* ta, float2* tb)
{
    float ha = a.hi, la = a.lo, hb = b ? b->hi : 0.f, lb = b ? b->lo : 0.f;
    warp_sum_acc(ha, la);
    if (b) warp_sum_acc(hb, lb);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
    float* shb = sh + 2 * nw;
    __syncthreads();
    if (lane == 0) {
        sh[2 * wid] = ha;
        sh[2 * wid + 1] = la;
        shb[2 * wid] = hb;
        shb[2 * wid + 1] = lb;
    }
    __syncthreads();
    if (threadIdx.x < 32) {
        const bool in = (int)threadIdx.x < nw;
        ha = in ? sh[2 * threadIdx.x] : 0.f;
        la = in ? sh[2 * threadIdx.x + 1] : 0.f;
        warp_sum_acc(ha, la);
        *ta = make_float2(ha, la);
        if (b) {
            hb = in ? shb[2 * threadIdx.x] : 0.f;
            lb = in ? shb[2 * threadIdx.x + 1] : 0.f;
            warp_sum_acc(hb, lb);
            *tb = make_float2(hb, lb);
        }
    }
}

__device__ __forceinline__ float2 block_pair_acc(const DotAcc& a, double* sh /* >= 2 doubles per warp */)
{
    float2 t = make_float2(0.f, 0.f), u;
    block_pair_acc2(a, nullptr, reinterpret_cast<float*>(sh), &t, &u);
    return t;
}

// The block total as a double (valid in thread 0).
__device__ __forceinline__ double block_sum_acc(const DotAcc& a, double* sh /* >= 2 doubles per warp */)
{
    const float2 t = block_pair_acc(a, sh);
    return (double)t.x + (double)t.y;
}

// Grid-wide deterministic reduction of the blocks' pair sums.  Each block
// stores its pair (v valid in thread 0) in the 8-byte slot part[bid]; the
// last block to arrive (atomic ticket) adds part[0..nparts) in a fixed
// order (warp 0: lane l takes l, l + 32, ..., then a butterfly over the
// lanes), stores the total in *out as a double, and re-arms the ticket
// counter for the next launch.  Consumers read the single scalar.
__device__ __forceinline__ float2 grid_pairs_sum(const double* part, int nparts)
{
    const float2* pp = reinterpret_cast<const float2*>(part);
    float hi = 0.f, lo = 0.f;
    for (int i = threadIdx.x; i < nparts; i += 32) {
        const float2 v = __ldcg(pp + i);
        pair_add(hi, lo, v.x, v.y);
    }
    warp_sum_acc(hi, lo);
    return make_float2(hi, lo);
}

__device__ __forceinline__ void grid_sum_finalize(float2 v, double* part, int bid, int nparts, unsigned int* counter,
                                                  double* out)
{
    __shared__ int am_last;
    if (threadIdx.x == 0) {
        reinterpret_cast<float2*>(part)[bid] = v;
        __threadfence();
        const unsigned int t = atomicAdd(counter, 1u);
        am_last = (t == (unsigned int)nparts - 1u);
    }
    __syncthreads();
    if (am_last && threadIdx.x < 32) {
        __threadfence();
        const float2 t = grid_pairs_sum(part, nparts);
        if (threadIdx.x == 0) {
            *out = (double)t.x + (double)t.y;
            *counter = 0u;
            __threadfence();
        }
    }
}

// Two totals with one ticket: the last block sums both partial arrays.
__device__ __forceinline__ void grid_sum_finalize2(float2 v0, float2 v1, double* part0, double* part1, int bid,
                                                   int nparts, unsigned int* counter, double* out0, double* out1)
{
    __shared__ int am_last2;
    if (threadIdx.x == 0) {
        reinterpret_cast<float2*>(part0)[bid] = v0;
        reinterpret_cast<float2*>(part1)[bid] = v1;
        __threadfence();
        const unsigned int t = atomicAdd(counter, 1u);
        am_last2 = (t == (unsigned int)nparts - 1u);
    }
    __syncthreads();
    if (am_last2 && threadIdx.x < 32) {
        __threadfence();
        const float2 t0 = grid_pairs_sum(part0, nparts);
        const float2 t1 = grid_pairs_sum(part1, nparts);
        if (threadIdx.x == 0) {
            *out0 = (double)t0.x + (double)t0.y;
            *out1 = (double)t1.x + (double)t1.y;
            *counter = 0u;
            __threadfence();
        }
    }
}

}  // namespace mh3d
