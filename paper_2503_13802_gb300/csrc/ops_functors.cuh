// Loader / storer functors and small device helpers shared by the runtime
// pencil kernels (ops.cu) and the compile-time specialised ones (ops_ct.cuh).
#pragma once

#include "ops_kernels.cuh"

namespace mh3d {

// ---------------------------------------------------------------------------
// Small helpers
// ---------------------------------------------------------------------------
__device__ __forceinline__ float2 ld2(const float* __restrict__ p, long long i, bool has2, int vec2)
{
    if (vec2 && has2) return *reinterpret_cast<const float2*>(p + i);
    return make_float2(p[i], has2 ? p[i + 1] : 0.f);
}
__device__ __forceinline__ void st2(float* __restrict__ p, long long i, bool has2, int vec2, float2 v)
{
    if (vec2 && has2) {
        *reinterpret_cast<float2*>(p + i) = v;
    } else {
        p[i] = v.x;
        if (has2) p[i + 1] = v.y;
    }
}

// a mod n for a in [-2, n + 1] (n >= 1): two steps either way cover n = 1.
__device__ __forceinline__ int wrap(int a, int n)
{
    if (a < 0) a += n;
    if (a < 0) a += n;
    if (a >= n) a -= n;
    if (a >= n) a -= n;
    return a;
}

// lambda * (R p)[i] at voxel (x, y, z).
__device__ __forceinline__ float reg_term(const RegArgs& g, const float* __restrict__ p, long long i, int x, int y,
                                          int z)
{
    const float pc = p[i];
    if (g.kind == 0) return g.lambda * pc;
    // T^T T = sum_a D_a^2, D_a the periodic second difference: stencil
    // (1, -4, 6, -4, 1) along each axis.
    const long long sy = g.nx, sz = (long long)g.nx * g.ny;
    const long long base = i - x - (long long)y * sy - (long long)z * sz;
    float acc = 0.f;
    {
        const long long r = base + (long long)y * sy + (long long)z * sz;
        acc += p[r + wrap(x - 2, g.nx)] - 4.f * p[r + wrap(x - 1, g.nx)] + 6.f * pc
             - 4.f * p[r + wrap(x + 1, g.nx)] + p[r + wrap(x + 2, g.nx)];
    }
    {
        const long long r = base + x + (long long)z * sz;
        acc += p[r + wrap(y - 2, g.ny) * sy] - 4.f * p[r + wrap(y - 1, g.ny) * sy] + 6.f * pc
             - 4.f * p[r + wrap(y + 1, g.ny) * sy] + p[r + wrap(y + 2, g.ny) * sy];
    }
    {
        const long long r = base + x + (long long)y * sy;
        acc += p[r + wrap(z - 2, g.nz) * sz] - 4.f * p[r + wrap(z - 1, g.nz) * sz] + 6.f * pc
             - 4.f * p[r + wrap(z + 1, g.nz) * sz] + p[r + wrap(z + 2, g.nz) * sz];
    }
    const bool shell = x < g.shell || y < g.shell || z < g.shell || x >= g.nx - g.shell || y >= g.ny - g.shell ||
                       z >= g.nz - g.shell;
    if (shell) acc += g.alpha * pc;
    return g.lambda * acc;
}

// The same at voxels x .. x + 3 of a row (x and nx multiples of 4, p 16-byte
// aligned): eleven float4 loads where reg_term takes 52 scalar ones.
__device__ __forceinline__ float4 reg_term4(const RegArgs& g, const float* __restrict__ p, long long i, int x, int y,
                                            int z)
{
    const int sy = g.nx, sz = g.nx * g.ny;
    const float* c0 = p + i;
    auto ld = [&](long long off) { return __ldg(reinterpret_cast<const float4*>(c0 + off)); };
    auto dy = [&](int d) { return ld((long long)(wrap(y + d, g.ny) - y) * sy); };
    auto dz = [&](int d) { return ld((long long)(wrap(z + d, g.nz) - z) * sz); };
    const float4 c = ld(0), l = ld(x == 0 ? g.nx - 4 : -4), r = ld(x + 4 == g.nx ? 4 - g.nx : 4);
    const float4 y0 = dy(-2), y1 = dy(-1), y3 = dy(1), y4 = dy(2), z0 = dz(-2), z1 = dz(-1), z3 = dz(1), z4 = dz(2);
    auto one = [&](float x0, float x1, float pc, float x3, float x4, float ya, float yb, float yc, float yd, float za,
                   float zb, float zc, float zd, int xx) {
        float acc = 0.f;
        acc += x0 - 4.f * x1 + 6.f * pc - 4.f * x3 + x4;
        acc += ya - 4.f * yb + 6.f * pc - 4.f * yc + yd;
        acc += za - 4.f * zb + 6.f * pc - 4.f * zc + zd;
        const bool shell = xx < g.shell || y < g.shell || z < g.shell || xx >= g.nx - g.shell ||
                           y >= g.ny - g.shell || z >= g.nz - g.shell;
        if (shell) acc += g.alpha * pc;
        return g.lambda * acc;
    };
    return make_float4(one(l.z, l.w, c.x, c.y, c.z, y0.x, y1.x, y3.x, y4.x, z0.x, z1.x, z3.x, z4.x, x),
                       one(l.w, c.x, c.y, c.z, c.w, y0.y, y1.y, y3.y, y4.y, z0.y, z1.y, z3.y, z4.y, x + 1),
                       one(c.x, c.y, c.z, c.w, r.x, y0.z, y1.z, y3.z, y4.z, z0.z, z1.z, z3.z, z4.z, x + 2),
                       one(c.y, c.z, c.w, r.x, r.y, y0.w, y1.w, y3.w, y4.w, z0.w, z1.w, z3.w, z4.w, x + 3));
}

// CG loop control at the start of an iteration's kernels.  Returns false
// when the loop is finished (every CTA of the kernel returns).  The first
// kernel of an iteration also evaluates the stopping rule and the CG beta
// (and, in the single-reduction form, alpha).  Every control word and scalar
// is read in one round of loads (values read before the done flag is tested
// are simply unused once the loop has ended).  The stopping test and
// alpha's cancellation-prone denominator are FP64.  With c.fp64 (the
// default) beta and alpha are FP64 quotients, rounded to FP32 only for the
// FP32 vector updates, and the recurrence keeps the FP64 alpha; otherwise
// the divisions run in FP32 on the split significands (ddiv_to_float,
// relative error below 3e-7), which keeps the narrow FP64 pipe of this part
// free of divides.  Every CTA computes them with the same operations, so all
// apply the same values.
__device__ __forceinline__ bool cg_enter(const CgCtl& c, bool first_kernel, float* beta, double* sh,
                                         float* alpha = nullptr)
{
    if (!first_kernel) return !*(volatile int*)&c.flags[0];
    const int done = *(volatile int*)&c.flags[0];
    const int it = *(volatile int*)&c.flags[1];
    const int gave_up = *(volatile int*)&c.flags[3];
    const double g_new = __ldcg(c.rr_new);
    const double bn = __ldcg(c.bn);
    const double ro = c.rr_old ? __ldcg(c.rr_old) : 0.0;
    const double dl = c.cgcg ? __ldcg(c.delta) : 0.0;
    const double ap = c.cgcg ? __ldcg(c.alpha_prev) : 0.0;
    if (done) return false;
    const bool lead = threadIdx.x == 0 && blockIdx.x == 0 && blockIdx.y == 0;
    if (gave_up) {   // a bounded wait gave up earlier: stop the loop
        if (lead) {
            c.flags[2] = MH3D_ERR_TIMEOUT;
            __threadfence();
            c.flags[0] = 1;
            if (c.use_cond) cudaGraphSetConditional(c.cond, 0);
        }
        return false;
    }
    int status = -1;
    if (!dbits_finite(g_new) || !dbits_finite(bn)) status = MH3D_ERR_NONFINITE;
    else if (dbits_zero(g_new) || dbits_zero(bn)) status = MH3D_OK;
    else if (c.tol2 > 0.0 && g_new <= c.tol2 * bn) status = MH3D_OK;   // ||r||^2 / ||A^T d||^2 <= tol^2
    else if (it >= c.max_iter) status = (c.tol2 > 0.0) ? MH3D_ERR_NOT_CONVERGED : MH3D_OK;
    if (lead && it < c.hist_cap) c.hist[it] = (bn > 0.0) ? sqrt(g_new / bn) : 0.0;
    if (status >= 0) {
        if (lead) {
            c.flags[2] = status;
            __threadfence();
            c.flags[0] = 1;
            if (c.use_cond) cudaGraphSetConditional(c.cond, 0);
        }
        return false;
    }
    // beta_i = gamma_i / gamma_{i-1}
    *beta = (it > 0) ? (c.fp64 ? (float)(g_new / ro) : ddiv_to_float(g_new, ro)) : 0.f;
    if (c.cgcg) {
        // alpha_i = gamma_i / (delta_i - beta_i gamma_i / alpha_{i-1})
        //         = gamma_i u / (delta_i u - gamma_i^2),  u = gamma_{i-1} alpha_{i-1}
        const double an = (it == 0) ? g_new : g_new * (ro * ap);
        const double ad = (it == 0) ? dl : fma(dl, ro * ap, -g_new * g_new);
        double a64 = 0.0;
        float a;
        if (c.fp64) {
            a64 = an / ad;
            a = (float)a64;
        } else {
            a = ddiv_to_float(an, ad);
            a64 = (double)a;
        }
        if (!isfinite(a) || !(a > 0.f)) {
            if (lead) {
                c.flags[2] = MH3D_ERR_NONFINITE;
                __threadfence();
                c.flags[0] = 1;
                if (c.use_cond) cudaGraphSetConditional(c.cond, 0);
            }
            return false;
        }
        if (lead) *c.alpha_out = a64;
        if (alpha) *alpha = a;
    }
    return true;
}

// cg_enter for a whole CTA (every thread calls it; c.flags set): thread 0
// evaluates the loop control and shares beta, alpha and the decision through
// shared memory, so the FP64 divides run once per CTA instead of once per
// thread (the FP64 pipe is narrow on this part).
__device__ __forceinline__ bool cg_enter_cta(const CgCtl& c, bool first_kernel, float* beta, float* alpha,
                                             float* sh3)
{
    if (threadIdx.x == 0) {
        float b = 0.f, al = 0.f;
        const bool go = cg_enter(c, first_kernel, &b, nullptr, &al);
        sh3[0] = b;
        sh3[1] = al;
        sh3[2] = go ? 1.f : 0.f;
    }
    __syncthreads();
    *beta = sh3[0];
    *alpha = sh3[1];
    return sh3[2] != 0.f;
}

// End of a CG iteration whose last pass is this kernel: the lead thread
// advances the completed-iteration counter (read only by later kernels).
// The hard bound ends the graph loop even if the first kernel of the next
// iteration, which normally stops it at max_iter, never ran.
__device__ __forceinline__ void cg_count_iteration(const CgCtl& c)
{
    if (threadIdx.x == 0 && blockIdx.x == 0 && blockIdx.y == 0) {
        const int it = c.flags[1] + 1;
        c.flags[1] = it;
        if (it > c.max_iter + 1) {
            c.flags[2] = MH3D_ERR_NOT_CONVERGED;
            if (c.use_cond) cudaGraphSetConditional(c.cond, 0);
        }
    }
}

// ---------------------------------------------------------------------------
// T pass
// ---------------------------------------------------------------------------
// Column pair p of a tile (run-time kernels).  nx even: columns x0 + 2p and
// x0 + 2p + 1, one 8-byte access; nx odd (rows not 8-byte aligned): columns
// x0 + p and x0 + p + P, so that consecutive lanes take consecutive columns
// of either access.
struct TCols {
    int x, second;       // first column, distance to the second
    bool has1, has2;
    __device__ __forceinline__ TCols(const TArgs& a, int x0, int p)
    {
        second = a.vec2 ? 1 : a.cols / 2;
        x = x0 + (a.vec2 ? 2 * p : p);
        has1 = x < a.nx;
        has2 = x + second < a.nx;
    }
    __device__ __forceinline__ float2 ld(const float* __restrict__ p, int i, int vec2) const
    {
        if (vec2) return *reinterpret_cast<const float2*>(p + i);
        return make_float2(p[i], has2 ? p[i + second] : 0.f);
    }
    __device__ __forceinline__ void st(float* __restrict__ p, int i, int vec2, float2 v) const
    {
        if (vec2) {
            *reinterpret_cast<float2*>(p + i) = v;
        } else {
            p[i] = v.x;
            if (has2) p[i + second] = v.y;
        }
    }
};

// Tile loader of a plain pass (in, times b).
struct TLoad {
    const TArgs* a;
    int base;            // voxel index of element 0, column 0 (grids hold at most 2^30 voxels)
    int x0;
    struct At {
        const TArgs* a;
        TCols c;
        int base, es;
        __device__ __forceinline__ float2 operator()(int e) const
        {
            if (!c.has1) return make_float2(0.f, 0.f);
            const int i = base + e * es, w = a->vec2;
            float2 v = c.ld(a->in, i, w);
            if (a->bin) {
                const float2 bb = c.ld(a->bin, i, w);
                v.x *= bb.x;
                v.y *= bb.y;
            }
            return v;
        }
    };
    __device__ __forceinline__ At at(int p) const
    {
        const TCols c(*a, x0, p);
        return At{a, c, base + c.x, (int)a->es};
    }
};

// The CG vector updates of a tile (TArgs.pupdate: MODE 1 p = r + beta p, 2
// the single-reduction form), the first stage's input into buf [n][P].  Four
// elements a step with every load before the stores, so that a thread keeps
// up to 24 loads in flight.
template <int MODE>
__device__ __forceinline__ void t_update(const TArgs& a, int base, int x0, int lgP, float beta, float alpha, float2* buf)
{
    constexpr int U = 4;
    const int w = a.vec2, de = (int)blockDim.x >> lgP, n = a.n;   // a thread keeps its column pair
    const TCols c(a, x0, (int)threadIdx.x & ((1 << lgP) - 1));
    const int es = (int)a.es, b0 = base + c.x;
    for (int e0 = (int)threadIdx.x >> lgP; e0 < n; e0 += U * de) {
        float2 rr[U], ss[U], pp[U], qq[U], xx[U], bb[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int e = e0 + u * de, i = b0 + e * es;
            if (e >= n || !c.has1) continue;
            rr[u] = c.ld(a.rvec, i, w);
            pp[u] = c.ld(a.pvec, i, w);
            if constexpr (MODE == 2) {
                ss[u] = c.ld(a.svec, i, w);
                qq[u] = c.ld(a.qdir, i, w);
                xx[u] = c.ld(a.xvec, i, w);
            }
            bb[u] = a.bin ? c.ld(a.bin, i, w) : make_float2(1.f, 1.f);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int e = e0 + u * de, i = b0 + e * es;
            if (e >= n) continue;
            float2 v = make_float2(0.f, 0.f);
            if (c.has1) {
                const float2 pn = make_float2(fmaf(beta, pp[u].x, rr[u].x), fmaf(beta, pp[u].y, rr[u].y));
                c.st(a.pvec, i, w, pn);
                v = pn;
                if constexpr (MODE == 2) {
                    const float2 qn = make_float2(fmaf(beta, qq[u].x, ss[u].x), fmaf(beta, qq[u].y, ss[u].y));
                    c.st(a.qdir, i, w, qn);
                    c.st(a.xvec, i, w, make_float2(fmaf(alpha, pn.x, xx[u].x), fmaf(alpha, pn.y, xx[u].y)));
                    v = make_float2(fmaf(-alpha, qn.x, rr[u].x), fmaf(-alpha, qn.y, rr[u].y));
                    c.st(a.rvec_w, i, w, v);
                }
                if (a.bin) {
                    v.x *= bb[u].x;
                    v.y *= bb[u].y;
                }
            }
            buf[(e << lgP) + ((int)threadIdx.x & ((1 << lgP) - 1))] = v;
        }
    }
}

// Tile storer of a plain pass (times b).
struct TStore {
    const TArgs* a;
    int base;
    int x0;
    struct At {
        const TArgs* a;
        TCols c;
        int base, es;
        __device__ __forceinline__ void operator()(int e, float2 v) const
        {
            if (!c.has1) return;
            const int i = base + e * es, w = a->vec2;
            if (a->bout) {
                const float2 bb = c.ld(a->bout, i, w);
                v.x *= bb.x;
                v.y *= bb.y;
            }
            c.st(a->out, i, w, v);
        }
    };
    __device__ __forceinline__ At at(int p) const
    {
        const TCols c(*a, x0, p);
        return At{a, c, base + c.x, (int)a->es};
    }
};

// The explicit normal operator's epilogue over a transformed tile buf [n][P]:
// q = b w + lambda R p, with p^T q (and p^T p for acc2); four elements a step
// with the loads of R = I first.
__device__ __forceinline__ void t_epilogue(const TArgs& a, int base, int x0, int lgP, const float2* buf, DotAcc* acc,
                                           DotAcc* acc2)
{
    constexpr int U = 4;
    const int w = a.vec2, de = (int)blockDim.x >> lgP, n = a.n;   // a thread keeps its column pair
    const int p = (int)threadIdx.x & ((1 << lgP) - 1);
    const TCols c(a, x0, p);
    if (!c.has1) return;
    const int es = (int)a.es, b0 = base + c.x;
    const bool plain = a.reg.kind == 0;
    for (int e0 = (int)threadIdx.x >> lgP; e0 < n; e0 += U * de) {
        float2 pp[U], bb[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int e = e0 + u * de, i = b0 + e * es;
            if (e >= n) continue;
            pp[u] = c.ld(a.pin, i, w);
            bb[u] = a.bout ? c.ld(a.bout, i, w) : make_float2(1.f, 1.f);
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int e = e0 + u * de, i = b0 + e * es;
            if (e >= n) continue;
            float2 v = buf[(e << lgP) + p];
            if (a.bout) {
                v.x *= bb[u].x;
                v.y *= bb[u].y;
            }
            if (plain) {
                v.x += a.reg.lambda * pp[u].x;
                v.y += a.reg.lambda * pp[u].y;
            } else {
                const int y = a.axis == 1 ? e : (int)blockIdx.y, z = a.axis == 1 ? (int)blockIdx.y : e;
                v.x += reg_term(a.reg, a.pin, i, c.x, y, z);
                if (c.has2) v.y += reg_term(a.reg, a.pin, i + c.second, c.x + c.second, y, z);
            }
            c.st(a.qvec, i, w, v);
            acc->add(pp[u].x, v.x);
            if (acc2) acc2->add(pp[u].x, pp[u].x);
            if (c.has2) {
                acc->add(pp[u].y, v.y);
                if (acc2) acc2->add(pp[u].y, pp[u].y);
            }
        }
    }
}

// ---------------------------------------------------------------------------
// X pass: loaders and storers
// ---------------------------------------------------------------------------
// Pencil p of a row-pair batch = rows (row0 + 2p, row0 + 2p + 1) as re/im.
struct RowPairLd {
    const float* v;
    int nx, row0, rows;
    __device__ __forceinline__ float2 operator()(int e, int p) const
    {
        const int r = row0 + 2 * p;
        float2 o = make_float2(0.f, 0.f);
        if (r < rows) o.x = v[(long long)r * nx + e];
        if (r + 1 < rows) o.y = v[(long long)(r + 1) * nx + e];
        return o;
    }
    struct At {
        const float* v;
        int nx;
        bool h1, h2;
        __device__ __forceinline__ float2 operator()(int e) const
        {
            return make_float2(h1 ? v[e] : 0.f, h2 ? v[nx + e] : 0.f);
        }
    };
    __device__ __forceinline__ At at(int p) const
    {
        const int r = row0 + 2 * p;
        return At{v + (long long)r * nx, nx, r < rows, r + 1 < rows};
    }
};
struct RowPairSt {
    float* v;
    int nx, row0, rows;
    __device__ __forceinline__ void operator()(int e, int p, float2 val) const
    {
        const int r = row0 + 2 * p;
        if (r < rows) v[(long long)r * nx + e] = val.x;
        if (r + 1 < rows) v[(long long)(r + 1) * nx + e] = val.y;
    }
    struct At {
        float* v;
        int nx;
        bool h1, h2;
        __device__ __forceinline__ void operator()(int e, float2 val) const
        {
            if (h1) v[e] = val.x;
            if (h2) v[nx + e] = val.y;
        }
    };
    __device__ __forceinline__ At at(int p) const
    {
        const int r = row0 + 2 * p;
        return At{v + (long long)r * nx, nx, r < rows, r + 1 < rows};
    }
};

// Forward: the portrait spectrum of pencil q = kk P + p (harmonic kk of a
// round) at bin m = sum_{j < s} A[m + j mx] Xhat_kk[m + j mx]   (the fold that
// realises P).
struct FoldLd {
    const float2* A;
    int ldA;
    const float2* __restrict__ xk;   // the round's first harmonic's spectrum
    int nx, mx, s, lgP, left;        // left: harmonics from the round's first on
    struct At {
        const float2* A;
        int ldA;
        const float2* __restrict__ xk;
        int mx, s;
        __device__ __forceinline__ float2 operator()(int m) const
        {
            float2 acc = c_mul(A[m * ldA], __ldg(xk + m));
            for (int j = 1; j < s; ++j) {
                const int w = m + j * mx;
                acc = c_add(acc, c_mul(A[w * ldA], __ldg(xk + w)));
            }
            return acc;
        }
    };
    // (a harmonic past the last folds with the last's spectrum and is not stored)
    __device__ __forceinline__ At at(int q) const
    {
        return At{A + (q & ((1 << lgP) - 1)), ldA, xk + min(q >> lgP, left - 1) * nx, mx, s};
    }
};

// One harmonic's portrait rows (row0 + 2p, row0 + 2p + 1) of a pencil.
// Windowed (padded plans): the portraits in memory are the field of view's,
// fmx samples a row; row r = z ny + y of the extended mesh is row
// (z - pz) fny + y - py, sample m is m - pm, and what lies outside the field
// of view is not stored and reads as zero.
struct PortraitRows {
    int row0, rows, mx;
    PortraitWin w;
    // the row's offset in memory, or -1
    __device__ __forceinline__ long long row(int r) const
    {
        if (r >= rows) return -1;
        if (!w.on) return (long long)r * mx;
        const int z = (int)w.dny.div((uint32_t)r), y = r - z * (int)w.dny.d;
        const int fz = z - w.pz, fy = y - w.py;
        if ((unsigned)fz >= (unsigned)w.fnz || (unsigned)fy >= (unsigned)w.fny) return -1;
        return ((long long)fz * w.fny + fy) * w.fmx;
    }
    __device__ __forceinline__ int m0() const { return w.on ? w.pm : 0; }
    __device__ __forceinline__ int len() const { return w.on ? w.fmx : mx; }
};

struct PortraitSt {
    float2* d;       // the harmonic's portraits
    float2 ph;       // e^{i theta_k}
    const PortraitRows& g;
    struct At {
        float2 *d0, *d1;   // the two rows, or null
        float2 ph;
        int m0, len;
        __device__ __forceinline__ void operator()(int m, float2 val) const
        {
            m -= m0;
            if ((unsigned)m >= (unsigned)len) return;
            if (d0) d0[m] = make_float2(ph.x * val.x, ph.y * val.x);
            if (d1) d1[m] = make_float2(ph.x * val.y, ph.y * val.y);
        }
    };
    __device__ __forceinline__ At at(int p) const
    {
        const long long i0 = g.row(g.row0 + 2 * p), i1 = g.row(g.row0 + 2 * p + 1);
        return At{i0 >= 0 ? d + i0 : nullptr, i1 >= 0 ? d + i1 : nullptr, ph, g.m0(), g.len()};
    }
};

// Adjoint: (Re(e^{-i theta} y[row]), Re(e^{-i theta} y[row+1])) at sample m.
struct PortraitKLd {
    const float2* __restrict__ d;
    float2 ph;
    const PortraitRows& g;
    struct At {
        const float2 *d0, *d1;
        float2 ph;
        int m0, len;
        __device__ __forceinline__ float2 operator()(int m) const
        {
            m -= m0;
            const bool in = (unsigned)m < (unsigned)len;
            const float2 z = make_float2(0.f, 0.f);
            const float2 y0 = in && d0 ? __ldg(d0 + m) : z, y1 = in && d1 ? __ldg(d1 + m) : z;
            return make_float2(fmaf(ph.x, y0.x, ph.y * y0.y), fmaf(ph.x, y1.x, ph.y * y1.y));
        }
    };
    __device__ __forceinline__ At at(int p) const
    {
        const long long i0 = g.row(g.row0 + 2 * p), i1 = g.row(g.row0 + 2 * p + 1);
        return At{i0 >= 0 ? d + i0 : nullptr, i1 >= 0 ? d + i1 : nullptr, ph, g.m0(), g.len()};
    }
};

// A round's portraits: pencil q = kk P + p of harmonic k0 + kk.
struct RoundSt {
    const XArgs& a;
    const PortraitRows& g;
    int k0;
    __device__ __forceinline__ PortraitSt::At at(int q) const
    {
        const int k = k0 + (q >> a.lgP);
        if (k >= a.K) return PortraitSt::At{nullptr, nullptr, make_float2(0.f, 0.f), 0, 0};
        return PortraitSt{a.dout + (long long)k * a.M, __ldg(a.phase + k), g}.at(q & ((1 << a.lgP) - 1));
    }
};
struct RoundKLd {
    const XArgs& a;
    const PortraitRows& g;
    int k0;
    __device__ __forceinline__ PortraitKLd::At at(int q) const
    {
        const int k = k0 + (q >> a.lgP);
        if (k >= a.K) return PortraitKLd::At{nullptr, nullptr, make_float2(0.f, 0.f), 0, 0};
        return PortraitKLd{a.din + (long long)k * a.M, __ldg(a.phase + k), g}.at(q & ((1 << a.lgP) - 1));
    }
};

// One harmonic's 2 P portrait rows, copied to shared memory [2 P][pitch] by
// 8-byte asynchronous copies, a warp per row.  What lies outside the field
// of view or past the last row is not written: the caller zeroes the buffer
// once.
__device__ __forceinline__ void stage_portraits(float2* raw, int pitch, const float2* __restrict__ d,
                                                const PortraitRows& g, int P)
{
    const int len = g.len();
    // short rows share a warp: 2^lgw lanes a row
    const int lgw = len >= 32 ? 5 : 32 - __clz(len - 1), lane = (int)threadIdx.x & ((1 << lgw) - 1);
    for (int rr = (int)threadIdx.x >> lgw; rr < 2 * P; rr += (int)blockDim.x >> lgw) {
        const long long o = g.row(g.row0 + rr);
        if (o < 0) continue;
        const float2* src = d + o;
        const uint32_t dst = (uint32_t)__cvta_generic_to_shared(raw + rr * pitch + g.m0());
        for (int m = lane; m < len; m += 1 << lgw)
            asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst + 8 * m), "l"(src + m) : "memory");
    }
}
// Those rows as the adjoint's pencils.
struct RawRowsLd {
    const float2* raw;
    float2 ph;
    int pitch;
    struct At {
        const float2* d;
        float2 ph;
        int pitch;
        __device__ __forceinline__ float2 operator()(int m) const
        {
            const float2 y0 = d[m], y1 = d[pitch + m];
            return make_float2(fmaf(ph.x, y0.x, ph.y * y0.y), fmaf(ph.x, y1.x, ph.y * y1.y));
        }
    };
    __device__ __forceinline__ At at(int p) const { return At{raw + 2 * p * pitch, ph, pitch}; }
};

// The same for the specialised adjoint (ops_ct.cuh), harmonic k0 + q / P.
struct PortraitLd {
    const float2* __restrict__ d;
    const float2* __restrict__ phase;
    long long M;
    int mx, row0, rows, P;
    __device__ __forceinline__ float2 operator()(int m, int q) const
    {
        const int kk = q / P, p = q - kk * P;
        const float2 ph = __ldg(phase + kk);
        const int r = row0 + 2 * p;
        const float2* dk = d + (long long)kk * M;
        float2 o = make_float2(0.f, 0.f);
        if (r < rows) {
            const float2 y = dk[(long long)r * mx + m];
            o.x = fmaf(ph.x, y.x, ph.y * y.y);
        }
        if (r + 1 < rows) {
            const float2 y = dk[(long long)(r + 1) * mx + m];
            o.y = fmaf(ph.x, y.x, ph.y * y.y);
        }
        return o;
    }
};

// Normal: out[m + a mx] = sum_b Q[m][a][b] A[m + b mx].
struct QLd {
    const float2* A;
    int ldA;
    const float2* __restrict__ Q;
    int mx, s;
    FastDiv dmx;
    struct At {
        const float2* A;
        int ldA;
        const float2* __restrict__ Q;
        int mx, s;
        FastDiv dmx;
        __device__ __forceinline__ float2 operator()(int w) const
        {
            const int a = (int)dmx.div((uint32_t)w), m = w - a * mx;
            const float2* qm = Q + (m * s + a) * s;
            float2 acc = make_float2(0.f, 0.f);
            for (int b = 0; b < s; ++b) acc = c_add(acc, c_mul(__ldg(qm + b), A[(m + b * mx) * ldA]));
            return acc;
        }
    };
    __device__ __forceinline__ At at(int p) const { return At{A + p, ldA, Q, mx, s, dmx}; }
};

// p^T q (and p^T p for acc2) of four voxels.
__device__ __forceinline__ void nrm_dots(const float4& p, const float4& q, DotAcc* acc, DotAcc* acc2)
{
    acc->add(p.x, q.x);
    acc->add(p.y, q.y);
    acc->add(p.z, q.z);
    acc->add(p.w, q.w);
    if (acc2) {
        acc2->add(p.x, p.x);
        acc2->add(p.y, p.y);
        acc2->add(p.z, p.z);
        acc2->add(p.w, p.w);
    }
}

// Normal epilogue q = b w + lambda R p over a tile of 2 P rows of w (pencil
// layout, row 2p the real and row 2p + 1 the imaginary part), accumulating
// p^T q (and p^T p for acc2), lanes along x.
__device__ __forceinline__ void nrm_epilogue_rt(const XArgs& a, int row0, int P, const float2* w, int ld, DotAcc* acc,
                                                DotAcc* acc2)
{
    const float* wf = reinterpret_cast<const float*>(w);
    const bool plain = a.reg.kind == 0;
    const int nx = a.nx, lane = (int)threadIdx.x & 31, nw = (int)blockDim.x >> 5;
    constexpr int U = 4;   // elements a step, their loads first
    // the stencil prior in groups of four voxels (reg_term4)
    const bool v4 = !plain && (nx & 3) == 0 && (((uintptr_t)a.pin | (uintptr_t)a.qout) & 15u) == 0;
    for (int rr = (int)threadIdx.x >> 5; rr < 2 * P && row0 + rr < a.rows; rr += nw) {   // a warp per row
        const int r = row0 + rr, i0 = r * nx;
        const int z = (int)a.dny.div((uint32_t)r), y = r - z * a.reg.ny;
        const float* wr = wf + 2 * (rr >> 1) + (rr & 1);
        if (v4) {
            for (int x = 4 * lane; x < nx; x += 128) {
                const float4 rt = reg_term4(a.reg, a.pin, i0 + x, x, y, z);
                const float4 pv = __ldg(reinterpret_cast<const float4*>(a.pin + i0 + x));
                float4 bv = make_float4(1.f, 1.f, 1.f, 1.f), q;
                if (a.b) bv = make_float4(a.b[i0 + x], a.b[i0 + x + 1], a.b[i0 + x + 2], a.b[i0 + x + 3]);
                q.x = fmaf(bv.x, wr[2 * x * ld], rt.x);
                q.y = fmaf(bv.y, wr[2 * (x + 1) * ld], rt.y);
                q.z = fmaf(bv.z, wr[2 * (x + 2) * ld], rt.z);
                q.w = fmaf(bv.w, wr[2 * (x + 3) * ld], rt.w);
                *reinterpret_cast<float4*>(a.qout + i0 + x) = q;
                nrm_dots(pv, q, acc, acc2);
            }
            continue;
        }
        for (int x0 = lane; x0 < nx; x0 += 32 * U) {
            float pv[U], bv[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int x = x0 + 32 * u;
                if (x >= nx) continue;
                pv[u] = a.pin[i0 + x];
                bv[u] = a.b ? a.b[i0 + x] : 1.f;
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int x = x0 + 32 * u;
                if (x >= nx) continue;
                const float v = wr[2 * x * ld];
                float q = a.b ? bv[u] * v : v;
                if (plain) q += a.reg.lambda * pv[u];
                else q += reg_term(a.reg, a.pin, i0 + x, x, y, z);
                a.qout[i0 + x] = q;
                acc->add(pv[u], q);
                if (acc2) acc2->add(pv[u], pv[u]);
            }
        }
    }
}

}  // namespace mh3d
