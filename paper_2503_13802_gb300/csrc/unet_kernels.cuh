// Kernels of the learned warm-start network: a small 3D U-Net with additive
// skips whose 3x3x3 convolutions run as implicit GEMMs on the tensor cores
// (bfloat16 operands, FP32 accumulation, mma.sync m16n8k16).
//
// Activations are channels-last bfloat16 volumes [D][H][W][C].  A
// convolution "same" (zero padding) with weights W[co][tap][ci] (tap =
// 9 (dz+1) + 3 (dy+1) + (dx+1)) is the GEMM
//     out[v][co] = sum_k A[v][k] Wt[k][co],   k = tap * Cin + ci,
// where A[v][k] = in[v + tap][ci] is gathered on the fly (never stored).
// The gather also forms the two special inputs of the decoder: a nearest x2
// upsampling of a half-resolution source, and the sum of two sources (the
// additive skip), rounded to bfloat16 as a stored sum would be.  The same
// kernel with negated taps and re-laid-out weights computes the gradient
// with respect to the input; the weight gradient is the GEMM
//     dW^T[k][co] = sum_v A[v][k] dY[v][co]
// split over voxel chunks into FP32 partials that a second kernel adds in a
// fixed order.
#pragma once

#include <cstdint>

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "fastdiv.h"
#include "halo_index.h"

namespace mh3d {
namespace unet {

constexpr int kBM = 128;   // GEMM rows per CTA (voxels, or weight rows in wgrad)
constexpr int kBK = 32;    // reduction depth per shared-memory stage
constexpr int kThreads = 256;
constexpr int kWChunk = 4096;   // voxels per CTA in the weight gradient

// Source of a convolution's input (the GEMM's gathered operand).
struct ConvSrc {
    const __nv_bfloat16* a = nullptr;   // [.][.][.][C] bfloat16
    const __nv_bfloat16* b = nullptr;   // second addend (skip), same shape as a, or null
    const float* f32 = nullptr;         // single-channel FP32 source instead of a (network input)
    const float* f32_scale = nullptr;   // device scalar multiplying the FP32 source (null: 1)
    int D = 0, H = 0, W = 0;            // resolution of the convolution (output)
    int C = 0;                          // source channels
    int up = 0;                         // 1: a is at half resolution (nearest x2 upsampling)
    int flip = 0;                       // 1: taps negated (gradient w.r.t. the input)
};

__device__ __forceinline__ float bf2f(__nv_bfloat16 v) { return __bfloat162float(v); }

// A[v][k] for one voxel (z, y, x) and k = tap * C + ci; 0 outside the volume.
__device__ __forceinline__ float gather1(const ConvSrc& s, int z, int y, int x, int k)
{
    const int tap = k / s.C, ci = k - tap * s.C;
    int dz = tap / 9 - 1, dy = (tap / 3) % 3 - 1, dx = tap % 3 - 1;
    if (s.flip) {
        dz = -dz;
        dy = -dy;
        dx = -dx;
    }
    const int zz = z + dz, yy = y + dy, xx = x + dx;
    if (zz < 0 || zz >= s.D || yy < 0 || yy >= s.H || xx < 0 || xx >= s.W) return 0.f;
    if (s.f32) return s.f32[((size_t)zz * s.H + yy) * s.W + xx] * (s.f32_scale ? *s.f32_scale : 1.f);
    size_t off;
    if (s.up)
        off = (((size_t)(zz >> 1) * (s.H >> 1) + (yy >> 1)) * (s.W >> 1) + (xx >> 1)) * s.C + ci;
    else
        off = (((size_t)zz * s.H + yy) * s.W + xx) * s.C + ci;
    float v = bf2f(s.a[off]);
    if (s.b) v = bf2f(__float2bfloat16(v + bf2f(s.b[off])));
    return v;
}

// Eight consecutive k (one tap, ci .. ci+7; needs C % 8 == 0) as 16 bytes.
__device__ __forceinline__ uint4 gather8(const ConvSrc& s, int z, int y, int x, int k)
{
    const int tap = k / s.C, ci = k - tap * s.C;
    int dz = tap / 9 - 1, dy = (tap / 3) % 3 - 1, dx = tap % 3 - 1;
    if (s.flip) {
        dz = -dz;
        dy = -dy;
        dx = -dx;
    }
    const int zz = z + dz, yy = y + dy, xx = x + dx;
    uint4 r = make_uint4(0, 0, 0, 0);
    if (zz < 0 || zz >= s.D || yy < 0 || yy >= s.H || xx < 0 || xx >= s.W) return r;
    size_t off;
    if (s.up)
        off = (((size_t)(zz >> 1) * (s.H >> 1) + (yy >> 1)) * (s.W >> 1) + (xx >> 1)) * s.C + ci;
    else
        off = (((size_t)zz * s.H + yy) * s.W + xx) * s.C + ci;
    r = *reinterpret_cast<const uint4*>(s.a + off);
    if (s.b) {
        const uint4 q = *reinterpret_cast<const uint4*>(s.b + off);
        __nv_bfloat162* pr = reinterpret_cast<__nv_bfloat162*>(&r);
        const __nv_bfloat162* pq = reinterpret_cast<const __nv_bfloat162*>(&q);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float2 u = __bfloat1622float2(pr[i]), w = __bfloat1622float2(pq[i]);
            pr[i] = __floats2bfloat162_rn(u.x + w.x, u.y + w.y);
        }
    }
    return r;
}

__device__ __forceinline__ uint32_t smem_addr(const void* p)
{
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void ldsm_x4(uint32_t r[4], const void* p)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(smem_addr(p)));
}

__device__ __forceinline__ void ldsm_x4_t(uint32_t r[4], const void* p)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(smem_addr(p)));
}

__device__ __forceinline__ void mma_bf16(float c[4], const uint32_t a[4], uint32_t b0, uint32_t b1)
{
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// One kBK-deep stage: warp w owns GEMM rows [16 w, 16 w + 16) and every
// column of the BN-wide tile.  sA is [kBM][kBK + 8] (row-major, m by k) or,
// with A_KMAJOR, [kBK][kBM + 8] (k by m); sB is [kBK][BN + 8] (k by n).
template <int BN, bool A_KMAJOR>
__device__ __forceinline__ void mma_stage(const __nv_bfloat16* sA, const __nv_bfloat16* sB, float (&acc)[BN / 8][4],
                                          int warp, int lane)
{
#pragma unroll
    for (int kk = 0; kk < kBK; kk += 16) {
        uint32_t a[4];
        if (A_KMAJOR) {
            const int row = kk + (lane & 7) + (lane >> 4) * 8;
            const int col = 16 * warp + ((lane >> 3) & 1) * 8;
            ldsm_x4_t(a, sA + row * (kBM + 8) + col);
        } else {
            const int row = 16 * warp + (lane & 15);
            const int col = kk + (lane >> 4) * 8;
            ldsm_x4(a, sA + row * (kBK + 8) + col);
        }
#pragma unroll
        for (int j = 0; j < BN / 16; ++j) {
            uint32_t b[4];
            const int row = kk + (lane & 7) + ((lane >> 3) & 1) * 8;
            const int col = j * 16 + (lane >> 4) * 8;
            ldsm_x4_t(b, sB + row * (BN + 8) + col);
            mma_bf16(acc[2 * j], a, b[0], b[1]);
            mma_bf16(acc[2 * j + 1], a, b[2], b[3]);
        }
    }
}

// Loads rows [k0, k0 + kBK) x columns [n0, n0 + BN) of a [Kpad][Npad] bfloat16
// weight matrix (Kpad a multiple of kBK, Npad a multiple of BN).
template <int BN>
__device__ __forceinline__ void load_weights(__nv_bfloat16* sB, const __nv_bfloat16* Wt, int Npad, int k0, int n0)
{
    constexpr int CH = BN / 8;
    for (int i = threadIdx.x; i < kBK * CH; i += kThreads) {
        const int r = i / CH, c = i % CH;
        *reinterpret_cast<uint4*>(sB + r * (BN + 8) + c * 8) =
            *reinterpret_cast<const uint4*>(Wt + (size_t)(k0 + r) * Npad + n0 + c * 8);
    }
}

// Convolution as GEMM: out[v][n] (n < N) = sum_k A[v][k] Wt[k][n] (+ bias,
// times the device scalar *oscale when given, ReLU).  Kvalid = 27 C; Wt is
// [Kpad][Npad] with zero rows k >= Kvalid.  OutT = __nv_bfloat16 (stored
// activations) or float.  Split K (part != null): blockIdx.z takes
// k in [z kl, (z + 1) kl) and writes its FP32 sums to part[z][v][n], which
// k_splitk_finish adds in split order before the epilogue.
template <int BN, class OutT>
__global__ void __launch_bounds__(kThreads) k_conv(ConvSrc src, const __nv_bfloat16* __restrict__ Wt, int Kpad,
                                                   int Npad, int N, const float* __restrict__ bias, int relu,
                                                   const float* __restrict__ oscale, OutT* __restrict__ out,
                                                   int kl, float* __restrict__ part)
{
    __shared__ __align__(16) __nv_bfloat16 sA[kBM * (kBK + 8)];
    __shared__ __align__(16) __nv_bfloat16 sB[kBK * (BN + 8)];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const long long V = (long long)src.D * src.H * src.W;
    const long long m0 = (long long)blockIdx.x * kBM;
    const int n0 = blockIdx.y * BN;
    const int Kvalid = 27 * src.C;
    const bool vec = (src.C % 8) == 0 && !src.f32;
    float acc[BN / 8][4];
#pragma unroll
    for (int t = 0; t < BN / 8; ++t) acc[t][0] = acc[t][1] = acc[t][2] = acc[t][3] = 0.f;
    const int kbeg = blockIdx.z * kl, kend = kbeg + kl < Kpad ? kbeg + kl : Kpad;
    for (int k0 = kbeg; k0 < kend; k0 += kBK) {
        if (vec) {
            for (int i = threadIdx.x; i < kBM * (kBK / 8); i += kThreads) {
                const int r = i / (kBK / 8), c = i % (kBK / 8);
                const long long v = m0 + r;
                const int k = k0 + c * 8;
                uint4 val = make_uint4(0, 0, 0, 0);
                if (v < V && k < Kvalid) {
                    const int x = (int)(v % src.W), y = (int)((v / src.W) % src.H), z = (int)(v / ((long long)src.W * src.H));
                    val = gather8(src, z, y, x, k);
                }
                *reinterpret_cast<uint4*>(sA + r * (kBK + 8) + c * 8) = val;
            }
        } else {
            for (int i = threadIdx.x; i < kBM * kBK; i += kThreads) {
                const int r = i / kBK, c = i % kBK;
                const long long v = m0 + r;
                const int k = k0 + c;
                float val = 0.f;
                if (v < V && k < Kvalid) {
                    const int x = (int)(v % src.W), y = (int)((v / src.W) % src.H), z = (int)(v / ((long long)src.W * src.H));
                    val = gather1(src, z, y, x, k);
                }
                sA[r * (kBK + 8) + c] = __float2bfloat16(val);
            }
        }
        load_weights<BN>(sB, Wt, Npad, k0, n0);
        __syncthreads();
        mma_stage<BN, false>(sA, sB, acc, warp, lane);
        __syncthreads();
    }
    // epilogue: fragment (row lane/4 [+8], columns 2 (lane%4) + {0, 1})
    if (part) {
        float* P = part + (size_t)blockIdx.z * V * N;
#pragma unroll
        for (int t = 0; t < BN / 8; ++t)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const long long v = m0 + 16 * warp + (lane >> 2) + 8 * h;
                if (v >= V) continue;
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const int n = n0 + t * 8 + 2 * (lane & 3) + e;
                    if (n < N) P[v * N + n] = acc[t][2 * h + e];
                }
            }
        return;
    }
    const float osc = oscale ? *oscale : 1.f;
#pragma unroll
    for (int t = 0; t < BN / 8; ++t) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const long long v = m0 + 16 * warp + (lane >> 2) + 8 * h;
            if (v >= V) continue;
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int n = n0 + t * 8 + 2 * (lane & 3) + e;
                if (n >= N) continue;
                float val = (acc[t][2 * h + e] + (bias ? bias[n] : 0.f)) * osc;
                if (relu) val = fmaxf(val, 0.f);
                if constexpr (sizeof(OutT) == 2)
                    out[v * N + n] = __float2bfloat16(val);
                else
                    out[v * N + n] = val;
            }
        }
    }
}

// ---------------------------------------------------------------------------
// One-channel source (the network input, or a one-channel gradient), on
// 8 x 4 x 4 output blocks: the block's input halo (10 x 6 x 6 voxels) and
// the weight matrix are staged in shared memory, and the 128 x 32 operand
// (27 taps, 5 zeros) is built from the halo explicitly.
constexpr int kTX = 8, kTY = 4, kTZ = 4;
constexpr int kHX = kTX + 2, kHY = kTY + 2, kHZ = kTZ + 2, kHV = kHX * kHY * kHZ;

// Shared-memory bytes of k_conv_tile<BN> for a weight matrix of Kpad rows
// (weights, two halo buffers and the operand tile).
template <int BN>
constexpr size_t tile_smem(int Kpad)
{
    return sizeof(__nv_bfloat16) * ((size_t)Kpad * (BN + 8) + 2 * (((kHV + 7) / 8) * 8) + kBM * (kBK + 8));
}

// Halo values a thread carries between tiles.
struct HaloRegs {
    static constexpr int kPer = (kHV + kThreads - 1) / kThreads;
    float v[kPer];
};

__device__ __forceinline__ void tile_origin(const ConvSrc& s, int t, int& x0, int& y0, int& z0)
{
    const int tilesX = (s.W + kTX - 1) / kTX, tilesY = (s.H + kTY - 1) / kTY;
    x0 = (t % tilesX) * kTX;
    t /= tilesX;
    y0 = (t % tilesY) * kTY;
    z0 = (t / tilesY) * kTZ;
}

// Global -> registers: the halo of the tile at (x0, y0, z0), zero outside,
// the skip addend summed and rounded as a stored sum would be.
__device__ __forceinline__ void halo_fetch(const ConvSrc& src, int x0, int y0, int z0, HaloRegs& h)
{
    const int Hs = src.up ? (src.H >> 1) : src.H, Ws = src.up ? (src.W >> 1) : src.W;
#pragma unroll
    for (int j = 0; j < HaloRegs::kPer; ++j) {
        const int hv = threadIdx.x + j * kThreads;
        float v = 0.f;
        if (hv < kHV) {
            const int hx = hv % kHX, hy = (hv / kHX) % kHY, hz = hv / (kHX * kHY);
            const int z = z0 - 1 + hz, y = y0 - 1 + hy, x = x0 - 1 + hx;
            if (z >= 0 && z < src.D && y >= 0 && y < src.H && x >= 0 && x < src.W) {
                if (src.f32) {
                    v = src.f32[((size_t)z * src.H + y) * src.W + x] * (src.f32_scale ? *src.f32_scale : 1.f);
                } else {
                    const size_t vox = src.up ? ((size_t)(z >> 1) * Hs + (y >> 1)) * Ws + (x >> 1)
                                              : ((size_t)z * src.H + y) * src.W + x;
                    v = bf2f(src.a[vox]);
                    if (src.b) v = bf2f(__float2bfloat16(v + bf2f(src.b[vox])));
                }
            }
        }
        h.v[j] = v;
    }
}

// Registers -> one halo buffer.
__device__ __forceinline__ void halo_store(__nv_bfloat16* sH, const HaloRegs& h)
{
#pragma unroll
    for (int j = 0; j < HaloRegs::kPer; ++j) {
        const int i = threadIdx.x + j * kThreads;
        if (i < kHV) sH[i] = __float2bfloat16(h.v[j]);
    }
}

// Persistent: each CTA stages the weight matrix once and walks output
// blocks blockIdx.x, blockIdx.x + gridDim.x, ...; while it multiplies one
// block, the next block's halo is in flight to registers, and lands in the
// other halo buffer afterwards.
template <int BN, class OutT>
__global__ void __launch_bounds__(kThreads, 2) k_conv_tile(ConvSrc src, const __nv_bfloat16* __restrict__ Wt, int Kpad,
                                                        int Npad, int N, const float* __restrict__ bias, int relu,
                                                        const float* __restrict__ oscale, OutT* __restrict__ out,
                                                        int ntiles)
{
    extern __shared__ __align__(16) unsigned char tile_raw[];
    constexpr int HB = ((kHV + 7) / 8) * 8;
    __nv_bfloat16* sW = reinterpret_cast<__nv_bfloat16*>(tile_raw);   // [Kpad][BN + 8]
    __nv_bfloat16* sH0 = sW + (size_t)Kpad * (BN + 8);                 // two [kHV] buffers
    __nv_bfloat16* sA = sH0 + 2 * HB;                                  // [kBM][kBK + 8]
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int n0 = blockIdx.y * BN;
    const int sgn = src.flip ? -1 : 1;
    const float osc = oscale ? *oscale : 1.f;

    for (int i = threadIdx.x; i < Kpad * (BN / 8); i += kThreads) {
        const int r = i / (BN / 8), c = i % (BN / 8);
        *reinterpret_cast<uint4*>(sW + r * (BN + 8) + c * 8) =
            *reinterpret_cast<const uint4*>(Wt + (size_t)r * Npad + n0 + c * 8);
    }
    int tile = blockIdx.x;
    if (tile >= ntiles) return;
    HaloRegs h;
    int x0, y0, z0;
    tile_origin(src, tile, x0, y0, z0);
    halo_fetch(src, x0, y0, z0, h);
    halo_store(sH0, h);
    __syncthreads();
    int cur = 0;
    for (;;) {
        const int next = tile + gridDim.x;
        int nx0 = 0, ny0 = 0, nz0 = 0;
        if (next < ntiles) {
            tile_origin(src, next, nx0, ny0, nz0);
            halo_fetch(src, nx0, ny0, nz0, h);
        }
        const __nv_bfloat16* sH = sH0 + cur * HB;
        float acc[BN / 8][4];
#pragma unroll
        for (int q = 0; q < BN / 8; ++q) acc[q][0] = acc[q][1] = acc[q][2] = acc[q][3] = 0.f;
        for (int i = threadIdx.x; i < kBM * kBK; i += kThreads) {
            const int mm = i / kBK, k = i % kBK;
            __nv_bfloat16 v = __float2bfloat16(0.f);
            if (k < 27) {
                const int tx = mm % kTX, ty = (mm / kTX) % kTY, tz = mm / (kTX * kTY);
                const int dz = sgn * (k / 9 - 1), dy = sgn * ((k / 3) % 3 - 1), dx = sgn * (k % 3 - 1);
                v = sH[((tz + 1 + dz) * kHY + (ty + 1 + dy)) * kHX + (tx + 1 + dx)];
            }
            sA[mm * (kBK + 8) + k] = v;
        }
        __syncthreads();
        mma_stage<BN, false>(sA, sW, acc, warp, lane);
#pragma unroll
        for (int q = 0; q < BN / 8; ++q) {
#pragma unroll
            for (int hh = 0; hh < 2; ++hh) {
                const int mm = 16 * warp + (lane >> 2) + 8 * hh;
                const int x = x0 + mm % kTX, y = y0 + (mm / kTX) % kTY, z = z0 + mm / (kTX * kTY);
                if (x >= src.W || y >= src.H || z >= src.D) continue;
                const long long v = ((long long)z * src.H + y) * src.W + x;
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const int n = n0 + q * 8 + 2 * (lane & 3) + e;
                    if (n >= N) continue;
                    float val = (acc[q][2 * hh + e] + (bias ? bias[n] : 0.f)) * osc;
                    if (relu) val = fmaxf(val, 0.f);
                    if constexpr (sizeof(OutT) == 2)
                        out[v * N + n] = __float2bfloat16(val);
                    else
                        out[v * N + n] = val;
                }
            }
        }
        if (next >= ntiles) break;
        // the other buffer was last read two tiles ago, before the previous barrier
        halo_store(sH0 + (cur ^ 1) * HB, h);
        __syncthreads();
        cur ^= 1;
        tile = next;
        x0 = nx0;
        y0 = ny0;
        z0 = nz0;
    }
}

__device__ __forceinline__ void lin_cp16(void* sdst, const void* gsrc, bool in)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_addr(sdst)), "l"(gsrc), "r"(in ? 16u : 0u)
                 : "memory");
}

// ---------------------------------------------------------------------------
// Tiled convolutions for sources of 8 n channels on mma.sync: one CTA per
// 8 x TY x 4 output block, eight warps of 32 voxels (two 16-row fragments,
// so that a weight fragment read from shared memory serves two products).
// The products of an output and their order are those of the kernels above
// (k16 steps in ascending tap and channel; with `split` > 0 a new sum every
// `split` steps, the sums added in order, as the split-K gather form does),
// so the three give the same bits.  What bounds them: the shared-memory
// reads of the fragments; tap offsets come from a table, and a halo unit's
// place and address are formed once per CTA, not per block.  Measured in the
// forward at 128x128x64, channels (16, 32, 64, 128), us a layer, against
// tiles of 128 voxels with one fragment a warp and the split-K gather form:
// 32 -> 32 at half resolution 70 -> 33, upsampled 64 -> 32 228 -> 53, 64 -> 64
// at a quarter 50 -> 20, 128 -> 128 at an eighth 50 -> 33.
//
// k_conv_halo keeps the whole weight matrix in shared memory (C <= 64) and
// walks blocks; k_conv_stream (C = 64 and 128 on coarse levels, a few blocks
// per SM) streams it tap by tap.
template <int TY>
struct HaloGeom {
    static constexpr int HX = kTX + 2, HY = TY + 2, HZ = kTZ + 2, HV = HX * HY * HZ, M = kTX * TY * kTZ;
};

// Shared-memory bytes of the two.
template <int C, int BN>
constexpr size_t conv_halo_smem(int Kpad)
{
    return sizeof(__nv_bfloat16) * ((size_t)Kpad * (BN + 8) + (size_t)HaloGeom<8>::HV * (C + 8) + 8) + sizeof(int) * 28;
}
constexpr int kStreamBN = 32;
template <int C>
constexpr size_t conv_stream_smem()
{
    return sizeof(__nv_bfloat16) * ((size_t)HaloGeom<4>::HV * (C + 8) + 3 * (size_t)C * (kStreamBN + 8)) + sizeof(int) * 28;
}

// A thread's halo units: unit i of the block is 8 channels of a halo voxel.
// rel: voxels from the block's first voxel (halo_index.h); pos: hx | hy << 8 |
// hz << 16; c8: the unit's first channel (kThreads is a multiple of C / 8, so
// a thread's units share it).
template <int C, int TY, int PER>
struct HaloUnits {
    using G = HaloGeom<TY>;
    static constexpr int kItems = G::HV * (C / 8);
    static_assert(kThreads % (C / 8) == 0, "a thread's units take the same channels");
    int rel[PER], pos[PER], c8;
    // the units first + j kThreads (j < PER)
    __device__ __forceinline__ void init(const ConvSrc& s, int first)
    {
        const int sh = s.up ? 1 : 0;
        c8 = first % (C / 8) * 8;
#pragma unroll
        for (int j = 0; j < PER; ++j) {
            const int i = first + j * kThreads, hv = i / (C / 8);
            const int hx = hv % G::HX, hy = (hv / G::HX) % G::HY, hz = hv / (G::HX * G::HY);
            pos[j] = i < kItems ? hx | hy << 8 | hz << 16 : -1;
            rel[j] = halo_rel(hx, hy, hz, sh, s.H >> sh, s.W >> sh);
        }
    }
};
__device__ __forceinline__ uint4 add_bf16x8(uint4 r, const uint4& q)   // the skip sum, rounded as a stored sum would be
{
    __nv_bfloat162* pr = reinterpret_cast<__nv_bfloat162*>(&r);
    const __nv_bfloat162* pq = reinterpret_cast<const __nv_bfloat162*>(&q);
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const float2 u = __bfloat1622float2(pr[e]), w = __bfloat1622float2(pq[e]);
        pr[e] = __floats2bfloat162_rn(u.x + w.x, u.y + w.y);
    }
    return r;
}
template <int C, int TY, int PER>
__device__ __forceinline__ void halo_load(const ConvSrc& s, const HaloUnits<C, TY, PER>& u, int x0, int y0, int z0,
                                          uint4 (&v)[PER])
{
    const int sh = s.up ? 1 : 0;
    const long long base = halo_base(x0, y0, z0, sh, s.H >> sh, s.W >> sh);
    const __nv_bfloat16 *a = s.a + halo_elem(base, 0, C, u.c8), *b = s.b ? s.b + halo_elem(base, 0, C, u.c8) : nullptr;
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        v[j] = make_uint4(0, 0, 0, 0);
        if (u.pos[j] < 0) continue;
        const int x = x0 - 1 + (u.pos[j] & 255), y = y0 - 1 + ((u.pos[j] >> 8) & 255), z = z0 - 1 + (u.pos[j] >> 16);
        if ((unsigned)x >= (unsigned)s.W || (unsigned)y >= (unsigned)s.H || (unsigned)z >= (unsigned)s.D) continue;
        const long long o = halo_elem(0, u.rel[j], C, 0);
        v[j] = *reinterpret_cast<const uint4*>(a + o);
        if (b) v[j] = add_bf16x8(v[j], *reinterpret_cast<const uint4*>(b + o));
    }
}
template <int C, int PER>
__device__ __forceinline__ void halo_put(__nv_bfloat16* sH, int first, int items, const uint4 (&v)[PER])
{
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        const int i = first + j * kThreads;
        if (i < items) *reinterpret_cast<uint4*>(sH + (i / (C / 8)) * (C + 8) + (i % (C / 8)) * 8) = v[j];
    }
}
// Tap t's halo offset in elements (t < 27).
template <int C, int TY>
__device__ __forceinline__ int tap_halo(int t, int sgn)
{
    using G = HaloGeom<TY>;
    const int dz = sgn * (t / 9 - 1), dy = sgn * ((t / 3) % 3 - 1), dx = sgn * (t % 3 - 1);
    return ((dz * G::HY + dy) * G::HX + dx) * (C + 8);
}

__device__ __forceinline__ void ldsm_a(uint32_t (&r)[4], uint32_t addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr));
}
__device__ __forceinline__ void ldsm_bt(uint32_t (&r)[4], uint32_t addr)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr));
}

// Epilogue of a 16-row fragment set: rows 16 mt + lane / 4 (+ 8) of the
// block, columns n0 + 8 q + 2 (lane % 4) + {0, 1}.
template <int TY, int NT, class OutT>
__device__ __forceinline__ void conv_store(const ConvSrc& s, const float (&acc)[NT][4], int mt, int lane, int x0, int y0,
                                           int z0, int n0, int N, const float* __restrict__ bias, int relu, float osc,
                                           OutT* __restrict__ out)
{
#pragma unroll
    for (int hh = 0; hh < 2; ++hh) {
        const int mm = 16 * mt + (lane >> 2) + 8 * hh;
        const int x = x0 + mm % kTX, y = y0 + (mm / kTX) % TY, z = z0 + mm / (kTX * TY);
        if (x >= s.W || y >= s.H || z >= s.D) continue;
        OutT* o = out + (((long long)z * s.H + y) * s.W + x) * N;
#pragma unroll
        for (int q = 0; q < NT; ++q) {
            const int n = n0 + q * 8 + 2 * (lane & 3);
            float v[2];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                v[e] = (acc[q][2 * hh + e] + (bias && n + e < N ? bias[n + e] : 0.f)) * osc;
                if (relu) v[e] = fmaxf(v[e], 0.f);
            }
            if constexpr (sizeof(OutT) == 2) {
                if ((N & 1) == 0) {
                    if (n < N) *reinterpret_cast<__nv_bfloat162*>(o + n) = __floats2bfloat162_rn(v[0], v[1]);
                    continue;
                }
            }
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                if (n + e >= N) continue;
                if constexpr (sizeof(OutT) == 2) o[n + e] = __float2bfloat16(v[e]);
                else o[n + e] = v[e];
            }
        }
    }
}

template <int TY>
__device__ __forceinline__ void block_origin(const ConvSrc& s, int t, int& x0, int& y0, int& z0)
{
    const int tx = (s.W + kTX - 1) / kTX, ty = (s.H + TY - 1) / TY;
    x0 = (t % tx) * kTX;
    t /= tx;
    y0 = (t % ty) * TY;
    z0 = (t / ty) * kTZ;
}

template <int C, int BN, class OutT>
__global__ void __launch_bounds__(kThreads, C <= 16 && BN <= 32 ? 2 : 1)
    k_conv_halo(ConvSrc src, const __nv_bfloat16* __restrict__ Wt, int Kpad, int Npad, int N,
                const float* __restrict__ bias, int relu, const float* __restrict__ oscale, OutT* __restrict__ out,
                int ntiles)
{
    extern __shared__ __align__(16) unsigned char ch_raw[];
    constexpr int TY = 8, CS = C + 8, NT = BN / 8, WS = BN + 8;
    using G = HaloGeom<TY>;
    constexpr int ITEMS = G::HV * (C / 8), PER = (ITEMS + kThreads - 1) / kThreads;
    constexpr bool PRE = C <= 32;   // the next block's halo in registers during this block's products
    static_assert(G::M == 32 * (kThreads / 32), "a warp per 32 voxels");
    __nv_bfloat16* sW = reinterpret_cast<__nv_bfloat16*>(ch_raw);   // [Kpad][BN + 8]
    __nv_bfloat16* sH = sW + (size_t)Kpad * WS;                      // [HV][C + 8]
    __nv_bfloat16* sZ = sH + (size_t)G::HV * CS;                     // 8 zeros
    int* toff = reinterpret_cast<int*>(sZ + 8);                      // tap offsets, bytes
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int n0 = blockIdx.y * BN;
    const float osc = oscale ? *oscale : 1.f;
    for (int i = threadIdx.x; i < Kpad * (BN / 8); i += kThreads) {
        const int r = i / (BN / 8), c = i % (BN / 8);
        *reinterpret_cast<uint4*>(sW + r * WS + c * 8) =
            *reinterpret_cast<const uint4*>(Wt + (size_t)r * Npad + n0 + c * 8);
    }
    if (threadIdx.x < 8) sZ[threadIdx.x] = __float2bfloat16(0.f);
    if (threadIdx.x < 27) toff[threadIdx.x] = 2 * tap_halo<C, TY>(threadIdx.x, src.flip ? -1 : 1);
    if (threadIdx.x == 27) toff[27] = 0;
    int tile = blockIdx.x;
    if (tile >= ntiles) return;
    HaloUnits<C, TY, PER> hu;
    hu.init(src, threadIdx.x);
    uint4 hv[PER];
    int x0, y0, z0;
    block_origin<TY>(src, tile, x0, y0, z0);
    halo_load(src, hu, x0, y0, z0, hv);
    // this lane's rows of the warp's two fragments
    uint32_t abase[2];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const int m = 32 * warp + 16 * i + (lane & 15);
        abase[i] = smem_addr(sH + ((m / (kTX * TY) + 1) * (G::HY * G::HX) + ((m / kTX) % TY + 1) * G::HX + m % kTX + 1) * CS);
    }
    const uint32_t bbase = smem_addr(sW + ((lane & 7) + ((lane >> 3) & 1) * 8) * WS + (lane >> 4) * 8);
    const uint32_t zrow = smem_addr(sZ);
    const int kh = lane >> 4;
    for (;;) {
        halo_put<C>(sH, threadIdx.x, ITEMS, hv);
        __syncthreads();
        const int next = tile + gridDim.x;
        int nx0 = 0, ny0 = 0, nz0 = 0;
        if (next < ntiles) block_origin<TY>(src, next, nx0, ny0, nz0);
        if (PRE && next < ntiles) halo_load(src, hu, nx0, ny0, nz0, hv);
        __syncwarp();   // (lanes load different units; ldmatrix and mma.sync are warp-wide)
        float acc[2][NT][4];
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int q = 0; q < NT; ++q) acc[i][q][0] = acc[i][q][1] = acc[i][q][2] = acc[i][q][3] = 0.f;
        auto step = [&](uint32_t a0, uint32_t a1, uint32_t b) {
            uint32_t fa[2][4];
            ldsm_a(fa[0], a0);
            ldsm_a(fa[1], a1);
#pragma unroll
            for (int j = 0; j < BN / 16; ++j) {
                uint32_t fb[4];
                ldsm_bt(fb, b + j * 32);
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    mma_bf16(acc[i][2 * j], fa[i], fb[0], fb[1]);
                    mma_bf16(acc[i][2 * j + 1], fa[i], fb[2], fb[3]);
                }
            }
        };
        if constexpr (C == 8) {
            // a step holds two taps, one per lane half; the 28th is zero
#pragma unroll 2
            for (int ks = 0; ks < 14; ++ks) {
                const int t = 2 * ks + kh, o = toff[t];
                step(t < 27 ? abase[0] + o : zrow, t < 27 ? abase[1] + o : zrow, bbase + ks * 16 * WS * 2);
            }
        } else {
            uint32_t b = bbase;
#pragma unroll 3
            for (int t = 0; t < 27; ++t) {
                const int o = toff[t] + 16 * kh;
#pragma unroll
                for (int c = 0; c < C / 16; ++c, b += 16 * WS * 2) step(abase[0] + o + 32 * c, abase[1] + o + 32 * c, b);
            }
        }
#pragma unroll
        for (int i = 0; i < 2; ++i)
            conv_store<TY>(src, acc[i], 2 * warp + i, lane, x0, y0, z0, n0, N, bias, relu, osc, out);
        if (next >= ntiles) break;
        __syncthreads();   // the halo has been read
        if (!PRE) halo_load(src, hu, nx0, ny0, nz0, hv);
        tile = next;
        x0 = nx0;
        y0 = ny0;
        z0 = nz0;
    }
}

// One 8 x 4 x 4 block and 32 outputs per CTA; warp (w & 3) takes voxels
// 32 (w & 3) .. + 31, w / 4 16 of the outputs.  Three weight buffers: tap
// t + 2 is copied while tap t multiplies, one barrier a tap.
template <int C, class OutT>
__global__ void __launch_bounds__(kThreads) k_conv_stream(ConvSrc src, const __nv_bfloat16* __restrict__ Wt, int Npad,
                                                          int N, const float* __restrict__ bias, int relu,
                                                          const float* __restrict__ oscale, OutT* __restrict__ out,
                                                          int split)
{
    extern __shared__ __align__(16) unsigned char cs_raw[];
    constexpr int TY = 4, CS = C + 8, BN = kStreamBN, WS = BN + 8, NT = 2;
    using G = HaloGeom<TY>;
    constexpr int ITEMS = G::HV * (C / 8), PER = 6;
    __nv_bfloat16* sH = reinterpret_cast<__nv_bfloat16*>(cs_raw);
    __nv_bfloat16* sW = sH + (size_t)G::HV * CS;   // three [C][BN + 8]
    int* toff = reinterpret_cast<int*>(sW + 3 * C * WS);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, wm = warp & 3, wn = warp >> 2;
    const int n0 = blockIdx.y * BN;
    const float osc = oscale ? *oscale : 1.f;
    auto stage_w = [&](int t) {
        if (t < 27) {
            __nv_bfloat16* d = sW + (t % 3) * C * WS;
#pragma unroll
            for (int i = threadIdx.x; i < C * (BN / 8); i += kThreads) {
                const int r = i / (BN / 8), c = i % (BN / 8);
                lin_cp16(d + r * WS + c * 8, Wt + (size_t)(t * C + r) * Npad + n0 + c * 8, true);
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    stage_w(0);
    stage_w(1);
    int x0, y0, z0;
    block_origin<TY>(src, blockIdx.x, x0, y0, z0);
    for (int first = threadIdx.x; first < ITEMS; first += PER * kThreads) {
        HaloUnits<C, TY, PER> hu;
        hu.init(src, first);
        uint4 hv[PER];
        halo_load(src, hu, x0, y0, z0, hv);
        halo_put<C>(sH, first, ITEMS, hv);
    }
    if (threadIdx.x < 27) toff[threadIdx.x] = 2 * tap_halo<C, TY>(threadIdx.x, src.flip ? -1 : 1);
    uint32_t abase[2];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const int m = 32 * wm + 16 * i + (lane & 15);
        abase[i] = smem_addr(sH + ((m / (kTX * TY) + 1) * (G::HY * G::HX) + ((m / kTX) % TY + 1) * G::HX + m % kTX + 1) * CS +
                             (lane >> 4) * 8);
    }
    const uint32_t bbase = smem_addr(sW + ((lane & 7) + ((lane >> 3) & 1) * 8) * WS + (lane >> 4) * 8 + wn * 16);
    float acc[2][NT][4], tot[2][NT][4];
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int q = 0; q < NT; ++q)
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[i][q][e] = tot[i][q][e] = 0.f;
    auto fold = [&]() {   // the split's sum joins the total, a new one starts
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int q = 0; q < NT; ++q)
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    tot[i][q][e] += acc[i][q][e];
                    acc[i][q][e] = 0.f;
                }
    };
    int left = split;
    for (int t = 0; t < 27; ++t) {
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        __syncthreads();   // tap t's weights have landed; tap t - 1's have been read
        stage_w(t + 2);
        const int o = toff[t];
        const uint32_t b = bbase + (t % 3) * C * WS * 2;
#pragma unroll
        for (int c = 0; c < C / 16; ++c) {
            uint32_t fa[2][4], fb[4];
            ldsm_a(fa[0], abase[0] + o + 32 * c);
            ldsm_a(fa[1], abase[1] + o + 32 * c);
            ldsm_bt(fb, b + c * 16 * WS * 2);
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                mma_bf16(acc[i][0], fa[i], fb[0], fb[1]);
                mma_bf16(acc[i][1], fa[i], fb[2], fb[3]);
            }
            if (--left == 0) {
                fold();
                left = split;
            }
        }
    }
    if (split > 0) {
        if (left != split) fold();
#pragma unroll
        for (int i = 0; i < 2; ++i)
            conv_store<TY>(src, tot[i], 2 * wm + i, lane, x0, y0, z0, n0 + 16 * wn, N, bias, relu, osc, out);
    } else {
#pragma unroll
        for (int i = 0; i < 2; ++i)
            conv_store<TY>(src, acc[i], 2 * wm + i, lane, x0, y0, z0, n0 + 16 * wn, N, bias, relu, osc, out);
    }
}

// out[v][n] = epilogue(sum over the S splits, in order, of part[z][v][n]).
template <class OutT>
__global__ void k_splitk_finish(const float* __restrict__ part, int S, long long VN, int N,
                                const float* __restrict__ bias, int relu, const float* __restrict__ oscale,
                                OutT* __restrict__ out)
{
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= VN) return;
    float a = 0.f;
    for (int z = 0; z < S; ++z) a += part[(size_t)z * VN + i];
    const int n = (int)(i % N);
    float val = (a + (bias ? bias[n] : 0.f)) * (oscale ? *oscale : 1.f);
    if (relu) val = fmaxf(val, 0.f);
    if constexpr (sizeof(OutT) == 2)
        out[i] = __float2bfloat16(val);
    else
        out[i] = val;
}

// Weight gradient, split over voxel chunks: part[chunk][k][n] =
// sum over the chunk's voxels of A[v][k] dY[v][n] (k < Kpad, n < N, dY is
// [V][N] bfloat16).  Grid (Kpad / kBM rounded up, chunks, N / BN rounded
// up): blockIdx.z takes outputs n0 = BN blockIdx.z .. n0 + BN - 1.
template <int BN>
__global__ void __launch_bounds__(kThreads) k_conv_wgrad(ConvSrc src, const __nv_bfloat16* __restrict__ dY, int N,
                                                         int Kpad, float* __restrict__ part)
{
    __shared__ __align__(16) __nv_bfloat16 sA[kBK * (kBM + 8)];   // [v][k]
    __shared__ __align__(16) __nv_bfloat16 sB[kBK * (BN + 8)];    // [v][n]
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const long long V = (long long)src.D * src.H * src.W;
    const int k0 = blockIdx.x * kBM, n0 = blockIdx.z * BN;
    const long long v0 = (long long)blockIdx.y * kWChunk;
    const long long v1 = v0 + kWChunk < V ? v0 + kWChunk : V;
    const int Kvalid = 27 * src.C;
    const bool vec = (src.C % 8) == 0 && !src.f32;
    const bool vecy = (N % 8) == 0;
    float acc[BN / 8][4];
#pragma unroll
    for (int t = 0; t < BN / 8; ++t) acc[t][0] = acc[t][1] = acc[t][2] = acc[t][3] = 0.f;
    for (long long vb = v0; vb < v1; vb += kBK) {
        if (vec) {
            for (int i = threadIdx.x; i < kBK * (kBM / 8); i += kThreads) {
                const int r = i / (kBM / 8), c = i % (kBM / 8);
                const long long v = vb + r;
                const int k = k0 + c * 8;
                uint4 val = make_uint4(0, 0, 0, 0);
                if (v < v1 && k < Kvalid) {
                    const int x = (int)(v % src.W), y = (int)((v / src.W) % src.H), z = (int)(v / ((long long)src.W * src.H));
                    val = gather8(src, z, y, x, k);
                }
                *reinterpret_cast<uint4*>(sA + r * (kBM + 8) + c * 8) = val;
            }
        } else {
            for (int i = threadIdx.x; i < kBK * kBM; i += kThreads) {
                const int r = i / kBM, c = i % kBM;
                const long long v = vb + r;
                const int k = k0 + c;
                float val = 0.f;
                if (v < v1 && k < Kvalid) {
                    const int x = (int)(v % src.W), y = (int)((v / src.W) % src.H), z = (int)(v / ((long long)src.W * src.H));
                    val = gather1(src, z, y, x, k);
                }
                sA[r * (kBM + 8) + c] = __float2bfloat16(val);
            }
        }
        if (vecy) {
            for (int i = threadIdx.x; i < kBK * (BN / 8); i += kThreads) {
                const int r = i / (BN / 8), c = i % (BN / 8);
                const long long v = vb + r;
                uint4 val = make_uint4(0, 0, 0, 0);
                if (v < v1 && n0 + c * 8 < N) val = *reinterpret_cast<const uint4*>(dY + v * N + n0 + c * 8);
                *reinterpret_cast<uint4*>(sB + r * (BN + 8) + c * 8) = val;
            }
        } else {
            for (int i = threadIdx.x; i < kBK * BN; i += kThreads) {
                const int r = i / BN, c = i % BN;
                const long long v = vb + r;
                sB[r * (BN + 8) + c] = (v < v1 && n0 + c < N) ? dY[v * N + n0 + c] : __float2bfloat16(0.f);
            }
        }
        __syncthreads();
        mma_stage<BN, true>(sA, sB, acc, warp, lane);
        __syncthreads();
    }
    float* P = part + (size_t)blockIdx.y * Kpad * N;
#pragma unroll
    for (int t = 0; t < BN / 8; ++t)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int k = k0 + 16 * warp + (lane >> 2) + 8 * h;
            if (k >= Kpad) continue;
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int n = n0 + t * 8 + 2 * (lane & 3) + e;
                if (n < N) P[(size_t)k * N + n] = acc[t][2 * h + e];
            }
        }
}

// ---------------------------------------------------------------------------
// Weight gradient from staged rows, for sources of 8 n channels.  The sums
// are the gather kernel's, product for product (chunks of kWChunk
// consecutive voxels, 16 voxels per mma in ascending order, chunks added in
// order), so the two give the same bits; what changes is how the operands
// reach the tensor cores.  One CTA takes a chunk, one dz, one slice of CL
// channels and BN outputs.  Blocks of 128 voxels (linear index) and their
// source voxels for the three dy -- 130 consecutive ones each, the linear
// shift of the tap -- are copied to shared memory once (cp.async, the next
// block under this block's products), and the three dx taps read the same
// rows: an A slice (16 weight rows x 16 voxels) is one ldmatrix.trans whose
// lanes point at their voxel's 16-byte row, or at a zero row where the tap
// leaves the volume (a 9-bit mask per voxel, formed with the block).  Warp =
// dy; a warp multiplies its three dx taps (CL = 8: two taps a slice).
// blockIdx.y past the slices sums the bias.
//
// What bounds it: a chunk is 256 dependent mma steps, so the instructions of
// a step times 256 on one warp per scheduler, whatever the layer; offsets
// and masks are therefore formed once per thread or block, not per step.
// The gather form spent that many block barriers and 27 gathers per voxel:
// at 64x64x64, channels (16, 32, 64), a layer took 270-460 us with it and
// takes 38-78 us here (a whole training step 5.51 -> 1.81 ms).
constexpr int kLV = 128;            // voxels per staged block
constexpr int kLR = kLV + 2;        // staged source voxels per dy
constexpr int kLS = 24;             // elements per staged voxel (16 + 8: eight rows hit distinct banks)
constexpr int kLT = 96;             // threads: one warp per dy
constexpr int kBiasT = 256;         // summands in flight of a bias chunk (k_bias_part's threads)
constexpr int kBiasY = (kBiasT + kLT - 1) / kLT;   // CTAs per chunk that carry them

template <int BN>
struct LinSmem {   // one of the two buffers, elements
    static constexpr int kSrc = 3 * kLR * kLS;
    static constexpr int kGrad = kLV * (BN + 8);
    static constexpr int kBuf = kSrc + kGrad + kLV;   // and the block's masks
    static constexpr size_t bytes() { return sizeof(__nv_bfloat16) * (2 * (size_t)kBuf + 8); }
};

__device__ __forceinline__ void ldsm_x2_t(uint32_t r[2], const void* p)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];"
                 : "=r"(r[0]), "=r"(r[1])
                 : "r"(smem_addr(p)));
}

// The block's output gradients into sG [128][BN + 8]: zero past v1 and N.
template <int BN, int T>
__device__ __forceinline__ void lin_stage_grad(__nv_bfloat16* sG, const __nv_bfloat16* __restrict__ dY, int N, int n0,
                                               int vb, int v1)
{
    constexpr int CH = BN / 8;
#pragma unroll
    for (int i0 = 0; i0 < kLV * CH; i0 += T) {
        const int i = i0 + threadIdx.x;
        if (kLV * CH % T != 0 && i >= kLV * CH) break;
        const int j = i / CH, c = n0 + (i % CH) * 8;
        __nv_bfloat16* d = sG + j * (BN + 8) + (i % CH) * 8;
        const bool in = vb + j < v1 && c < N;
        const __nv_bfloat16* g = dY + (in ? (size_t)(vb + j) * N + c : 0);
        if ((N & 7) == 0) {
            lin_cp16(d, g, in);
        } else {
            uint32_t w[4] = {0, 0, 0, 0};
#pragma unroll
            for (int e = 0; e < 8; ++e)
                if (in && c + e < N) w[e / 2] |= (uint32_t)(*reinterpret_cast<const uint16_t*>(g + e)) << (16 * (e & 1));
            *reinterpret_cast<uint4*>(d) = make_uint4(w[0], w[1], w[2], w[3]);
        }
    }
}

// The B fragments (all BN outputs) of voxels kk .. kk + 15.
template <int BN>
__device__ __forceinline__ void grad_frags(uint32_t (&b)[BN / 8][2], const __nv_bfloat16* sG, int kk, int lane)
{
    const int row = kk + (lane & 7) + ((lane >> 3) & 1) * 8;
    if constexpr (BN == 8) {
        ldsm_x2_t(b[0], sG + row * (BN + 8));
    } else {
#pragma unroll
        for (int j = 0; j < BN / 16; ++j) {
            uint32_t r[4];
            ldsm_x4_t(r, sG + row * (BN + 8) + j * 16 + (lane >> 4) * 8);
            b[2 * j][0] = r[0];
            b[2 * j][1] = r[1];
            b[2 * j + 1][0] = r[2];
            b[2 * j + 1][1] = r[3];
        }
    }
}

// The bias gradient's chunk sums as k_bias_part forms them: summand t
// (< per, the largest multiple of N within kBiasT) adds the chunk's elements
// t, t + per, ... in order; k_wgrad_lin_reduce combines them.
__device__ __forceinline__ void lin_bias(const __nv_bfloat16* __restrict__ dY, int N, int v0, int v1, int t,
                                         float* __restrict__ bvs)
{
    const int per = (kBiasT / N) * N;
    if (t >= kBiasT) return;
    float s = 0.f;
    if (t < per) {
        constexpr int U = 32;   // loads in flight
        const __nv_bfloat16* p = dY + (size_t)v0 * N + t;
        int left = ((v1 - v0) * N - t + per - 1) / per;
        for (; left >= U; left -= U, p += U * per) {
            __nv_bfloat16 q[U];
#pragma unroll
            for (int u = 0; u < U; ++u) q[u] = p[u * per];
#pragma unroll
            for (int u = 0; u < U; ++u) s += bf2f(q[u]);
        }
        for (; left > 0; --left, p += per) s += bf2f(*p);
    }
    bvs[(size_t)blockIdx.x * kBiasT + t] = s;
}

// MODE: 0 a plain source, 1 a half-resolution source read by nearest x2
// upsampling, 2 the rounded sum of two sources (loaded to registers before
// a block's products and summed into the other buffer after them).
template <int CL, int BN, int MODE>
__global__ void __launch_bounds__(kLT) k_wgrad_lin(ConvSrc src, const __nv_bfloat16* __restrict__ dY, int N, int Kpad,
                                                   FastDiv fw, FastDiv fh, float* __restrict__ part,
                                                   float* __restrict__ bvs)
{
    static_assert(CL == 8 || CL == 16, "channel slice");
    extern __shared__ __align__(16) unsigned char wl_raw[];
    constexpr int NT = BN / 8, U = CL == 16 ? 3 : 2, CH = CL / 8;
    constexpr int SG = LinSmem<BN>::kSrc, SM = SG + LinSmem<BN>::kGrad, BUF = LinSmem<BN>::kBuf;
    constexpr int IT = (3 * kLR * CH + kLT - 1) / kLT;
    __nv_bfloat16* sm = reinterpret_cast<__nv_bfloat16*>(wl_raw);
    __nv_bfloat16* sZ = sm + 2 * BUF;   // 8 zeros
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int D = src.D, H = src.H, W = src.W, C = src.C, V = D * H * W;
    const int v0 = blockIdx.x * kWChunk, v1 = min(v0 + kWChunk, V);
    const int nsl = C / CL;
    if ((int)blockIdx.y >= 3 * nsl) {
        if (blockIdx.z == 0) lin_bias(dY, N, v0, v1, ((int)blockIdx.y - 3 * nsl) * kLT + threadIdx.x, bvs);
        return;
    }
    const int slice = (int)blockIdx.y / 3, dz = (int)blockIdx.y % 3 - 1;
    const int n0 = blockIdx.z * BN;
    if (threadIdx.x < 8) sZ[threadIdx.x] = __float2bfloat16(0.f);

    // this thread's staged units: for dy the source voxels vb - 1 + (dz H +
    // dy) W + j, j < 130 (zero outside [0, V); a shift that crosses a face is
    // replaced by the zero row where it is read)
    int rel[IT], dst[IT];
#pragma unroll
    for (int i = 0; i < IT; ++i) {
        const int q = threadIdx.x + i * kLT, c8 = q % CH, dyi = q / CH / kLR, j = q / CH - dyi * kLR;
        rel[i] = -1 + j + (dz * H + dyi - 1) * W;
        dst[i] = q < 3 * kLR * CH ? (dyi * kLR + j) * kLS + c8 * 8 : -1;
    }
    const int ch0 = slice * CL + (CH == 2 ? (threadIdx.x & 1) * 8 : 0);   // kLT is even: c8 = thread parity
    const __nv_bfloat16* sa = src.a + ch0;
    uint4 ra[MODE == 2 ? IT : 1], rb[MODE == 2 ? IT : 1];
    auto stage = [&](int vb, __nv_bfloat16* buf) {
#pragma unroll
        for (int i = 0; i < IT; ++i) {
            const int u = vb + rel[i];
            const bool in = dst[i] >= 0 && (unsigned)u < (unsigned)V;
            if constexpr (MODE == 2) {
                ra[i] = rb[i] = make_uint4(0, 0, 0, 0);
                if (in) {
                    ra[i] = *reinterpret_cast<const uint4*>(sa + (size_t)u * C);
                    rb[i] = *reinterpret_cast<const uint4*>(src.b + ch0 + (size_t)u * C);
                }
            } else if (dst[i] >= 0) {
                size_t off = 0;
                if (MODE == 1 && in) {
                    const int yz = (int)fw.div(u), x = u - yz * W, z = (int)fh.div(yz), y = yz - z * H;
                    off = (size_t)(((z >> 1) * (H >> 1) + (y >> 1)) * (W >> 1) + (x >> 1)) * C;
                } else if (in) {
                    off = (size_t)u * C;
                }
                lin_cp16(buf + dst[i], sa + off, in);
            }
        }
        lin_stage_grad<BN, kLT>(buf + SG, dY, N, n0, vb, v1);
        asm volatile("cp.async.commit_group;" ::: "memory");
        // the voxels' masks: bit 3 dy + dx set where the tap stays inside
        for (int j = threadIdx.x; j < kLV; j += kLT) {
            const int v = vb + j, yz = (int)fw.div(v), x = v - yz * W, z = (int)fh.div(yz), y = yz - z * H;
            uint32_t m = 0;
            if (v < v1 && (unsigned)(z + dz) < (unsigned)D) {
                const uint32_t mx = (x > 0 ? 1u : 0u) | 2u | (x < W - 1 ? 4u : 0u);
                m = (y > 0 ? mx : 0u) | mx << 3 | (y < H - 1 ? mx << 6 : 0u);
            }
            reinterpret_cast<uint16_t*>(buf + SM)[j] = (uint16_t)m;
        }
    };
    auto finish = [&](__nv_bfloat16* buf) {   // MODE 2: the rounded sums into the buffer
        if constexpr (MODE == 2) {
#pragma unroll
            for (int i = 0; i < IT; ++i) {
                if (dst[i] < 0) continue;
                __nv_bfloat162* pr = reinterpret_cast<__nv_bfloat162*>(&ra[i]);
                const __nv_bfloat162* pq = reinterpret_cast<const __nv_bfloat162*>(&rb[i]);
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const float2 a = __bfloat1622float2(pr[e]), b = __bfloat1622float2(pq[e]);
                    pr[e] = __floats2bfloat162_rn(a.x + b.x, a.y + b.y);
                }
                *reinterpret_cast<uint4*>(buf + dst[i]) = ra[i];
            }
        }
    };

    float acc[U][NT][4];
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
        for (int t = 0; t < NT; ++t) acc[u][t][0] = acc[u][t][1] = acc[u][t][2] = acc[u][t][3] = 0.f;
    // this lane's voxel of an A slice: rr of its 16; mh: its 8-row half
    const int rr = (lane & 7) + 8 * (lane >> 4), mh = (lane >> 3) & 1;
    const uint32_t zrow = smem_addr(sZ);

    stage(v0, sm);
    finish(sm);
    int cur = 0;
    for (int vb = v0; vb < v1; vb += kLV, cur ^= 1) {
        const bool more = vb + kLV < v1;
        if (more) {
            stage(vb + kLV, sm + (cur ^ 1) * BUF);
            asm volatile("cp.async.wait_group 1;" ::: "memory");
        } else {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
        }
        __syncthreads();
        const __nv_bfloat16* buf = sm + cur * BUF;
        const uint32_t row = smem_addr(buf + (warp * kLR + rr + 1) * kLS + (CL == 16 ? mh * 8 : 0));   // dx = 0
        const uint16_t* msk = reinterpret_cast<const uint16_t*>(buf + SM) + rr;
#pragma unroll
        for (int ks = 0; ks < kLV / 16; ++ks) {
            uint32_t b[NT][2];
            grad_frags<BN>(b, buf + SG, 16 * ks, lane);
            const uint32_t mk = ((uint32_t)msk[16 * ks] >> (3 * warp)) & 7u;
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int dxi = CL == 16 ? u : 2 * u + mh;   // CL = 8: the halves carry two taps (3: none)
                const uint32_t p = (mk >> dxi) & 1u ? row + (16 * ks + dxi - 1) * kLS * 2 : zrow;
                uint32_t a[4];
                asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                             : "=r"(a[0]), "=r"(a[1]), "=r"(a[2]), "=r"(a[3])
                             : "r"(p));
#pragma unroll
                for (int t = 0; t < NT; ++t) mma_bf16(acc[u][t], a, b[t][0], b[t][1]);
            }
        }
        if (more) finish(sm + (cur ^ 1) * BUF);
        __syncthreads();
    }
    // fragment (row lane / 4 [+ 8], columns 2 (lane % 4) + {0, 1})
    float* P = part + (size_t)blockIdx.x * Kpad * N;
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
        for (int t = 0; t < NT; ++t)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int half = e >> 1, r = (lane >> 2);
                const int dxi = CL == 16 ? u : 2 * u + half;
                if (dxi > 2) continue;
                const int k = (9 * (dz + 1) + 3 * warp + dxi) * C + slice * CL + (CL == 16 ? r + 8 * half : r);
                const int n = n0 + t * 8 + 2 * (lane & 3) + (e & 1);
                if (n < N) P[(size_t)k * N + n] = acc[u][t][e];
            }
}

// The same for one-channel sources (the FP32 network input): the nine
// (dz, dy) rows of a block are staged as scalars, two threads build a
// voxel's 27 taps as one row of the operand (16 each), and warp w multiplies
// taps 16 (w & 1) .. + 15 with outputs 8 (w / 2) .. + 7.
constexpr int kC1T = 256;
template <int BN>
__global__ void __launch_bounds__(kC1T) k_wgrad_lin1(ConvSrc src, const __nv_bfloat16* __restrict__ dY, int N, int Kpad,
                                                     FastDiv fw, FastDiv fh, float* __restrict__ part,
                                                     float* __restrict__ bvs)
{
    constexpr int NT = BN / 8, IT = (9 * kLR + kC1T - 1) / kC1T;
    static_assert(2 * NT <= kC1T / 32, "a warp per (tap half, output tile)");
    __shared__ __align__(16) __nv_bfloat16 sS[9 * kLR + 6];
    __shared__ __align__(16) __nv_bfloat16 sA[kLV * (kBK + 8)];
    __shared__ __align__(16) __nv_bfloat16 sG[2][kLV * (BN + 8)];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int D = src.D, H = src.H, W = src.W, V = D * H * W;
    const int v0 = blockIdx.x * kWChunk, v1 = min(v0 + kWChunk, V);
    if (blockIdx.y > 0) {
        if (blockIdx.z == 0) lin_bias(dY, N, v0, v1, threadIdx.x, bvs);
        return;
    }
    const int n0 = blockIdx.z * BN;
    const float fsc = src.f32_scale ? *src.f32_scale : 1.f;
    float f[IT];
    auto fetch = [&](int vb) {
#pragma unroll
        for (int i = 0; i < IT; ++i) {
            const int q = threadIdx.x + i * kC1T, r = q / kLR, j = q - r * kLR;
            const int u = vb - 1 + j + ((r / 3 - 1) * H + (r % 3 - 1)) * W;
            float val = 0.f;
            if (q < 9 * kLR && (unsigned)u < (unsigned)V) {
                if (src.f32) {
                    val = src.f32[u] * fsc;
                } else {
                    int o = u;
                    if (src.up) {
                        const int yz = (int)fw.div(u), x = u - yz * W, z = (int)fh.div(yz), y = yz - z * H;
                        o = ((z >> 1) * (H >> 1) + (y >> 1)) * (W >> 1) + (x >> 1);
                    }
                    val = bf2f(src.a[o]);
                    if (src.b) val = bf2f(__float2bfloat16(val + bf2f(src.b[o])));
                }
            }
            f[i] = val;
        }
    };
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
    fetch(v0);
    lin_stage_grad<BN, kC1T>(sG[0], dY, N, n0, v0, v1);
    asm volatile("cp.async.commit_group;" ::: "memory");
    int cur = 0;
    const int un = warp & 1, nt = warp >> 1, jv = threadIdx.x & (kLV - 1), half = threadIdx.x / kLV;
    for (int vb = v0; vb < v1; vb += kLV, cur ^= 1) {
#pragma unroll
        for (int i = 0; i < IT; ++i) {
            const int q = threadIdx.x + i * kC1T;
            if (q < 9 * kLR) sS[q] = __float2bfloat16(f[i]);
        }
        __syncthreads();
        if (vb + kLV < v1) {
            fetch(vb + kLV);
            lin_stage_grad<BN, kC1T>(sG[cur ^ 1], dY, N, n0, vb + kLV, v1);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
        {   // taps 16 half .. + 15 of this thread's voxel, zero where they leave the volume
            const int v = vb + jv, yz = (int)fw.div(v), x = v - yz * W, z = (int)fh.div(yz), y = yz - z * H;
            uint32_t m = 0;
            if (v < v1) {
                const uint32_t mx = (x > 0 ? 1u : 0u) | 2u | (x < W - 1 ? 4u : 0u);
                const uint32_t my = (y > 0 ? mx : 0u) | mx << 3 | (y < H - 1 ? mx << 6 : 0u);
                m = (z > 0 ? my : 0u) | my << 9 | (z < D - 1 ? my << 18 : 0u);
            }
            const uint16_t* sp = reinterpret_cast<const uint16_t*>(sS) + jv;
            uint32_t w[8];
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                // tap 16 half + i: its row (tap / 3) and dx + 1 (tap % 3); taps past 26 read row 8
                const int o0 = (i / 3) * kLR + i % 3, k1 = 16 + i < 27 ? 16 + i : 26, o1 = (k1 / 3) * kLR + k1 % 3;
                const uint32_t t = sp[half ? o1 : o0];
                const uint32_t b = (m >> (16 * half + i)) & 1u ? t : 0u;
                if (i & 1) w[i / 2] |= b << 16;
                else w[i / 2] = b;
            }
            uint4* d = reinterpret_cast<uint4*>(sA + jv * (kBK + 8) + 16 * half);
            d[0] = make_uint4(w[0], w[1], w[2], w[3]);
            d[1] = make_uint4(w[4], w[5], w[6], w[7]);
        }
        asm volatile("cp.async.wait_group 1;" ::: "memory");
        __syncthreads();
        if (nt < NT) {
#pragma unroll
            for (int ks = 0; ks < kLV / 16; ++ks) {
                uint32_t b[2], a[4];
                ldsm_x2_t(b, sG[cur] + (16 * ks + (lane & 15)) * (BN + 8) + nt * 8);
                ldsm_x4_t(a, sA + (16 * ks + (lane & 7) + (lane >> 4) * 8) * (kBK + 8) + un * 16 + ((lane >> 3) & 1) * 8);
                mma_bf16(acc, a, b[0], b[1]);
            }
        }
        __syncthreads();
    }
    if (nt >= NT) return;
    float* P = part + (size_t)blockIdx.x * Kpad * N;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const int k = 16 * un + (lane >> 2) + 8 * (e >> 1);
        const int n = n0 + nt * 8 + 2 * (lane & 3) + (e & 1);
        if (k < 27 && n < N) P[(size_t)k * N + n] = acc[e];
    }
}

// gW[n][k] = sum over chunks, in order, of part[chunk][k][n] (as
// k_wgrad_reduce); the last block's sums gb[n] over
// the chunks of the bias summands, each chunk's in k_bias_part's order.
static __global__ void __launch_bounds__(256) k_wgrad_lin_reduce(const float* __restrict__ part, int chunks, int Kpad,
                                                          int Kvalid, int N, const float* __restrict__ bvs,
                                                          float* __restrict__ gW, float* __restrict__ gb)
{
    if (blockIdx.x == gridDim.x - 1) {
        __shared__ float t_s[2048];   // [chunks of a round][N]
        const int per = (kBiasT / N) * N, cr = 2048 / N;
        float s = 0.f;
        for (int c0 = 0; c0 < chunks; c0 += cr) {
            const int nc = chunks - c0 < cr ? chunks - c0 : cr;
            for (int i = threadIdx.x; i < nc * N; i += 256) {
                const float* q = bvs + (size_t)(c0 + i / N) * kBiasT;
                float t = 0.f;
#pragma unroll 8
                for (int j = i % N; j < per; j += N) t += q[j];
                t_s[i] = t;
            }
            __syncthreads();
            if ((int)threadIdx.x < N) {
#pragma unroll 8
                for (int c = 0; c < nc; ++c) s += t_s[c * N + threadIdx.x];
            }
            __syncthreads();
        }
        if ((int)threadIdx.x < N) gb[threadIdx.x] = s;
        return;
    }
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= Kvalid * N) return;
    const int k = i / N, n = i % N;
    const float* q = part + i;   // (c Kpad + k) N + n
    const size_t cs = (size_t)Kpad * N;
    float s = 0.f;
    int c = 0;
    constexpr int U = 16;   // loads in flight
    for (; c + U <= chunks; c += U) {
        float w[U];
#pragma unroll
        for (int u = 0; u < U; ++u) w[u] = q[(c + u) * cs];
#pragma unroll
        for (int u = 0; u < U; ++u) s += w[u];
    }
    for (; c < chunks; ++c) s += q[c * cs];
    gW[(size_t)n * Kvalid + k] = s;
}

// grad[n][k] (k < Kvalid: the parameter layout W[co][tap][ci]) = sum over
// chunks, in chunk order, of part[chunk][k][n].
static __global__ void k_wgrad_reduce(const float* __restrict__ part, int chunks, int Kpad, int Kvalid, int N,
                               float* __restrict__ grad)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= Kvalid * N) return;
    const int k = i / N, n = i % N;
    float s = 0.f;
    for (int c = 0; c < chunks; ++c) s += part[((size_t)c * Kpad + k) * N + n];
    grad[(size_t)n * Kvalid + k] = s;
}

// Bias gradient: part[b][n] = sum over block b's voxels of dY[v][n]; then
// grad[n] = sum over blocks in order.  The block reads its chunk of dY as one
// contiguous run: thread t (t < per, per the largest multiple of N within
// the block) always lands on channel t % N, and the threads of a channel are
// combined in thread order.
static __global__ void k_bias_part(const __nv_bfloat16* __restrict__ dY, long long V, int N, float* __restrict__ part)
{
    __shared__ float red[kThreads];
    const long long v0 = (long long)blockIdx.x * kWChunk;
    const long long v1 = v0 + kWChunk < V ? v0 + kWChunk : V;
    const int per = (kThreads / N) * N;
    float s = 0.f;
    if ((int)threadIdx.x < per)
        for (long long i = v0 * N + threadIdx.x; i < v1 * N; i += per) s += bf2f(dY[i]);
    red[threadIdx.x] = s;
    __syncthreads();
    if ((int)threadIdx.x < N) {
        float t = 0.f;
        for (int j = threadIdx.x; j < per; j += N) t += red[j];
        part[(size_t)blockIdx.x * N + threadIdx.x] = t;
    }
}

static __global__ void k_bias_reduce(const float* __restrict__ part, int blocks, int N, float* __restrict__ grad)
{
    const int n = blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= N) return;
    float s = 0.f;
    for (int b = 0; b < blocks; ++b) s += part[(size_t)b * N + n];
    grad[n] = s;
}

// 2x2x2 mean pool of [D][H][W][C] (D, H, W even) into [D/2][H/2][W/2][C].
static __global__ void k_pool(const __nv_bfloat16* __restrict__ in, int D, int H, int W, int C,
                       __nv_bfloat16* __restrict__ out)
{
    const long long n = (long long)(D / 2) * (H / 2) * (W / 2) * C;
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int c = (int)(i % C);
    long long v = i / C;
    const int x = (int)(v % (W / 2));
    v /= (W / 2);
    const int y = (int)(v % (H / 2));
    const int z = (int)(v / (H / 2));
    float s = 0.f;
    for (int a = 0; a < 2; ++a)
        for (int b = 0; b < 2; ++b)
            for (int e = 0; e < 2; ++e)
                s += bf2f(in[(((size_t)(2 * z + a) * H + (2 * y + b)) * W + (2 * x + e)) * C + c]);
    out[i] = __float2bfloat16(s * 0.125f);
}

// g[v][c] = skip[v][c] + gp[parent(v)][c] / 8: gradient of a volume that
// feeds both a 2x2x2 mean pool (gradient gp) and an additive skip (skip).
static __global__ void k_pool_grad_add(const __nv_bfloat16* __restrict__ skip, const __nv_bfloat16* __restrict__ gp, int D,
                                int H, int W, int C, __nv_bfloat16* __restrict__ g)
{
    const long long n = (long long)D * H * W * C;
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int c = (int)(i % C);
    long long v = i / C;
    const int x = (int)(v % W);
    v /= W;
    const int y = (int)(v % H);
    const int z = (int)(v / H);
    const size_t pi = (((size_t)(z >> 1) * (H >> 1) + (y >> 1)) * (W >> 1) + (x >> 1)) * C + c;
    g[i] = __float2bfloat16(bf2f(skip[i]) + bf2f(gp[pi]) * 0.125f);
}

// Gradient of a nearest x2 upsampling: g[z][y][x][c] = sum of the 8 children
// of fine-grid gradient gf ([2D][2H][2W][C]).
static __global__ void k_up_grad(const __nv_bfloat16* __restrict__ gf, int D, int H, int W, int C,
                          __nv_bfloat16* __restrict__ g)
{
    const long long n = (long long)D * H * W * C;
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int c = (int)(i % C);
    long long v = i / C;
    const int x = (int)(v % W);
    v /= W;
    const int y = (int)(v % H);
    const int z = (int)(v / H);
    float s = 0.f;
    for (int a = 0; a < 2; ++a)
        for (int b = 0; b < 2; ++b)
            for (int e = 0; e < 2; ++e)
                s += bf2f(gf[(((size_t)(2 * z + a) * (2 * H) + (2 * y + b)) * (2 * W) + (2 * x + e)) * C + c]);
    g[i] = __float2bfloat16(s);
}

// out = g where y > 0 else 0 (ReLU gradient; g itself is kept, a skip may
// need it unmasked).
static __global__ void k_relu_grad(__nv_bfloat16* __restrict__ out, const __nv_bfloat16* __restrict__ g,
                            const __nv_bfloat16* __restrict__ y, long long n)
{
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = bf2f(y[i]) > 0.f ? g[i] : __float2bfloat16(0.f);
}

// The elementwise kernels above on 8 channels a thread (C a multiple of 8):
// one 16-byte access per voxel and operand instead of eight 2-byte ones, and
// the voxel's coordinates once (divisions by multiplication); the sums run
// per channel in the same order.  The scalar forms keep other channel counts.
struct Vol8 {   // index math of [D][H][W][C / 8] units
    FastDiv dc, dw, dh;
    int n;   // units
    Vol8(int D, int H, int W, int C) : dc(C / 8), dw(W), dh(H), n(D * H * W * (C / 8)) {}
    __device__ __forceinline__ void split(int i, int& c8, int& x, int& y, int& z) const
    {
        const int v = (int)dc.div((uint32_t)i);
        c8 = i - v * (int)dc.d;
        const int q = (int)dw.div((uint32_t)v);
        x = v - q * (int)dw.d;
        z = (int)dh.div((uint32_t)q);
        y = q - z * (int)dh.d;
    }
};
__device__ __forceinline__ void add8(float (&s)[8], uint4 q)
{
    const __nv_bfloat162* p = reinterpret_cast<const __nv_bfloat162*>(&q);
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const float2 f = __bfloat1622float2(p[e]);
        s[2 * e] += f.x;
        s[2 * e + 1] += f.y;
    }
}
__device__ __forceinline__ uint4 pack8(const float (&s)[8], float f)
{
    uint4 r;
    __nv_bfloat162* p = reinterpret_cast<__nv_bfloat162*>(&r);
#pragma unroll
    for (int e = 0; e < 4; ++e) p[e] = __floats2bfloat162_rn(s[2 * e] * f, s[2 * e + 1] * f);
    return r;
}
// The 8 children of each coarse unit summed times f: the mean pool (f = 1/8)
// and the gradient of the upsampling (f = 1).  g: the coarse volume.
static __global__ void k_sum8_v8(const uint4* __restrict__ in, Vol8 g, float f, uint4* __restrict__ out)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= g.n) return;
    int c8, x, y, z;
    g.split(i, c8, x, y, z);
    const int C8 = (int)g.dc.d, W = 2 * (int)g.dw.d, H = 2 * (int)g.dh.d;
    const uint4* p = in + (((size_t)(2 * z) * H + 2 * y) * W + 2 * x) * C8 + c8;
    uint4 q[8];
#pragma unroll
    for (int a = 0; a < 8; ++a) q[a] = p[(((size_t)(a >> 2) * H + ((a >> 1) & 1)) * W + (a & 1)) * C8];
    float s[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int a = 0; a < 8; ++a) add8(s, q[a]);
    out[i] = pack8(s, f);
}
static __global__ void k_pool_grad_add_v8(const uint4* __restrict__ skip, const uint4* __restrict__ gp, Vol8 g,
                                          uint4* __restrict__ out)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= g.n) return;
    int c8, x, y, z;
    g.split(i, c8, x, y, z);
    const int C8 = (int)g.dc.d, W = (int)g.dw.d >> 1, H = (int)g.dh.d >> 1;
    const uint4 a = skip[i], b = gp[(((size_t)(z >> 1) * H + (y >> 1)) * W + (x >> 1)) * C8 + c8];
    uint4 r;
    const __nv_bfloat162* pa = reinterpret_cast<const __nv_bfloat162*>(&a);
    const __nv_bfloat162* pb = reinterpret_cast<const __nv_bfloat162*>(&b);
    __nv_bfloat162* pr = reinterpret_cast<__nv_bfloat162*>(&r);
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const float2 u = __bfloat1622float2(pa[e]), v = __bfloat1622float2(pb[e]);
        pr[e] = __floats2bfloat162_rn(u.x + v.x * 0.125f, u.y + v.y * 0.125f);
    }
    out[i] = r;
}
static __global__ void k_relu_grad_v8(uint4* __restrict__ out, const uint4* __restrict__ g, const uint4* __restrict__ y,
                                      long long n8)
{
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n8) return;
    uint4 a = g[i];
    const uint4 b = y[i];
    __nv_bfloat16* pa = reinterpret_cast<__nv_bfloat16*>(&a);
    const __nv_bfloat16* pb = reinterpret_cast<const __nv_bfloat16*>(&b);
#pragma unroll
    for (int e = 0; e < 8; ++e)
        if (!(bf2f(pb[e]) > 0.f)) pa[e] = __float2bfloat16(0.f);
    out[i] = a;
}

// Loss sum((out - t)^2) / (2 V) per block in FP64 partials; gradient
// g = (out - t) / V as bfloat16.  The target is multiplied by the device
// scalar *tscale when given.
static __global__ void k_mse(const float* __restrict__ out, const float* __restrict__ t, const float* __restrict__ tscale,
                      long long V, __nv_bfloat16* __restrict__ g, double* __restrict__ part)
{
    __shared__ double red[kThreads];
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    double s = 0.0;
    if (i < V) {
        const float d = out[i] - t[i] * (tscale ? *tscale : 1.f);
        g[i] = __float2bfloat16(d / (float)V);
        s = (double)d * d;
    }
    red[threadIdx.x] = s;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) part[blockIdx.x] = red[0] / (2.0 * (double)V);
}

// Per-block FP64 partial sums of in[i]^2.
static __global__ void k_sumsq_part(const float* __restrict__ in, long long V, double* __restrict__ part)
{
    __shared__ double red[kThreads];
    double s = 0.0;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < V; i += (long long)gridDim.x * blockDim.x) {
        const double v = in[i];
        s += v * v;
    }
    red[threadIdx.x] = s;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) part[blockIdx.x] = red[0];
}

constexpr int kScaleMax = 304;   // most partial sums of the RMS
constexpr int kScaleT = 512;     // k_scales' threads

// r = RMS of the input from the partials; scales = {1 / r, r gain, 1 / (r gain)}
// (r = 1 for an all-zero input).  One block; the partials add up in a tree (one
// after the other they are a chain of 304 FP64 additions: 13.1 us against 4.3).
static __global__ void __launch_bounds__(kScaleT) k_scales(const double* __restrict__ part, int nb, long long V,
                                                           float gain, float* __restrict__ scales)
{
    __shared__ double ps[kScaleT];
    ps[threadIdx.x] = (int)threadIdx.x < nb ? part[threadIdx.x] : 0.0;
    __syncthreads();
    for (int w = kScaleT / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) ps[threadIdx.x] += ps[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x != 0) return;
    const double s = ps[0];
    double r = sqrt(s / (double)V);
    if (!(r > 0.0)) r = 1.0;
    scales[0] = (float)(1.0 / r);
    scales[1] = (float)(r * gain);
    scales[2] = (float)(1.0 / (r * gain));
}

// Wt[k][n] (forward) = W[n][k] for k < 27 Cin, n < Cout; zero padding.
// With transpose_io (gradient w.r.t. the input): k = tap * Cout + co,
// n = ci, Wt[k][n] = W[co][tap][ci].
static __global__ void k_prep_weights(const float* __restrict__ W, int Cin, int Cout, int Kpad, int Npad, int transpose_io,
                               __nv_bfloat16* __restrict__ Wt)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= Kpad * Npad) return;
    const int k = i / Npad, n = i % Npad;
    float v = 0.f;
    if (!transpose_io) {
        if (k < 27 * Cin && n < Cout) v = W[(size_t)n * 27 * Cin + k];
    } else {
        if (k < 27 * Cout && n < Cin) {
            const int tap = k / Cout, co = k % Cout;
            v = W[((size_t)co * 27 + tap) * Cin + n];
        }
    }
    Wt[i] = __float2bfloat16(v);
}

// One operand matrix of the network, all of them written by one launch of
// k_prep_all (forty launches of a microsecond or two before): kind 0 the
// implicit-GEMM matrix of k_prep_weights, 1 the tcgen05 layout (C8P, NP; see
// umma_conv.cuh), 2 its paired-tap layout.  K = 27 Cs rows and N columns of the
// matrix carry weights; blocks [block0, next job's block0).
struct PrepJob {
    int kind, transpose, cin, cout, K, N, Npad, Cs, C8P, NP, sgn, total, block0;
    long long woff;
    __nv_bfloat16* dst;
};
static __global__ void k_prep_all(const PrepJob* __restrict__ jobs, int njobs, const float* __restrict__ theta)
{
    __shared__ int job_s;
    if (threadIdx.x == 0) {
        int lo = 0, hi = njobs - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) / 2;
            if (jobs[mid].block0 <= (int)blockIdx.x) lo = mid;
            else hi = mid - 1;
        }
        job_s = lo;
    }
    __syncthreads();
    const PrepJob& q = jobs[job_s];
    const int i = ((int)blockIdx.x - q.block0) * blockDim.x + threadIdx.x;
    if (i >= q.total) return;
    const float* W = theta + q.woff;
    int k = -1, n = 0;   // row and column of the matrix; -1: padding
    if (q.kind == 0) {
        k = i / q.Npad;
        n = i % q.Npad;
    } else if (q.kind == 1) {
        const int j = i % 8, c = (i / (8 * q.NP)) % q.C8P, tap = i / (8 * q.NP * q.C8P), ci = 8 * c + j;
        n = (i / 8) % q.NP;
        if (ci < q.Cs) k = tap * q.Cs + ci;
    } else {
        const int j = i % 8, c = (i / (8 * q.NP)) % 2, g = (i / (16 * q.NP)) % 2, pzx = i / (32 * q.NP);
        const int pz = pzx / 3, px = pzx % 3, p = g == 0 ? c : (c == 0 ? 2 : -1);
        n = (i / 8) % q.NP;
        if (p >= 0 && j < q.Cs) {
            const int dz = q.sgn * (pz - 1), dy = q.sgn * (p - 1), dx = q.sgn * (px - 1);
            k = (9 * (dz + 1) + 3 * (dy + 1) + (dx + 1)) * q.Cs + j;
        }
    }
    float v = 0.f;
    if (k >= 0 && k < q.K && n < q.N) {
        if (!q.transpose) {
            v = W[(size_t)n * 27 * q.cin + k];
        } else {
            const int tap = k / q.cout, co = k % q.cout;
            v = W[((size_t)co * 27 + tap) * q.cin + n];
        }
    }
    q.dst[i] = __float2bfloat16(v);
}

// Adam (FP32 master weights): m = b1 m + (1 - b1) g, v = b2 v + (1 - b2) g^2,
// theta -= lr (m / (1 - b1^t)) / (sqrt(v / (1 - b2^t)) + eps).
static __global__ void k_adam(float* __restrict__ theta, float* __restrict__ m, float* __restrict__ v,
                       const float* __restrict__ g, long long n, float lr, float b1, float b2, float eps, float c1,
                       float c2)
{
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    theta[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

}  // namespace unet
}  // namespace mh3d
