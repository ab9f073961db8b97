// 3x3x3 convolutions of the warm-start network on the fifth-generation
// tensor cores: tcgen05.mma (kind::f16, bfloat16 operands, FP32
// accumulation) reading both operands from shared memory through matrix
// descriptors and accumulating in tensor memory (TMEM); the epilogue reads
// the accumulators back with tcgen05.ld.
//
// The GEMM of one tile.  A tile is 8 x 16 voxels (x, y) of one z plane; TMEM
// lane m = 8 (y - y0) + x - x0.  An input plane p enters three output planes,
// p + 1, p and p - 1 (taps dz = -1, 0, 1; the walk runs down z for a flipped
// operand, so that every output still adds its planes in the order dz = -1, 0,
// 1).  For every (dy, dx) and 16 input channels, with t the tap's dz + 1,
//     D_{p + 1 - t}[m][n] += sum_{c < 16} in[p][y + dy][x + dx][c] W[n][t, dy, dx][c]
// for the three t together is one tcgen05.mma with M = 128, N = 3 NP, K = 16
// (NP >= the output channels, a multiple of 16).
//
// Accumulators: output plane o has the NP columns of TMEM slot o mod 3, so a
// plane's MMA covers all three slots; which t a slot takes turns with p, and
// the weights hold five groups t = 2, 1, 0, 2, 1 of which the B descriptor
// starts at group 2 - (p + 1) mod 3.  After plane p's MMAs output p - 1 is
// complete: the epilogue reads its slot and stores zeros there.
//
// Operand layout (no swizzle, K-major canonical layout: 8 rows x 16 bytes
// per core matrix, rows 16 bytes apart, core matrices along M `SBO` and
// along K `LBO` bytes apart):
//   halo: input planes of 18 x 10 voxels, each [chunk of 8 channels][18 y][10
//         x][8]: eight x neighbours are a core matrix, the next y row is SBO =
//         160 bytes on, so the A operand of a tap is its plane started at voxel
//         (1 + dy, 1 + dx) -- a descriptor offset, no data movement -- and the
//         tap's second 8 channels sit LBO = 180 voxels on;
//   weights: [dy, dx][chunk][5 groups][NP][8], the B operand of (dy, dx, chunk
//         pair) one descriptor, its second 8 channels 5 NP rows on.
// Chunks are padded to an even count with zeros (8 channels: one zero
// chunk; the FP32 single-channel network input: channel 0 of chunk 0).
//
// A CTA of 128 threads walks a column of tiles with two staged planes: one is
// multiplied while the next is staged (1.4 input voxels staged per output
// voxel).  The columns' planes are one sequence, of which every CTA takes an
// equal run; a run of R outputs multiplies R + 2 planes.
// What bounds it: the MMAs' reads of A from shared memory.  Back to back on one
// CTA a K = 16 MMA with M = 128 takes 39, 44, 48, 56 and 96 cycles for N = 16, 48,
// 64, 96 and 192 whatever its A offset, so the three dz of a plane in one MMA
// cost little more than one; nine of them with their commit and wait, a
// plane's chain, take 69, 72, 101 and 142 cycles each for N = 16, 48, 96 and 192.
// Issued from a branch on the thread index instead of elect.sync: 45 and 79
// for N = 16.
// Measured, a whole forward of channels (16, 32, 64, 128) at 128x128x64: 650 us
// with one MMA a tap, 559 with three.  Every output bit stays.
// The wait on an mbarrier is bounded (%globaltimer): on expiry the CTA
// records MH3D_ERR_TIMEOUT in *status, frees its TMEM and returns.
#pragma once

#include <cstdint>

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "bulk.cuh"
#include "unet_kernels.cuh"

namespace mh3d {
namespace unet {
namespace umma {

constexpr int kM = 128;                       // voxels per tile (TMEM lanes)
constexpr int kX = 8, kY = 16;                // the tile's extents
constexpr int kHX = kX + 2, kHV = kHX * (kY + 2);   // a staged plane: 180 voxels
constexpr int kSlots = 2;                     // staged planes
constexpr int kGroups = 5;                    // weight groups t = 2, 1, 0, 2, 1
constexpr int kT = 128;                       // threads per CTA

template <int C8P, int NP>
struct Geom {
    static_assert(C8P % 2 == 0 && NP % 16 == 0 && NP >= 16 && NP <= 64, "operand shape");
    static constexpr int kWUnits = 9 * C8P * kGroups * NP;   // 16-byte units
    static constexpr int kPlane = C8P * kHV;                 // 16-byte units of a staged plane
    static constexpr int kCols = NP == 16 ? 64 : 4 * NP;     // TMEM columns: 3 NP, to a power of two
    static constexpr int kPer = (kPlane + kT - 1) / kT;      // units a thread stages
    static constexpr size_t smem() { return 128 + (size_t)kWUnits * 16 + (size_t)kSlots * kPlane * 16; }
};

// One thread of a converged warp.
__device__ __forceinline__ bool elect_one()
{
    uint32_t r;
    asm volatile(
        "{\n"
        " .reg .pred p;\n"
        " elect.sync _|p, 0xffffffff;\n"
        " selp.u32 %0, 1, 0, p;\n"
        "}\n"
        : "=r"(r));
    return r != 0;
}

// ---- tcgen05 primitives (inline PTX) ----------------------------------------

__device__ __forceinline__ void tmem_alloc(uint32_t* dst_smem, uint32_t ncols)
{
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(dst_smem)),
                 "r"(ncols)
                 : "memory");
}
__device__ __forceinline__ void tmem_relinquish()
{
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols)
{
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// D (TMEM) (+)= A (smem) B (smem); accumulate = 0 overwrites D.
__device__ __forceinline__ void mma_f16(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                        uint32_t accumulate)
{
    asm volatile(
        "{\n"
        " .reg .pred p;\n"
        " setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n"
        "}\n" ::"r"(d_tmem),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}

// Arrives once on the mbarrier when every MMA this thread issued so far has
// completed.
__device__ __forceinline__ void mma_commit(uint64_t* bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
                 : "memory");
}

// 16 consecutive FP32 columns of this warp's 32 lanes (lane i: TMEM lane
// base + i).
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16])
{
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}
// Zeros into those columns.
__device__ __forceinline__ void tmem_zero16(uint32_t taddr)
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1};" ::"r"(
                     taddr),
                 "r"(0)
                 : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// Shared-memory matrix descriptor: start address, leading (K) and stride
// (M/N) byte offsets, the fixed 0b001 at bits 46-48, no swizzle.
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo, uint32_t sbo)
{
    return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | (1ull << 46);
}

// Instruction descriptor of kind::f16: FP32 D (bits 4-5 = 1), bfloat16 A
// and B (bits 7-9, 10-12 = 1), both K-major, N / 8 at bits 17-22, M / 16
// at bits 24-28.
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// ---- staging ---------------------------------------------------------------

// Asynchronous 16-byte copy global -> shared (cp.async, L2 only); src_bytes
// 0 fills the 16 bytes with zeros without reading.
__device__ __forceinline__ void cp_async16(void* sdst, const void* gsrc, uint32_t src_bytes)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(sdst)), "l"(gsrc), "r"(src_bytes)
                 : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// ---- the kernel --------------------------------------------------------------

// Epilogue of one tile: warp w holds TMEM lanes 32 w .. 32 w + 31, columns
// acc .. acc + NP - 1 = output channels; x, y: the lane's voxel.  The columns
// are zero afterwards.
template <int NP, class OutT>
__device__ __forceinline__ void epilogue(const ConvSrc& src, uint32_t acc, int z, int y, int x, int N,
                                         const float* __restrict__ bias, int relu, float osc, OutT* __restrict__ out)
{
    const int warp = threadIdx.x >> 5;
    const long long v = ((long long)z * src.H + y) * src.W + x;
#pragma unroll
    for (int c0 = 0; c0 < NP; c0 += 16) {
        float a[16];
        __syncwarp();   // lanes outside the volume leave an iteration early; tcgen05.ld and .st are warp-wide
        tmem_ld16(acc + ((uint32_t)(32 * warp) << 16) + (uint32_t)c0, a);
        tmem_ld_wait();
        tmem_zero16(acc + ((uint32_t)(32 * warp) << 16) + (uint32_t)c0);
        if (x >= src.W || y >= src.H) continue;
#pragma unroll
        for (int j = 0; j < 16; ++j) {
            const int n = c0 + j;
            a[j] = (a[j] + ((bias && n < N) ? bias[n] : 0.f)) * osc;
            if (relu) a[j] = fmaxf(a[j], 0.f);
        }
        if constexpr (sizeof(OutT) == 2) {
            if (N % 8 == 0) {   // whole 16-byte groups of channels (the voxel's row is 16-byte aligned)
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    if (c0 + 8 * h >= N) break;
                    uint4 pk;
                    __nv_bfloat162* q = reinterpret_cast<__nv_bfloat162*>(&pk);
#pragma unroll
                    for (int i = 0; i < 4; ++i) q[i] = __floats2bfloat162_rn(a[8 * h + 2 * i], a[8 * h + 2 * i + 1]);
                    *reinterpret_cast<uint4*>(out + v * N + c0 + 8 * h) = pk;
                }
                continue;
            }
        }
#pragma unroll
        for (int j = 0; j < 16; ++j) {
            const int n = c0 + j;
            if (n >= N) break;
            if constexpr (sizeof(OutT) == 2)
                out[v * N + n] = __float2bfloat16(a[j]);
            else
                out[v * N + n] = a[j];
        }
    }
    __syncwarp();   // the caller's next tcgen05 instruction is warp-wide
}

// The 9 x C8P / 2 MMAs of one plane into the three accumulators at column
// acc, committed to `bar` (one thread).  g0: the first weight group.
// Descriptor start addresses count 16-byte units, so offsets add to the low
// field.
//
// Paired taps (sources of at most 8 channels, whose second chunk is zero
// padding): one MMA takes two taps of the same dx and neighbouring y -- row
// offsets 0 and 1, the second chunk LBO = one row on -- and a second MMA the
// third row with a zero second chunk: 6 MMAs a plane instead of 9.  The paired
// weights ([3 px][2 g][2 c][5 groups][NP][8]) are indexed by plane offsets, the
// flip folded in.  (The third row's second chunk is the row below it, one past
// the halo for the last tile row, where the zeroed second chunk plane begins.)
template <int C8P, int NP>
__device__ __forceinline__ void issue_mmas(uint32_t acc, uint32_t sP_a, uint32_t sW_a, int g0, int sgn, int pair,
                                           uint64_t* bar)
{
    constexpr uint32_t kIdesc = idesc_bf16(kM, 3 * NP);
    const uint64_t b0 = smem_desc(sW_a, kGroups * NP * 16, 128) + (uint64_t)(g0 * NP);
    if (pair) {
        const uint64_t a0 = smem_desc(sP_a, kHX * 16, kHX * 16);
#pragma unroll
        for (int px = 0; px < 3; ++px)
#pragma unroll
            for (int g = 0; g < 2; ++g)
                mma_f16(acc, a0 + (uint64_t)(2 * g * kHX + px), b0 + (uint64_t)((px * 2 + g) * 2 * kGroups * NP), kIdesc, 1);
    } else {
        const uint64_t a0 = smem_desc(sP_a, kHV * 16, kHX * 16) + (uint64_t)(kHX + 1);
#pragma unroll
        for (int yx = 0; yx < 9; ++yx) {
            const uint64_t at = a0 + (uint64_t)(int64_t)(sgn * ((yx / 3 - 1) * kHX + yx % 3 - 1));
#pragma unroll
            for (int ks = 0; ks < C8P / 2; ++ks)
                mma_f16(acc, at + (uint64_t)(2 * ks * kHV), b0 + (uint64_t)((yx * C8P + 2 * ks) * kGroups * NP), kIdesc, 1);
        }
    }
    mma_commit(bar);
}

// Wu: [27][C8P][NP][8] bfloat16 (k_prep_umma), Wpair: [3 pz][3 px][2 g][2 c][NP][8]
// (k_prep_umma_pair) or null; out: [V][N] channels last.
//
// Staging: 16-byte units, channels 8 c .. 8 c + 7 of a halo voxel, zero
// outside the volume; only the cv chunks that carry channels (the padding
// chunks are zeroed once).  A unit's place in the plane does not change along
// the column, so a thread's offsets are formed once per column.  Plain and
// upsampled bfloat16 sources: one cp.async a unit.  The skip sum (rounded to
// bfloat16, as a stored sum would be; not upsampled) and the FP32 input
// (rounded to bfloat16, channel 0) need arithmetic: their units are loaded
// into registers, combined and stored.
template <int C8P, int NP, class OutT>
__global__ void __launch_bounds__(kT) k_conv_umma(ConvSrc src, const __nv_bfloat16* __restrict__ Wu, int N,
                                                  const float* __restrict__ bias, int relu,
                                                  const float* __restrict__ oscale, OutT* __restrict__ out,
                                                  int ntx, int nty, int* status, const __nv_bfloat16* __restrict__ Wpair)
{
    using G = Geom<C8P, NP>;
    constexpr int U = G::kPer;
    extern __shared__ unsigned char umma_raw[];
    __shared__ __align__(8) uint64_t mbar;
    __shared__ uint32_t tmem_base_s;
    unsigned char* base =
        reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(umma_raw) + 127) & ~uintptr_t(127));
    uint4* sW = reinterpret_cast<uint4*>(base);                  // [9][C8P][kGroups][NP]
    uint4* sH = sW + G::kWUnits;                                 // [kSlots][C8P][kHV]
    const int tid = threadIdx.x, warp = tid >> 5;
    const int pair = Wpair != nullptr ? 1 : 0;
    const int sgn = src.flip ? -1 : 1;

    if (warp == 0) {
        tmem_alloc(&tmem_base_s, G::kCols);
        tmem_relinquish();
    }
    if (tid == 0) {
        mbar_init(&mbar, 1);
        fence_barrier_init();
    }
    const int cv = src.f32 ? 1 : src.C / 8;   // chunks carrying channels
    {
        // unit (a, g, n) of the layout is row n of tap row t(g) of a; a = (dy, dx,
        // chunk), or (px, g, c) of the paired taps
        const uint4* w4 = reinterpret_cast<const uint4*>(pair ? Wpair : Wu);
        const int na = pair ? 3 * 2 * 2 : 9 * C8P;
        for (int i = tid; i < na * kGroups * NP; i += kT) {
            const int n = i % NP, ag = i / NP, a = ag / kGroups, g = ag - a * kGroups;
            sW[i] = w4[((5 - g) % 3 * na + a) * NP + n];
        }
        const int pad = (C8P - cv) * kHV;
        for (int q = 0; q < kSlots; ++q)
            for (int i = tid; i < pad; i += kT) sH[q * G::kPlane + cv * kHV + i] = make_uint4(0, 0, 0, 0);
    }
    fence_proxy_async_smem();   // generic-proxy writes -> visible to the tensor core
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_base_s;
    const uint32_t sW_a = smem_u32(sW), sH_a = smem_u32(sH);
    const float osc = oscale ? *oscale : 1.f;
    const float fsc = src.f32 && src.f32_scale ? *src.f32_scale : 1.f;
    const int sh = src.up ? 1 : 0;
    const long long plane8 = (long long)(src.H >> sh) * (src.W >> sh) * cv;   // 16-byte units of a source plane
    const uint4* ga = reinterpret_cast<const uint4*>(src.a);
    const uint4* gb = reinterpret_cast<const uint4*>(src.b);

    int j = 0;   // planes so far: staged slot j & 1, phase j & 1 of the barrier
    bool ok = true;
    auto wait_plane = [&](int t) {   // plane t's MMAs have completed (one thread spins)
        ok = __syncthreads_and(tid != 0 || mbar_wait(&mbar, t & 1, status));
        tc_fence_after();
        return ok;
    };
    const bool rev = src.flip && !pair;   // (the paired weights hold the flip)
    auto real = [&](int p) { return rev ? src.D - 1 - p : p; };   // the walk's plane p
    // this CTA's run of the ntx x nty columns' planes
    const long long total = (long long)ntx * nty * src.D;
    long long pos = total * blockIdx.x / gridDim.x;
    const long long end = total * (blockIdx.x + 1) / gridDim.x;
    while (pos < end && ok) {
        const int q = (int)(pos / src.D), zb = (int)(pos - (long long)q * src.D);
        const int ze = (int)min((long long)src.D, zb + (end - pos)), x0 = (q % ntx) * kX, y0 = (q / ntx) * kY;
        pos += ze - zb;
        // this thread's units: place in a source plane (-1: outside) and in a slot
        int goff[U], soff[U];
#pragma unroll
        for (int k = 0; k < U; ++k) {
            const int i = tid + k * kT, hv = i / cv, c = i - hv * cv;
            const int xx = x0 + hv % kHX - 1, yy = y0 + hv / kHX - 1;
            const bool in = (unsigned)xx < (unsigned)src.W && (unsigned)yy < (unsigned)src.H;
            soff[k] = i < kHV * cv ? c * kHV + hv : -1;
            goff[k] = in ? ((yy >> sh) * (src.W >> sh) + (xx >> sh)) * cv + c : -1;
        }
        uint4 va[U], vb[U];
        auto fetch = [&](int z) {   // register-staged sources: the loads of source plane z
            if (!src.b && !src.f32) return;
            const bool zin = (unsigned)z < (unsigned)src.D;
#pragma unroll
            for (int k = 0; k < U; ++k) {
                const bool use = zin && soff[k] >= 0 && goff[k] >= 0;
                va[k] = vb[k] = make_uint4(0, 0, 0, 0);
                if (src.f32) {
                    if (use) va[k].x = __float_as_uint(__ldg(src.f32 + z * plane8 + goff[k]));
                } else if (use) {
                    va[k] = __ldg(ga + z * plane8 + goff[k]);
                    vb[k] = __ldg(gb + z * plane8 + goff[k]);
                }
            }
        };
        auto put = [&](int z, int slot) {   // the plane into its slot
            uint4* d = sH + slot * G::kPlane;
            const bool zin = (unsigned)z < (unsigned)src.D;
#pragma unroll
            for (int k = 0; k < U; ++k) {
                if (soff[k] < 0) continue;
                const bool in = zin && goff[k] >= 0;
                if (src.f32) {
                    // (a zero outside the volume stays +0 whatever the scale's sign)
                    const __nv_bfloat16 b = __float2bfloat16(__uint_as_float(va[k].x) * fsc);
                    d[soff[k]] = make_uint4(in ? (uint32_t)(*reinterpret_cast<const uint16_t*>(&b)) : 0u, 0, 0, 0);
                } else if (src.b) {
                    __nv_bfloat162* pr = reinterpret_cast<__nv_bfloat162*>(&va[k]);
                    const __nv_bfloat162* pq = reinterpret_cast<const __nv_bfloat162*>(&vb[k]);
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const float2 a = __bfloat1622float2(pr[e]), b = __bfloat1622float2(pq[e]);
                        pr[e] = __floats2bfloat162_rn(a.x + b.x, a.y + b.y);
                    }
                    d[soff[k]] = va[k];
                } else {
                    cp_async16(d + soff[k], ga + (in ? (z >> sh) * plane8 + goff[k] : 0), in ? 16u : 0u);
                }
            }
        };
        fetch(real(zb - 1));
        put(real(zb - 1), j & 1);
        const int m = 32 * warp + (tid & 31), ex = x0 + m % kX, ey = y0 + m / kX;   // this thread's output voxel
        const uint32_t tlane = tmem + ((uint32_t)(32 * warp) << 16);
        __syncwarp();   // (staging skips the units a lane does not have)
#pragma unroll
        for (int c0 = 0; c0 < 3 * NP; c0 += 16) tmem_zero16(tlane + (uint32_t)c0);
        for (int p = zb - 1; p <= ze; ++p, ++j) {
            tmem_st_wait();
            cp_async_wait_all();
            fence_proxy_async_smem();
            tc_fence_before();
            __syncthreads();
            if (warp == 0 && elect_one()) {
                tc_fence_after();
                issue_mmas<C8P, NP>(tmem, sH_a + (uint32_t)((j & 1) * G::kPlane * 16), sW_a, 2 - (p + 1) % 3, sgn, pair,
                                    &mbar);
            }
            if (p < ze) {   // into the other slot, whose MMAs have completed
                fetch(real(p + 1));
                put(real(p + 1), (j + 1) & 1);
            }
            if (!wait_plane(j)) break;
            const uint32_t acc = (uint32_t)((p + 2) % 3 * NP);   // output p - 1
            if (p > zb) {
                epilogue<NP>(src, tmem + acc, real(p - 1), ey, ex, N, bias, relu, osc, out);
            } else {
#pragma unroll
                for (int c0 = 0; c0 < NP; c0 += 16) tmem_zero16(tlane + acc + (uint32_t)c0);
            }
        }
        if (!ok) break;
        tmem_st_wait();
    }
    cp_async_wait_all();   // no copy lands after the CTA has gone
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        tmem_dealloc(tmem, G::kCols);
    }
}

}  // namespace umma
}  // namespace unet
}  // namespace mh3d
