// Weight layouts of the tcgen05 convolution (umma_conv.cuh).
#include "umma_launch.h"

namespace mh3d {
namespace unet {
namespace {

// The paired-tap weights of a source of at most 8 channels:
// Wp[pz][px][g][c][n][j], plane offsets (pz, p, px) of the halo, p = 0 and 1
// for g = 0 (c = 0, 1) and p = 2 for g = 1 (c = 0; c = 1 zero); the tap is
// the one applied at offset (pz - 1, p - 1, px - 1) = sgn (dz, dy, dx).
__global__ void k_prep_umma_pair(const __nv_bfloat16* __restrict__ Wt, int Npad, int Cs, int N, int NP, int sgn,
                                 __nv_bfloat16* __restrict__ Wp)
{
    const int total = 9 * 2 * 2 * NP * 8;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= total) return;
    const int j = i % 8, n = (i / 8) % NP, c = (i / (8 * NP)) % 2, g = (i / (16 * NP)) % 2, pzx = i / (32 * NP);
    const int pz = pzx / 3, px = pzx % 3;
    const int p = g == 0 ? c : (c == 0 ? 2 : -1);
    __nv_bfloat16 v = __float2bfloat16(0.f);
    if (p >= 0 && j < Cs && n < N) {
        const int dz = sgn * (pz - 1), dy = sgn * (p - 1), dx = sgn * (px - 1);
        const int tap = 9 * (dz + 1) + 3 * (dy + 1) + (dx + 1);
        v = Wt[(size_t)(tap * Cs + j) * Npad + n];
    }
    Wp[i] = v;
}

// Wu[tap][c][n][j] = Wt[(tap * Cs + 8 c + j) * Npad + n] (zero past Cs
// source channels or N output channels); Wt is the implicit-GEMM matrix
// [Kpad][Npad] of the mma.sync kernels (forward or input-gradient layout).
__global__ void k_prep_umma(const __nv_bfloat16* __restrict__ Wt, int Npad, int Cs, int N, int C8P, int NP,
                            __nv_bfloat16* __restrict__ Wu)
{
    const int total = 27 * C8P * NP * 8;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= total) return;
    const int j = i % 8, n = (i / 8) % NP, c = (i / (8 * NP)) % C8P, tap = i / (8 * NP * C8P);
    const int ci = 8 * c + j;
    __nv_bfloat16 v = __float2bfloat16(0.f);
    if (ci < Cs && n < N) v = Wt[(size_t)(tap * Cs + ci) * Npad + n];
    Wu[i] = v;
}

unsigned prep_blocks(int n) { return (unsigned)((n + 255) / 256); }

}  // namespace

void launch_prep_umma(const __nv_bfloat16* Wt, int Npad, int Cs, int N, const UmmaW& u, cudaStream_t st)
{
    k_prep_umma<<<prep_blocks(27 * u.c8p * u.np * 8), 256, 0, st>>>(Wt, Npad, Cs, N, u.c8p, u.np, u.w);
    if (u.wp) k_prep_umma_pair<<<prep_blocks(9 * 2 * 2 * u.np * 8), 256, 0, st>>>(Wt, Npad, Cs, N, u.np, u.sgn, u.wp);
}

}  // namespace unet
}  // namespace mh3d
