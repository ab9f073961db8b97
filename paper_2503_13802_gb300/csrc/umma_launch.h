// Launches of the tcgen05 convolution (umma_conv.cuh).  The kernel's
// instantiations are compiled in files of their own, one per (chunk planes,
// accumulator columns): umma_c2_n16.cu .. umma_c4_n64.cu.
#pragma once

#include <algorithm>
#include <cstdlib>

#include "mh3d_internal.h"
#include "unet_kernels.cuh"

namespace mh3d {
namespace unet {

// Weights of one convolution in the tcgen05 kernel's B-operand layout
// ([27][c8p][np][8] bfloat16, umma_conv.cuh); w null: that kernel is not
// used for it.
struct UmmaW {
    __nv_bfloat16* w = nullptr;
    __nv_bfloat16* wp = nullptr;   // paired-tap layout (sources of at most 8 channels), or null
    int c8p = 0, np = 0;
    int sgn = 1;                   // -1: the input-gradient (flipped) operand
};

inline int smem_optin()
{
    static int v = -1;
    if (v < 0) {
        int dev = 0;
        cudaGetDevice(&dev);
        if (cudaDeviceGetAttribute(&v, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess) v = 48 * 1024;
    }
    return v;
}

// Paired taps for sources of at most 8 channels (MH3D_UMMA_PAIR=0: off).
inline bool umma_pair()
{
    const char* e = std::getenv("MH3D_UMMA_PAIR");
    return !(e && e[0] == '0');
}

// One convolution (OutT float or __nv_bfloat16) with its operands in u.
template <int C8P, int NP, class OutT>
cudaError_t launch_umma_nb(const ConvSrc& s, const UmmaW& u, int N, const float* bias, int relu, const float* oscale,
                           OutT* out, int* status, cudaStream_t st);

// The operands' layouts (Wt: the implicit-GEMM matrix of the mma.sync kernels).
void launch_prep_umma(const __nv_bfloat16* Wt, int Npad, int Cs, int N, const UmmaW& u, cudaStream_t st);

}  // namespace unet
}  // namespace mh3d
