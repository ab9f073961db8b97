// Places of a convolution block's halo in its source volume.
#pragma once

#include <cstdint>

#include <cuda_runtime.h>

namespace mh3d {
namespace unet {

// Halo voxel (hx, hy, hz) of a block, counted in source voxels from the
// block's first voxel; Hs x Ws is a source plane, sh = 1 reads a half-resolution source
// (block origins are even, so halving commutes with the offset).  A volume has
// fewer than 2^30 voxels, so the offset of any voxel inside it fits; one that
// lies outside may wrap (unsigned arithmetic) and is never read.
__host__ __device__ __forceinline__ int halo_rel(int hx, int hy, int hz, int sh, int Hs, int Ws)
{
    const uint32_t z = (uint32_t)((hz - 1) >> sh), y = (uint32_t)((hy - 1) >> sh), x = (uint32_t)((hx - 1) >> sh);
    return (int)((z * (uint32_t)Hs + y) * (uint32_t)Ws + x);
}

// The block's first voxel (x0, y0, z0) in the source.
__host__ __device__ __forceinline__ long long halo_base(int x0, int y0, int z0, int sh, int Hs, int Ws)
{
    return ((long long)(z0 >> sh) * Hs + (y0 >> sh)) * Ws + (x0 >> sh);
}

// The element of channel c: 64 bits, since C channels of 2^30 voxels are not
// counted in 32.
__host__ __device__ __forceinline__ long long halo_elem(long long base, int rel, int C, int c)
{
    return (base + rel) * C + c;
}

}  // namespace unet
}  // namespace mh3d
