"""Element offsets of the halo convolutions' source reads (halo_index.h), on
the host against Python's integers: every halo voxel inside the volume, for
blocks in the corners and the middle, at sizes where a slice or a row alone
passes 2^31 elements.  (An offset formed in 32 bits is 4 GB off there:
4 x 2898 x 2898 x 64 = 2^31 + 2,507,776.)"""
import ctypes
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2503_13802_gb300", "csrc")
SOURCE = """
#include "halo_index.h"
using namespace mh3d::unet;
extern "C" long long element(int x0, int y0, int z0, int hx, int hy, int hz, int sh, int Hs, int Ws, int C, int c)
{
    return halo_elem(halo_base(x0, y0, z0, sh, Hs, Ws), 0, C, c) + halo_elem(0, halo_rel(hx, hy, hz, sh, Hs, Ws), C, 0);
}
"""
# (nx, ny, nz), channels, upsampled, rows of a block (8: resident weights, 4: streamed)
CASES = [
    ((2898, 2898, 5), 64, 0, 8),
    ((2048, 2048, 9), 128, 0, 4),
    ((8192, 8192, 5), 16, 0, 8),
    ((2097152, 11, 6), 128, 0, 4),
    ((4100, 4100, 60), 64, 1, 8),
    ((1073741822, 1, 1), 8, 0, 8),
    ((10, 14, 6), 16, 1, 8),
]


@pytest.fixture(scope="module")
def element(tmp_path_factory):
    from paper_2503_13802_gb300 import build

    if not os.path.exists(build.nvcc()):
        pytest.skip("nvcc not available")
    d = tmp_path_factory.mktemp("halo")
    src, so = str(d / "halo.cu"), str(d / "halo.so")
    with open(src, "w") as f:
        f.write(SOURCE)
    subprocess.run([build.nvcc(), "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-I" + CSRC, "-o", so, src], check=True)
    f = ctypes.CDLL(so).element
    f.restype = ctypes.c_longlong
    return f


@pytest.mark.parametrize("n,C,up,TY", CASES)
def test_halo_offsets_are_exact(n, C, up, TY, element):
    W, H, D = n
    Ws, Hs = W >> up, H >> up

    def origins(m, step):
        last = (m - 1) // step * step
        return sorted({0, last // 2 // step * step, last})

    for x0 in origins(W, 8):
        for y0 in origins(H, TY):
            for z0 in origins(D, 4):
                for hz in range(6):
                    for hy in range(TY + 2):
                        for hx in (0, 1, 8, 9):
                            x, y, z = x0 - 1 + hx, y0 - 1 + hy, z0 - 1 + hz
                            if not (0 <= x < W and 0 <= y < H and 0 <= z < D):
                                continue
                            want = (((z >> up) * Hs + (y >> up)) * Ws + (x >> up)) * C + C - 8
                            assert element(x0, y0, z0, hx, hy, hz, up, Hs, Ws, C, C - 8) == want, (x, y, z)
