"""The four-wide vector kernels' edges: lengths around multiples of four and of
the grid, and vectors that are not 16-byte aligned (one element a thread).
The sums are float-pair products and pair additions: exact products, a
relative error of about 2^-44 per addition against the sum of the magnitudes;
1e-11 of it leaves room for the 2^17 additions of the longest."""
import numpy as np
import pytest

from tests._cases import gpu_plan, params

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n", [1, 3, 4, 5, 1023, 4098, 100003])
@pytest.mark.parametrize("off", [0, 1])
def test_dot_of_any_length_and_alignment(n, off):
    from paper_2503_13802_gb300 import mh3d_dot

    g = torch.Generator(device="cuda").manual_seed(n + off)
    a = torch.randn(n + 1, generator=g, device="cuda")[off:off + n]
    b = torch.randn(n + 1, generator=g, device="cuda")[:n]
    a64, b64 = a.cpu().numpy().astype(np.float64), b.cpu().numpy().astype(np.float64)
    plan = gpu_plan(params((36, 18, 6), kmin=2, kmax=3))
    got = mh3d_dot(plan, a, b)
    assert abs(got - float(np.dot(a64, b64))) <= 1e-11 * float(np.dot(np.abs(a64), np.abs(b64)))
