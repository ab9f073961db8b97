"""The drive-axis passes of any subset factor, up to eight harmonics a round,
against the FP64 oracle: one harmonic, rounds that are exactly full and last
rounds of one and of several harmonics, portrait rows of 1 to 108 samples
(none, one and two transform stages), 16 and 8 row pairs a CTA, row counts
that leave a ragged last CTA.

Tolerance 1e-5 (relative L2), as for the passes' other lengths: at most six
transforms of at most four stages, a few roundings of 2^-24 each."""
import pytest

import oracle
import workloads as W
from tests._cases import gpu_plan, oracle_geom, params, rel_l2, sens_map

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

TOL = 1e-5
CASES = {
    "s6_k1": params((96, 3, 9), s=6, r=1, kmin=2, kmax=2, theta=[0.3]),
    "s8_k8": params((64, 12, 8), s=8, r=3, kmin=2, kmax=9),
    "s12_k9": params((108, 6, 4), s=12, r=11, kmin=2, kmax=10),
    "s6_k17": params((162, 4, 9), s=6, kmin=2, kmax=18),
    "s16_one_sample": params((16, 6, 4), s=16, r=5, kmin=2, kmax=6),
    "s6_8_pairs": params((192, 144, 96), s=6, kmin=2, kmax=5),
    "short_k9": params((16, 81, 64), s=1, kmin=2, kmax=10),
    "short_k11": params((54, 27, 16), s=1, kmin=2, kmax=12),
    "short_s3": params((162, 9, 8), s=3, r=2, kmin=2, kmax=4),
    "row96": params((96, 18, 16), s=1, kmin=2, kmax=6),
    "row108": params((216, 9, 4), s=2, r=1, kmin=2, kmax=6),
    "short_s4": params((32, 36, 27), s=4, r=1, kmin=2, kmax=17),
    "short_ragged": params((18, 3, 9), s=2, r=1, kmin=2, kmax=6),
}


@pytest.mark.parametrize("name", list(CASES))
def test_rounds_match_oracle(name):
    from paper_2503_13802_gb300 import mh3d_adjoint, mh3d_forward

    p = CASES[name]
    g = oracle_geom(p)
    b = sens_map(p)
    plan = gpu_plan(p, b)
    x, y = W.random_volume(g.shape, 51), W.random_portraits(g.portrait_shape, 52)
    d = torch.empty(g.portrait_shape, dtype=torch.complex64, device="cuda")
    mh3d_forward(plan, torch.as_tensor(x, dtype=torch.float32, device="cuda").contiguous(), d)
    assert rel_l2(d.cpu().numpy(), oracle.forward(g, x, b)) <= TOL
    rho = torch.empty(g.shape, dtype=torch.float32, device="cuda")
    mh3d_adjoint(plan, torch.as_tensor(y, dtype=torch.complex64, device="cuda").contiguous(), rho)
    assert rel_l2(rho.cpu().numpy(), oracle.adjoint(g, y, b)) <= TOL
