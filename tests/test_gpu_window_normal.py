"""The drive-axis normal pass of padded plans (portraits in shared memory only)
against the FP64 oracle: every subset factor of its own kernel, one harmonic,
a last round that is not full, row groups inside, across and outside the
window, an odd row count, and solves of a fixed and a tolerance-driven length.

Tolerance 1e-5 (relative L2), as for the passes that it joins: six transforms
of at most four stages, a few roundings of 2^-24 each."""
import numpy as np
import pytest

import oracle
import workloads as W
from tests._cases import oracle_geom, params, rel_l2

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

TOL = 1e-5


@pytest.mark.parametrize("p,pad", [
    (params((36, 5, 7), s=1, kmin=2, kmax=2, theta=[0.7]), (0, 2, 1)),
    (params((128, 20, 9), s=2, kmin=2, kmax=9), (8, 2, 0)),
    (params((60, 50, 3), s=2, r=1, kmin=2, kmax=18), (6, 2, 3)),
    (params((66, 7, 11), s=3, r=1, kmin=2, kmax=6), (3, 1, 8)),
    (params((136, 16, 5), s=4, r=3, kmin=2, kmax=4), (4, 16, 2)),
])
def test_window_normal_matches_oracle(p, pad):
    from paper_2503_13802_gb300 import Plan, make_opts, mh3d_normal, mh3d_solve

    g = oracle_geom(p)
    ge = oracle.padded_geometry(g, pad)
    b = W.sensitivity(tuple(ge.n), ge.voxel_mm, kind="gaussian")
    plan = Plan(p["n"], voxel_mm=p["voxel"], ds_factor=p["s"], ds_offset=p["r"], k_min=p["kmin"], k_max=p["kmax"],
                gamma_per_mm=p["gamma"], gammaA=p["gammaA"], transverse_ratio=p["tratio"], theta=p["theta"],
                sensitivity=b, pad=pad)
    x = W.random_volume(ge.shape, 31)
    xd = torch.as_tensor(x, dtype=torch.float32, device="cuda").contiguous()
    q = torch.empty(ge.shape, dtype=torch.float32, device="cuda")
    mh3d_normal(plan, xd, q, make_opts(lam=2e-2, reg_kind=0, normal_mode=1))
    clean = oracle.padded_forward(g, pad, x, b)
    ref = oracle.padded_adjoint(g, pad, clean, b) + 2e-2 * np.asarray(x)
    assert rel_l2(q.cpu().numpy(), ref) <= TOL
    # a fixed count of iterations and a tolerance that the same count meets
    d = torch.as_tensor(clean.astype(np.complex64), device="cuda").contiguous()
    a, c = (torch.empty(ge.shape, dtype=torch.float32, device="cuda") for _ in range(2))
    info = mh3d_solve(plan, d, make_opts(lam=1e-2, lam_relative=True, max_iter=5, fixed_iters=True), a)
    assert info["iters"] == 5 and len(info["history"]) == 6
    info = mh3d_solve(plan, d, make_opts(lam=1e-2, lam_relative=True, max_iter=5, rel_tol=1e-30), c)
    assert info["iters"] == 5
    assert torch.equal(a, c)
