"""Padded plans whose passes read and write the field of view's window, in the
forms with passes of their own: portrait lengths of three radices (no joint
normal pass), subset factors from five on, short portrait rows, each with both
priors, against the FP64 oracle.

Tolerance 1e-5 (relative L2), as for the other lengths: at most six transforms
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
    (params((300, 4, 3), s=2, r=1, kmin=2, kmax=6), (12, 2, 0)),     # 162 samples: three radices
    (params((420, 3, 4), s=2, kmin=2, kmax=4), (6, 0, 1)),           # 216
    (params((84, 4, 10), s=6, r=5, kmin=2, kmax=4), (12, 1, 1)),
    (params((80, 7, 8), s=8, r=2, kmin=2, kmax=12), (8, 1, 0)),
    (params((36, 5, 7), s=2, r=1, kmin=2, kmax=11), (6, 2, 1)),      # rows of 24 samples
])
def test_windowed_forms_match_oracle(p, pad):
    from paper_2503_13802_gb300 import Plan, make_opts, mh3d_adjoint, mh3d_forward, mh3d_normal

    g = oracle_geom(p)
    ge = oracle.padded_geometry(g, pad)
    b = W.sensitivity(tuple(ge.n), ge.voxel_mm, kind="gaussian")
    plan = Plan(p["n"], voxel_mm=p["voxel"], ds_factor=p["s"], ds_offset=p["r"], k_min=p["kmin"], k_max=p["kmax"],
                gamma_per_mm=p["gamma"], gammaA=p["gammaA"], transverse_ratio=p["tratio"], theta=p["theta"],
                sensitivity=b, pad=pad)
    x, y = W.random_volume(ge.shape, 61), W.random_portraits(g.portrait_shape, 62).astype(np.complex64)
    xd = torch.as_tensor(x, dtype=torch.float32, device="cuda").contiguous()
    d = torch.empty(g.portrait_shape, dtype=torch.complex64, device="cuda")
    mh3d_forward(plan, xd, d)
    clean = oracle.padded_forward(g, pad, x, b)
    assert rel_l2(d.cpu().numpy(), clean) <= TOL
    rho = torch.empty(ge.shape, dtype=torch.float32, device="cuda")
    mh3d_adjoint(plan, torch.as_tensor(y, device="cuda").contiguous(), rho)
    assert rel_l2(rho.cpu().numpy(), oracle.padded_adjoint(g, pad, y.astype(np.complex128), b)) <= TOL
    nx = oracle.padded_adjoint(g, pad, clean, b)
    q = torch.empty(ge.shape, dtype=torch.float32, device="cuda")
    for kind in (0, 1):
        mh3d_normal(plan, xd, q, make_opts(lam=2e-2, reg_kind=kind, alpha=0.7, normal_mode=1))
        ref = nx + 2e-2 * oracle.reg_apply(ge, np.asarray(x, dtype=np.float64), kind, 0.7, 2)
        assert rel_l2(q.cpu().numpy(), ref) <= TOL, kind
