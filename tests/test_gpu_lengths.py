"""The run-time passes over the lengths where they change form, against the
FP64 oracle: transforms of no, one, two, three and four stages, odd x lengths,
every subset factor with its own kernel (1 to 4) and one without (6), more
harmonics than a round holds, columns and rows that leave ragged tiles,
padded plans whose passes read the field of view's window.

Tolerance 1e-5 (relative L2): an output passes through at most six transforms
of at most four stages, each adding a few roundings of 2^-24 relative, about
24 x 4 x 6e-8 = 6e-6 at worst and their root sum, 1e-6, as a rule."""
import numpy as np
import pytest

import oracle
import workloads as W
from tests._cases import gpu_plan, oracle_geom, params, rel_l2, sens_map

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

TOL = 1e-5
CASES = {
    "two_stage": params((36, 18, 54), s=1, kmin=2, kmax=4),
    "one_stage": params((12, 16, 9), s=2, r=1, kmin=2, kmax=3, theta=[0.4, -1.2]),
    "odd_x": params((81, 6, 27), s=3, r=2, kmin=2, kmax=4),
    "s4": params((144, 6, 36), s=4, r=1, kmin=2, kmax=8),
    "s6": params((108, 4, 12), s=6, r=5, kmin=2, kmax=4),
    "rounds": params((24, 9, 48), s=1, kmin=2, kmax=17),
    "three_stage": params((324, 4, 6), s=2, kmin=2, kmax=3),
    "four_stage": params((729, 2, 3), s=3, r=1, kmin=2, kmax=3),
    "longest": params((1024, 2, 2), s=4, kmin=2, kmax=3),
    "long_yz": params((8, 648, 3), s=2, kmin=2, kmax=3),
    "unit_yz": params((54, 1, 1), s=2, r=1, kmin=2, kmax=4),
}


def _dev(a, dtype):
    return torch.as_tensor(np.ascontiguousarray(a)).to(device="cuda", dtype=dtype).contiguous()


@pytest.mark.parametrize("name", list(CASES))
def test_run_time_passes_match_oracle(name):
    from paper_2503_13802_gb300 import make_opts, mh3d_adjoint, mh3d_forward, mh3d_normal

    p = CASES[name]
    g = oracle_geom(p)
    b = sens_map(p)
    plan = gpu_plan(p, b)
    x, y = W.random_volume(g.shape, 11), W.random_portraits(g.portrait_shape, 12)
    d = torch.empty(g.portrait_shape, dtype=torch.complex64, device="cuda")
    mh3d_forward(plan, _dev(x, torch.float32), d)
    assert rel_l2(d.cpu().numpy(), oracle.forward(g, x, b)) <= TOL
    rho = torch.empty(g.shape, dtype=torch.float32, device="cuda")
    mh3d_adjoint(plan, _dev(y, torch.complex64), rho)
    assert rel_l2(rho.cpu().numpy(), oracle.adjoint(g, y, b)) <= TOL
    q = torch.empty(g.shape, dtype=torch.float32, device="cuda")
    for kind in (0, 1):
        oo = oracle.SolveOpts(lam=2e-2, reg_kind=kind, alpha=0.7)
        for mode in (0, 1):
            mh3d_normal(plan, _dev(x, torch.float32), q, make_opts(lam=2e-2, reg_kind=kind, alpha=0.7,
                                                                  normal_mode=mode))
            assert rel_l2(q.cpu().numpy(), oracle.normal_apply(g, x, b, oo)) <= TOL, (kind, mode)


@pytest.mark.parametrize("p,pad", [
    (params((24, 12, 36), s=1, kmin=2, kmax=4), (6, 3, 9)),
    (params((120, 4, 24), s=4, r=1, kmin=2, kmax=8), (12, 1, 6)),
    (params((63, 5, 21), s=3, r=2, kmin=2, kmax=4), (9, 2, 3)),
    (params((4, 12, 9), s=2, r=1, kmin=2, kmax=3, theta=[0.4, -1.2]), (4, 2, 0)),
])
def test_windowed_passes_of_padded_plans_match_oracle(p, pad):
    """The passes read and write the field of view's portraits inside the
    extended grid (sizes without specialised kernels)."""
    from paper_2503_13802_gb300 import Plan, make_opts, mh3d_adjoint, mh3d_forward, mh3d_normal

    g = oracle_geom(p)
    ge = oracle.padded_geometry(g, pad)
    b = W.sensitivity(tuple(ge.n), ge.voxel_mm, kind="gaussian")
    plan = Plan(p["n"], voxel_mm=p["voxel"], ds_factor=p["s"], ds_offset=p["r"], k_min=p["kmin"], k_max=p["kmax"],
                gamma_per_mm=p["gamma"], gammaA=p["gammaA"], transverse_ratio=p["tratio"], theta=p["theta"],
                sensitivity=b, pad=pad)
    x, y = W.random_volume(ge.shape, 21), W.random_portraits(g.portrait_shape, 22).astype(np.complex64)
    d = torch.empty(g.portrait_shape, dtype=torch.complex64, device="cuda")
    mh3d_forward(plan, _dev(x, torch.float32), d)
    assert rel_l2(d.cpu().numpy(), oracle.padded_forward(g, pad, x, b)) <= TOL
    rho = torch.empty(ge.shape, dtype=torch.float32, device="cuda")
    mh3d_adjoint(plan, _dev(y, torch.complex64), rho)
    assert rel_l2(rho.cpu().numpy(), oracle.padded_adjoint(g, pad, y.astype(np.complex128), b)) <= TOL
    q = torch.empty(ge.shape, dtype=torch.float32, device="cuda")
    mh3d_normal(plan, _dev(x, torch.float32), q, make_opts(lam=2e-2, reg_kind=0, normal_mode=1))
    ref = oracle.padded_adjoint(g, pad, oracle.padded_forward(g, pad, x, b), b) + 2e-2 * np.asarray(x)
    assert rel_l2(q.cpu().numpy(), ref) <= TOL
