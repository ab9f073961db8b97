"""Performance cases: the work that a user of this framework has it do, each
case one call (or one training step) through the public entry points.

Every case is a dict of plain values.  `kind` names the entry point:
  forward, adjoint   the portrait operators A and A^T (mh3d_forward, mh3d_adjoint)
  solve              conjugate gradients on the normal equations (mh3d_solve)
  apg                the paper's accelerated projected gradient (mh3d_solve, solver 1)
  batch              many volumes in one call (mh3d_solve_batched)
  general            conjugate gradients on the three-component model with
                     caller-supplied PSFs (mh3d_general_solve)
  infer, train       the learned warm start's network: inference, and one
                     gradient and Adam step
`nx, ny, nz` is the field of view, `s` / `r` the drive-axis downsampling and
its offset, `K` the number of harmonics (k = 2 .. K + 1), `sens` whether a
receive sensitivity weights the volume, `px, py, pz` the boundary padding per
side.  Iterative cases run a fixed number of iterations, as the
fixed-iteration workload of `workloads` does, so that a pass is the same
amount of work on any code.

`exact` restates the model in FP64 with numpy and torch alone: the Langevin
derivatives by their pole sum, circular convolutions by torch's FFT, plain CG
and projected gradient, torch's conv3d for the network.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2503_13802_gb300 import mh3d as M
from paper_2503_13802_gb300.unet import UNet

GAMMA, GAMMA_A, RATIO = 1.387016, 2.0, 0.5   # the package's default scanner (1 mm voxels)
LAM = 1e-3                                   # regularisation weight relative to ||A||^2, as in the workloads
SNR_DB = 25.0
GAIN = 0.5                                   # output gain of the scaled network calls
# lengths 2^a 3^b from 16 to 256, roughly evenly spaced in their logarithm
LENGTHS = (16, 18, 24, 27, 32, 36, 48, 54, 64, 72, 81, 96, 108, 128, 144, 162, 192, 216, 243, 256)
BATCH_CLASSES = ((64, 64, 64), (96, 96, 64), (128, 128, 64), (192, 192, 96))   # workloads.BATCH_SIZE_CLASSES


def _case(name, kind, n, **kw):
    c = dict(name=name, kind=kind, nx=n[0], ny=n[1], nz=n[2], s=1, r=0, K=4, sens=False, px=0, py=0, pz=0, iters=0)
    c.update(kw)
    return c


def listed():
    return [
        # the smallest volume of the workloads: previews and tests; launch and call latency
        _case("forward_32", "forward", (32, 32, 32)),
        # one forward model of the benchmark workload: simulating a scan, checking a fit
        _case("forward_128", "forward", (128, 128, 64), s=2, K=8, sens=True),
        # its adjoint: a back-projection image, the right-hand side of every solve, the network's input
        _case("adjoint_128", "adjoint", (128, 128, 64), s=2, K=8, sens=True),
        # the precision workload: a large head-sized volume, all rows kept, sixteen harmonics
        _case("forward_256", "forward", (256, 256, 128), K=16),
        # a grid of mixed 2- and 3-powers kept every third row with an offset: a scanner whose
        # field of view is no power of two
        _case("adjoint_ragged", "adjoint", (162, 108, 81), s=3, r=1, K=5, sens=True),
        # the benchmark: one reconstruction of the 128 x 128 x 64 workload from device portraits
        _case("solve_128", "solve", (128, 128, 64), s=2, K=8, sens=True, iters=12),
        # the same field of view with boundary padding (model grid 144 x 144 x 72), the paper's remedy
        # for objects at the edge
        _case("solve_padded", "solve", (128, 128, 64), s=2, K=8, sens=True, px=8, py=8, pz=4, iters=6),
        # the paper's own solver: rho >= 0 with the second-difference and boundary prior
        _case("apg_96", "apg", (96, 96, 64), s=2, K=8, sens=True, iters=20),
        # throughput service: eight uneven volumes in one call
        dict(name="batch_8", kind="batch", K=8, s=2, iters=12,
             sizes="64x64x64,128x128x64,96x96x64,192x192x96,64x64x64,96x96x64,128x128x64,64x64x64"),
        # tensor-PSF model: a calibrated or simulated PSF that is not separable
        _case("general_128", "general", (128, 128, 64), s=2, K=8, sens=True, iters=3),
        # the learned warm start at inference: the four-level network of the learned benchmark
        dict(name="infer_128", kind="infer", nx=128, ny=128, nz=64, channels="16,32,64,128"),
        # its training: one gradient and one Adam step of the default three-level network
        dict(name="train_64", kind="train", nx=64, ny=64, nz=64, channels="16,32,64"),
    ]


def _grid(rng, most, least=1 << 12, s_choices=(1, 2, 3, 4)):
    """A grid of LENGTHS of `least` to `most` voxels and a downsampling factor that divides its drive axis."""
    while True:
        n = tuple(rng.choice(LENGTHS) for _ in range(3))
        s = rng.choice(s_choices)
        if n[0] % s == 0 and n[0] // s >= 8 and least <= n[0] * n[1] * n[2] <= most:
            return n, s


def draw(rng):
    """One more case: the operators over grids of 4096 to 8.4 M voxels (2- and 3-powers), 2 to 16 harmonics, s = 1
    to 4; the solvers over grids of up to 1.05 M voxels; batches of 2 to 8 volumes of the four classes; networks of
    three and four levels on grids of 32 to 128 voxels a side."""
    kind = rng.choice(("forward", "adjoint", "forward", "adjoint", "solve", "solve", "apg", "batch", "general",
                       "infer", "train"))
    if kind in ("forward", "adjoint"):
        while True:
            n, s = _grid(rng, 256 * 256 * 128)
            K = rng.randint(2, 16)
            if n[0] * n[1] * n[2] // s * K <= 256 * 256 * 128 * 16:
                break
        c = _case("", kind, n, s=s, r=rng.randrange(s), K=K, sens=rng.random() < 0.6)
    elif kind in ("solve", "apg"):
        n, s = _grid(rng, 128 * 128 * 64, 1 << 15, (1, 2, 2, 3))
        c = _case("", kind, n, s=s, r=rng.randrange(s), K=rng.randint(3, 9), sens=rng.random() < 0.6,
                  iters=rng.randint(4, 12))
    elif kind == "general":
        n, s = _grid(rng, 128 * 128 * 64, 1 << 15, (1, 2, 2, 3))
        c = _case("", kind, n, s=s, r=rng.randrange(s), K=rng.randint(2, 8), sens=rng.random() < 0.6,
                  iters=rng.randint(1, 3))
    elif kind == "batch":
        v = [rng.choice(BATCH_CLASSES) for _ in range(rng.randint(2, 8))]
        while sum(a * b * c for a, b, c in v) > 7_000_000:
            v.remove(max(v))
        c = dict(kind=kind, K=rng.randint(4, 8), s=2, iters=rng.randint(6, 12),
                 sizes=",".join("%dx%dx%d" % t for t in v or [BATCH_CLASSES[0]]))
    else:
        big = kind == "infer"
        base = rng.choice((8, 16))
        ch = [base << l for l in range(rng.choice((3, 4)))]
        while True:
            n = [8 * rng.randint(4, 16) for _ in range(3)]
            if n[0] * n[1] * n[2] <= (1 << 20 if big else 1 << 18):
                break
        c = dict(kind=kind, nx=n[0], ny=n[1], nz=n[2], channels=",".join(map(str, ch)))
    c.pop("name", None)
    return c


# ---------------------------------------------------------------------------
# Inputs (all from the seed)
# ---------------------------------------------------------------------------
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _coords(n):
    return torch.arange(n, device="cuda", dtype=torch.float64) - (n - 1) / 2.0


def _phantom(n, gen, blobs=40):
    """Sum of Gaussian blobs (sigma U(1.5, 4) voxels, amplitude U(0.2, 1)), float32 [nz][ny][nx]."""
    u = torch.rand((5, blobs), generator=gen, device="cuda", dtype=torch.float64)
    sig = 1.5 + 2.5 * u[0]
    g = []
    for a in range(3):
        lim = (n[a] / 2.0 - 3.0 * sig).clamp_min(0.0)
        c = -lim + 2.0 * lim * u[1 + a]
        g.append(torch.exp(-((_coords(n[a])[None] - c[:, None]) ** 2) / (2.0 * sig[:, None] ** 2)))
    return torch.einsum("b,bz,by,bx->zyx", 0.2 + 0.8 * u[4], g[2], g[1], g[0]).float().contiguous()


def _sens(n):
    """Receive sensitivity: a Gaussian of 0.6 of the grid, float32 [nz][ny][nx]."""
    g = [torch.exp(-_coords(m) ** 2 / (2.0 * (0.6 * m) ** 2)) for m in n]
    return (g[2][:, None, None] * g[1][None, :, None] * g[0][None, None, :]).float().contiguous()


def _grid_of(c):
    return (c["nx"] + 2 * c["px"], c["ny"] + 2 * c["py"], c["nz"] + 2 * c["pz"])


def _theta(K):
    return [float(t) for t in np.linspace(-2.5, 2.0, K)]


def _portrait_shape(c):
    return (c["K"], c["nz"], c["ny"], c["nx"] // c["s"])


def _complex_noise(shape, gen):
    return torch.view_as_complex(torch.randn(shape + (2,), generator=gen, device="cuda") * math.sqrt(0.5))


def _noisy(clean, gen):
    """Portraits at SNR_DB: circular complex noise over all harmonics jointly."""
    rms = clean.abs().double().pow(2).mean().sqrt().float()
    return (clean + _complex_noise(tuple(clean.shape), gen) * (rms * 10.0 ** (-SNR_DB / 20.0))).contiguous()


def _plan(c, sens):
    return M.Plan((c["nx"], c["ny"], c["nz"]), ds_factor=c["s"], ds_offset=c["r"], k_min=2, k_max=c["K"] + 1,
                  theta=_theta(c["K"]), sensitivity=sens, pad=(c["px"], c["py"], c["pz"]))


def _volumes(c):
    """The batch's volumes as solve cases."""
    return [_case("", "solve", tuple(map(int, t.split("x"))), s=c["s"], K=c["K"], sens=True, iters=c["iters"])
            for t in c["sizes"].split(",")]


def _general_psf(c):
    """(h_k)_j samples [K][3][nz][ny][nx], float32 on the GPU: the separable harmonic PSFs as the drive component and
    their transverse slopes, scaled, as the other two, so that all three components have a PSF's size and decay."""
    m = _model(_geometry(c))
    x, y, z = m["hx"], m["hy"], m["hz"]
    out = torch.empty((c["K"], 3, c["nz"], c["ny"], c["nx"]), dtype=torch.float32, device="cuda")
    hx, hy, hz = (torch.as_tensor(v, device="cuda") for v in (x, y, z))
    dy = 0.5 * (torch.roll(hy, -1) - torch.roll(hy, 1))
    dz = 0.5 * (torch.roll(hz, -1) - torch.roll(hz, 1))
    for j, (py, pz) in enumerate(((hy, hz), (dy, hz), (hy, dz))):
        t = pz[:, None] * py[None, :]
        for k in range(c["K"]):
            out[k, j] = (t[:, :, None] * hx[k][None, None, :]).float()
    return out


def _general_norm2(c):
    """An upper bound of ||A||^2 of the general model with |b_j| <= 1 (the weight lambda is relative to it)."""
    return 3.0 * _model(_geometry(c))["norm2"]


def _bvec(c, gen):
    """Three smooth sensitivity components (drive-axis coil strongest), float32 [3][nz][ny][nx]."""
    b = _sens(_grid_of(c))
    w = 0.2 + 0.1 * torch.rand(2, generator=gen, device="cuda")
    return torch.stack([b, w[0] * b * b, w[1] * torch.sqrt(b)]).contiguous()


def _channels(c):
    return tuple(int(v) for v in c["channels"].split(","))


def _layers(ch):
    """(cin, cout) of every convolution in parameter order."""
    L = len(ch)
    io = []
    for l in range(L):
        io += [(1 if l == 0 else ch[l - 1], ch[l]), (ch[l], ch[l])]
    for l in range(L - 2, -1, -1):
        io += [(ch[l + 1], ch[l]), (ch[l], ch[l])]
    return io + [(ch[0], 1)]


def _params(ch, gen):
    """He-normal weights and small biases, one flat float32 vector."""
    parts = []
    for ci, co in _layers(ch):
        parts.append(torch.randn(co * 27 * ci, generator=gen, device="cuda") * (2.0 / (27 * ci)) ** 0.5)
        parts.append(torch.randn(co, generator=gen, device="cuda") * 0.02)
    return torch.cat(parts).contiguous()


def _inputs(c, seed):
    """The tensors of one case."""
    g = _gen(seed)
    kind = c["kind"]
    if kind in ("infer", "train"):
        n = (c["nx"], c["ny"], c["nz"])
        # a back-projection-like volume of large, arbitrary scale and a smooth target
        vol = _phantom(n, g) + 0.05 * torch.randn((n[2], n[1], n[0]), generator=g, device="cuda")
        return dict(inp=(300.0 * vol).contiguous(), target=(150.0 * _phantom(n, g)).contiguous(),
                    theta=_params(_channels(c), g))
    if kind == "batch":
        return [_inputs(v, int(seed) * 64 + i) for i, v in enumerate(_volumes(c))]
    sens = _sens(_grid_of(c)) if c["sens"] else None
    if kind == "forward":
        return dict(rho=_phantom(_grid_of(c), g), sens=sens)
    if kind == "adjoint":
        return dict(d=_complex_noise(_portrait_shape(c), g), sens=sens)
    if kind == "general":
        bvec = _bvec(c, g) if c["sens"] else None
        rho = _phantom(_grid_of(c), g)
        h = _general_psf(c)
        clean = _Gen64(c, h, bvec).forward(rho.double()).to(torch.complex64)
        return dict(h=h, bvec=bvec, d=_noisy(clean, g))
    rho = _phantom(_grid_of(c), g)
    clean = _Sep64(c, sens).forward(rho.double()).to(torch.complex64)
    return dict(d=_noisy(clean, g), sens=sens)


def _opts(c):
    if c["kind"] == "apg":
        # the paper's prior (alpha 4, two-voxel shell) and a step below 1 / ||M||^2 that a program keeps per plan
        return M.make_opts(reg_kind=1, alpha=4.0, shell=2, lam=LAM, lam_relative=True, solver=1, max_iter=c["iters"],
                           fixed_iters=True, apg_tau=_apg_tau(c))
    if c["kind"] == "general":
        return M.make_opts(lam=LAM * _general_norm2(c), max_iter=c["iters"], fixed_iters=True)
    return M.make_opts(lam=LAM, lam_relative=True, max_iter=c["iters"], fixed_iters=True)


def _apg_tau(c):
    # lambda_max(T^T T) = 48 for the three periodic second differences, alpha on the shell
    return 0.99 / (_model(_geometry(c))["norm2"] * (1.0 + LAM * (48.0 + 4.0)))


def prepare(case, seed):
    c = case
    kind = c["kind"]
    t = _inputs(c, seed)
    if kind in ("infer", "train"):
        net = UNet((c["nx"], c["ny"], c["nz"]), *_channels(c))
        net.set_params(t["theta"])
        st = dict(kind=kind, net=net, inp=t["inp"])
        if kind == "infer":
            st["out"] = torch.empty(net.shape, dtype=torch.float32, device="cuda")
        else:
            st.update(target=t["target"], grad=torch.empty(net.nparam, dtype=torch.float32, device="cuda"))
        return st
    if kind == "batch":
        plans = [_plan(v, x["sens"]) for v, x in zip(_volumes(c), t)]
        return dict(kind=kind, plans=plans, ds=[x["d"] for x in t], opts=_opts(c),
                    rhos=[torch.empty(p.shape, dtype=torch.float32, device="cuda") for p in plans])
    plan = _plan(c, None if kind == "general" else t["sens"])
    st = dict(kind=kind, plan=plan)
    if kind == "forward":
        st.update(rho=t["rho"], d=torch.empty(plan.portrait_shape, dtype=torch.complex64, device="cuda"))
        return st
    st.update(d=t["d"], rho=torch.empty(plan.shape, dtype=torch.float32, device="cuda"))
    if kind == "general":
        M.mh3d_general_set_psf(plan, t["h"].cpu().numpy())
        st["bvec"] = t["bvec"]
    if kind != "adjoint":
        st["opts"] = _opts(c)
    return st


def run(state):
    kind = state["kind"]
    if kind == "forward":
        return M.mh3d_forward(state["plan"], state["rho"], state["d"])
    if kind == "adjoint":
        return M.mh3d_adjoint(state["plan"], state["d"], state["rho"])
    if kind in ("solve", "apg"):
        info = M.mh3d_solve(state["plan"], state["d"], state["opts"], state["rho"])
        return {"rho": state["rho"], "iters": info["iters"]}
    if kind == "batch":
        infos = M.mh3d_solve_batched(state["plans"], state["ds"], state["opts"], state["rhos"])
        return {"rhos": state["rhos"], "iters": [i["iters"] for i in infos]}
    if kind == "general":
        info = M.mh3d_general_solve(state["plan"], state["d"], state["opts"], state["rho"], bvec=state["bvec"])
        return {"rho": state["rho"], "iters": info["iters"]}
    if kind == "infer":
        state["net"].forward_scaled(state["inp"], GAIN, state["out"])
        return state["out"]
    loss = state["net"].loss_grad_scaled(state["inp"], state["target"], GAIN, grad=state["grad"])
    state["net"].adam_step(1e-3)
    return {"grad": state["grad"], "loss": loss}


# ---------------------------------------------------------------------------
# Work: each input read once, each output written once
# ---------------------------------------------------------------------------
def _fft_flops(n, lines):
    return 5.0 * n * math.log2(max(n, 2)) / 2.0 * lines   # real data: half of a complex transform


def _op_flops(c):
    """One application of A (A^T costs the same): the transverse convolutions, the drive-axis transform, and per
    harmonic a multiply and the transform of the kept rows."""
    nx, ny, nz = _grid_of(c)
    N, mx = nx * ny * nz, nx // c["s"]
    t = 2 * _fft_flops(ny, N // ny) + 2 * _fft_flops(nz, N // nz) + _fft_flops(nx, ny * nz)
    return t + c["K"] * (_fft_flops(mx, ny * nz) + 4.0 * N)


def work(case):
    c = case
    kind = c["kind"]
    if kind in ("infer", "train"):
        ch = _channels(c)
        V = c["nx"] * c["ny"] * c["nz"]
        L = len(ch)
        level = [l for l in range(L) for _ in range(2)] + [l for l in range(L - 2, -1, -1) for _ in range(2)] + [0]
        flops = sum(2.0 * 27 * ci * co * (V >> 3 * l) for (ci, co), l in zip(_layers(ch), level))
        npar = sum(co * 27 * ci + co for ci, co in _layers(ch))
        if kind == "infer":
            return {"bytes": 4.0 * (2 * V + npar), "flops": flops}
        return {"bytes": 4.0 * (2 * V + 7 * npar), "flops": 3.0 * flops}   # parameters, moments and gradient
    if kind == "batch":
        w = [work(v) for v in _volumes(c)]
        return {k: sum(x[k] for x in w) for k in ("bytes", "flops")}
    nx, ny, nz = _grid_of(c)
    N = nx * ny * nz
    KM = c["K"] * c["nz"] * c["ny"] * (c["nx"] // c["s"])
    if kind == "general":
        nb = 3 if c["sens"] else 1
        spectra = 8.0 * c["K"] * nb * N / 2   # the PSF spectra, once (conjugate-symmetric halves)
        f = _fft_flops
        full = f(nx, ny * nz) + f(ny, nx * nz) + f(nz, nx * ny)
        op = (nb + c["K"] / c["s"]) * full + c["K"] * nb * 4.0 * N
        return {"bytes": spectra + 8.0 * KM + 4.0 * N * (1 + (nb if nb == 3 else 0)),
                "flops": (2 * c["iters"] + 1) * op + 10.0 * N * c["iters"]}
    byts = 8.0 * KM + 4.0 * N * (2 if c["sens"] else 1)
    if kind in ("forward", "adjoint"):
        return {"bytes": byts, "flops": _op_flops(c)}
    # A^T d, then per iteration the normal operator (each axis transformed forth and back) and five vector updates
    if c["px"] or c["py"] or c["pz"]:
        it = 2 * _op_flops(c)
    else:
        it = 2 * (_fft_flops(nx, ny * nz) + _fft_flops(ny, nx * nz) + _fft_flops(nz, nx * ny)) + 4.0 * c["s"] * N
    return {"bytes": byts, "flops": _op_flops(c) + c["iters"] * (it + 14.0 * N)}


# ---------------------------------------------------------------------------
# The model in FP64, with numpy and torch alone
# ---------------------------------------------------------------------------
def _langevin_deriv(k, x):
    """L^(k)(x), k >= 1, by the poles of coth at i pi n: sum_n 2 Re[(-1)^k k! (x - i pi n)^-(k+1)], the tail by the
    midpoint Euler-Maclaurin form."""
    x = np.asarray(x, dtype=np.float64)
    NP = 4000
    sg = (-1.0) ** k * math.factorial(k)
    n = np.arange(NP, 0, -1, dtype=np.float64)
    acc = (2.0 * sg * ((x[:, None] - 1j * math.pi * n[None, :]) ** (-(k + 1))).real).sum(axis=1)
    a = NP + 0.5
    z = x - 1j * math.pi * a
    acc += 2.0 * sg * (1j * z ** (-k)).real / (k * math.pi)
    acc -= 2.0 * sg * (1j * math.pi * (k + 1) * z ** (-(k + 2))).real / 24.0
    return acc


def _offsets(n):
    i = np.arange(n, dtype=np.float64)
    return np.where(2 * i < n, i, i - n)


def _geometry(c):
    return _grid_of(c) + (c["s"], c["K"])


@functools.lru_cache(maxsize=64)
def _model(geometry):
    """Sampled one-dimensional kernels and ||A||^2 (b = 1) of a geometry (nx, ny, nz, s, K)."""
    nx, ny, nz, s, K = geometry
    hx = np.stack([GAMMA_A ** k / math.factorial(k - 1) * _langevin_deriv(k, GAMMA * _offsets(nx))
                   for k in range(2, K + 2)])
    hy, hz = (3.0 * _langevin_deriv(1, GAMMA * RATIO * _offsets(n)) for n in (ny, nz))
    X = np.fft.fft(hx, axis=1).reshape(K, s, nx // s)   # bin m + a nx/s at [a][m]
    B = np.einsum("kam,kbm->mab", X.conj(), X) / s
    norm2 = float(np.linalg.eigvalsh(B).max() * (np.abs(np.fft.fft(hy)) ** 2).max()
                  * (np.abs(np.fft.fft(hz)) ** 2).max())
    return dict(hx=hx, hy=hy, hz=hz, norm2=norm2)


def _phases(K):
    return [complex(math.cos(t), math.sin(t)) for t in _theta(K)]


class _Sep64:
    """The separable model's operators on a case's grid."""

    def __init__(self, c, sens):
        self.c = c
        self.m = _model(_geometry(c))
        self.b = None if sens is None else sens.double()
        rf = lambda v: torch.fft.rfft(torch.as_tensor(v, device="cuda"))   # noqa: E731
        self.X, self.Y, self.Z = rf(self.m["hx"]), rf(self.m["hy"]), rf(self.m["hz"])

    def _conv(self, v, H, dim):
        shape = [1, 1, 1]
        shape[dim] = -1
        return torch.fft.irfft(torch.fft.rfft(v, dim=dim) * H.view(shape), n=v.shape[dim], dim=dim)

    def _window(self):
        c = self.c
        p = c["px"] // c["s"]
        return (slice(c["pz"], c["pz"] + c["nz"]), slice(c["py"], c["py"] + c["ny"]),
                slice(p, p + c["nx"] // c["s"]))

    def forward(self, rho):
        c = self.c
        v = rho if self.b is None else rho * self.b
        F = torch.fft.rfft(self._conv(self._conv(v, self.Y, 1), self.Z, 0), dim=2)
        nx = rho.shape[2]
        out = torch.empty(_portrait_shape(c), dtype=torch.complex128, device="cuda")
        for k, ph in enumerate(_phases(c["K"])):
            out[k] = ph * torch.fft.irfft(F * self.X[k], n=nx, dim=2)[..., c["r"]::c["s"]][self._window()]
        return out

    def adjoint(self, d):
        c = self.c
        nx, ny, nz = _grid_of(c)
        acc = 0.0
        for k, ph in enumerate(_phases(c["K"])):
            u = torch.zeros((nz, ny, nx), dtype=torch.float64, device="cuda")
            u[..., c["r"]::c["s"]][self._window()] = (d[k] * ph.conjugate()).real
            acc = acc + torch.fft.rfft(u, dim=2) * self.X[k].conj()
        v = torch.fft.irfft(acc, n=nx, dim=2)
        v = self._conv(self._conv(v, self.Z.conj(), 0), self.Y.conj(), 1)
        return v if self.b is None else v * self.b


class _Gen64:
    """The three-component model's operators."""

    def __init__(self, c, h, bvec):
        self.c = c
        self.H = torch.fft.rfftn(h[:, :3 if bvec is not None else 1].double(), dim=(2, 3, 4))
        self.b = bvec.double() if bvec is not None else None

    def forward(self, rho):
        c = self.c
        w = rho[None] if self.b is None else rho[None] * self.b
        W = torch.fft.rfftn(w, dim=(1, 2, 3))
        out = torch.empty(_portrait_shape(c), dtype=torch.complex128, device="cuda")
        for k, ph in enumerate(_phases(c["K"])):
            out[k] = ph * torch.fft.irfftn((self.H[k] * W).sum(0), s=rho.shape, dim=(0, 1, 2))[..., c["r"]::c["s"]]
        return out

    def adjoint(self, d):
        c = self.c
        acc = 0.0
        for k, ph in enumerate(_phases(c["K"])):
            u = torch.zeros((c["nz"], c["ny"], c["nx"]), dtype=torch.float64, device="cuda")
            u[..., c["r"]::c["s"]] = (d[k] * ph.conjugate()).real
            acc = acc + torch.fft.rfftn(u, dim=(0, 1, 2))[None] * self.H[k].conj()
        v = torch.fft.irfftn(acc, s=(c["nz"], c["ny"], c["nx"]), dim=(1, 2, 3))
        return v[0] if self.b is None else (v * self.b).sum(0)


def _cg64(normal, rhs, iters):
    x, r = torch.zeros_like(rhs), rhs.clone()
    p, rr = r.clone(), (rhs * rhs).sum()
    for _ in range(iters):
        q = normal(p)
        a = rr / (p * q).sum()
        x += a * p
        r -= a * q
        rn = (r * r).sum()
        p = r + (rn / rr) * p
        rr = rn
    return x


def _prior64(c, v):
    """T^T T + alpha P^T P with alpha = 4 and a two-voxel shell."""
    out = torch.zeros_like(v)
    for dim in range(3):
        d = torch.roll(v, 1, dim) - 2.0 * v + torch.roll(v, -1, dim)
        out += torch.roll(d, 1, dim) - 2.0 * d + torch.roll(d, -1, dim)
    shell = torch.ones_like(v)
    shell[2:-2, 2:-2, 2:-2] = 0.0
    return out + 4.0 * shell * v


def _net64(ch, theta, x):
    """The network on [1, 1, D, H, W]; theta a flat vector (autograd follows it)."""
    ws, o = [], 0
    for ci, co in _layers(ch):
        w = theta[o:o + co * 27 * ci].view(co, 3, 3, 3, ci).permute(0, 4, 1, 2, 3)
        ws.append((w, theta[o + co * 27 * ci:o + co * 27 * ci + co]))
        o += co * 27 * ci + co
    it = iter(ws)
    conv = lambda v: torch.nn.functional.conv3d(v, *next(it), padding=1)   # noqa: E731
    skips = []
    for l in range(len(ch)):
        x = torch.relu(conv(x if l == 0 else torch.nn.functional.avg_pool3d(x, 2)))
        x = torch.relu(conv(x))
        skips.append(x)
    for l in range(len(ch) - 2, -1, -1):
        for dim in (2, 3, 4):
            x = x.repeat_interleave(2, dim=dim)
        x = torch.relu(conv(x))
        x = torch.relu(conv(x + skips[l]))
    return conv(x)


def _exact_solve(c, t):
    op = _Sep64(c, t["sens"])
    lam = LAM * op.m["norm2"]
    rhs = op.adjoint(t["d"].to(torch.complex128))
    if c["kind"] == "apg":
        tau = _apg_tau(c)
        x = torch.zeros_like(rhs)
        y = x
        for k in range(1, c["iters"] + 1):
            xn = torch.clamp(y - tau * (op.adjoint(op.forward(y)) + lam * _prior64(c, y) - rhs), min=0.0)
            y = xn + k / (k + 3.0) * (xn - x)
            x = xn
        return x
    return _cg64(lambda p: op.adjoint(op.forward(p)) + lam * p, rhs, c["iters"])


def exact(case, seed):
    c = case
    kind = c["kind"]
    t = _inputs(c, seed)
    if kind == "forward":
        return _Sep64(c, t["sens"]).forward(t["rho"].double())
    if kind == "adjoint":
        return _Sep64(c, t["sens"]).adjoint(t["d"].to(torch.complex128))
    if kind in ("solve", "apg"):
        return {"rho": _exact_solve(c, t), "iters": None}
    if kind == "batch":
        return {"rhos": [_exact_solve(v, x) for v, x in zip(_volumes(c), t)], "iters": None}
    if kind == "general":
        op = _Gen64(c, t["h"], t["bvec"])
        lam = LAM * _general_norm2(c)
        rhs = op.adjoint(t["d"].to(torch.complex128))
        return {"rho": _cg64(lambda p: op.adjoint(op.forward(p)) + lam * p, rhs, c["iters"]), "iters": None}
    r = float(t["inp"].double().pow(2).mean().sqrt())
    theta = t["theta"].double().requires_grad_(kind == "train")
    with torch.set_grad_enabled(kind == "train"):
        out = _net64(_channels(c), theta, t["inp"].double()[None, None] / r)[0, 0]
        if kind == "infer":
            return r * GAIN * out
        loss = (out - t["target"].double() / (r * GAIN)).pow(2).mean() / 2.0
        loss.backward()
    return {"grad": theta.grad, "loss": float(loss.detach())}
