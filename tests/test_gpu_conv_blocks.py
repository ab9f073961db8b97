"""The halo-block and weight-streaming convolutions against the gather kernel:
the same 16-product steps in the same order (the streaming form also in the
same split-K groups), so every output is equal bit for bit.  Sizes at the
edges: volumes smaller than a block, one voxel more than blocks, output
tiles with remainders, every channel count the block kernels take."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

CASES = [
    # (nx, ny, nz), cin, cout, mode
    ((1, 1, 1), 16, 16, "plain"),
    ((8, 8, 4), 8, 16, "plain"),
    ((9, 9, 5), 8, 9, "skip"),
    ((17, 3, 7), 16, 33, "plain"),
    ((10, 14, 6), 16, 64, "up"),
    ((7, 8, 9), 32, 1, "plain"),
    ((24, 15, 4), 32, 63, "skip"),
    ((9, 5, 3), 64, 8, "plain"),
    ((40, 40, 20), 64, 32, "up"),
    ((88, 56, 21), 64, 64, "plain"),     # blocks for every SM
    ((5, 9, 4), 64, 41, "skip"),         # streamed weights
    ((6, 4, 10), 64, 32, "up"),
]


def _both(monkeypatch, run):
    monkeypatch.setenv("MH3D_UNET_UMMA", "0")
    got = []
    for gather in ("0", "1"):
        monkeypatch.setenv("MH3D_UNET_GATHER", gather)
        got.append(run())
    return got


@pytest.mark.parametrize("n,cin,cout,mode", CASES)
def test_block_convolutions_equal_the_gather_kernel(n, cin, cout, mode, monkeypatch):
    from paper_2503_13802_gb300.unet import mh3d_unet_conv_forward, mh3d_unet_conv_input_grad

    nx, ny, nz = n
    V = nx * ny * nz
    g = torch.Generator(device="cuda").manual_seed(nx + 5 * cin + cout)
    rnd = lambda m: torch.randn(m, generator=g, device="cuda").to(torch.bfloat16)   # noqa: E731
    kw = dict(src=rnd((V // 8 if mode == "up" else V) * cin))
    if mode == "up":
        kw["up"] = 1
    if mode == "skip":
        kw["skip"] = rnd(V * cin)
    W = torch.randn(cout * 27 * cin, generator=g, device="cuda") / (27 * cin) ** 0.5
    b = torch.randn(cout, generator=g, device="cuda")
    dy = rnd(V * cout)

    def run():
        out = torch.full((V * cout,), float("nan"), device="cuda")
        gin = torch.full((V * cin,), float("nan"), device="cuda")
        mh3d_unet_conv_forward(n, cin, cout, W, b, out, relu=True, **kw)
        mh3d_unet_conv_input_grad(n, cin, cout, dy, W, gin)
        return out, gin

    a, r = _both(monkeypatch, run)
    assert torch.equal(a[0], r[0]) and torch.equal(a[1], r[1])


def test_streamed_split_k_equals_the_gather_kernel_through_the_network(monkeypatch):
    """A network of 64 and 128 channels: its coarse levels are split along K
    on the gather kernel and streamed in the same groups otherwise."""
    from paper_2503_13802_gb300.unet import UNet

    n, ch = (40, 32, 32), (64, 64, 128)
    g = torch.Generator(device="cuda").manual_seed(5)
    x = torch.randn(n[0] * n[1] * n[2], generator=g, device="cuda")
    t = torch.randn(n[0] * n[1] * n[2], generator=g, device="cuda")

    def run():
        net = UNet(n, *ch)
        gp = torch.Generator(device="cuda").manual_seed(6)
        net.set_params(torch.randn(net.nparam, generator=gp, device="cuda") * 0.02)
        out = torch.empty(net.V, dtype=torch.float32, device="cuda")
        net.forward(x, out)
        grad = torch.empty(net.nparam, dtype=torch.float32, device="cuda")
        net.loss_grad(x, t, grad)
        return out, grad

    a, r = _both(monkeypatch, run)
    assert bool(torch.isfinite(a[0]).all()) and float(a[0].abs().max()) > 0
    assert torch.equal(a[0], r[0]) and torch.equal(a[1], r[1])
