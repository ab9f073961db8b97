"""The tcgen05 convolution's walk through the volume against FP64: edge tiles
(warps with lanes outside the volume) with 16, 32 and 64 accumulator columns,
one plane a CTA, runs that start inside a column of tiles, both for the
forward (walking up z) and the input gradient (the flipped operand walks
down).

Operands are exact in bfloat16, so only the FP32 accumulation of at most
27 x 32 products differs: relative L2 <= 1e-5, as for the network's layers."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

CASES = [
    # (nx, ny, nz), cin, cout
    ((9, 17, 5), 16, 16),        # one plane a CTA, edge tiles on both axes
    ((3, 2, 1), 8, 24),          # smaller than a tile: paired taps, 32 columns
    ((99, 18, 3), 32, 64),       # 64 columns
    ((104, 33, 61), 16, 8),      # more planes than CTAs: runs start inside columns
    ((101, 31, 70), 8, 16),      # the same on the paired taps
]


def _conv64(x, w, nx, ny, nz):
    """x [nz][ny][nx][cin], w [cout][27][cin] in FP64."""
    k = w.reshape(w.shape[0], 3, 3, 3, -1).permute(0, 4, 1, 2, 3)
    return torch.nn.functional.conv3d(x.permute(3, 0, 1, 2)[None], k, padding=1)[0].permute(1, 2, 3, 0)


@pytest.mark.parametrize("n,cin,cout", CASES)
def test_walk_matches_fp64(n, cin, cout, monkeypatch):
    from paper_2503_13802_gb300.unet import mh3d_unet_conv_forward, mh3d_unet_conv_input_grad

    monkeypatch.setenv("MH3D_UNET_UMMA", "1")
    nx, ny, nz = n
    V = nx * ny * nz
    g = torch.Generator(device="cuda").manual_seed(nx + cin + cout)
    src = torch.randn(V * cin, generator=g, device="cuda").to(torch.bfloat16)
    dy = torch.randn(V * cout, generator=g, device="cuda").to(torch.bfloat16)
    w = (torch.randn(cout * 27 * cin, generator=g, device="cuda") / (27 * cin) ** 0.5).to(torch.bfloat16).float()
    out = torch.full((V * cout,), float("nan"), device="cuda")
    mh3d_unet_conv_forward(n, cin, cout, w, None, out, src=src)
    w64 = w.double().reshape(cout, 27, cin)
    ref = _conv64(src.double().reshape(nz, ny, nx, cin), w64, nx, ny, nz).reshape(-1)
    assert float((out.double() - ref).norm() / ref.norm()) <= 1e-5
    gin = torch.full((V * cin,), float("nan"), device="cuda")
    mh3d_unet_conv_input_grad(n, cin, cout, dy, w, gin)
    wt = w64.flip(1).permute(2, 1, 0).contiguous()   # the transposed convolution
    ref = _conv64(dy.double().reshape(nz, ny, nx, cout), wt, nx, ny, nz).reshape(-1)
    assert float((gin.double() - ref).norm() / ref.norm()) <= 1e-5
