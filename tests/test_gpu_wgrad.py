"""The staged-row weight gradient against the gather kernel: both add the
same products in the same order (chunks of 4096 voxels, 16 voxels per mma,
chunks in order), so every weight and bias gradient is equal bit for bit.
Sizes at the edges: rows shorter than an mma step, volumes of one voxel more
or less than a chunk or a block, channel slices of 8 and 16, output tiles of
8, 16 and 32 with remainders, one-channel sources."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

CASES = [
    # (nx, ny, nz), cin, cout, mode
    ((4, 4, 4), 16, 16, "plain"),
    ((6, 2, 10), 8, 9, "plain"),
    ((241, 17, 1), 16, 8, "plain"),      # 4097 voxels: a chunk and one voxel
    ((63, 5, 13), 24, 24, "skip"),       # 4095 voxels, slices of 8 channels
    ((2, 64, 66), 48, 33, "plain"),      # rows of two voxels, two output tiles
    ((20, 12, 18), 64, 64, "up"),
    ((128, 4, 4), 40, 1, "skip"),
    ((130, 2, 2), 8, 32, "up"),
    ((7, 9, 11), 1, 16, "f32"),
    ((66, 64, 2), 1, 33, "f32"),
    ((12, 10, 8), 1, 8, "plain"),
    ((16, 6, 4), 1, 3, "up"),
    ((1, 1, 1), 16, 16, "plain"),
]


@pytest.mark.parametrize("n,cin,cout,mode", CASES)
def test_staged_rows_equal_the_gather_kernel(n, cin, cout, mode, monkeypatch):
    from paper_2503_13802_gb300.unet import mh3d_unet_conv_weight_grad

    nx, ny, nz = n
    g = torch.Generator(device="cuda").manual_seed(nx + 7 * cin + cout)
    V = nx * ny * nz
    rnd = lambda m: torch.randn(m, generator=g, device="cuda").to(torch.bfloat16)   # noqa: E731
    kw = dict(src_f32=torch.randn(V, generator=g, device="cuda")) if mode == "f32" else dict(src=rnd(
        (V // 8 if mode == "up" else V) * cin))
    if mode == "up":
        kw["up"] = 1
    if mode == "skip":
        kw["skip"] = rnd(V * cin)
    dy = rnd(V * cout)
    got = []
    for gather in ("0", "1"):
        monkeypatch.setenv("MH3D_UNET_GATHER", gather)
        gW = torch.full((cout * 27 * cin,), float("nan"), device="cuda")
        gb = torch.full((cout,), float("nan"), device="cuda")
        mh3d_unet_conv_weight_grad(n, cin, cout, dy, gW, gb, **kw)
        got.append((gW, gb))
    assert torch.equal(got[0][0], got[1][0]) and torch.equal(got[0][1], got[1][1])
