"""Sums of one sign over long reductions. The tensor cores' accumulators are truncated when an MMA adds to them, so such a sum
comes out low by an amount that grows with its length; the kernels cut long reductions into parts. Every entry is compared
with 64-bit sums of the library's own codes: within 1e-5 of it (all terms have one sign, so the sum is the sum of their sizes),
the bound of every other layer."""
import pytest
import torch

pytestmark = pytest.mark.gpu
TOL = 1e-5


@pytest.fixture(scope="module")
def ctx():
    import paper_2004_04729_b200 as dbp
    c = dbp.Context(0)
    yield c
    c.close()


def _positive(gen, dtype, *shape, scale=1.0):
    return (torch.randn(*shape, generator=gen, device="cuda").abs() * scale).to(torch.bfloat16 if dtype == "bf16" else torch.float32)


def _layer(ctx, dtype, B, Ci, Co, H, W, k):
    """delta, X, W all positive, the codes and the step size of a call with seed 3 and scale 1."""
    import paper_2004_04729_b200 as dbp
    gen = torch.Generator(device="cuda")
    gen.manual_seed(B + Ci + Co)
    d = _positive(gen, dtype, B, Co, H, W, scale=1e-3)
    X, Wt = _positive(gen, dtype, B, Ci, H, W), _positive(gen, dtype, Co, Ci, k, k)
    q = dbp.nsd_quantize(ctx, d, 3, 1.0)
    return d, X, Wt, dbp.nsd_decode_dense(ctx, q, d.shape), q.delta.double().item()


def _some(n):
    """A few channels, the first and the last among them."""
    return torch.unique(torch.linspace(0, n - 1, min(n, 7), device="cuda").long())


def _shifted(t, dy, dx):
    """t[..., y + dy, x + dx], zero outside."""
    return torch.nn.functional.pad(t, (1, 1, 1, 1))[..., 1 + dy:t.shape[-2] + 1 + dy, 1 + dx:t.shape[-1] + 1 + dx]


def _check_dW(dW, codes, delta, X, k):
    co, ci = _some(dW.shape[0]), _some(dW.shape[1])
    q, x = codes[:, co].double(), X[:, ci].double()
    for ky in range(k):
        for kx in range(k):
            ref = delta * torch.einsum("bcyx,bdyx->cd", q, x if k == 1 else _shifted(x, ky - 1, kx - 1))
            rel = ((dW[co][:, ci][:, :, ky, kx].double() - ref) / ref).abs().max().item()
            assert rel <= TOL, (ky, kx, rel)


@pytest.mark.parametrize("dtype,B,Ci,Co,H,W", [
    ("f32", 64, 512, 512, 28, 28),      # 50176 positions in two pieces on 48 tiles
    ("f32", 256, 64, 64, 56, 56),       # both pieces in one tile
    ("f32", 130, 128, 72, 56, 56),      # a ragged tile of output channels
    ("bf16", 64, 512, 512, 28, 28),
    ("bf16", 256, 128, 128, 56, 56)])
def test_3x3_weight_gradients(ctx, dtype, B, Ci, Co, H, W):
    import paper_2004_04729_b200 as dbp
    d, X, Wt, codes, delta = _layer(ctx, dtype, B, Ci, Co, H, W, 3)
    for need_dX in (False, True):       # the dW kernel by itself, and sharing the SMs with dX where it does
        out = dbp.dithered_conv_backward(ctx, d, X, Wt, 3, 1.0, need_dX=need_dX)
        _check_dW(out["dW"], codes, delta, X, 3)
    assert ctx.last_device_status() == (0, 0)


@pytest.mark.parametrize("dtype,B,Ci,Co,H,W", [
    ("bf16", 1024, 64, 64, 56, 56),     # quantization and products in one kernel, whose dW accumulators live as long as it does
    ("bf16", 400, 72, 200, 56, 56),     # the same with two panels of output channels
    ("bf16", 1500, 512, 512, 14, 14),   # few tiles, long reductions
    ("f32", 700, 512, 512, 14, 14)])
def test_1x1_weight_gradients(ctx, dtype, B, Ci, Co, H, W):
    import paper_2004_04729_b200 as dbp
    d, X, Wt, codes, delta = _layer(ctx, dtype, B, Ci, Co, H, W, 1)
    _check_dW(dbp.dithered_conv_backward(ctx, d, X, Wt, 3, 1.0)["dW"], codes, delta, X, 1)
    assert ctx.last_step()[1] == int((codes != 0).sum())
    assert ctx.last_device_status() == (0, 0)


def _check_dX(dX, codes, delta, W, k):
    """The first and the last image, a few channels, every position."""
    ci, im = _some(dX.shape[1]), torch.tensor([0, dX.shape[0] - 1], device="cuda")
    q, w = codes[im].double(), W[:, ci].double()
    ref = sum(torch.einsum("bcyx,cd->bdyx", q if k == 1 else _shifted(q, 1 - ky, 1 - kx), w[:, :, ky, kx]) for ky in range(k) for kx in range(k))
    rel = ((dX[im][:, ci].double() - delta * ref) / (delta * ref)).abs().max().item()
    assert rel <= TOL, rel


@pytest.mark.parametrize("dtype,B,Ci,Co,H,W", [
    ("f32", 8, 128, 512, 28, 28),       # the low pieces of the weights in a pass of their own
    ("f32", 3, 72, 520, 9, 31),         # the same, ragged
    ("f32", 8, 128, 1000, 28, 28),      # the reduction in two parts
    ("f32", 2, 200, 2100, 5, 62),       # in four; rows as long as the kernel takes
    ("f32", 4, 64, 2048, 28, 28),       # few channels: no longer both pieces on one accumulator's lanes
    ("f32", 40, 24, 5000, 4, 4),        # in eight; several images per patch
    ("bf16", 4, 128, 2048, 28, 28), ("bf16", 2, 40, 1030, 17, 12)])
def test_3x3_input_gradients(ctx, dtype, B, Ci, Co, H, W):
    import paper_2004_04729_b200 as dbp
    d, X, Wt, codes, delta = _layer(ctx, dtype, B, Ci, Co, H, W, 3)
    out = dbp.dithered_conv_backward(ctx, d, X, Wt, 3, 1.0, flags=dbp.DBP_DX_F32 | dbp.DBP_FORCE_DENSE * (Co % 8 == 0))
    _check_dX(out["dX"], codes, delta, Wt, 3)
    alone = dbp.dithered_conv_backward(ctx, d, X, Wt, 3, 1.0, need_dW=False, flags=dbp.DBP_DX_F32)["dX"]
    assert torch.equal(alone, out["dX"])         # one order of the sums, whatever else is asked for
    assert ctx.last_device_status() == (0, 0)


def test_3x3_input_gradient_of_more_channels_than_the_parts_hold(ctx):
    """fp32 from 7169 output channels on: the gather kernels; the tensor cores' when those are insisted on (540 MMAs a part)."""
    import paper_2004_04729_b200 as dbp
    d, X, Wt, codes, delta = _layer(ctx, "f32", 1, 8, 7176, 5, 5, 3)
    _check_dX(dbp.dithered_conv_backward(ctx, d, X, Wt, 3, 1.0)["dX"], codes, delta, Wt, 3)
    _check_dX(dbp.dithered_conv_backward(ctx, d, X, Wt, 3, 1.0, flags=dbp.DBP_FORCE_DENSE)["dX"], codes, delta, Wt, 3)


@pytest.mark.parametrize("Ci,Co", [(128, 512), (128, 1024), (256, 72)])
def test_stride_2_input_gradients_in_parts(ctx, Ci, Co):
    """The phase images of a stride-2 layer go through the same passes and parts; positions (y, x) of dX take the taps whose
    parity fits."""
    import paper_2004_04729_b200 as dbp
    B, H, W = 2, 12, 20
    d, _, Wt, codes, delta = _layer(ctx, "f32", B, Ci, Co, H // 2, W // 2, 3)
    X = torch.ones(B, Ci, H, W, device="cuda")
    dX = dbp.dithered_conv_backward(ctx, d, X, Wt, 3, 1.0, stride=2)["dX"]
    ci = _some(Ci)
    up = torch.zeros(B, Co, H, W, dtype=torch.float64, device="cuda")
    up[:, :, ::2, ::2] = codes.double()
    ref = delta * sum(torch.einsum("bcyx,cd->bdyx", _shifted(up, 1 - ky, 1 - kx), Wt[:, ci, ky, kx].double()) for ky in range(3) for kx in range(3))
    assert ((dX[:, ci].double() - ref).abs() <= TOL * ref).all()


@pytest.mark.parametrize("dtype,B,N,K,want", [
    ("f32", 8192, 16, 64, "dW"), ("f32", 2, 60000, 72, "dX"),       # one tile's reduction on warp-level MMAs
    ("f32", 16384, 300, 256, "dW"), ("f32", 300, 8192, 256, "dX"),  # the longest parts of the CTA-wide kernel
    ("f32", 260, 8300, 128, "both"), ("f32", 70, 16500, 130, "both"), ("bf16", 300, 20000, 256, "dX"),     # dX in parts
    ("bf16", 96, 24577, 131, "both"),
    ("bf16", 32768, 320, 512, "dW"), ("bf16", 300, 8192, 512, "dX")])
def test_linear_layers(ctx, dtype, B, N, K, want):
    import paper_2004_04729_b200 as dbp
    d, X, Wt, codes, delta = _layer(ctx, dtype, B, K, N, 1, 1, 1)
    out = dbp.dithered_linear_backward(ctx, d.view(B, N), X.view(B, K), Wt.view(N, K), 3, 1.0, need_dW=want != "dX", need_dX=want != "dW",
                                       flags=dbp.DBP_DX_F32)
    if want != "dX":
        _check_dW(out["dW"].view(N, K, 1, 1), codes, delta, X, 1)
    if want != "dW":
        _check_dX(out["dX"].view(B, K, 1, 1), codes, delta, Wt, 1)
        for _ in range(3):                       # the parts are added in one order
            again = dbp.dithered_linear_backward(ctx, d.view(B, N), X.view(B, K), Wt.view(N, K), 3, 1.0, need_dW=want != "dX", flags=dbp.DBP_DX_F32)
            assert torch.equal(again["dX"], out["dX"])
    assert ctx.last_device_status() == (0, 0)


@pytest.mark.parametrize("dtype,B,Ci,Co,H,W", [
    ("f32", 2, 72, 8192, 8, 8), ("f32", 2, 264, 8200, 9, 12), ("f32", 3, 40, 16500, 5, 5),    # whole words or not, two and three parts
    ("bf16", 2, 136, 20000, 8, 8), ("bf16", 5, 24, 8257, 5, 7)])
def test_1x1_input_gradients(ctx, dtype, B, Ci, Co, H, W):
    import paper_2004_04729_b200 as dbp
    d, X, Wt, codes, delta = _layer(ctx, dtype, B, Ci, Co, H, W, 1)
    out = dbp.dithered_conv_backward(ctx, d, X, Wt, 3, 1.0, flags=dbp.DBP_DX_F32)
    _check_dX(out["dX"], codes, delta, Wt, 1)
    _check_dW(out["dW"], codes, delta, X, 1)
    for _ in range(3):
        assert torch.equal(dbp.dithered_conv_backward(ctx, d, X, Wt, 3, 1.0, flags=dbp.DBP_DX_F32)["dX"], out["dX"])
    assert ctx.last_device_status() == (0, 0)
