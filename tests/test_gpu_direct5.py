"""5x5 layers of few channels (both products in one launch on the dense codes): parity with the oracle at the edges of the
kernel's register tiles, with a folded ReLU mask, each product by itself and more images than CTAs."""
import numpy as np
import pytest
import torch

import oracle
import workloads as wl

pytestmark = pytest.mark.gpu
TOL = 1e-5


@pytest.fixture(scope="module")
def ctx():
    import paper_2004_04729_b200 as dbp
    c = dbp.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("B,Ci,Co,H,W,dtype", [
    (3, 1, 6, 32, 32, "f32"), (5, 6, 16, 16, 16, "f32"),     # LeNet-5-like
    (2, 3, 5, 7, 9, "f32"),                                  # odd everything: rows of 9, an odd input channel, dW size % 4 != 0
    (2, 1, 1, 1, 1, "f32"), (1, 12, 32, 18, 18, "f32"), (2, 2, 3, 5, 2, "bf16"), (300, 2, 4, 6, 6, "f32"), (3, 7, 12, 9, 8, "bf16")])
def test_layers_of_few_channels(ctx, B, Ci, Co, H, W, dtype):
    import paper_2004_04729_b200 as dbp
    L = wl.conv_layer(B, Ci, Co, H, W, 5, data_seed=B + Ci + Co + H, scale=2.0, seed=4, dtype=dtype)
    mask = (np.random.default_rng(B + H).random(L.delta.shape) < 0.6) if dtype == "f32" else np.ones(L.delta.shape, bool)
    dz = (L.delta * mask).astype(np.float32)
    tdt = torch.bfloat16 if dtype == "bf16" else torch.float32
    d, X, Wt = (torch.from_numpy(np.ascontiguousarray(a)).to(tdt).cuda() for a in (L.delta, L.X, L.W))
    m = torch.from_numpy(mask.astype(np.uint8)).cuda()
    def call(**kw):
        if dtype == "f32":
            ctx.set_relu_mask(m)
        return dbp.dithered_conv_backward(ctx, d, X, Wt, L.seed, L.scale, flags=dbp.DBP_DX_F32, **kw)
    out = call(need_db=True)
    D, nnz = ctx.last_step()
    assert ctx.last_device_status() == (0, 0)
    D = np.float32(D)
    codes, onnz, _ = oracle.nsd_codes(dz, L.seed, D)
    assert nnz == onnz
    ref = oracle.conv_backward(codes, D, L.X, L.W, with_abs=True)
    for key in ("dW", "dX", "db"):
        g = out[key].double().cpu().numpy()
        assert np.linalg.norm(g - ref[key]) <= TOL * np.linalg.norm(ref[key]) + 1e-30, key
        assert np.all(np.abs(g - ref[key]) <= TOL * ref["S_" + key] + 1e-30), key
    assert torch.equal(call(need_dW=False)["dX"], out["dX"])
    assert (call(need_dX=False)["dW"] - out["dW"]).abs().max().item() <= 1e-5 * out["dW"].abs().max().item() + 1e-30


@pytest.mark.parametrize("B,Ci,Co,H,W,dtype", [
    (149, 6, 16, 16, 16, "f32"), (310, 6, 16, 16, 16, "bf16"), (160, 1, 6, 32, 32, "f32"), (301, 3, 5, 7, 9, "f32"),
    (150, 12, 32, 18, 18, "f32"), (299, 2, 16, 9, 12, "bf16")])
def test_more_images_than_sms(ctx, B, Ci, Co, H, W, dtype):
    test_layers_of_few_channels(ctx, B, Ci, Co, H, W, dtype)


@pytest.mark.parametrize("B,Ci,Co,H,W", [(3, 6, 16, 16, 16), (5, 1, 6, 32, 28), (2, 3, 5, 6, 8), (1, 2, 1, 2, 4), (150, 4, 12, 12, 12),
                                         (2, 3, 5, 8, 10)])          # (rows that are no whole vectors: routed first)
def test_gradient_routed_by_the_statistics(ctx, B, Ci, Co, H, W):
    """A network's 5x5 layer below a pool: the step size of the routed gradient (1e-6 of the one in 64 bits), and, with that step
    size given, the count and the products of the routed gradient (the codes are the same, so the products are sums of the same terms:
    fp32 sums agree to 1e-5)."""
    import paper_2004_04729_b200 as dbp
    g = torch.Generator(device="cuda").manual_seed(B + 7 * Co + H)
    rnd = lambda *s: torch.randn(*s, generator=g, device="cuda")
    mask = (torch.rand(B, Co, H, W, generator=g, device="cuda") < 0.6).to(torch.uint8)
    argmax = torch.randint(0, 4, (B, Co, H // 2, W // 2), generator=g, device="cuda", dtype=torch.int8)
    X, Wt, n = rnd(B, Ci, H, W), rnd(Co, Ci, 5, 5), Co * (H // 2) * (W // 2)
    X2, W2, top = rnd(B, n), rnd(10, n) / n ** 0.5, rnd(B, 10)
    for first_dX in (True, False):
        net = dbp.network_backward(ctx, ["conv", "linear"], [X, X2], [Wt, W2], [mask, None], [argmax, None], top, 2.0, 5,
                                   first_layer_dX=first_dX, with_sparse=False)
        step = ctx.last_step()
        above = dbp.dithered_linear_backward(ctx, top, X2, W2, dbp.layer_seed(5, 1), 2.0)
        assert torch.equal(above["dX"], net[1]["dX"])
        routed = dbp.maxpool2x2_backward(ctx, above["dX"].view(argmax.shape), argmax)
        want = 2.0 * (routed * mask).double().std(unbiased=False).item()
        assert abs(step[0] - want) <= 1e-6 * want
        ctx.set_relu_mask(mask)
        ref = dbp.dithered_conv_backward(ctx, routed, X, Wt, dbp.layer_seed(5, 0), 0.0, delta_in=torch.tensor([step[0]], device="cuda"))
        assert step[1] == ctx.last_step()[1]
        for key in ("dW", "dX") if first_dX else ("dW",):
            assert (net[0][key] - ref[key]).norm().item() <= TOL * ref[key].norm().item(), key
        assert first_dX or net[0]["dX"] is None
    assert ctx.last_device_status() == (0, 0)


def _pooled(ctx, g, argmax, delta, X, Wt, dW=None, dX=None, db=None, *, scale=2.0, delta_in=None, q=None, flags=0, seed=5, sizes=None, address=None,
            null=()):
    """The C entry point: nothing of it is checked in Python. `address`: delta's, where it is not the tensor's own."""
    import paper_2004_04729_b200.binding as b
    B, Co, H, W = delta.shape
    at = lambda t: None if t is None else t.data_ptr()
    s = sizes or (B, X.shape[1], Co, H, W)
    k = Wt.shape[2]
    return b.load_library().dithered_conv_backward_pooled(ctx._h, at(g), at(argmax), address or at(delta),
                                                          None if "X" in null else at(X), None if "W" in null else at(Wt), *s, k, (k - 1) // 2, seed,
                                                          scale, at(delta_in), q.c() if q else None, at(dW), at(dX), at(db), flags)


def _pooled_layer(B, Ci, Co, H, W, k):
    g = torch.Generator(device="cuda").manual_seed(B + 7 * Co + H + k)
    rnd = lambda *s: torch.randn(*s, generator=g, device="cuda")
    argmax = torch.randint(0, 4, (B, Co, H // 2, W // 2), generator=g, device="cuda", dtype=torch.int8)
    return g, rnd(B, Co, H // 2, W // 2), argmax, rnd(B, Ci, H, W), rnd(Co, Ci, k, k)


@pytest.mark.parametrize("k", [1, 3, 5])
def test_refused_pooled_calls_write_nothing(ctx, k):
    """What the layer's call refuses is refused before the routing kernel: delta keeps its values and nothing is launched."""
    import paper_2004_04729_b200 as dbp
    import paper_2004_04729_b200.binding as b
    _, g, argmax, X, Wt = _pooled_layer(3, 4, 6, 8, 12, k)
    room = torch.full((3 * 6 * 8 * 12 + 4,), 7.0, device="cuda")
    delta = room[:-4].view(3, 6, 8, 12)
    whole = dict(dW=torch.empty_like(Wt), dX=torch.empty_like(X), q=dbp.SparseGradient(delta.numel()))
    bad = dbp.SparseGradient(delta.numel())
    bad._c.values = bad.values.data_ptr() + 1
    at = delta.data_ptr()
    torch.cuda.synchronize()
    before = b.load_library().dbp_kernel_launches()
    for wrong in (dict(null=("X",)), dict(null=("W",)), dict(flags=dbp.DBP_FORCE_SPARSE | dbp.DBP_FORCE_DENSE), dict(scale=0.0),
                  dict(scale=float("nan")), dict(address=at + 4), dict(address=at + 8), dict(dW=room[1:]), dict(dX=room[2:]), dict(q=bad),
                  dict(sizes=(0, 4, 6, 8, 12)), dict(sizes=(3, 0, 6, 8, 12)), dict(sizes=(3, 4, -6, 8, 12)), dict(sizes=(3, 4, 6, 8, 5000))):
        assert _pooled(ctx, g, argmax, delta, X, Wt, **{**whole, **wrong}) == -1, wrong
    assert _pooled(ctx, g, argmax, delta, X, Wt, **whole, flags=dbp.DBP_FORCE_DENSE) == -2       # (six output channels)
    assert _pooled(ctx, g, argmax, delta, X, Wt, **whole, sizes=(3, 4, 6, 7, 12)) == -2
    assert b.load_library().dbp_kernel_launches() == before
    torch.cuda.synchronize()
    assert bool((room == 7.0).all())


@pytest.mark.parametrize("k,B,Ci,Co,H,W,how", [
    (5, 3, 6, 16, 16, 16, ""), (5, 150, 4, 12, 12, 12, ""), (5, 200, 3, 24, 20, 36, ""),       # routed by the statistics; several tiles a block
    (5, 4, 2, 5, 8, 8, "mask"), (5, 4, 2, 5, 8, 8, "argmax"), (5, 4, 2, 5, 8, 8, "g"), (5, 4, 2, 5, 8, 10, ""),      # ... not these: routed first
    (5, 4, 2, 5, 8, 8, "given"), (5, 4, 2, 5, 8, 8, "sparse"), (3, 5, 20, 24, 12, 8, ""), (3, 5, 20, 24, 12, 8, "sparse"), (1, 4, 9, 17, 6, 14, "")])
def test_pooled_calls(ctx, k, B, Ci, Co, H, W, how):
    """dithered_conv_backward_pooled against the routed gradient's own call with the same step size: the written delta and the bias
    gradient are the same bits, the products sums of the same terms (1e-5). The buffer is used again with other gradients, which have to be
    the ones that are quantized. `how`: the operand that starts off its boundary, or the option that is set."""
    import paper_2004_04729_b200 as dbp
    gen, g, argmax, X, Wt = _pooled_layer(B, Ci, Co, H, W, k)
    delta = torch.full((B, Co, H, W), 9.0, device="cuda")
    dW, dX, db = torch.empty_like(Wt), torch.empty_like(X), torch.empty(Co, device="cuda")
    off = lambda t, by: torch.cat([t.new_zeros(int(by)), t.reshape(-1)])[int(by):].view(t.shape)          # starts `by` elements into its storage
    for turn in range(3):
        g = torch.randn(g.shape, generator=gen, device="cuda")
        mask = (torch.rand(B, Co, H, W, generator=gen, device="cuda") < 0.6).to(torch.uint8)
        am, mk, gg = off(argmax, how == "argmax"), off(mask, how == "mask"), off(g, how == "g")
        given = torch.tensor([0.5], device="cuda") if how == "given" else None
        q = dbp.SparseGradient(delta.numel()) if how == "sparse" else None
        ctx.set_relu_mask(mk)
        assert _pooled(ctx, gg, am, delta, X, Wt, dW, dX, db, scale=0.0 if how == "given" else 2.0, delta_in=given, q=q, seed=turn) == 0
        step = ctx.last_step()
        routed = dbp.maxpool2x2_backward(ctx, g, argmax)
        assert torch.equal(delta, routed)
        want = 0.5 if how == "given" else 2.0 * (routed * mask).double().std(unbiased=False).item()
        assert abs(step[0] - want) <= 1e-6 * want
        ctx.set_relu_mask(mask)
        ref = dbp.dithered_conv_backward(ctx, routed, X, Wt, turn, 0.0, delta_in=torch.tensor([step[0]], device="cuda"), need_db=True)
        assert step[1] == ctx.last_step()[1]
        assert torch.equal(db, ref["db"])
        for got, key in ((dW, "dW"), (dX, "dX")):
            assert (got - ref[key]).norm().item() <= TOL * ref[key].norm().item(), key
        if q is not None:
            assert q.nnz.item() == step[1] and q.delta.item() == step[0]
    assert ctx.last_device_status() == (0, 0)
