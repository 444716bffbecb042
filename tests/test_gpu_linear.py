"""Linear layers on the tensor-core kernel that runs both products in one launch (bf16 of any size, fp32 beyond the
two-launch path): parity with the oracle at the edges of its tiles. Delta and nnz come back through dbp_last_step and
the oracle's codes, given that Delta, stand behind every gradient entry."""
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


@pytest.mark.parametrize("dtype,B,N,K", [
    ("bf16", 1, 1, 1), ("bf16", 128, 64, 64), ("bf16", 129, 65, 71), ("bf16", 33, 300, 264), ("bf16", 700, 10, 257),
    ("bf16", 640, 136, 520),           # dW split along the reduction
    ("bf16", 36, 2470, 320), ("bf16", 2560, 1280, 512),      # more tiles than SMs: two accumulators in flight
    ("bf16", 4225, 2200, 1032),        # tiles of 256 rows: the last of dX holds one row, the last columns are eight
    ("bf16", 4225, 2200, 1030),        # the same, rows of X and W re-written, plain stores
    ("bf16", 6418, 3208, 360),         # the same in parts
    ("f32", 257, 513, 65), ("f32", 131, 1003, 131), ("f32", 20000, 7, 12), ("f32", 256, 1000, 2048), ("f32", 513, 260, 8)])
def test_both_products_and_the_bias_gradient(ctx, dtype, B, N, K):
    import paper_2004_04729_b200 as dbp
    L = wl.linear_layer(B, N, K, data_seed=B + 3 * N + 7 * K, scale=2.0, seed=11, dtype=dtype)
    tdt = torch.bfloat16 if dtype == "bf16" else torch.float32
    d, X, W = (torch.from_numpy(np.ascontiguousarray(a)).to(tdt).cuda() for a in (L.delta, L.X, L.W))
    out = dbp.dithered_linear_backward(ctx, d, X, W, L.seed, L.scale, need_db=True, flags=dbp.DBP_DX_F32)
    D, nnz = ctx.last_step()
    assert ctx.last_device_status() == (0, 0)
    D = np.float32(D)
    want = oracle.step_size(L.delta, L.scale)
    assert abs(float(D) - float(want)) <= 1e-6 * float(want)
    codes, onnz, _ = oracle.nsd_codes(L.delta, L.seed, D)
    assert nnz == onnz
    ref = oracle.linear_backward(codes, D, L.X, L.W, with_abs=True)
    for key in ("dW", "dX", "db"):
        g = out[key].double().cpu().numpy()
        assert np.linalg.norm(g - ref[key]) <= TOL * np.linalg.norm(ref[key]) + 1e-30, key
        assert np.all(np.abs(g - ref[key]) <= TOL * ref["S_" + key] + 1e-30), key
    # one product at a time, a given step size (no statistics kernel), bf16 dX: the same numbers
    step = torch.tensor([float(D)], device="cuda")
    only_x = dbp.dithered_linear_backward(ctx, d, X, W, L.seed, 0.0, delta_in=step, need_dW=False, flags=dbp.DBP_DX_F32)
    only_w = dbp.dithered_linear_backward(ctx, d, X, W, L.seed, 0.0, delta_in=step, need_dX=False)
    assert torch.equal(only_x["dX"], out["dX"])
    assert (only_w["dW"] - out["dW"]).abs().max().item() <= 1e-5 * out["dW"].abs().max().item() + 1e-30
    if dtype == "bf16":
        low = dbp.dithered_linear_backward(ctx, d, X, W, L.seed, L.scale)
        assert torch.equal(low["dX"], out["dX"].to(torch.bfloat16))


@pytest.mark.parametrize("B,N,K", [(1198, 241, 1992), (1089, 456, 1344), (2602, 548, 816), (64, 100, 72)])
def test_weight_gradients_of_one_or_two_parts_are_the_same_bits_every_time(ctx, B, N, K):
    """Layers whose estimate hardly differs between more and fewer parts, and one of one part."""
    import paper_2004_04729_b200 as dbp
    rng = np.random.default_rng(B)
    d, X, W = (torch.from_numpy(rng.standard_normal(s).astype(np.float32)).bfloat16().cuda() for s in ((B, N), (B, K), (N, K)))
    outs = [dbp.dithered_linear_backward(ctx, d, X, W, 3, 2.0)["dW"] for _ in range(12)]
    for dW in outs[1:]:
        assert torch.equal(dW, outs[0])
