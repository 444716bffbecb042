"""1x1 and 3x3 layers of either type with channel counts and planes that no tile or 16-byte row fits, as the calls run by
default (no sparse structure, no forced path): parity with the oracle. Delta and nnz come back through dbp_last_step and
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


@pytest.mark.parametrize("B,Ci,Co,H,W,k", [
    (2, 72, 136, 27, 19, 1),      # odd planes
    (3, 130, 33, 8, 8, 1),        # channel counts on neither side a multiple of 8
    (5, 3, 5, 4, 6, 1),           # dW rows no multiple of 16 bytes
    (2, 300, 70, 5, 5, 1),        # three tiles of input channels, two accumulators' worth
    (9, 20, 24, 1, 2, 1),         # the smallest plane
    (4, 64, 40, 3, 3, 1), (1, 257, 129, 16, 12, 1),
    (3, 41, 56, 13, 5, 1),        # one position behind a whole chunk, rows that start anywhere
    (30, 257, 250, 31, 33, 1),    # the same in tiles of 256 input channels, pairs of chunks across images
    (2, 3, 8, 6, 6, 3), (2, 12, 20, 9, 9, 3), (3, 130, 65, 7, 5, 3), (2, 65, 67, 8, 8, 3), (4, 10, 6, 2, 3, 3),
    (1, 33, 129, 20, 17, 3), (3, 9, 1, 6, 7, 3)])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_layers_of_awkward_sizes(ctx, dtype, B, Ci, Co, H, W, k):
    import paper_2004_04729_b200 as dbp
    L = wl.conv_layer(B, Ci, Co, H, W, k, data_seed=B + Ci + 3 * Co + H, scale=2.0, seed=5, dtype=dtype)
    tdt = torch.bfloat16 if dtype == "bf16" else torch.float32
    d, X, Wt = (torch.from_numpy(np.ascontiguousarray(a)).to(tdt).cuda() for a in (L.delta, L.X, L.W))
    out = dbp.dithered_conv_backward(ctx, d, X, Wt, L.seed, L.scale, need_db=True, flags=dbp.DBP_DX_F32)
    D, nnz = ctx.last_step()
    assert ctx.last_device_status() == (0, 0)
    D = np.float32(D)
    codes, onnz, _ = oracle.nsd_codes(L.delta, L.seed, D)
    assert nnz == onnz
    ref = oracle.conv_backward(codes, D, L.X, L.W, with_abs=True)
    for key in ("dW", "dX", "db"):
        g = out[key].double().cpu().numpy()
        assert np.linalg.norm(g - ref[key]) <= TOL * np.linalg.norm(ref[key]) + 1e-30, key
        assert np.all(np.abs(g - ref[key]) <= TOL * ref["S_" + key] + 1e-30), key
    # a given step size (no statistics kernel), each product by itself, dW overlapped: the same numbers
    step = torch.tensor([float(D)], device="cuda")
    only_x = dbp.dithered_conv_backward(ctx, d, X, Wt, L.seed, 0.0, delta_in=step, need_dW=False, need_db=True, flags=dbp.DBP_DX_F32)
    only_w = dbp.dithered_conv_backward(ctx, d, X, Wt, L.seed, 0.0, delta_in=step, need_dX=False, need_db=True)
    both = dbp.dithered_conv_backward(ctx, d, X, Wt, L.seed, L.scale, flags=dbp.DBP_DW_ASYNC)
    ctx.join()
    assert torch.equal(only_x["dX"], out["dX"]) and torch.equal(only_x["db"], out["db"]) and torch.equal(only_w["db"], out["db"])
    top = out["dW"].abs().max().item()
    for r in (only_w, both):
        assert (r["dW"] - out["dW"]).abs().max().item() <= 1e-5 * top
    assert torch.equal(both["dX"], out["dX"].to(both["dX"].dtype))


@pytest.mark.parametrize("B,Ci,Co,H,W,stride", [
    (64, 8, 10, 28, 28, 1),       # 1.6 MB of codes in rows of 16 channels, 1.0 MB in rows of 10
    (128, 16, 9, 32, 32, 1),      # 4.2 MB in rows of 16 channels, 2.4 MB in rows of 9
    (64, 8, 10, 56, 56, 2)])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_codes_whose_padded_rows_are_much_larger(dtype, B, Ci, Co, H, W, stride):
    """3x3 layers whose codes lie in rows padded to 16 bytes, at sizes where the padding is more than any rounding of the
    workspace's size: on a context of their own, so that no earlier, larger call has made room for them."""
    import paper_2004_04729_b200 as dbp
    L = wl.conv_layer(B, Ci, Co, H, W, 3, data_seed=B + Co + H, scale=2.0, seed=11, dtype=dtype, stride=stride)
    tdt = torch.bfloat16 if dtype == "bf16" else torch.float32
    d, X, Wt = (torch.from_numpy(np.ascontiguousarray(a)).to(tdt).cuda() for a in (L.delta, L.X, L.W))
    own = dbp.Context(0)
    try:
        out = dbp.dithered_conv_backward(own, d, X, Wt, L.seed, L.scale, need_db=True, flags=dbp.DBP_DX_F32, stride=stride)
        D, nnz = own.last_step()
        assert own.last_device_status() == (0, 0)
    finally:
        own.close()
    D = np.float32(D)
    codes, onnz, _ = oracle.nsd_codes(L.delta, L.seed, D)
    assert nnz == onnz
    ref = oracle.conv_backward(codes, D, L.X, L.W, with_abs=True) if stride == 1 else \
        oracle.conv_backward_strided(codes, D, L.X, L.W, stride, with_abs=True)
    for key in ("dW", "dX", "db"):
        g = out[key].double().cpu().numpy()
        assert np.all(np.abs(g - ref[key]) <= TOL * ref["S_" + key] + 1e-30), key
