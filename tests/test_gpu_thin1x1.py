"""Thin bf16 1x1 layers, which one kernel quantizes and multiplies: parity with the oracle at the edges of its range (channel
counts and planes that end inside a tile, one and two accumulators, the fewest tiles), and the same numbers as the separate
kernels that a bias gradient or an fp32 dX asks for."""
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
    c.profile_enable(True)
    yield c
    c.close()


@pytest.mark.parametrize("B,Ci,Co,H,W", [
    (300, 8, 8, 8, 8),            # the fewest channels and positions of a chunk; one chunk per tile
    (598, 64, 64, 8, 8),          # two chunks per tile, the last tile of two images
    (300, 72, 136, 9, 8),         # planes of 64 + 8 positions; output channels that end inside the second stage
    (301, 200, 72, 8, 9),         # two accumulators of input channels, three and a half panels
    (303, 136, 40, 8, 8),         # three panels: the fourth does not exist
    (297, 256, 64, 8, 8),         # the most input channels
    (600, 64, 512, 8, 8),         # the most output channels; all of tensor memory
    (24, 64, 256, 28, 28)])
def test_thin_layers(ctx, B, Ci, Co, H, W):
    import paper_2004_04729_b200 as dbp
    L = wl.conv_layer(B, Ci, Co, H, W, 1, data_seed=B + Ci + 3 * Co + H, scale=2.0, seed=5, dtype="bf16")
    d, X, Wt = (torch.from_numpy(np.ascontiguousarray(a)).bfloat16().cuda() for a in (L.delta, L.X, L.W))
    ctx.profile_read()
    out = dbp.dithered_conv_backward(ctx, d, X, Wt, L.seed, L.scale)
    D, nnz = ctx.last_step()
    assert ctx.last_device_status() == (0, 0)
    pr = ctx.profile_read()
    assert pr["fused"][1] == 1 and pr["dx_dense"][1] == 0 and pr["quantize"][1] == 0, pr
    D = np.float32(D)
    codes, onnz, _ = oracle.nsd_codes(L.delta, L.seed, D)
    assert nnz == onnz
    ref = oracle.conv_backward(codes, D, L.X, L.W, with_abs=True)
    g = out["dW"].double().cpu().numpy()
    assert np.all(np.abs(g - ref["dW"]) <= TOL * ref["S_dW"] + 1e-30)
    g = out["dX"].double().cpu().numpy()
    assert np.all(np.abs(g - ref["dX"]) <= 2.0 ** -8 * np.abs(ref["dX"]) + TOL * ref["S_dX"] + 1e-30)
    # a given step size, dW overlapped, a step size of zero
    step = torch.tensor([float(D)], device="cuda")
    again = dbp.dithered_conv_backward(ctx, d, X, Wt, L.seed, 0.0, delta_in=step, flags=dbp.DBP_DW_ASYNC)
    apart = dbp.dithered_conv_backward(ctx, d, X, Wt, L.seed, L.scale, need_db=True)
    ctx.join()
    top = out["dW"].abs().max().item()
    assert ctx.profile_read()["fused"][1] == 1
    for r in (again, apart):
        assert (r["dW"] - out["dW"]).abs().max().item() <= 1e-5 * top
    assert torch.equal(again["dX"], out["dX"])
    none = dbp.dithered_conv_backward(ctx, torch.zeros_like(d), X, Wt, L.seed, L.scale)
    assert not none["dW"].any() and not none["dX"].any() and ctx.last_step()[1] == 0


@pytest.mark.parametrize("B,Ci,Co,H,W", [(300, 72, 136, 9, 8), (598, 64, 64, 8, 8), (24, 64, 256, 28, 28)])
def test_thin_layers_clip_and_count(ctx, B, Ci, Co, H, W):
    """A stage that holds a code out of range is decided again with care: every code and the counts are as if each element
    had been decided by itself, in the first and the last places of rows, chunks, stages and images."""
    import paper_2004_04729_b200 as dbp
    L = wl.conv_layer(B, Ci, Co, H, W, 1, data_seed=B + Ci, scale=2.0, seed=7, dtype="bf16")
    delta = L.delta.copy()
    at = [(0, 0, 0, 0), (0, 0, H - 1, W - 1), (0, Co - 1, 0, 1), (B - 1, Co - 1, H - 1, W - 1), (B // 2, Co // 2, H // 2, W // 2),
          (1, min(63, Co - 1), 0, 0), (1, min(64, Co - 1), 0, 7)]
    for i, a in enumerate(at):
        delta[a] = (-1.0) ** i * (1.0 if i < 5 else 0.0635)      # far out of range, and about its edge: 0.0635 is 127 steps
    d, X, Wt = (torch.from_numpy(np.ascontiguousarray(a)).bfloat16().cuda() for a in (delta, L.X, L.W))
    delta = d.float().cpu().numpy()
    D = np.float32(5e-4)
    codes, nnz, sat = oracle.nsd_codes(delta, L.seed, D)
    assert sat >= 5
    out = dbp.dithered_conv_backward(ctx, d, X, Wt, L.seed, 0.0, delta_in=torch.tensor([float(D)], device="cuda"))
    assert ctx.last_step() == (float(D), nnz)
    assert ctx.last_device_status()[1] == sat
    ref = oracle.conv_backward(codes, D, L.X, L.W, with_abs=True)
    g = out["dW"].double().cpu().numpy()
    assert np.all(np.abs(g - ref["dW"]) <= TOL * ref["S_dW"] + 1e-30)
    g = out["dX"].double().cpu().numpy()
    assert np.all(np.abs(g - ref["dX"]) <= 2.0 ** -8 * np.abs(ref["dX"]) + TOL * ref["S_dX"] + 1e-30)
