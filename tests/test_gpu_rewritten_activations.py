"""Activations that are re-written before the weight-gradient kernels read them (two bf16 pieces of fp32 values, planes that are no
multiple of 16 bytes, stacked tiny planes, stride-2 phases): on whichever stream that is done, X is read after its producer and the
buffer is not written again before the kernels of an earlier call have read it."""
import numpy as np
import pytest
import torch

import oracle
import workloads as wl

pytestmark = pytest.mark.gpu
TOL = 1e-5

# B, Ci, Co, H, W (of X), k, stride, dtype: small ones, re-written beside the quantizer, and ones of 2^25 multiply-adds and more
LAYERS = [(4, 72, 40, 9, 11, 1, 1, "f32"), (3, 64, 48, 7, 7, 3, 1, "bf16"), (2, 40, 64, 20, 20, 3, 1, "f32"), (8, 32, 64, 4, 4, 3, 1, "f32"),
          (4, 128, 64, 14, 14, 3, 2, "bf16"), (4, 64, 40, 14, 14, 1, 2, "bf16"),
          (16, 72, 136, 27, 19, 1, 1, "f32"), (16, 128, 128, 7, 7, 3, 1, "bf16"), (8, 128, 64, 14, 14, 3, 1, "f32"), (64, 64, 64, 4, 4, 3, 1, "f32"),
          (8, 128, 64, 14, 14, 3, 2, "bf16"), (32, 128, 192, 14, 14, 1, 2, "bf16"), (8, 64, 64, 28, 28, 3, 2, "f32")]


@pytest.fixture(scope="module")
def ctx():
    import paper_2004_04729_b200 as dbp
    c = dbp.Context(0)
    yield c
    c.close()


def _layer(i, seed):
    B, Ci, Co, H, W, k, stride, dtype = LAYERS[i]
    rng = np.random.default_rng(100 * i + seed)
    tdt = torch.bfloat16 if dtype == "bf16" else torch.float32
    put = lambda a: torch.from_numpy(a.astype(np.float32)).to(tdt).cuda()
    return (put(rng.laplace(0.0, 1e-3, (B, Co, H // stride, W // stride))), put(np.maximum(rng.standard_normal((B, Ci, H, W)), 0)),
            put(rng.standard_normal((Co, Ci, k, k)) * 0.1), stride)


def _call(ctx, layer, seed, flags=0, X=None):
    import paper_2004_04729_b200 as dbp
    d, Xl, W, stride = layer
    return dbp.dithered_conv_backward(ctx, d, Xl if X is None else X, W, seed, 2.0, flags=flags | dbp.DBP_DX_F32, stride=stride)


def _same(a, b):
    assert torch.equal(a["dX"], b["dX"])
    # the parts of dW arrive in any order
    assert (a["dW"] - b["dW"]).abs().max().item() <= 1e-5 * b["dW"].abs().max().item()


@pytest.fixture(scope="module")
def alone(ctx):
    """Every layer with two inputs by itself, checked against the oracle."""
    out = {}
    for i, (_, _, _, _, _, _, stride, _) in enumerate(LAYERS):
        for seed in (1, 2):
            layer = _layer(i, seed)
            r = _call(ctx, layer, seed)
            torch.cuda.synchronize()
            D, _ = ctx.last_step()
            d, X, W = (t.float().cpu().numpy() for t in layer[:3])
            codes, _, _ = oracle.nsd_codes(d, seed, np.float32(D))
            if stride == 1:
                ref = oracle.conv_backward(codes, np.float32(D), X, W, with_abs=True)
                assert np.all(np.abs(r["dW"].double().cpu().numpy() - ref["dW"]) <= TOL * ref["S_dW"] + 1e-30)
            else:
                ref = oracle.conv_backward_strided(codes, np.float32(D), X, W, stride)
                g = r["dW"].double().cpu().numpy()
                assert np.linalg.norm(g - ref["dW"]) <= TOL * np.linalg.norm(ref["dW"])
            out[i, seed] = layer, r
    return out


@pytest.mark.parametrize("i", range(len(LAYERS)))
def test_activations_still_being_written_when_the_call_is_made(ctx, alone, i):
    layer, ref = alone[i, 1]
    X = torch.zeros_like(layer[1])
    big = torch.randn(4096, 4096, device="cuda")
    torch.cuda.synchronize()
    for _ in range(4):                       # some hundred microseconds in front of the copy that makes X
        big = big @ big * 1e-2
    X.copy_(layer[1])
    out = _call(ctx, layer, 1, X=X)
    X.zero_()                                # in stream order behind the joined call, which must have read X by then
    torch.cuda.synchronize()
    _same(out, ref)


def test_overlapped_and_joined_calls_in_turn(ctx, alone):
    """Both sets of buffers, each re-used by other layers with other data while earlier dW kernels may still run."""
    import paper_2004_04729_b200 as dbp
    order = [(i, seed) for seed in (1, 2) for i in range(len(LAYERS))] * 2
    for pattern in ("aj", "aaj", "ja", "aaja", "jjaaa"):
        outs = []
        for n, key in enumerate(order):
            overlapped = pattern[n % len(pattern)] == "a"
            outs.append(_call(ctx, alone[key][0], key[1], dbp.DBP_DW_ASYNC if overlapped else 0))
        ctx.join()
        torch.cuda.synchronize()
        assert ctx.last_device_status() == (0, 0)
        for key, out in zip(order, outs):
            _same(out, alone[key][1])
