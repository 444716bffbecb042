"""3x3 input gradients whose patches share halos, whose reduction over output channels is split over a cluster of CTAs, or
whose weight pieces share the accumulator, or that leave by whole blocks: parity with the oracle and bit-identical repeats."""
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
    (1, 512, 512, 7, 7, "bf16"), (9, 256, 512, 7, 7, "bf16"), (5, 200, 320, 4, 6, "bf16"),    # clusters, partial last patches
    (3, 128, 576, 2, 2, "bf16"),                                                              # nine blocks of channels over a cluster
    (30, 512, 136, 2, 2, "f32"), (7, 136, 512, 4, 4, "f32"), (2, 264, 128, 14, 14, "f32"),
    (1, 128, 128, 1, 1, "f32"),
    (3, 64, 64, 13, 32, "f32"), (2, 40, 72, 9, 11, "f32"), (1, 3, 200, 33, 62, "f32"),       # both weight pieces in one MMA:
    (9, 56, 352, 16, 16, "f32"), (12, 16, 88, 30, 30, "f32"), (6, 38, 98, 12, 12, "f32"),    # ... in whole blocks or not, as dW asks
    (9, 40, 72, 6, 24, "bf16"), (5, 200, 72, 6, 25, "f32"), (40, 130, 136, 5, 5, "f32"),       # dX and dW share every SM, or not
    (3, 64, 72, 26, 26, "f32"), (2, 72, 136, 7, 56, "bf16"), (1, 256, 128, 12, 59, "f32"), (1, 136, 72, 9, 60, "bf16"),   # half an SM: widest rows
    (3, 40, 24, 9, 56, "bf16"), (2, 72, 16, 10, 28, "bf16"), (2, 24, 24, 22, 60, "bf16"),      # dX by whole blocks: partial last
    (2, 136, 40, 11, 16, "f32"), (9, 136, 64, 4, 8, "f32"), (1, 64, 8, 31, 48, "f32"),        # patches, several images, ragged rows
    (69, 98, 274, 2, 2, "f32"), (33, 136, 520, 2, 3, "bf16"), (60, 200, 392, 1, 4, "f32"),    # rows of several images: no kernel row above or
    (50, 130, 456, 5, 1, "f32"), (33, 128, 312, 7, 7, "f32"), (17, 72, 500, 4, 5, "bf16"),    # ... below, one column, ragged images and channels,
    (14, 896, 352, 9, 9, "f32"), (24, 136, 1000, 2, 2, "f32")])                                # ... clusters of two to eight, wide tiles
def test_input_gradient(ctx, B, Ci, Co, H, W, dtype):
    import paper_2004_04729_b200 as dbp
    L = wl.conv_layer(B, Ci, Co, H, W, 3, data_seed=B + Ci + 5 * Co + H, scale=2.0, seed=9, dtype=dtype)
    tdt = torch.bfloat16 if dtype == "bf16" else torch.float32
    d, X, Wt = (torch.from_numpy(np.ascontiguousarray(a)).to(tdt).cuda() for a in (L.delta, L.X, L.W))
    out = dbp.dithered_conv_backward(ctx, d, X, Wt, L.seed, L.scale, flags=dbp.DBP_DX_F32)
    D, _ = ctx.last_step()
    assert ctx.last_device_status() == (0, 0)
    codes, _, _ = oracle.nsd_codes(L.delta, L.seed, np.float32(D))
    ref = oracle.conv_backward(codes, np.float32(D), L.X, L.W, with_abs=True)
    for key in ("dX", "dW"):
        g = out[key].double().cpu().numpy()
        assert np.linalg.norm(g - ref[key]) <= TOL * np.linalg.norm(ref[key]) + 1e-30, key
        assert np.all(np.abs(g - ref[key]) <= TOL * ref["S_" + key] + 1e-30), key
    for kw in ({"need_dW": False}, {"need_dW": False}, {"flags": dbp.DBP_DW_ASYNC}, {}):
        again = dbp.dithered_conv_backward(ctx, d, X, Wt, L.seed, L.scale, **kw)["dX"]
        ctx.join()
        assert torch.equal(again, out["dX"].to(again.dtype)), kw


@pytest.mark.parametrize("B,Ci,Co,H,W,dtype", [
    (50, 72, 136, 8, 8, "bf16"), (41, 130, 72, 7, 9, "f32"),           # images of one block: several code buffers, ragged channels
    (70, 40, 200, 3, 5, "bf16"), (33, 16, 65, 8, 16, "f32"),           # ... and of two blocks, one output channel past a panel
    (3, 7, 130, 12, 11, "bf16"), (2, 129, 129, 20, 9, "f32"),          # channels that are no multiple of four in dW's rows
    (2, 1, 65, 5, 4, "f32"), (2, 4, 72, 3, 6, "bf16"), (3, 13, 40, 6, 6, "f32"),      # ... rows of one to four groups of channels, the last one empty
    (2, 332, 1000, 4, 5, "bf16"),                                      # ... more groups than the finishing kernel has threads
    (2, 24, 72, 24, 24, "f32"), (2, 40, 130, 9, 44, "bf16"),           # segments of 192 positions, of 128 for the next quantizer's sake, of 128
    (3, 200, 72, 13, 13, "f32"), (2, 16, 48, 24, 24, "f32"), (2, 16, 72, 5, 62, "bf16")])       # ... of a whole image, one panel, the widest rows
def test_weight_gradient_of_a_whole_sm(ctx, B, Ci, Co, H, W, dtype):
    """An overlapped call's dW kernel has the SMs to itself, and so has that of a call without dX, with other segments. Twice each: the
    next call adds into a scratch that the one before put back to zero. (Tolerance: fp32 sums of exact products, as above.)"""
    import paper_2004_04729_b200 as dbp
    L = wl.conv_layer(B, Ci, Co, H, W, 3, data_seed=B + Ci + 3 * Co + H, scale=2.0, seed=11, dtype=dtype)
    tdt = torch.bfloat16 if dtype == "bf16" else torch.float32
    d, X, Wt = (torch.from_numpy(np.ascontiguousarray(a)).to(tdt).cuda() for a in (L.delta, L.X, L.W))
    ref = None
    for kw in 2 * (dict(flags=dbp.DBP_DW_ASYNC), dict(need_dX=False)):
        out = dbp.dithered_conv_backward(ctx, d, X, Wt, L.seed, L.scale, **kw)
        ctx.join()
        D, _ = ctx.last_step()
        if ref is None:
            codes, _, _ = oracle.nsd_codes(L.delta, L.seed, np.float32(D))
            ref = oracle.conv_backward(codes, np.float32(D), L.X, L.W, with_abs=True)
        g = out["dW"].double().cpu().numpy()
        assert np.linalg.norm(g - ref["dW"]) <= TOL * np.linalg.norm(ref["dW"]) + 1e-30
        assert np.all(np.abs(g - ref["dW"]) <= TOL * ref["S_dW"] + 1e-30)
    assert ctx.last_device_status() == (0, 0)


def test_threads_launch_the_same_kernels_with_other_sizes():
    """Two threads, a context and a stream each, with layers whose kernels are the same functions with different amounts of shared
    memory: every call goes through, and dX has the bits that it has alone (dW's partial sums meet in any order: fp32 sums)."""
    import threading
    import paper_2004_04729_b200 as dbp
    shapes = [[(70, 128, 256, 8, 8), (40, 72, 136, 14, 14), (8, 16, 128, 24, 24)], [(33, 128, 64, 2, 3), (5, 96, 72, 5, 5), (4, 64, 72, 7, 20)]]
    errors = []

    def work(which):
        try:
            stream = torch.cuda.Stream()
            with torch.cuda.stream(stream):
                ctx = dbp.Context(0, stream)
                gen = torch.Generator(device="cuda").manual_seed(which)
                rnd = lambda *s: torch.randn(*s, generator=gen, device="cuda")
                layers = [(rnd(B, Co, H, W), rnd(B, Ci, H, W), rnd(Co, Ci, 3, 3)) for B, Ci, Co, H, W in shapes[which]]
                first = [None] * len(layers)
                for turn in range(200):
                    for i, (d, X, Wt) in enumerate(layers):
                        out = dbp.dithered_conv_backward(ctx, d, X, Wt, 7, 2.0)
                        if turn % 20 == 0:
                            if first[i] is None:
                                first[i] = {k: out[k].clone() for k in ("dX", "dW")}
                            assert torch.equal(out["dX"], first[i]["dX"])
                            assert (out["dW"] - first[i]["dW"]).norm().item() <= TOL * first[i]["dW"].norm().item()
                assert ctx.last_device_status() == (0, 0)
                ctx.close()
        except BaseException as e:                       # (an assertion in a thread would be lost)
            errors.append(e)

    threads = [threading.Thread(target=work, args=(t,)) for t in (0, 1)]
    for t in threads: t.start()
    for t in threads: t.join()
    assert not errors, errors
