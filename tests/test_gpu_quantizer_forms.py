"""Every form in which the quantizers write codes for the product kernels, at the edges of its tiles and runs and with codes out of
range among them: the counts are the oracle's, and the products are those of the oracle's codes."""
import numpy as np
import pytest
import torch

import oracle
import workloads as wl

pytestmark = pytest.mark.gpu
TOL = 1e-5                       # relative to the sum of the terms' magnitudes; a bf16 dX is rounded once more (2^-8)


@pytest.fixture(scope="module")
def ctx():
    import paper_2004_04729_b200 as dbp
    c = dbp.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("B,Ci,Co,H,W,k,dtype,mask", [
    # position-major, planes of a multiple of eight or four elements
    (3, 16, 72, 8, 8, 3, "bf16", False), (2, 24, 136, 12, 18, 3, "bf16", False), (5, 16, 64, 14, 14, 3, "bf16", False),
    (2, 16, 40, 14, 14, 3, "f32", True), (1, 8, 66, 16, 17, 3, "f32", False), (3, 40, 72, 26, 26, 3, "f32", True),
    # ... whole images of small planes, several to a tile, and the copy with rows of zeros
    (301, 16, 136, 2, 2, 3, "f32", True), (150, 24, 512, 4, 4, 3, "f32", True), (77, 16, 128, 2, 6, 3, "f32", False),
    (610, 16, 64, 4, 4, 3, "bf16", False), (310, 16, 72, 2, 2, 3, "bf16", False),
    # ... odd planes: runs of channels of one image, in one round and two; with the copy; channels that are no multiple of 8
    (3, 16, 64, 7, 7, 3, "bf16", False), (2, 24, 96, 13, 13, 3, "bf16", False), (2, 16, 40, 21, 37, 3, "f32", True),
    (9, 16, 72, 3, 5, 3, "f32", True), (2, 16, 30, 7, 7, 3, "f32", True), (1, 16, 24, 33, 41, 3, "bf16", False),
    (150, 16, 184, 5, 5, 3, "bf16", False), (150, 16, 184, 5, 5, 3, "f32", True),      # ... runs of 64 and 56 channels, two to a block
    # planes at a padded pitch: a multiple of four, odd ones of less and of more than a run, tensors that end within a vector, second
    # runs of a block, the smallest
    (3, 24, 40, 14, 14, 1, "bf16", False), (7, 16, 72, 2, 6, 1, "bf16", False), (2, 24, 40, 10, 18, 1, "f32", True),
    (5, 16, 72, 7, 7, 1, "bf16", False), (4, 16, 24, 27, 19, 1, "f32", True), (1, 16, 16, 23, 45, 1, "bf16", False),
    (3, 24, 41, 5, 5, 1, "f32", False), (2, 16, 9, 7, 9, 1, "bf16", False),
    (9, 16, 7, 59, 59, 1, "bf16", False), (33, 16, 20, 53, 53, 1, "bf16", False), (33, 16, 20, 53, 53, 1, "f32", True),
    (1, 8, 3, 1, 2, 1, "bf16", False), (1001, 48, 9, 1, 1, 1, "bf16", False), (4003, 72, 463, 1, 1, 1, "f32", True),
    # planes back to back, with a last tile that is not whole and a tail shorter than a vector
    (3, 24, 40, 16, 16, 1, "bf16", False), (2, 16, 24, 24, 20, 1, "f32", True), (300, 200, 90, 1, 1, 1, "f32", True),
    (523, 72, 41, 1, 1, 1, "bf16", False), (600, 260, 257, 1, 1, 1, "f32", False),
    # bytes
    (5, 3, 7, 9, 11, 5, "f32", True), (130, 6, 16, 16, 16, 5, "f32", True)])
def test_forms(ctx, B, Ci, Co, H, W, k, dtype, mask):
    import paper_2004_04729_b200 as dbp
    linear = H == W == 1
    L = wl.conv_layer(B, Ci, Co, H, W, k, data_seed=B + Ci + 3 * Co + H, scale=2.0, seed=11, dtype=dtype)
    tdt = torch.bfloat16 if dtype == "bf16" else torch.float32
    delta = L.delta.copy()
    flat = delta.reshape(-1)
    n = flat.size
    places = sorted({0, 1, H * W - 1, min(n - 1, H * W), n // 3, n // 2 + 1, n - 2, n - 1, min(n - 1, 4095), min(n - 1, 4097)})
    for i, a in enumerate(places):
        flat[a] = (-1.0) ** i * (1.0 if i % 2 else 0.0635)       # far out of range, and about its edge (127 steps)
    m = (np.random.default_rng(3).random(delta.shape) < 0.8).astype(np.uint8) if mask else None
    d, X, Wt = (torch.from_numpy(np.ascontiguousarray(a)).to(tdt).cuda() for a in (delta, L.X, L.W))
    dz = d.float().cpu().numpy() * (m if mask else 1.0).astype(np.float32) if mask else d.float().cpu().numpy()
    D = np.float32(5e-4)
    step = torch.tensor([float(D)], device="cuda")
    codes, nnz, sat = oracle.nsd_codes(dz, L.seed, D)
    assert sat > 0
    if mask:
        tm = torch.from_numpy(m).cuda()
        ctx.set_relu_mask(tm)
    args = (d.view(B, Co), X.view(B, Ci), Wt.view(Co, Ci)) if linear else (d, X, Wt)
    fn = dbp.dithered_linear_backward if linear else dbp.dithered_conv_backward
    out = fn(ctx, *args, L.seed, 0.0, delta_in=step)
    assert ctx.last_step() == (float(D), nnz)
    assert ctx.last_device_status()[1] == sat
    ref = oracle.conv_backward(codes, D, X.float().cpu().numpy(), Wt.float().cpu().numpy(), with_abs=True)
    g = out["dW"].double().cpu().numpy().reshape(ref["dW"].shape)
    assert np.all(np.abs(g - ref["dW"]) <= TOL * ref["S_dW"] + 1e-30)
    g = out["dX"].double().cpu().numpy().reshape(ref["dX"].shape)
    rounded = 2.0 ** -8 * np.abs(ref["dX"]) if dtype == "bf16" else 0.0
    assert np.all(np.abs(g - ref["dX"]) <= rounded + TOL * ref["S_dX"] + 1e-30)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("n", [1, 31, 1023, 1024, 1025, 1024 * 37 + 511, 1024 * 8 * 1200])
def test_sparse_form(ctx, n, dtype):
    """Whole segments without a code out of range, with some, and the last, partial one."""
    import paper_2004_04729_b200 as dbp
    tdt = torch.bfloat16 if dtype == "bf16" else torch.float32
    x = np.random.default_rng(n).laplace(0.0, 1e-3, n).astype(np.float32)
    for i, a in enumerate({0, n // 2, n - 1, max(0, n - 1025)}):
        x[a] = (-1.0) ** i * (1.0 if i % 2 else 0.0635)
    d = torch.from_numpy(x).to(tdt).cuda()
    D = np.float32(5e-4)
    codes, nnz, sat = oracle.nsd_codes(d.float().cpu().numpy(), 5, D)
    q = dbp.nsd_quantize(ctx, d, 5, 0.0, delta_in=torch.tensor([float(D)], device="cuda"))
    assert q.nnz.item() == nnz and ctx.last_device_status()[1] == sat
    assert np.array_equal(dbp.nsd_decode_dense(ctx, q).cpu().numpy().reshape(-1), codes)


@pytest.mark.parametrize("masked", [False, True])
def test_step_size_of_a_large_tensor_beside_an_earlier_dw(ctx, masked):
    """Large fp32 gradients are added up by fewer blocks while an earlier call's dW is outstanding: the step size and the count keep their
    bits, and the step size is the one in 64 bits to 1e-6. (Ragged planes: the last tile of the sums is not whole.)"""
    import paper_2004_04729_b200 as dbp
    g = torch.Generator(device="cuda").manual_seed(3)
    delta = torch.randn(16, 128, 111, 111, generator=g, device="cuda") + 0.25
    X, W = torch.randn(16, 8, 111, 111, generator=g, device="cuda"), torch.randn(128, 8, 1, 1, generator=g, device="cuda")
    mask = (torch.rand(delta.shape, generator=g, device="cuda") < 0.6).to(torch.uint8) if masked else None
    steps = []
    for flags in (0, dbp.DBP_DW_ASYNC, dbp.DBP_DW_ASYNC):          # the last call comes behind an outstanding dW
        ctx.set_relu_mask(mask)
        out = dbp.dithered_conv_backward(ctx, delta, X, W, 11, 2.0, flags=flags)
        if len(steps) == 1:
            steps.append(None)
            continue
        ctx.join()
        steps.append(ctx.last_step())
    assert steps[0] == steps[2]
    want = 2.0 * (delta * mask if masked else delta).double().std(unbiased=False).item()
    assert abs(steps[0][0] - want) <= 1e-6 * want
    assert ctx.last_device_status() == (0, 0)
