"""GPU parity of the tensor path's routes for channel counts that are no multiple of 16, output rows without 16-byte
alignment, and full-range unsigned bytes with padding (bit-exact against the CPU oracle)."""
import numpy as np
import pytest

from psb_testlib import compare, gpu_layer, oracle_layer

pytestmark = pytest.mark.gpu

# (N, C, H, W, O, K, stride, pad, layout, dtype, largest magnitude, shortcut dtype or None, levels or None)
CASES = [
    (3, 100, 9, 13, 150, 3, 1, 1, 1, np.uint8, 255, None, None),       # rows of 2-byte units, two channel blocks
    (2, 17, 11, 9, 33, 3, 1, 1, 1, np.uint8, 255, np.uint8, None),     # single bytes, padded to one K block
    (4, 31, 13, 12, 20, 5, 2, 2, 0, np.uint8, 255, np.int8, None),     # planar in and out, 4-byte units
    (5, 36, 8, 7, 100, 1, 1, 0, 1, np.int8, 127, np.uint8, None),      # plain matrix product, rows of 4-byte units
    (2, 64, 12, 11, 64, 3, 1, 1, 1, np.uint8, 255, None, None),        # no repacking, the flip only
    (4, 96, 15, 9, 72, 3, 2, 1, 1, np.uint8, 200, np.uint8, None),     # partly filled last channel block, in_max < 255
    (3, 40, 7, 9, 24, 3, 1, 1, 1, np.uint8, 255, None, (0, 3, 4)),     # draw-count map on flipped, repacked rows
    (150, 333, 1, 1, 31, 1, 1, 0, 1, np.uint8, 255, None, None),       # fully connected, odd everything
    (4, 16, 9, 9, 48, 1, 1, 0, 1, np.uint8, 15, None, None),           # rows narrower than a K block
]


@pytest.mark.parametrize("want", [("q",), ("q", "f32", "acc")])
@pytest.mark.parametrize("case", CASES)
def test_odd_layers_on_the_tensor_path(case, want, oracle):
    import paper_1904_02205_b200 as psb

    N, C, H, W, O, K, stride, pad, layout, dtype, top, res_dtype, levels = case
    ctx = psb.Context(0)
    rng = np.random.default_rng(C * 7 + O)
    w = rng.normal(0, np.sqrt(2.0 / (C * K * K)), size=(O, C, K, K)).astype(np.float32)
    x = rng.integers(0 if dtype == np.uint8 else -top, top + 1, size=(N, C, H, W) if layout == 0 else (N, H, W, C)).astype(dtype)
    oh, ow = (H + 2 * pad - K) // stride + 1, (W + 2 * pad - K) // stride + 1
    res = None
    if res_dtype is not None:
        lo = 0 if res_dtype == np.uint8 else -128
        res = rng.integers(lo, lo + 256, size=(N, O, oh, ow) if layout == 0 else (N, oh, ow, O)).astype(res_dtype)
    kmap = None if levels is None else rng.choice(levels, size=(N, oh, ow)).astype(np.uint8)
    args = (w, x, layout, 1, stride, pad, 5, 3, list(levels or (3,)), kmap, 3, rng.uniform(0.5, 1.5, O).astype(np.float32),
            rng.normal(0, 0.5, O).astype(np.float32), True, np.float32(0.02), 0, 255)
    o = oracle_layer(oracle, *args, residual=res, res_scale=np.float32(0.3))
    g = gpu_layer(psb, ctx, *args, psb.PSB_DT_U8, residual=res, res_scale=np.float32(0.3), in_max=top, path=psb.PSB_PATH_TENSOR,
                  want=want)
    compare(g, o, list(levels or (3,)))
    assert g["path"] == psb.PSB_PATH_TENSOR
    ctx.close()


def test_rows_that_start_at_odd_addresses(oracle):
    """An input tensor at an address the copy engine cannot take is repacked first."""
    import torch

    import paper_1904_02205_b200 as psb

    ctx = psb.Context(0)
    rng = np.random.default_rng(3)
    w = rng.normal(0, 0.2, size=(32, 48, 1, 1)).astype(np.float32)
    x = rng.integers(0, 16, size=(200, 48)).astype(np.uint8)
    flat = torch.zeros(200 * 48 + 16, dtype=torch.uint8, device=ctx.device)
    wt = ctx.sample_weights(torch.from_numpy(w).to(ctx.device), seed=1, level_mask=8)
    ctx.set_sample_map(None, 3)
    one = torch.ones(32, device=ctx.device)
    W, eb, _ = oracle.sample_level(w, 1, 0, 3)
    acc = x.astype(np.int64) @ W.reshape(32, 48).astype(np.int64).T
    for shift in (1, 4, 7, 8):
        flat[shift:shift + x.size] = torch.from_numpy(x.ravel()).to(ctx.device)
        got = ctx.gemm(wt, flat[shift:shift + x.size].view(200, 48), one, one, False, 1.0, 0, 255, in_max=15,
                       path=psb.PSB_PATH_TENSOR, want=("acc",))["acc"].cpu().numpy()
        assert ctx.device_status() == 0 and np.array_equal(got, acc)
    wt.free()
    ctx.close()


@pytest.mark.parametrize("case", [
    # (N, H, W, C, O, shortcut dtype, exp_bits, log2k, in_max): several tiles per SM, ragged last rows and channel tiles
    (19, 56, 55, 64, 64, np.uint8, 4, 3, 15), (30, 49, 41, 32, 80, np.int8, 4, 3, 15), (19, 56, 55, 64, 64, np.int8, 3, 0, 15),
    (8, 57, 61, 128, 144, np.uint8, 4, 6, 15), (19, 56, 57, 256, 64, np.int8, 4, 6, 127),
])
@pytest.mark.parametrize("signed_out", [False, True])
def test_shortcut_tiles_through_shared_memory(case, signed_out, oracle):
    """Layers with a shortcut and enough tiles for the staged output stage: two to four planes, 32- and 64-bit
    recombination, a second channel tile that is partly or wholly beyond the channels."""
    import torch

    import paper_1904_02205_b200 as psb

    N, H, W, C, O, res_dtype, exp_bits, log2k, top = case
    assert -(-N * H * W // 128) * -(-O // 64) >= 3 * 148
    ctx = psb.Context(0)
    rng = np.random.default_rng(O + H)
    w = rng.normal(0, np.sqrt(2.0 / C), size=(O, C, 1, 1)).astype(np.float32)
    x = rng.integers(0, top + 1, size=(N, H, W, C)).astype(np.uint8)
    lo = 0 if res_dtype == np.uint8 else -128
    res = rng.integers(lo, lo + 256, size=(N, H, W, O)).astype(res_dtype)
    scale, bias = rng.uniform(0.5, 1.5, O).astype(np.float32), rng.normal(0, 0.5, O).astype(np.float32)
    dev = lambda t: torch.from_numpy(t).to(ctx.device)
    wt = ctx.sample_weights(dev(w), seed=5, layer_id=3, level_mask=1 << log2k, exp_bits=exp_bits)
    ctx.set_sample_map(None, log2k)
    qmin, qmax = (-100, 101) if signed_out else (0, 15)
    inv_step = np.float32(0.5)
    q = ctx.conv2d(wt, dev(x), psb.PSB_LAYOUT_NHWC, 1, 0, dev(scale), dev(bias), not signed_out, inv_step, qmin, qmax,
                   out_dtype=psb.PSB_DT_S8 if signed_out else psb.PSB_DT_U8, residual=dev(res), residual_scale=0.3, in_max=top,
                   path=psb.PSB_PATH_TENSOR)["q"].cpu().numpy()
    assert ctx.device_status() == 0
    # first and last image against the oracle
    for n in (0, N - 1):
        o = oracle_layer(oracle, w, x[n:n + 1], 1, 1, 1, 0, 5, 3, [log2k], None, log2k, scale, bias, not signed_out, inv_step, qmin,
                         qmax, residual=res[n:n + 1], res_scale=np.float32(0.3), exp_bits=exp_bits)
        assert np.array_equal(q[n:n + 1].astype(np.int32), o["q"])
    wt.free()
    ctx.close()


@pytest.mark.parametrize("case", [
    # (N, C, H, W, O, K, stride, shortcut dtype, exp_bits, log2k, largest byte, sums that fit 32 bits), each with and without an
    # addend where the bytes are unsigned, three planes, then two and four
    (19, 3, 112, 111, 64, 7, 2, np.uint8, 4, 3, 255, False), (19, 3, 112, 111, 64, 7, 2, np.int8, 4, 0, 255, True),
    (13, 12, 40, 39, 144, 3, 1, np.int8, 4, 4, 255, False), (13, 12, 40, 39, 144, 3, 1, np.uint8, 4, 1, 15, True),
    (13, 12, 40, 39, 144, 3, 1, np.uint8, 4, 3, -127, True), (13, 12, 40, 39, 144, 5, 1, np.uint8, 4, 4, -127, False),
    (13, 12, 40, 39, 144, 3, 1, np.uint8, 3, 2, 255, True), (19, 3, 112, 111, 64, 7, 2, np.uint8, 4, 6, 255, False),
])
@pytest.mark.parametrize("signed_out", [False, True])
def test_shortcut_of_a_flat_k_axis(case, signed_out, oracle):
    """Filters with fewer than 16 input channels, a shortcut, and enough tiles for the staged output stage."""
    import torch

    import paper_1904_02205_b200 as psb

    N, C, H, W, O, K, stride, res_dtype, exp_bits, log2k, top, fits = case
    oh, ow = (H + 2 * (K // 2) - K) // stride + 1, (W + 2 * (K // 2) - K) // stride + 1
    assert -(-N * oh * ow // 128) * -(-O // 64) >= 3 * 148 and O % 16 == 0
    ctx = psb.Context(0)
    rng = np.random.default_rng(O + H + log2k)
    w = rng.normal(0, np.sqrt(2.0 / (C * K * K)), size=(O, C, K, K)).astype(np.float32)
    x = rng.integers(min(top, 0), abs(top) + 1, size=(N, H, W, C)).astype(np.uint8 if top > 0 else np.int8)
    lo = 0 if res_dtype == np.uint8 else -128
    res = rng.integers(lo, lo + 256, size=(N, oh, ow, O)).astype(res_dtype)
    scale, bias = rng.uniform(0.5, 1.5, O).astype(np.float32), rng.normal(0, 0.5, O).astype(np.float32)
    # the output stage's bound: row sums of |W| in units of 256, each contribution rounded up
    sums = np.abs(oracle.sample_level(w, 5, 3, log2k, exp_bits=exp_bits)[0].astype(np.int64)).reshape(O, -1)
    assert (int((-(-sums // 256)).sum(1).max()) * 256 * abs(top) < 1 << 31) == fits
    assert fits or int(sums.sum(1).max()) * abs(top) >= 1 << 31
    dev = lambda t: torch.from_numpy(t).to(ctx.device)
    wt = ctx.sample_weights(dev(w), seed=5, layer_id=3, level_mask=1 << log2k, exp_bits=exp_bits)
    ctx.set_sample_map(None, log2k)
    qmin, qmax = (-100, 101) if signed_out else (0, 255)
    inv_step = np.float32(32.0 / abs(top))
    q = ctx.conv2d(wt, dev(x), psb.PSB_LAYOUT_NHWC, stride, K // 2, dev(scale), dev(bias), not signed_out, inv_step, qmin, qmax,
                   out_dtype=psb.PSB_DT_S8 if signed_out else psb.PSB_DT_U8, residual=dev(res), residual_scale=0.3, in_max=abs(top),
                   path=psb.PSB_PATH_TENSOR)["q"].cpu().numpy()
    assert ctx.device_status() == 0
    # first and last image against the oracle
    for n in (0, N - 1):
        o = oracle_layer(oracle, w, x[n:n + 1], 1, 1, stride, K // 2, 5, 3, [log2k], None, log2k, scale, bias, not signed_out, inv_step,
                         qmin, qmax, residual=res[n:n + 1], res_scale=np.float32(0.3), exp_bits=exp_bits)
        assert np.array_equal(q[n:n + 1].astype(np.int32), o["q"])
        assert len(np.unique(q[n])) > 50
    wt.free()
    ctx.close()


@pytest.mark.parametrize("case", [
    # (N, C, H, W, stride, dtype, shortcut dtype or None): odd channel counts, one row or column, long strips, wide sums
    (2, 37, 9, 11, 1, np.uint8, None), (1, 5, 7, 1, 2, np.int8, None), (3, 64, 1, 13, 1, np.uint8, np.int8),
    (1, 8, 61, 9, 1, np.int8, np.uint8), (2, 12, 64, 33, 2, np.uint8, None), (130, 48, 14, 15, 1, np.uint8, None),
    (2, 39, 30, 17, 2, np.uint8, np.uint8),
])
@pytest.mark.parametrize("log2k,flat", [(4, False), (6, True)])
def test_depthwise_strips(case, log2k, flat, oracle):
    """flat: all weights near the window's top, so that the sums do not fit 32 bits."""
    import paper_1904_02205_b200 as psb

    N, C, H, W, stride, dtype, res_dtype = case
    ctx = psb.Context(0)
    rng = np.random.default_rng(C * 3 + H)
    w = rng.normal(0, 0.3, size=(C, 1, 3, 3)).astype(np.float32)
    if flat:
        w = (np.sign(w) * rng.uniform(1.5, 1.99, size=w.shape)).astype(np.float32)
    lo, hi = (0, 256) if dtype == np.uint8 else (-128, 128)
    x = rng.integers(lo, hi, size=(N, H, W, C)).astype(dtype)
    oh, ow = (H - 1) // stride + 1, (W - 1) // stride + 1
    res = None
    if res_dtype is not None:
        lo = 0 if res_dtype == np.uint8 else -128
        res = rng.integers(lo, lo + 256, size=(N, oh, ow, C)).astype(res_dtype)
    args = (w, x, 1, C, stride, 1, 5, 3, [log2k], None, log2k, rng.uniform(0.5, 1.5, C).astype(np.float32),
            rng.normal(0, 0.5, C).astype(np.float32), False, np.float32(0.05 if not flat else 0.01), -100, 101)
    o = oracle_layer(oracle, *args, residual=res, res_scale=np.float32(0.3))
    g = gpu_layer(psb, ctx, *args, psb.PSB_DT_S8, residual=res, res_scale=np.float32(0.3), want=("q",))
    compare(g, o, [log2k])
    ctx.close()


@pytest.mark.parametrize("case", [
    # (N, H, W, C, O, K, shortcut dtype or None, in_max): several tiles per SM on rows sorted by level
    (19, 56, 57, 64, 64, 1, np.uint8, 15), (30, 49, 41, 32, 80, 1, np.int8, 15), (19, 56, 57, 64, 48, 3, None, 15),
    (8, 57, 61, 128, 144, 1, np.uint8, 127),
])
@pytest.mark.parametrize("levels", [(0, 2, 4), (5, 6)])
def test_sorted_rows_through_shared_memory(case, levels, oracle):
    import torch

    import paper_1904_02205_b200 as psb

    N, H, W, C, O, K, res_dtype, top = case
    assert -(-N * H * W // 128) * -(-O // 64) >= 3 * 148
    ctx = psb.Context(0)
    rng = np.random.default_rng(O + H + levels[0])
    w = rng.normal(0, np.sqrt(2.0 / (C * K * K)), size=(O, C, K, K)).astype(np.float32)
    x = rng.integers(0, top + 1, size=(N, H, W, C)).astype(np.uint8)
    scale, bias = rng.uniform(0.5, 1.5, O).astype(np.float32), rng.normal(0, 0.5, O).astype(np.float32)
    res = None
    if res_dtype is not None:
        lo = 0 if res_dtype == np.uint8 else -128
        res = rng.integers(lo, lo + 256, size=(N, H, W, O)).astype(res_dtype)
    kmap = rng.choice(levels, size=(N, H, W)).astype(np.uint8)
    dev = lambda t: torch.from_numpy(t).to(ctx.device)
    wt = ctx.sample_weights(dev(w), seed=5, layer_id=3, level_mask=sum(1 << l for l in levels))
    run = lambda: ctx.conv2d(wt, dev(x), psb.PSB_LAYOUT_NHWC, 1, K // 2, dev(scale), dev(bias), True, np.float32(0.2), 0, 15,
                             residual=None if res is None else dev(res), residual_scale=0.3, in_max=top, path=psb.PSB_PATH_TENSOR)
    ctx.set_sample_map(dev(kmap))
    q = run()["q"].cpu().numpy()
    assert ctx.device_status() == 0
    for n in (0, N - 1):
        o = oracle_layer(oracle, w, x[n:n + 1], 1, 1, 1, K // 2, 5, 3, list(levels), kmap[n:n + 1], levels[0], scale, bias, True,
                         np.float32(0.2), 0, 15, residual=None if res is None else res[n:n + 1], res_scale=np.float32(0.3))
        assert np.array_equal(q[n:n + 1].astype(np.int32), o["q"])
    # a level that was not sampled is reported; the other locations keep their results
    bad = kmap.copy()
    bad[1, 3, :200] = 1
    ctx.set_sample_map(dev(bad))
    again = run()["q"].cpu().numpy()
    assert ctx.device_status() == psb.PSB_ERR_BAD_K
    assert np.array_equal(again[2:], q[2:])
    ctx.set_sample_map(None, 0)
    wt.free()
    ctx.close()


@pytest.mark.parametrize("case", [
    # (N, C, H, W, O, K, stride, levels or None): padded full-range unsigned bytes on 1 .. 127 locations, the activation
    # tile mostly beyond them
    (1, 24, 1, 1, 40, 3, 1, None), (2, 20, 4, 4, 30, 3, 1, None), (1, 100, 7, 7, 150, 3, 1, None), (2, 37, 7, 9, 70, 5, 1, None),
    (1, 24, 21, 11, 33, 3, 2, None), (3, 17, 6, 7, 64, 3, 1, (0, 3)),
])
def test_few_locations_of_padded_full_range_bytes(case, oracle):
    import paper_1904_02205_b200 as psb

    N, C, H, W, O, K, stride, levels = case
    ctx = psb.Context(0)
    rng = np.random.default_rng(C + O)
    w = rng.normal(0, np.sqrt(2.0 / (C * K * K)), size=(O, C, K, K)).astype(np.float32)
    x = rng.integers(0, 256, size=(N, H, W, C)).astype(np.uint8)
    oh, ow = (H + 2 * (K // 2) - K) // stride + 1, (W + 2 * (K // 2) - K) // stride + 1
    assert N * oh * ow < 128
    kmap = None if levels is None else rng.choice(levels, size=(N, oh, ow)).astype(np.uint8)
    args = (w, x, 1, 1, stride, K // 2, 5, 3, list(levels or (4,)), kmap, 4, rng.uniform(0.5, 1.5, O).astype(np.float32),
            rng.normal(0, 0.5, O).astype(np.float32), True, np.float32(0.02), 0, 255)
    o = oracle_layer(oracle, *args)
    for want in (("q",), ("q", "f32", "acc")):
        g = gpu_layer(psb, ctx, *args, psb.PSB_DT_U8, path=psb.PSB_PATH_TENSOR, want=want)
        compare(g, o, list(levels or (4,)))
        assert g["path"] == psb.PSB_PATH_TENSOR
    ctx.close()


@pytest.mark.parametrize("case", [
    # (N, C, H, W, O, K, largest magnitude, levels or None, tensor path): both sides of the line that PSB_PATH_AUTO draws
    (1, 64, 20, 15, 64, 3, 255, None, True), (1, 64, 20, 14, 64, 3, 255, None, False), (2, 256, 7, 7, 256, 3, 255, None, True),
    (1, 32, 4, 7, 32, 3, 255, None, False), (1, 100, 7, 7, 150, 3, 255, None, False), (1, 100, 8, 8, 150, 3, 255, None, True),
    (31, 512, 1, 1, 2048, 1, 15, None, True), (4, 512, 1, 1, 2048, 1, 15, None, False), (10, 52, 14, 14, 60, 1, 15, None, True),
    (1, 12, 10, 10, 128, 5, 255, None, True), (1, 12, 7, 7, 128, 5, 255, None, False), (1, 48, 6, 6, 16, 3, 255, (0, 3), False),
    (1, 48, 12, 12, 64, 3, 255, (0, 3), True),
])
def test_line_between_the_paths(case, oracle):
    import paper_1904_02205_b200 as psb

    N, C, H, W, O, K, top, levels, tensor = case
    ctx = psb.Context(0)
    rng = np.random.default_rng(C + O + H)
    w = rng.normal(0, np.sqrt(2.0 / (C * K * K)), size=(O, C, K, K)).astype(np.float32)
    x = rng.integers(0, top + 1, size=(N, H, W, C)).astype(np.uint8)
    kmap = None if levels is None else rng.choice(levels, size=(N, H, W)).astype(np.uint8)
    args = (w, x, 1, 1, 1, K // 2, 5, 3, list(levels or (3,)), kmap, 3, rng.uniform(0.5, 1.5, O).astype(np.float32),
            rng.normal(0, 0.5, O).astype(np.float32), True, np.float32(0.02), 0, 255)
    g = gpu_layer(psb, ctx, *args, psb.PSB_DT_U8, in_max=top, want=("q", "acc"))
    compare(g, oracle_layer(oracle, *args), list(levels or (3,)))
    assert g["path"] == (psb.PSB_PATH_TENSOR if tensor else psb.PSB_PATH_SHIFT_ADD)
    ctx.close()


@pytest.mark.parametrize("case", [
    # (channels, largest byte, signed input, shortcut, draw-count map): sums whose lower two planes fit 32 bits, at the limit
    # (16383 x channels x byte just below 2^31) and just beyond it, with and without an addend, and sums that fit as a whole
    (1024, 255, False, False, False), (1040, 255, False, False, False), (1024, 255, False, True, True), (1024, 127, True, True, False),
    (8736, 15, False, False, False), (8752, 15, False, True, False), (960, 255, False, True, False), (8736, 15, False, True, True),
    (16, 255, False, True, False), (16, 255, False, False, True), (1040, 255, False, True, True),
])
def test_large_sums_are_rounded_once(case, oracle):
    """Accumulators near 2^36 that differ by a few units in the last place of their fp32 value: codes show each of them."""
    import torch

    import paper_1904_02205_b200 as psb

    C, amax, signed, shortcut, with_map = case
    ctx = psb.Context(0)
    rng = np.random.default_rng(C + amax)
    O, H, W = 80, 15, 20
    # a third of the weights small: their activations vary, the others' do not
    small = rng.random(C) < 0.34
    small[0] = False
    exps = np.where(small, rng.integers(-15, -6, size=(O, C)), rng.integers(-2, 1, size=(O, C)))
    exps[:, 0] = 0
    w = (np.exp2(exps) * (1.0 + rng.random((O, C)))).astype(np.float32).reshape(O, C, 1, 1)
    dt = np.int8 if signed else np.uint8
    x = np.where(small, rng.integers(0, amax + 1, size=(1, H, W, C)), amax).astype(dt)
    res = rng.integers(0, 4, size=(1, H, W, O)).astype(np.uint8) if shortcut else None
    levels = (2, 4) if with_map else (4,)
    kmap = rng.choice(levels, size=(1, H, W)).astype(np.uint8) if with_map else None
    Ws = {l: oracle.sample_level(w, 3, 0, l)[0] for l in levels}
    eb = oracle.sample_level(w, 3, 0, 4)[1]
    g = oracle.geom(x.shape, oracle.NHWC, oracle.S8 if signed else oracle.U8, w.shape, 1, 1, 0)
    acc = oracle.conv_acc(x, g, Ws, kmap=kmap, uniform_log2k=4)
    scale = np.exp2(4.0 - eb.astype(np.float64)).astype(np.float32)
    mid = np.median(acc.reshape(-1, O) if kmap is None else acc.reshape(-1, O)[kmap.ravel() == 4], axis=0)
    bias = (-mid.astype(np.float32)).astype(np.float32)
    step = max(1.0, float(np.exp2(np.floor(np.log2(mid.max())) - 23)))
    inv_step = np.float32(1.0 / step)
    _, q = oracle.epilogue(acc, g, scale, bias, eb, False, inv_step, -128, 127, kmap=kmap, uniform_log2k=4, residual=res,
                           residual_scale=np.float32(step))
    assert len(np.unique(q)) > 50
    cu = lambda a: None if a is None else torch.from_numpy(a).to(ctx.device)
    wt = ctx.sample_weights(cu(w), seed=3, layer_id=0, level_mask=sum(1 << l for l in levels))
    ctx.set_sample_map(cu(kmap), 4)
    got = ctx.conv2d(wt, cu(x), psb.PSB_LAYOUT_NHWC, 1, 0, cu(scale), cu(bias), False, float(inv_step), -128, 127, out_dtype=psb.PSB_DT_S8,
                     residual=cu(res), residual_scale=step, in_max=amax, path=psb.PSB_PATH_TENSOR, want=("q",))["q"]
    assert ctx.device_status() == 0
    assert np.array_equal(got.cpu().numpy().astype(np.int32), q)
    ctx.set_sample_map(None, 4)
    wt.free()
    ctx.close()


@pytest.mark.parametrize("want", [("q", "f32"), ("f32",)])
@pytest.mark.parametrize("case", CASES + [
    (3, 128, 12, 11, 192, 3, 1, 1, 1, np.uint8, 15, np.uint8, None),      # whole 16-byte pieces, streamed planes
    (2, 64, 13, 11, 68, 1, 1, 0, 1, np.uint8, 127, np.int8, None),        # rows of 16 bytes of fp32, 4 of codes
    (2, 64, 13, 11, 80, 3, 2, 1, 1, np.int8, 127, None, (0, 2, 4)),       # a draw-count map
    (2, 96, 9, 14, 64, 1, 1, 0, 1, np.uint8, 255, np.uint8, (6, 2)),      # levels of three and of four planes
    (2, 160, 20, 11, 48, 3, 1, 1, 0, np.uint8, 15, np.uint8, None),       # planar
    (2, 3, 21, 19, 36, 7, 2, 3, 1, np.uint8, 255, None, None),            # flat K axis
])
def test_real_valued_outputs(case, want, oracle):
    import paper_1904_02205_b200 as psb

    N, C, H, W, O, K, stride, pad, layout, dtype, top, res_dtype, levels = case
    ctx = psb.Context(0)
    rng = np.random.default_rng(C * 11 + O)
    w = rng.normal(0, np.sqrt(2.0 / (C * K * K)), size=(O, C, K, K)).astype(np.float32)
    x = rng.integers(0 if dtype == np.uint8 else -top, top + 1, size=(N, C, H, W) if layout == 0 else (N, H, W, C)).astype(dtype)
    oh, ow = (H + 2 * pad - K) // stride + 1, (W + 2 * pad - K) // stride + 1
    res = None
    if res_dtype is not None:
        lo = 0 if res_dtype == np.uint8 else -128
        res = rng.integers(lo, lo + 256, size=(N, O, oh, ow) if layout == 0 else (N, oh, ow, O)).astype(res_dtype)
    kmap = None if levels is None else rng.choice(levels, size=(N, oh, ow)).astype(np.uint8)
    for relu, qmin, qmax, dt in ((True, 0, 255, psb.PSB_DT_U8), (False, -100, 90, psb.PSB_DT_S8)):
        args = (w, x, layout, 1, stride, pad, 5, 3, list(levels or (3,)), kmap, 3, rng.uniform(0.5, 1.5, O).astype(np.float32),
                rng.normal(0, 0.5, O).astype(np.float32), relu, np.float32(0.02), qmin, qmax)
        o = oracle_layer(oracle, *args, residual=res, res_scale=np.float32(0.3))
        g = gpu_layer(psb, ctx, *args, dt, residual=res, res_scale=np.float32(0.3), in_max=top, path=psb.PSB_PATH_TENSOR, want=want)
        compare(g, o, list(levels or (3,)))
        assert np.array_equal(g["f32"], o["f32"])       # rounded operations only, in the same order
    ctx.close()


@pytest.mark.parametrize("case", [
    # (N, C, H, W, O, K, pad, largest byte, levels, exp_bits): one, two and four planes, three in 64 bits (with and without an addend)
    (2, 64, 13, 11, 68, 1, 0, 15, (0, 1), 1), (2, 48, 13, 11, 72, 3, 1, 255, (0, 3), 3), (2, 96, 9, 14, 50, 1, 0, 255, (5, 6), 4),
    (1, 1040, 13, 11, 64, 1, 0, 255, (4, 3), 4), (1, 8752, 5, 7, 36, 1, 0, 15, (4, 2), 4), (2, 8, 21, 19, 36, 3, 1, 255, (6, 5), 4),
])
@pytest.mark.parametrize("layout", [0, 1])
@pytest.mark.parametrize("with_map", [False, True])
def test_real_valued_outputs_of_other_recombinations(case, layout, with_map, oracle):
    import paper_1904_02205_b200 as psb

    N, C, H, W, O, K, pad, top, levels, exp_bits = case
    ctx = psb.Context(0)
    rng = np.random.default_rng(C * 11 + O)
    w = rng.normal(0, np.sqrt(2.0 / (C * K * K)), size=(O, C, K, K)).astype(np.float32)
    x = rng.integers(0, top + 1, size=(N, C, H, W) if layout == 0 else (N, H, W, C)).astype(np.uint8)
    res = rng.integers(0, 256, size=(N, O, H, W) if layout == 0 else (N, H, W, O)).astype(np.uint8)
    kmap = rng.choice(levels, size=(N, H, W)).astype(np.uint8) if with_map else None
    used = list(levels) if with_map else [levels[0]]
    args = (w, x, layout, 1, 1, pad, 5, 3, used, kmap, levels[0], rng.uniform(0.5, 1.5, O).astype(np.float32),
            rng.normal(0, 0.5, O).astype(np.float32), True, np.float32(0.02), 0, 255)
    o = oracle_layer(oracle, *args, residual=res, res_scale=np.float32(0.3), exp_bits=exp_bits)
    g = gpu_layer(psb, ctx, *args, psb.PSB_DT_U8, residual=res, res_scale=np.float32(0.3), in_max=top, path=psb.PSB_PATH_TENSOR,
                  want=("q", "f32"), exp_bits=exp_bits)
    compare(g, o, used)
    assert np.array_equal(g["f32"], o["f32"])       # rounded operations only, in the same order
    ctx.close()


@pytest.mark.parametrize("shortcut", [False, True])
@pytest.mark.parametrize("levels", [(0,), (0, 2)])
def test_long_rows_of_small_sums_with_an_addend(shortcut, levels, oracle):
    """Full-range bytes on rows too long for two planes to fit 32 bits together, but whose sums do: one weight at the window's top."""
    import paper_1904_02205_b200 as psb

    C, O, H, W = 1056, 48, 11, 13
    ctx = psb.Context(0)
    rng = np.random.default_rng(4)
    w = (rng.normal(0, 1, size=(O, C, 1, 1)) * 2.0 ** -9).astype(np.float32)
    w[0, 0] = 1.5
    x = rng.integers(0, 256, size=(1, H, W, C)).astype(np.uint8)
    res = rng.integers(-128, 128, size=(1, H, W, O)).astype(np.int8) if shortcut else None
    kmap = rng.choice(levels, size=(1, H, W)).astype(np.uint8) if len(levels) > 1 else None
    assert C * 128 * 16383 >= 1 << 31
    for l in levels:
        sums = np.abs(oracle.sample_level(w, 5, 3, l)[0].astype(np.int64)).reshape(O, -1)
        assert int((-(-sums // 256)).sum(1).max()) * 256 * 255 < 1 << 31
    args = (w, x, 1, 1, 1, 0, 5, 3, list(levels), kmap, 0, np.ones(O, np.float32), np.zeros(O, np.float32), False, np.float32(8.0), -100, 101)
    o = oracle_layer(oracle, *args, residual=res, res_scale=np.float32(0.01))
    g = gpu_layer(psb, ctx, *args, psb.PSB_DT_S8, residual=res, res_scale=np.float32(0.01), in_max=255, path=psb.PSB_PATH_TENSOR, want=("q",))
    compare(g, o, list(levels))
    assert len(np.unique(o["q"])) > 50
    ctx.close()
