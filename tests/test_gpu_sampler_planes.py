"""GPU parity of filters that are kept as digit planes only (sampler, export, matrix products with few rows) and of the
batched sampler under the sampling options, bit-exact against the CPU oracle."""
import numpy as np
import pytest

from psb_testlib import compare, gpu_layer, oracle_layer

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("case", [
    # (rows, features, outputs, levels, signed input, map): lane groups of 1 .. 32, several segments of features
    (1, 16, 5, (3,), False, False), (3, 47, 70, (0,), True, False), (5, 130, 64, (6,), False, False),
    (4, 512, 33, (4,), True, False), (7, 9000, 10, (3,), False, False), (6, 200, 40, (0, 2, 4), False, True),
])
def test_few_rows_from_the_digit_planes(case, oracle):
    import paper_1904_02205_b200 as psb

    M, C, O, levels, signed, with_map = case
    ctx = psb.Context(0)
    rng = np.random.default_rng(C + O)
    w = rng.normal(0, np.sqrt(2.0 / C), size=(O, C, 1, 1)).astype(np.float32)
    x = rng.integers(-128, 128, size=(M, 1, 1, C)).astype(np.int8) if signed else rng.integers(0, 256, size=(M, 1, 1, C)).astype(np.uint8)
    kmap = rng.choice(levels, size=(M, 1, 1)).astype(np.uint8) if with_map else None
    args = (w, x, 1, 1, 1, 0, 5, 3, list(levels), kmap, levels[0], rng.uniform(0.5, 1.5, O).astype(np.float32),
            rng.normal(0, 0.5, O).astype(np.float32), True, np.float32(0.02), 0, 255)
    o = oracle_layer(oracle, *args)
    g = gpu_layer(psb, ctx, *args, psb.PSB_DT_U8, path=psb.PSB_PATH_SHIFT_ADD)
    compare(g, o, list(levels))
    ctx.close()


@pytest.mark.parametrize("opts", [dict(prob_bits=8, underflow=1), dict(prob_bits=4, exp_bits=3), dict(prob_bits=6, deterministic=1),
                                  dict(underflow=1, exp_bits=2), dict(prob_bits=5)])
@pytest.mark.parametrize("log2k", [0, 1, 2, 4, 6])
def test_one_level_under_options_alone_and_in_a_batch(opts, log2k, oracle):
    import torch

    import paper_1904_02205_b200 as psb

    ctx = psb.Context(0)
    rng = np.random.default_rng(log2k)
    shapes = [(70, 36, 3, 3), (33, 64, 1, 1), (16, 3, 5, 5), (130, 30, 1, 1)]
    ws = [rng.normal(0, 0.1, size=s).astype(np.float32) for s in shapes]
    ws[1][3, 5] = 0.0
    exp_bits = opts.get("exp_bits", 4)
    more = {k: v for k, v in opts.items() if k != "exp_bits"}
    dev = [torch.from_numpy(w).to(ctx.device) for w in ws]
    handles = [ctx.sample_weights(t, seed=9, layer_id=i, level_mask=1 << log2k, norm=i & 1, **opts) for i, t in enumerate(dev)]
    batch = ctx.sample_batch_create(dev, handles)
    for seed in (9, 1234567890123):
        if seed != 9:
            ctx.sample_batch_run(batch, seed)
        for i, w in enumerate(ws):
            W, eb = oracle.sample_level_ex(w, seed, i, log2k, exp_bits=exp_bits, norm=i & 1, **more)[:2]
            got, base = ctx.weights_export(handles[i], log2k)
            assert np.array_equal(got.cpu().numpy().astype(np.int64), W) and np.array_equal(base.cpu().numpy(), eb)
    assert ctx.device_status() == 0
    ctx.sample_batch_free(batch)
    for h in handles:
        h.free()
    ctx.close()


@pytest.mark.parametrize("case", [
    # (N, C, H, W, O, K, stride, layout, levels, signed input): flat and tap-major K axes, patches in pieces of 1, 4 and 16
    # bytes, one segment of the axis and two, locations that are no multiple of the block's four
    (1, 3, 9, 7, 17, 5, 2, 0, (3,), False), (2, 7, 4, 5, 40, 3, 1, 1, (0,), True), (1, 17, 5, 5, 70, 3, 1, 1, (6,), False),
    (3, 36, 3, 4, 33, 3, 2, 0, (4,), True), (1, 64, 7, 7, 130, 5, 1, 1, (2,), False), (1, 1000, 2, 3, 9, 3, 1, 1, (3,), False),
    (2, 24, 6, 5, 20, 3, 1, 0, (0, 2, 4), False), (1, 4, 8, 8, 12, 7, 3, 1, (1, 5), True), (1, 48, 1, 1, 64, 1, 1, 1, (3,), False),
    (1, 16, 30, 31, 8, 3, 1, 1, (3,), False),
])
def test_filters_with_taps_from_the_digit_planes(case, oracle):
    import paper_1904_02205_b200 as psb

    N, C, H, W, O, K, stride, layout, levels, signed = case
    ctx = psb.Context(0)
    rng = np.random.default_rng(C * 5 + O)
    w = rng.normal(0, np.sqrt(2.0 / (C * K * K)), size=(O, C, K, K)).astype(np.float32)
    lo, hi, dt = (-128, 128, np.int8) if signed else (0, 256, np.uint8)
    x = rng.integers(lo, hi, size=(N, C, H, W) if layout == 0 else (N, H, W, C)).astype(dt)
    oh, ow = (H + 2 * (K // 2) - K) // stride + 1, (W + 2 * (K // 2) - K) // stride + 1
    res = rng.integers(0, 256, size=(N, O, oh, ow) if layout == 0 else (N, oh, ow, O)).astype(np.uint8)
    kmap = rng.choice(levels, size=(N, oh, ow)).astype(np.uint8) if len(levels) > 1 else None
    args = (w, x, layout, 1, stride, K // 2, 5, 3, list(levels), kmap, levels[0], rng.uniform(0.5, 1.5, O).astype(np.float32),
            rng.normal(0, 0.5, O).astype(np.float32), True, np.float32(0.02), 0, 255)
    o = oracle_layer(oracle, *args, residual=res, res_scale=np.float32(0.3))
    before = ctx.launch_count()
    g = gpu_layer(psb, ctx, *args, psb.PSB_DT_U8, residual=res, res_scale=np.float32(0.3), path=psb.PSB_PATH_SHIFT_ADD)
    compare(g, o, list(levels))
    # sampling, one export per level, one launch for the layer and one for a planar input: nothing is put together first
    planar = 1 if layout == 0 and C > 1 and H * W > 1 else 0
    assert ctx.launch_count() - before <= 2 + len(levels) + 1 + planar
    ctx.close()


def test_few_locations_at_odd_addresses(oracle):
    import torch

    import paper_1904_02205_b200 as psb

    ctx = psb.Context(0)
    rng = np.random.default_rng(3)
    w = rng.normal(0, 0.1, size=(32, 48, 3, 3)).astype(np.float32)
    x = rng.integers(0, 256, size=(1, 4, 5, 48)).astype(np.uint8)
    wt = ctx.sample_weights(torch.from_numpy(w).to(ctx.device), seed=1, level_mask=8)
    ctx.set_sample_map(None, 3)
    one = torch.ones(32, device=ctx.device)
    W = {3: oracle.sample_level(w, 1, 0, 3)[0]}
    acc = oracle.conv_acc(x, oracle.geom(x.shape, oracle.NHWC, oracle.U8, w.shape, 1, 1, 1), W, uniform_log2k=3)
    flat = torch.zeros(x.size + 16, dtype=torch.uint8, device=ctx.device)
    for shift in (0, 1, 4, 6):
        flat[shift:shift + x.size] = torch.from_numpy(x.ravel()).to(ctx.device)
        got = ctx.conv2d(wt, flat[shift:shift + x.size].view(x.shape), 1, 1, 1, one, one, False, 1.0, 0, 255,
                         path=psb.PSB_PATH_SHIFT_ADD, want=("acc",))["acc"].cpu().numpy()
        assert ctx.device_status() == 0 and np.array_equal(got, acc)
    wt.free()
    ctx.close()


@pytest.mark.parametrize("case", [
    # (norm, rows, channels, filter size, launches): both sides of the lines of the sampling without an exponent pass
    (0, 128, 256, 1, 1), (0, 129, 256, 1, 2), (0, 3, 257, 1, 2), (1, 9, 1536, 1, 1), (1, 65, 1537, 1, 2), (1, 64, 2048, 1, 1),
    (1, 64, 2049, 1, 2), (1, 295, 1537, 1, 2), (1, 296, 1537, 1, 1), (1, 147, 256, 3, 1), (1, 147, 257, 3, 2), (1, 148, 257, 3, 1),
    (1, 296, 4096, 1, 1), (1, 296, 4097, 1, 2),
])
def test_windows_found_by_the_sampler_or_by_a_pass_of_their_own(case, oracle):
    import torch

    import paper_1904_02205_b200 as psb

    norm, O, C, K, launches = case
    ctx = psb.Context(0)
    rng = np.random.default_rng(O + C)
    w = rng.normal(0, 0.1, size=(O, C, K, K)).astype(np.float32)
    w *= np.exp2(rng.integers(-3, 4, size=(O, 1, 1, 1))).astype(np.float32)
    before = ctx.launch_count()
    wt = ctx.sample_weights(torch.from_numpy(w).to(ctx.device), seed=3, layer_id=2, level_mask=8, norm=norm)
    assert ctx.launch_count() - before == launches
    W, eb, _ = oracle.sample_level(w, 3, 2, 3, norm=norm)
    got, base = ctx.weights_export(wt, 3)
    assert np.array_equal(got.cpu().numpy().astype(np.int64), W) and np.array_equal(base.cpu().numpy(), eb)
    assert ctx.device_status() == 0
    wt.free()
    ctx.close()


@pytest.mark.parametrize("opts", [dict(prob_bits=8, underflow=1), dict(prob_bits=4, underflow=1, exp_bits=3), dict(underflow=1, exp_bits=3),
                                  dict(exp_bits=1), dict(prob_bits=8, exp_bits=2), dict()])
@pytest.mark.parametrize("levels", [(0, 1, 2, 3, 4), (3, 6), (5,), (3,)])
def test_decoding_and_counting_at_their_edges(opts, levels, oracle):
    """Weights around the window's floor, the grid's carry, the largest and smallest exponents, in rows cut into whole quads
    and not, under one and several levels; both passes of a layer and the single one."""
    import torch

    import paper_1904_02205_b200 as psb

    ctx = psb.Context(0)
    mask = sum(1 << l for l in levels)
    exp_bits = opts.get("exp_bits", 4)
    more = {k: v for k, v in opts.items() if k != "exp_bits"}
    for norm, top, shape in ((0, 0, (5, 37, 3, 3)), (1, 0, (9, 1028, 1, 1)), (0, 127, (70, 700, 1, 1)), (1, -120, (300, 44, 3, 1))):
        rng = np.random.default_rng(shape[1] + top + 200)
        # magnitudes down to well below the floor, mantissas at 0, at the top of the grid and anywhere
        exps = np.maximum(top - rng.integers(0, (1 << exp_bits) + 12, size=shape), -126)
        exps.flat[0] = top
        mant = rng.choice([0, 1, 0x7FFFFF, 0x7FC000, 0x7F8000, 0x7BFFFF, 0x004000, 0x040000, 0x3FFFFF], size=shape)
        mant = np.where(rng.random(shape) < 0.5, mant, rng.integers(0, 1 << 23, size=shape))
        bits = (rng.integers(0, 2, size=shape) << 31) | ((exps + 127) << 23) | mant
        bits = np.where(rng.random(shape) < 0.05, bits & 0x807FFFFF, bits)            # zeros and sub-normals
        w = bits.astype(np.uint32).view(np.float32)
        wt = ctx.sample_weights(torch.from_numpy(w).to(ctx.device), seed=7, layer_id=4, level_mask=mask, norm=norm, **opts)
        for l in levels:
            W, eb = oracle.sample_level_ex(w, 7, 4, l, exp_bits=exp_bits, norm=norm, **more)[:2]
            got, base = ctx.weights_export(wt, l)
            assert np.array_equal(got.cpu().numpy().astype(np.int64), W) and np.array_equal(base.cpu().numpy(), eb)
        assert ctx.device_status() == 0
        wt.free()
    ctx.close()


@pytest.mark.parametrize("opts", [dict(prob_bits=b, underflow=b % 2, exp_bits=4 - b % 3) for b in (1, 2, 3, 5, 6, 7)] +
                         [dict(prob_bits=3, deterministic=1, underflow=1), dict(prob_bits=8, deterministic=1), dict(prob_bits=4, deterministic=1, exp_bits=3)])
@pytest.mark.parametrize("levels", [(0, 1, 2, 3, 4, 5, 6), (1, 5), (6,), (4,), (0,)])
def test_comparators_of_other_widths(opts, levels, oracle):
    """Widths whose words end inside a level (3, 5, 6 bits) and at one, one level and several; no draws at all."""
    test_decoding_and_counting_at_their_edges(opts, levels, oracle)


@pytest.mark.parametrize("case", [
    # (rows, channels, filter size): one to six rows in a block of eight warps, one to four in a block of four, which share them out;
    # tap-major planes, then flat K axes
    (40, 300, 1), (1300, 160, 1), (2000, 160, 1), (2500, 160, 1), (3100, 160, 1), (30, 20, 3), (1000, 2400, 1), (1900, 2100, 1),
    (4600, 1000, 1), (40, 3, 7), (64, 12, 5), (2400, 15, 3),
])
def test_windows_of_rows_that_warps_share(case, oracle):
    test_windows_found_by_the_sampler_or_by_a_pass_of_their_own((1, *case, 1), oracle)


@pytest.mark.parametrize("scale", [1, 3, 9])
@pytest.mark.parametrize("opts", [dict(), dict(norm=1, prob_bits=5, underflow=1), dict(prob_bits=8)])
def test_batches_of_any_size(scale, opts, oracle):
    """The blocks of a batch are cut by the weights of all its layers: 22 thousand, 142 thousand and 1.1 million here, every kind of filter
    among them, rows that no block holds as a whole and rows that many fit into one."""
    import torch

    import paper_1904_02205_b200 as psb

    ctx = psb.Context(0)
    rng = np.random.default_rng(scale)
    shapes = [((24 * scale, 3, 7, 7), 1), ((32 * scale, 1, 3, 3), 32 * scale), ((16 * scale, 70 * scale, 3, 3), 1), ((33, 17 * scale, 1, 1), 1),
              ((64 * scale, 48 * scale, 1, 1), 1), ((24, 6, 3, 3), 4), ((10, 300 * scale, 1, 1), 1), ((150, 4, 1, 1), 1)]
    ws = [(rng.normal(0, 0.1, size=s) * np.exp2(rng.integers(-3, 4, size=(s[0], 1, 1, 1)))).astype(np.float32) for s, _ in shapes]
    dev = [torch.from_numpy(w).to(ctx.device) for w in ws]
    hs = [ctx.sample_weights(d, groups=g, seed=1, layer_id=i, level_mask=0b1001, **opts) for i, (d, (_, g)) in enumerate(zip(dev, shapes))]
    batch = ctx.sample_batch_create(dev, hs)
    for seed in (7, 8):
        ctx.sample_batch_run(batch, seed)
        for i, (w, h) in enumerate(zip(ws, hs)):
            for level in (0, 3):
                W, eb = oracle.sample_level_ex(w, seed, i, level, **opts)[:2]
                got, base = ctx.weights_export(h, level)
                assert np.array_equal(got.cpu().numpy().astype(np.int64), W) and np.array_equal(base.cpu().numpy(), eb), (i, level)
    assert ctx.device_status() == 0
    ctx.sample_batch_free(batch)
    for h in hs:
        h.free()
    ctx.close()
