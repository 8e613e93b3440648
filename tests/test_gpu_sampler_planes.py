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
