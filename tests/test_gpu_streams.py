"""Work buffers: layers on several streams of one context, on more streams than it keeps buffers for, and in graphs that
are captured on a stream the context has not met."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


class Layers:
    """Layers that need every work buffer between them: planar input, repacked rows, a flat K axis, a draw-count map."""

    def __init__(self, psb, ctx, images):
        import torch

        self.psb, self.ctx, self.torch = psb, ctx, torch
        rng = np.random.default_rng(images)
        dev = lambda a: torch.from_numpy(a).to(ctx.device)
        self.specs = []
        for c, o, hw, k, layout, levels in ((48, 40, 14, 3, 0, (3,)), (37, 24, 13, 3, 1, (3,)), (3, 16, 17, 7, 1, (3,)),
                                            (32, 64, 12, 3, 1, (0, 2, 4)), (5, 32, 15, 5, 0, (1, 4))):
            w = dev(rng.normal(0, 0.1, size=(o, c, k, k)).astype(np.float32))
            x = dev(rng.integers(0, 16, size=(images, c, hw, hw) if layout == 0 else (images, hw, hw, c)).astype(np.uint8))
            kmap = None if len(levels) == 1 else dev(rng.choice(levels, size=(images, hw, hw)).astype(np.uint8))
            wt = ctx.sample_weights(w, seed=7, level_mask=sum(1 << l for l in levels))
            one = torch.ones(o, device=ctx.device)
            shape = (images, o, hw, hw) if layout == 0 else (images, hw, hw, o)
            self.specs.append((wt, x, layout, k // 2, one, kmap, levels[0], {"q": torch.empty(shape, dtype=torch.uint8, device=ctx.device)}))

    def run(self, i):
        wt, x, layout, pad, one, kmap, log2k, out = self.specs[i]
        self.ctx.set_sample_map(kmap, log2k)
        self.ctx.conv2d(wt, x, layout, 1, pad, one, one, True, 0.05, 0, 15, in_max=15, path=self.psb.PSB_PATH_TENSOR, out=out)

    def clear(self):
        for s in self.specs:
            s[-1]["q"].zero_()

    def results(self):
        self.torch.cuda.synchronize()
        return [s[-1]["q"].cpu().numpy() for s in self.specs]

    def reference(self):
        for i in range(len(self.specs)):
            self.run(i)
        return self.results()

    def free(self):
        self.ctx.set_sample_map(None, 0)
        for s in self.specs:
            s[0].free()


def _same(got, ref):
    return all(np.array_equal(a, b) for a, b in zip(got, ref))


def test_interleaved_streams_and_more_streams_than_buffers():
    import torch

    import paper_1904_02205_b200 as psb

    ctx = psb.Context(0)
    a, b = Layers(psb, ctx, 9), Layers(psb, ctx, 4)
    ref_a, ref_b = a.reference(), b.reference()
    assert all(r.any() for r in ref_a + ref_b)
    s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
    for _ in range(3):
        a.clear()
        b.clear()
        torch.cuda.synchronize()
        for i in range(len(a.specs)):
            with torch.cuda.stream(s1):
                a.run(i)
            with torch.cuda.stream(s2):
                b.run(i)
        assert _same(a.results(), ref_a) and _same(b.results(), ref_b)
    streams = [torch.cuda.Stream() for _ in range(11)]
    for s in streams + streams[:2]:
        a.clear()
        torch.cuda.synchronize()
        with torch.cuda.stream(s):
            for i in range(len(a.specs)):
                a.run(i)
        assert _same(a.results(), ref_a)
    assert ctx.device_status() == 0
    a.free()
    b.free()
    ctx.close()


def test_capture_on_a_stream_not_met_before():
    """After a pass on one stream the same calls are captured on another; the graph keeps its buffers when later calls
    need larger ones and when other streams take sets over."""
    import torch

    import paper_1904_02205_b200 as psb

    ctx = psb.Context(0)
    a, big = Layers(psb, ctx, 5), Layers(psb, ctx, 23)
    ref, ref_big = a.reference(), big.reference()
    side = torch.cuda.Stream()
    g = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(g, stream=side):
        for i in range(len(a.specs)):
            a.run(i)

    def replay():
        a.clear()
        torch.cuda.synchronize()
        g.replay()
        return a.results()

    assert _same(replay(), ref)
    # larger calls on the stream of the capture, then on ten others
    for s in [side] + [torch.cuda.Stream() for _ in range(10)]:
        big.clear()
        torch.cuda.synchronize()
        with torch.cuda.stream(s):
            for i in range(len(big.specs)):
                big.run(i)
        assert _same(big.results(), ref_big)
    assert _same(replay(), ref)
    # an order that was sorted on the captured stream before a replay still stands after it
    big.clear()
    with torch.cuda.stream(side):
        big.run(3)
        g.replay()
        big.specs[3][-1]["q"].zero_()
        wt, x, layout, pad, one, kmap, log2k, out = big.specs[3]
        ctx.conv2d(wt, x, layout, 1, pad, one, one, True, 0.05, 0, 15, in_max=15, path=psb.PSB_PATH_TENSOR, out=out)
    assert np.array_equal(big.results()[3], ref_big[3])
    assert ctx.device_status() == 0
    del g
    a.free()
    big.free()
    ctx.close()


def test_captured_sampling_replayed_after_later_calls():
    """One window per layer, in a graph that samples a handle and a batch twice each: replays, with eager calls between them,
    give the filters of the seeds that were captured."""
    import torch

    import paper_1904_02205_b200 as psb

    ctx = psb.Context(0)
    rng = np.random.default_rng(5)
    w = [torch.from_numpy(rng.normal(0, 0.1, size=s).astype(np.float32)).to(ctx.device)
         for s in ((64, 64, 3, 3), (72, 40, 3, 3), (33, 300, 1, 1))]
    alone = ctx.sample_weights(w[0], seed=1, level_mask=8)
    kept = [ctx.sample_weights(a, seed=1, layer_id=i, level_mask=8) for i, a in enumerate(w)]
    batch = ctx.sample_batch_create(w, kept)

    def calls(seeds):
        for seed in seeds:
            ctx.sample_weights(w[0], seed=seed, level_mask=8, into=alone)
            ctx.sample_batch_run(batch, seed)

    def filters():
        torch.cuda.synchronize()
        return [ctx.weights_export(h, 3)[0].cpu().numpy() for h in [alone] + kept]

    calls([3])
    ref = filters()
    assert all(r.any() for r in ref)
    g = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(g, stream=torch.cuda.Stream()):
        calls([2, 3])
    for eager in ([], [], [4, 5]):
        calls(eager)
        torch.cuda.synchronize()
        g.replay()
        assert _same(filters(), ref)
    assert ctx.device_status() == 0
    del g
    ctx.sample_batch_free(batch)
    for h in [alone] + kept:
        h.free()
    ctx.close()
