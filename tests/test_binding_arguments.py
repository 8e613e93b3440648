"""What the Python binding accepts and hands to the library (no GPU needed)."""
from types import SimpleNamespace

import pytest
import torch

import paper_1904_02205_b200.binding as B


def _epilogue(want, inv_step=1.0, residual_scale=0.0, out=None):
    t = torch.ones(4)
    return B.Context._epilogue(SimpleNamespace(device="cpu"), (2, 4), t, t, True, inv_step, 0, 15, B.PSB_DT_U8, None,
                               residual_scale, want, out)


@pytest.mark.parametrize("want,kinds", [(("q",), "q"), ("q", "q"), ("f32", "f32"), ("acc", "acc"), ("q+f32", "q f32"),
                                        (["f32", "acc"], "f32 acc"), ({"q": 1}, "q")])
def test_wanted_outputs_as_a_sequence_or_one_text(want, kinds):
    assert sorted(_epilogue(want)[1]) == sorted(kinds.split())


@pytest.mark.parametrize("inv_step,residual_scale", [(1e39, 0.0), (1.0, -1e300), (float("inf"), 0.0), (0.25, 3.0)])
def test_floats_beyond_fp32_become_infinities(inv_step, residual_scale):
    ep, _ = _epilogue(("q",), inv_step, residual_scale)
    head = (B.PSB_DT_U8, 15, 2, 4, 0)
    assert B._block(B._GEMM_BLOCK, B.psb_gemm_desc, head, ep) == bytes(B.psb_gemm_desc(*head, B.psb_epilogue(*ep)))


class _Filter:
    """A stand-in for a CUDA tensor."""
    is_cuda, dtype = True, torch.float32

    def __init__(self, *shape):
        self.shape = torch.Size(shape)

    def is_contiguous(self):
        return True

    def dim(self):
        return len(self.shape)

    def data_ptr(self):
        return 256


def test_filters_of_more_than_four_dimensions_pass_their_first_four(monkeypatch):
    seen = []

    def sample(ctx, w, shape, *rest):
        seen.append(shape)
        return 0

    monkeypatch.setattr(B, "_stream", lambda s: 0)
    ctx = SimpleNamespace(handle=None, lib=SimpleNamespace(psb_sample_weights=sample, packed_sample_weights=sample))
    wt = B.Context.sample_weights(ctx, _Filter(6, 5, 1, 1, 1))
    assert seen == [bytes(B.psb_wshape(6, 5, 1, 1, 1))] and wt.shape == (6, 5, 1, 1, 1, 1)
    wt.handle = None
    with pytest.raises(IndexError):
        B.Context.sample_weights(ctx, _Filter(6, 5, 3))


def test_the_library_functions_take_argument_structures():
    """load_library() is public: its functions take the structures of psb.h, by value or by reference."""
    lib = B.load_library()
    conv, gemm, shape, cfg = B.psb_conv_desc(), B.psb_gemm_desc(), B.psb_wshape(), B.psb_sample_cfg()
    for call in (lambda p: lib.psb_conv2d(None, None, None, p(conv), None),
                 lambda p: lib.psb_gemm(None, None, None, p(gemm), None),
                 lambda p: lib.psb_sample_weights(None, None, p(shape), p(cfg), None, None)):
        assert call(lambda s: s) == B.PSB_ERR_INVALID_ARG and call(B.C.byref) == B.PSB_ERR_INVALID_ARG
