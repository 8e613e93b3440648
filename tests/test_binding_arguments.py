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
