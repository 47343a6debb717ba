"""What dwf_autotune leaves behind on a lattice that streams, and after a call
that failed."""
import pytest
import torch

import synth
from paper_2103_05034_gb300 import _lib, ops
from paper_2103_05034_gb300._lib import DWF_EINVAL, DWF_ETIMEOUT, DWFError, F32

pytestmark = pytest.mark.gpu


@pytest.fixture
def ctx():
    L = (8, 16, 16, 32)
    c = ops.Context(L, 16, 1.8, synth.random_gauge(L, 0.3, 11))
    yield c
    c.close()


def test_a_streaming_choice_comes_with_one_that_does_not(ctx):
    assert ops.dwf_get_hop_scalar_variant(ctx, F32) == 0
    v, ms = ops.dwf_autotune(ctx, F32, 5)
    s = ops.dwf_get_hop_scalar_variant(ctx, F32)
    assert ms > 0
    # variant 0 streams here: it either won, and a scalar variant stands beside it, or another is everybody's
    assert (0 < s < _lib.HOP_VARIANTS) if v == 0 else s == 0
    x = torch.randn(2 * ctx.half_numel(), device="cuda")

    def filtered():
        return ops.cheby_filter(ctx, torch.zeros_like(x), x, 1, 1.0, 90.0, 4, 0.1)

    tuned = filtered()
    ops.dwf_set_hop_variant(ctx, F32, v)
    assert ops.dwf_get_hop_scalar_variant(ctx, F32) == 0
    ops.dwf_set_hop_scalar_variant(ctx, F32, s)  # the choice as a program restores it
    assert torch.equal(filtered(), tuned)
    with pytest.raises(DWFError) as e:
        ops.dwf_set_hop_scalar_variant(ctx, F32, _lib.HOP_VARIANTS)
    assert e.value.code == DWF_EINVAL


def test_a_tuner_call_that_fails_leaves_the_choice(ctx):
    ops.dwf_set_hop_variant(ctx, F32, 7)
    assert _lib.lib().dwf_selftest_raise_timeout(ctx.h, ops._stream()) == 0
    torch.cuda.synchronize()
    with pytest.raises(DWFError) as e:
        ops.dwf_autotune(ctx, F32, 1)
    assert e.value.code == DWF_ETIMEOUT
    assert _lib.lib().dwf_get_hop_variant(ctx.h, F32) == 7
