"""Whom a hopping launch's wait that gave up is reported to.  The flag is raised
from the host, on the stream, while the calls under test are queued behind a
sleeping kernel: no device wait runs out."""
import pytest
import torch

import synth
from paper_2103_05034_gb300 import _lib, ops
from paper_2103_05034_gb300._lib import COARSE_CG, DWF_ETIMEOUT, DWFError, F32

pytestmark = pytest.mark.gpu

L, LS = (4, 4, 4, 4), 8


def _raise_later(ctx):
    """The flag goes up about 0.1 s from now, in stream order."""
    torch.cuda._sleep(200_000_000)
    assert _lib.lib().dwf_selftest_raise_timeout(ctx.h, ops._stream()) == 0


@pytest.fixture
def ctx():
    c = ops.Context(L, LS, 1.8, synth.random_gauge(L, 0.3, 11))
    yield c
    torch.cuda.synchronize()
    c.close()


def _timeout(f):
    with pytest.raises(DWFError) as e:
        f()
    assert e.value.code == DWF_ETIMEOUT


ASYNC = {
    "dhop": lambda c, o, i: ops.dwf_dhop(c, o, i, 0, 0, 1),
    "mpc": lambda c, o, i: ops.dwf_mpc(c, o, i, 0.1, 0, 1),
    "mpcdag": lambda c, o, i: ops.dwf_mpcdag_mpc(c, o, i, 0.1, 1),
    "ddw": lambda c, o, i: ops.dwf_ddw(c, o, i, 0.1, 0, 1),
    "filter": lambda c, o, i: ops.cheby_filter(c, o, i, 1, 1.0, 80.0, 3, 0.1),
}


@pytest.mark.parametrize("op", ASYNC)
def test_status_reports_an_asynchronous_call(ctx, op):
    full = op in ("ddw", "filter")
    x = torch.randn(2 * ctx.half_numel() if full else ctx.half_numel(), device="cuda")
    out = torch.zeros_like(x)
    ASYNC[op](ctx, out, x)  # sizes the workspaces
    ops.dwf_status(ctx)
    torch.cuda._sleep(200_000_000)
    ASYNC[op](ctx, out, x)
    assert _lib.lib().dwf_selftest_raise_timeout(ctx.h, ops._stream()) == 0
    _timeout(lambda: ops.dwf_status(ctx))
    ops.dwf_status(ctx)  # reported once
    ASYNC[op](ctx, out, x)
    ops.dwf_status(ctx)


def test_next_hopping_call_reports_when_nobody_asked(ctx):
    x = torch.randn(ctx.half_numel(), device="cuda")
    out = torch.zeros_like(x)
    assert _lib.lib().dwf_selftest_raise_timeout(ctx.h, ops._stream()) == 0
    torch.cuda.synchronize()
    _timeout(lambda: ops.dwf_dhop(ctx, out, x, 0, 0, 1))
    ops.dwf_dhop(ctx, out, x, 0, 0, 1)
    ops.dwf_status(ctx)


def test_synchronising_calls_report_their_own_launches(ctx):
    """Each of these synchronises at its end, after its last hopping launch."""
    n = 2 * ctx.half_numel()
    g = torch.Generator(device="cuda").manual_seed(3)
    eta = torch.randn(8 * n, dtype=torch.float64, device="cuda", generator=g)
    p = ops.mg_params((2, 2, 2, 2), 8, 0.1, lambda_lo=0.5, lambda_max=80.0, filter_order=4, smooth=(0.5, 80.0, 4),
                      coarse_tol=1e-3, coarse_maxiter=8, coarse_solver=COARSE_CG)
    mg = ops.MG(ctx, p, eta)
    x = torch.randn(n, device="cuda", generator=g)
    out = torch.zeros_like(x)
    half = torch.randn(ctx.half_numel(), dtype=torch.float64, device="cuda", generator=g)
    basis = torch.randn(8 * n, device="cuda", generator=g)
    calls = {
        "smooth": lambda: ops.mg_smooth(mg, out, x),
        "precondition": lambda: ops.mg_precondition(mg, out, x),
        "norm2": lambda: ops.dwf_norm2(ctx, x),
        "normal": lambda: ops.rbcg_normal_solve(ctx, torch.zeros_like(half), half, 0.1, 1e-8),
        "autotune": lambda: ops.dwf_autotune(ctx, F32, 1),
        "coarse_build": lambda: ops.coarse_build(ctx, basis, 8, 4, (2, 2, 2, 2), 0.1),
    }
    for f in calls.values():
        f()
        _raise_later(ctx)
        _timeout(f)
        ops.dwf_status(ctx)
        f()
