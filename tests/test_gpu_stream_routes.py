"""Which hopping launches the streaming kernel takes, and the branches of it that
a lattice reaches only if it does: rows of a single x-segment (the wrap-around
inside the tile), several masses in one launch, |out|^2 of several fields.

Tolerances: as between the kernels in test_gpu_stream.py, less than 1e-6 in the
norm per hopping application.  The force is bilinear in fields after at most
three of them: 2 * 3e-6."""
import pytest
import torch

import synth
from paper_2103_05034_gb300 import ops
from paper_2103_05034_gb300._lib import F16S, F32

pytestmark = pytest.mark.gpu

SCALAR = 3
# FP32 at Ls 8 (six sites a row, and five), 16 (four and three), 24 (two); FP16 at Ls 8
SINGLE = [((12, 16, 16, 32), 8, F32, 1), ((10, 16, 16, 64), 8, F32, 2), ((12, 16, 16, 24), 8, F16S, 3), ((8, 16, 16, 32), 16, F32, 1),
          ((6, 16, 16, 32), 16, F32, 1), ((8, 16, 16, 16), 16, F32, 3), ((4, 16, 16, 64), 24, F32, 1), ((4, 16, 16, 48), 24, F32, 3)]
# several segments, the shapes of test_gpu_stream.py
WIDE = [((24, 12, 8, 48), 8, F32, 1), ((22, 12, 8, 64), 8, F32, 1), ((24, 12, 8, 48), 8, F16S, 1), ((16, 16, 16, 16), 16, F32, 1),
        ((14, 16, 16, 32), 16, F32, 1), ((12, 12, 12, 24), 16, F32, 1), ((16, 2, 16, 192), 16, F32, 1),
        ((8, 16, 16, 48), 24, F32, 1), ((34, 4, 8, 96), 24, F32, 1)]


def _field(n, prec, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(n, device="cuda", generator=g).to(torch.float16 if prec == F16S else torch.float32)


def _rel(a, b):
    return float((a.double() - b.double()).norm() / b.double().norm())


def _counted(ctx, f):
    """f()'s result, its launches and how many of them streamed."""
    ops.dwf_reset_counters(ctx)
    r = f()
    return r, ops.dwf_counters(ctx)[0], ops.dwf_streamed_launches(ctx)


@pytest.mark.parametrize("L,Ls,prec,nrhs", SINGLE + WIDE)
def test_every_plain_launch_streams(L, Ls, prec, nrhs):
    ctx = ops.Context(L, Ls, 1.8, synth.random_gauge(L, 0.3, 11))
    half = _field(nrhs * ctx.half_numel(), prec, 1)
    full = _field(2 * nrhs * ctx.half_numel(), prec, 2)
    calls = [lambda p=p, d=d: ops.dwf_dhop(ctx, torch.zeros_like(half), half, p, d, nrhs) for p in (0, 1) for d in (0, 1)]
    for d in (0, 1):
        calls.append(lambda d=d: ops.dwf_mpc(ctx, torch.zeros_like(half), half, 0.05, d, nrhs))
        calls.append(lambda d=d: ops.dwf_ddw(ctx, torch.zeros_like(full), full, 0.3, d, nrhs))
    calls.append(lambda: ops.dwf_hdw(ctx, torch.zeros_like(full), full, 1.0, nrhs))
    tol = 2.0 ** -11 if prec == F16S else 1e-6
    for f in calls:
        ops.dwf_set_hop_variant(ctx, prec, 0)
        got, launches, streamed = _counted(ctx, f)
        assert launches == streamed > 0
        ops.dwf_set_hop_variant(ctx, prec, SCALAR)
        want, _, none = _counted(ctx, f)
        assert none == 0
        assert _rel(got, want) < 2 * tol
    ctx.close()


@pytest.mark.parametrize("L,Ls,prec", [((4, 4, 4, 8), 16, F32), ((8, 8, 8, 16), 8, F32), ((12, 12, 12, 24), 4, F32),
                                       ((16, 16, 16, 32), 16, F16S)])
def test_other_launches_do_not(L, Ls, prec):
    ctx = ops.Context(L, Ls, 1.8, synth.random_gauge(L, 0.3, 11))
    x = _field(ctx.half_numel(), prec, 1)
    _, launches, streamed = _counted(ctx, lambda: ops.dwf_mpc(ctx, torch.zeros_like(x), x, 0.05))
    assert launches == 2 and streamed == 0
    ctx.close()


def test_launches_that_end_in_a_chebyshev_step_do_not():
    """Of a step's four hopping launches the last two end in the recurrence."""
    L, Ls = (8, 16, 16, 32), 16
    ctx = ops.Context(L, Ls, 1.8, synth.random_gauge(L, 0.3, 11))
    x = _field(2 * ctx.half_numel(), F32, 3)
    counts = {}
    for order in (1, 6):
        _, _, counts[order] = _counted(ctx, lambda: ops.cheby_filter(ctx, torch.zeros_like(x), x, 1, 1.0, 90.0, order, 0.1))
    assert counts[1] == 4 and counts[6] == 4 + 5 * 2
    ctx.close()


@pytest.mark.parametrize("L,Ls", [((8, 16, 16, 16), 16), ((4, 16, 16, 48), 24)])
def test_batched_solve_with_several_masses_streams(L, Ls):
    """The batch's step lengths come from |M_pc p|^2 of every field, each with
    its own mass, reduced by the streaming kernel: the solves converge to their
    FP64 residual and in as many iterations as with the scalar kernel (checks
    are eight iterations apart, two apart at most)."""
    ctx = ops.Context(L, Ls, 1.8, synth.random_gauge(L, 0.3, 11))
    masses, tol, n = [0.2, 1.0, 0.5], 1e-9, ctx.half_numel()
    phi = _field(3 * n, F32, 5).double()
    res = {}
    for v in (0, SCALAR):
        ops.dwf_set_hop_variant(ctx, F32, v)
        x = torch.zeros_like(phi)
        stats, _, streamed = _counted(ctx, lambda: ops.rbcg_normal_solve_batch(ctx, x, phi, masses, tol))
        assert (streamed > 0) == (v == 0)
        res[v] = [s["iterations"] for s in stats]
        for i, m in enumerate(masses):
            xi, pi = x[i * n:(i + 1) * n], phi[i * n:(i + 1) * n]
            r = pi - ops.dwf_mpcdag_mpc(ctx, torch.zeros_like(xi), xi.contiguous(), m)
            assert float(r.norm() / pi.norm()) <= 1.01 * tol
    for a, b in zip(res[0], res[SCALAR]):
        assert abs(a - b) <= 16
    ctx.close()


def test_force_of_several_masses_streams():
    L, Ls = (8, 16, 16, 16), 16
    ctx = ops.Context(L, Ls, 1.8, synth.random_gauge(L, 0.3, 11))
    X = _field(3 * ctx.half_numel(), F32, 6)
    out = {}
    for v in (0, SCALAR):
        ops.dwf_set_hop_variant(ctx, F32, v)
        force = torch.zeros(L[3], L[2], L[1], L[0], 4, 3, 3, dtype=torch.complex128, device="cuda")
        _, _, streamed = _counted(ctx, lambda: ops.dwf_force(ctx, force, X, [0.01, 0.2, 1.0]))
        assert streamed == (3 if v == 0 else 0)
        out[v] = torch.view_as_real(force)
    assert _rel(out[0], out[SCALAR]) < 6e-6
    ctx.close()
