"""The streaming hopping kernel (the untuned default on lattices that fill the
GPU) against the scalar kernel (variant 3, itself tested against the oracle):
every epilogue, whole and ragged x-segments, wrap-around in y and z, several
right-hand sides.

Tolerance: both kernels add the eight neighbour terms of an output in FP32,
some 60 additions of products; with eps = 2^-24 and independent roundings each
is within about sqrt(60) eps = 5e-7 of the exact sum in the norm, so the two
differ by less than 1e-6 per hopping application.  FP16 storage rounds each
stored result to 2^-11, where a difference in FP32 can move a value by one
unit: the norm of the difference stays below 2^-11.
"""
import numpy as np
import pytest
import torch

import synth
from paper_2103_05034_gb300 import ops
from paper_2103_05034_gb300._lib import F16S, F32, SOLVE_MIXED_F32

pytestmark = pytest.mark.gpu

REF = 3
SHAPES = [  # whole segments; ragged ones; a lattice of one y-tile
    ((24, 12, 8, 48), 8, F32), ((22, 12, 8, 64), 8, F32), ((24, 12, 8, 48), 8, F16S),
    ((16, 16, 16, 16), 16, F32), ((14, 16, 16, 32), 16, F32), ((12, 12, 12, 24), 16, F32), ((16, 2, 16, 192), 16, F32),
    ((8, 16, 16, 48), 24, F32), ((34, 4, 8, 96), 24, F32),
]


def _context(L, Ls):
    return ops.Context(L, Ls, 1.8, synth.random_gauge(L, 0.3, 11))


def _field(ctx, halves, prec, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    dt = torch.float16 if prec == F16S else torch.float32
    return torch.randn(halves * ctx.half_numel(), device="cuda", generator=g).to(dt)


def _rel(a, b):
    return float((a.double() - b.double()).norm() / b.double().norm())


@pytest.mark.parametrize("L,Ls,prec", SHAPES)
def test_stream_matches_scalar_kernel(L, Ls, prec):
    ctx = _context(L, Ls)
    half, full = _field(ctx, 3, prec, 1), _field(ctx, 2, prec, 2)
    n = ctx.half_numel()

    def results():
        out = []
        for parity in (0, 1):
            for dag in (0, 1):
                out.append(ops.dwf_dhop(ctx, torch.zeros_like(half[:n]), half[:n], parity, dag))
        for dag in (0, 1):
            out.append(ops.dwf_mpc(ctx, torch.zeros_like(half), half, 0.05, dag, 3))
            out.append(ops.dwf_ddw(ctx, torch.zeros_like(full), full, 0.3, dag))
        out.append(ops.dwf_hdw(ctx, torch.zeros_like(full), full, 1.0))
        return out

    ops.dwf_set_hop_variant(ctx, prec, 0)
    got = results()
    again = results()
    ops.dwf_set_hop_variant(ctx, prec, REF)
    tol = 2.0 ** -11 if prec == F16S else 1e-6
    for a, r, b in zip(got, again, results()):
        assert torch.equal(a, r)
        assert _rel(a, b) < 2 * tol


@pytest.mark.parametrize("L,Ls", [((24, 12, 8, 48), 8), ((14, 16, 16, 32), 16), ((34, 4, 8, 96), 24)])
def test_stream_fused_chebyshev_and_cg(L, Ls):
    """The Chebyshev and CG epilogues and the fused reductions: a filter and a
    solve.  A filter of order n amplifies the FP32 difference of its operator
    applications at most about 2 n-fold; a solve to 1e-10 fixes x to 1e-10 over
    the smallest singular value, above 0.02 at this mass."""
    ctx = _context(L, Ls)
    full = _field(ctx, 2, F32, 3)
    b = _field(ctx, 2, F32, 4).double()

    def results():
        f = ops.cheby_filter(ctx, torch.zeros_like(full), full, 1, 1.0, 90.0, 6, 0.1)
        x = torch.zeros_like(b)
        st = ops.rbcg_solve(ctx, x, b, 0.1, 1e-10, policy=SOLVE_MIXED_F32)
        assert st["true_residual"] <= 1e-10
        return f, x

    ops.dwf_set_hop_variant(ctx, F32, 0)
    f0, x0 = results()
    ops.dwf_set_hop_variant(ctx, F32, REF)
    f1, x1 = results()
    assert _rel(f0, f1) < 2 * 6 * 2e-6
    assert _rel(x0, x1) < 2 * 1e-10 / 0.02
