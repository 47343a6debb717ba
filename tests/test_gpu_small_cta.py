"""The FP64 hopping kernels for small lattices against each other, and the
one-sweep inverse of the fifth-dimension matrix with its fallback."""
import numpy as np
import pytest
import torch

import synth
from oracle import dwf
from paper_2103_05034_gb300 import layout, ops
from paper_2103_05034_gb300._lib import F32, F64

from gpu_helpers import dev_to_half, half_dev, rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,Ls,nrhs", [
    # directions against small CTAs
    ((4, 4, 4, 4), 16, 5), ((6, 2, 4, 6), 24, 3), ((6, 4, 4, 6), 8, 5), ((8, 4, 6, 4), 4, 6),
    # small CTAs against large ones
    ((8, 8, 8, 8), 16, 12), ((6, 10, 8, 8), 24, 14), ((8, 8, 8, 16), 8, 12), ((16, 8, 8, 16), 4, 12)])
def test_fp64_kernels_agree(L, Ls, nrhs):
    """One right-hand side and nrhs of them fall on different sides of the lines
    between the FP64 kernels: the same products, added in another order.  Some 60
    additions at 2^-53 each: 1e-15 in the norm per application, 1e-14 allowed."""
    ctx = ops.Context(L, Ls, 1.8, synth.random_gauge(L, 0.3, 5))
    n = ctx.half_numel()
    g = torch.Generator(device="cuda").manual_seed(1)
    x = torch.randn(2 * nrhs * n, dtype=torch.float64, device="cuda", generator=g)
    h = x[:nrhs * n]
    many = [(ops.dwf_mpc(ctx, torch.zeros_like(h), h, 0.1, d, nrhs), n, lambda o, v, d=d: ops.dwf_mpc(ctx, o, v, 0.1, d))
            for d in (0, 1)]
    many += [(ops.dwf_ddw(ctx, torch.zeros_like(x), x, 0.3, d, nrhs), 2 * n,
              lambda o, v, d=d: ops.dwf_ddw(ctx, o, v, 0.3, d)) for d in (0, 1)]
    many.append((ops.dwf_hdw(ctx, torch.zeros_like(x), x, 0.3, nrhs), 2 * n, lambda o, v: ops.dwf_hdw(ctx, o, v, 0.3)))
    many.append((ops.cheby_filter(ctx, torch.zeros_like(x), x, nrhs, 1.0, 90.0, 3, 0.1), 2 * n,
                 lambda o, v: ops.cheby_filter(ctx, o, v, 1, 1.0, 90.0, 3, 0.1)))
    for all_, w, f in many:
        for r in (0, nrhs - 1):
            one = f(torch.zeros(w, dtype=torch.float64, device="cuda"), x[r * w:(r + 1) * w].clone())
            want = all_[r * w:(r + 1) * w]
            assert float((one - want).norm() / want.norm()) < 1e-14


@pytest.mark.parametrize("prec,tol", [(F64, 1e-12), (F32, 1e-6)])
@pytest.mark.parametrize("M5,mf", [(1.8, 0.0), (1.8, 1.0), (1.8, -0.5), (4.5, 0.01), (3.9, 20.0)])
def test_inverse_either_side_of_the_one_sweep_line(prec, tol, M5, mf):
    """d = 5 - M5 above and below 1, masses above and below d^Ls: the general
    two-sweep path is taken for the last two.  That path recovers v_q from
    F_q - F_{q-1}/d, so its error grows by up to d^-Ls, and by the mass."""
    L, Ls = (4, 4, 2, 2), 8
    tol *= max(1.0, (5 - M5) ** -Ls, abs(mf))
    U = synth.random_gauge(L, 0.5, 8)
    ctx = ops.Context(L, Ls, M5, U)
    psi = synth.gaussian_spinor(L, Ls, 3)
    pe = dwf.project_parity(psi, L, 0)
    for dag, f in ((0, dwf.mpc), (1, dwf.mpc_dag)):
        inp = half_dev(psi, L, 0, prec)
        out = ops.dwf_mpc(ctx, torch.zeros_like(inp), inp, mf, dag)
        assert rel(dev_to_half(out, Ls), layout.to_half(f(U, pe, M5, mf), L, 0)) < tol
