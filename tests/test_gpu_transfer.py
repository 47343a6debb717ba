"""Restriction and prolongation of one field by the cluster-split kernels
against the same projectors in 64 bits: block sizes on either side of the
splits, basis sizes around the warps' shares, both precisions, and pointers
that are only 8-byte aligned (the general kernels).

Tolerance: n-term FP32 sums of products of O(1) numbers taken 16 at a time and
then in FP64: eps = 6e-8 times sqrt(16) for random signs, 1e-6 allowed in the
norm; FP64 1e-13 (the restriction's result is rounded to FP32: 6e-8)."""
import numpy as np
import pytest
import torch

import synth
from paper_2103_05034_gb300 import ops
from paper_2103_05034_gb300._lib import F32, F64

pytestmark = pytest.mark.gpu


def _blocks(L, block):
    """Coarse site of every site of a full field in storage order (even, then odd)."""
    x, y, z, t = np.meshgrid(*(np.arange(n) for n in L), indexing="ij")
    lex = x + L[0] * (y + L[1] * (z + L[2] * t))
    Lc = [L[m] // block[m] for m in range(4)]
    xc = x // block[0] + Lc[0] * (y // block[1] + Lc[1] * (z // block[2] + Lc[2] * (t // block[3])))
    order = np.argsort(lex.ravel())
    xc, par = xc.ravel()[order], ((x + y + z + t) % 2).ravel()[order]
    return torch.from_numpy(np.concatenate([xc[par == 0], xc[par == 1]])).cuda(), int(np.prod(Lc))


@pytest.mark.parametrize("prec", [F32, F64])
@pytest.mark.parametrize("L,Ls,block,nb,shift", [
    ((4, 4, 4, 4), 4, (2, 2, 2, 2), 5, 0), ((8, 4, 4, 8), 8, (4, 4, 4, 4), 32, 0), ((8, 8, 4, 4), 24, (4, 2, 2, 2), 24, 0),
    ((4, 4, 4, 4), 16, (4, 4, 4, 4), 64, 0), ((16, 16, 16, 8), 4, (2, 2, 2, 2), 8, 0), ((8, 4, 4, 8), 8, (2, 1, 1, 1), 9, 0),
    ((8, 4, 4, 8), 8, (4, 4, 4, 4), 16, 2),
])
def test_restrict_and_prolong_one_field(prec, L, Ls, block, nb, shift):
    if prec == F64 and shift:
        pytest.skip("FP64 numbers are 16 bytes")
    ctx = ops.Context(L, Ls, 1.8, synth.random_gauge(L, 0.3, 5))
    xc, nc = _blocks(L, block)
    dt = torch.float32 if prec == F32 else torch.float64
    g = torch.Generator(device="cuda").manual_seed(3)
    n = 2 * ctx.half_numel()
    basis = torch.randn(nb * n + shift, dtype=dt, device="cuda", generator=g)[shift:]
    f = torch.randn(n + shift, dtype=dt, device="cuda", generator=g)[shift:]
    c = torch.randn(2 * nc * nb, dtype=torch.float32, device="cuda", generator=g)
    P = torch.view_as_complex(basis.double().reshape(nb, -1, 12 * Ls, 2))
    v = torch.view_as_complex(f.double().reshape(-1, 12 * Ls, 2))

    got = ops.dwf_restrict(ctx, torch.zeros_like(c), f, basis, nb, block)
    want = torch.zeros(nc, nb, dtype=torch.complex128, device="cuda")
    for j in range(nb):
        want[:, j].index_add_(0, xc, (P[j].conj() * v).sum(1))
    got = torch.view_as_complex(got.double().reshape(nc, nb, 2))
    assert float((got - want).norm() / want.norm()) < 1e-6

    w = torch.view_as_complex(c.double().reshape(nc, nb, 2))
    full = torch.stack([P[j] * w[xc, j, None] for j in range(nb)]).sum(0)
    for acc in (0, 1):
        out = ops.dwf_prolong(ctx, f.clone() if not shift else torch.cat([f[:shift], f])[shift:], c, basis, nb, block,
                              accumulate=acc)
        ref = full + v if acc else full
        out = torch.view_as_complex(out.double().reshape(-1, 12 * Ls, 2))
        assert float((out - ref).norm() / ref.norm()) < (1e-6 if prec == F32 else 1e-13)
