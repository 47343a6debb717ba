"""The complex-split tensor-core coarse stencil where a CTA takes more than one
quad of sites (the accumulator is drained and reused), against the FP32 stencil
on the CUDA cores.

Tolerance: both factors of a product are rounded to TF32 (2^-11 relative), so
each product is off by at most 2^-10 and, with independent signs, a sum of them
by less in the norm: 1e-3."""
import pytest
import torch

import synth
from paper_2103_05034_gb300 import ops
from paper_2103_05034_gb300._lib import F32, TF32

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nrhs", [16, 32])
@pytest.mark.parametrize("L", [(8, 8, 8, 24), (12, 8, 12, 28)])  # 192 and 504 quads on 152 SMs
def test_several_quads_a_cta(L, nrhs):
    ctx = ops.Context(L, 4, 1.8, synth.random_gauge(L, 0.3, 5))
    n = 2 * ctx.half_numel()
    g = torch.Generator(device="cuda").manual_seed(2)
    basis = torch.randn(32 * n, dtype=torch.float64, device="cuda", generator=g)
    for h, sign in ((slice(0, 16 * n), 1), (slice(16 * n, 32 * n), -1)):
        ops.dwf_chiral_project(ctx, basis[h], basis[h], sign, 16)
    ops.block_orthonormalise(ctx, basis, 32, 16, (2, 2, 2, 2))
    C = ops.coarse_build(ctx, basis, 32, 16, (2, 2, 2, 2), 0.1)
    x = torch.randn(C.nc * 32 * nrhs * 2, device="cuda", generator=g)
    want = ops.coarse_apply(C, torch.zeros_like(x), x, nrhs, F32)
    for _ in range(2):
        got = ops.coarse_apply(C, torch.zeros_like(x), x, nrhs, TF32)
        ops.coarse_apply_status(C)
        assert float((got - want).norm() / want.norm()) < 1e-3
