"""Workloads of the library on one GPU, each one pass through a public entry point.

A case is a dict of plain values; `kind` says which entry point it calls:

  op      one operator application: dwf_dhop, dwf_mpc, dwf_mpcdag_mpc, dwf_ddw, dwf_hdw
  solve   a red-black CG solve to the accuracy of an HMC accept/reject step (rbcg_solve)
  batch   the pseudofermion solves of one gauge field, a mass each (rbcg_normal_solve_batch)
  force   the fermion force of several pseudofermions (dwf_force)
  filter  the Chebyshev filter of a subspace setup (cheby_filter)
  vcycle  one V(1,1) cycle of the HDCR multigrid (mg_precondition)
  coarse  the little Dirac operator on many right-hand sides (coarse_apply)

Fields are complex Gaussians (sources, pseudofermions); links are U = exp(i eps H) with H from Gaussian
coefficients of the Gell-Mann matrices, on lattices longer than 16 the field of a smaller lattice repeated.
"""
import math

import torch

from paper_2103_05034_gb300 import ops
from paper_2103_05034_gb300._lib import COARSE_CG, F16S, F32, F64, SOLVE_MIXED_F32, TF32

M5 = 1.8
EPS = 0.2  # smooth links, like the smeared stand-in ensembles
PREC = {"f64": F64, "f32": F32, "f16": F16S}
REAL = {"f64": torch.float64, "f32": torch.float32, "f16": torch.float16}
BYTES = {"f64": 16, "f32": 8, "f16": 4}  # of one complex number
MASSES = (0.01, 0.05, 0.2, 1.0)          # the Hasenbusch-style masses of the force workload


def listed():
    return [
        # the smallest call there is: the parity lattice, where launches and latency are all
        {"name": "mpc_f64_4x4x4x4_ls8", "kind": "op", "op": "mpc", "prec": "f64", "L": "4x4x4x4", "Ls": 8, "nrhs": 1,
         "dagger": False, "mf": 0.01, "tuned": False},
        # the inner operator of the CG on the 16^3 test volume, as a context gives it without tuning
        {"name": "mpcdag_f32_16x16x16x32_ls16", "kind": "op", "op": "mpcdag", "prec": "f32", "L": "16x16x16x32", "Ls": 16,
         "nrhs": 1, "dagger": False, "mf": 0.01, "tuned": False},
        # the same operator on the largest multigrid volume, tuned as a production run does it; far larger than L2
        {"name": "mpcdag_f32_24x24x24x48_ls24", "kind": "op", "op": "mpcdag", "prec": "f32", "L": "24x24x24x48", "Ls": 24,
         "nrhs": 1, "dagger": False, "mf": 0.00078, "tuned": True},
        # H_DW of three fields on a lattice whose extents divide nothing evenly, at a short fifth dimension
        {"name": "hdw_f32_12x6x10x14_ls8_n3", "kind": "op", "op": "hdw", "prec": "f32", "L": "12x6x10x14", "Ls": 8, "nrhs": 3,
         "dagger": False, "mf": 0.02, "tuned": False},
        # the inner operator of the FP16-storage CG
        {"name": "mpcdag_f16_16x16x16x32_ls16", "kind": "op", "op": "mpcdag", "prec": "f16", "L": "16x16x16x32", "Ls": 16,
         "nrhs": 1, "dagger": False, "mf": 0.01, "tuned": False},
        # D_DW^dag in FP64: true residuals and the FP64 solves
        {"name": "ddwdag_f64_8x8x8x16_ls24", "kind": "op", "op": "ddw", "prec": "f64", "L": "8x8x8x16", "Ls": 24, "nrhs": 1,
         "dagger": True, "mf": 0.00078, "tuned": False},
        # a whole mixed-precision solve on the 16^3 test volume
        {"name": "rbcg_16x16x16x32_ls16", "kind": "solve", "L": "16x16x16x32", "Ls": 16, "mf": 0.01, "tol": 1e-12},
        # the four pseudofermion solves of a molecular dynamics step on a small volume
        {"name": "normal_batch_8x8x8x16_ls16", "kind": "batch", "L": "8x8x8x16", "Ls": 16, "npf": 4, "tol": 1e-12},
        # the force of that step on the 16^3 test volume, in single precision
        {"name": "force_f32_16x16x16x32_ls16", "kind": "force", "prec": "f32", "L": "16x16x16x32", "Ls": 16, "npf": 4},
        # two vectors of the subspace setup through a filter
        {"name": "filter_f32_12x12x12x24_ls16_n2", "kind": "filter", "prec": "f32", "L": "12x12x12x24", "Ls": 16, "nrhs": 2,
         "order": 40, "mf": 0.01},
        # the preconditioner of the HDCR solve; a fixed number of coarse iterations
        {"name": "vcycle_16x16x16x16_ls16_nb32", "kind": "vcycle", "L": "16x16x16x16", "Ls": 16, "block": 4, "nb": 32,
         "smooth": 20, "coarse_iters": 24, "mf": 0.01},
        # the coarse operator of 512 sites on 32 right-hand sides: the tensor-core stencil
        {"name": "coarse_tf32_nc512_nb32_n32", "kind": "coarse", "prec": "tf32", "L": "8x8x8x16", "Ls": 4, "block": 2, "nb": 32,
         "nrhs": 32, "mf": 0.01},
    ]


def _even(rng, lo, hi):
    """An even extent, evenly spread over the logarithm."""
    return 2 * round(math.exp(rng.uniform(math.log(lo), math.log(hi))) / 2)


def _lattice(rng, lo, hi, most):
    """Four extents and Ls, of at most `most` 5D sites."""
    while True:
        L, Ls = [_even(rng, lo, hi) for _ in range(3)] + [_even(rng, lo, 1.5 * hi)], rng.choice((4, 8, 16, 16, 24, 24))
        if math.prod(L) * Ls <= most:
            return "x".join(map(str, L)), Ls


def draw(rng):
    kind = rng.choice(("op", "op", "op", "op", "solve", "batch", "force", "filter", "vcycle", "coarse"))
    mf = round(math.exp(rng.uniform(math.log(0.001), math.log(0.2))), 5)
    if kind == "op":
        op, prec = rng.choice(("dhop", "mpc", "mpcdag", "ddw", "hdw")), rng.choice(("f64", "f32", "f32", "f32", "f16"))
        L, Ls = _lattice(rng, 4, 24, 2e6 if prec == "f64" else 8e6)
        nrhs = rng.choice((1, 1, 2, 3, 5)) if math.prod(map(int, L.split("x"))) * Ls < 2e6 else 1
        return {"kind": kind, "op": op, "prec": prec, "L": L, "Ls": Ls, "nrhs": nrhs,
                "dagger": op in ("dhop", "mpc", "ddw") and rng.random() < 0.5, "mf": mf, "tuned": rng.random() < 0.3}
    if kind == "solve":
        L, Ls = _lattice(rng, 4, 16, 1e6)
        return {"kind": kind, "L": L, "Ls": Ls, "mf": max(mf, 0.01), "tol": 1e-12}
    if kind == "batch":
        L, Ls = _lattice(rng, 4, 12, 3e5)
        return {"kind": kind, "L": L, "Ls": Ls, "npf": rng.choice((2, 3, 4)), "tol": 1e-12}
    if kind == "force":
        prec = rng.choice(("f32", "f64"))
        L, Ls = _lattice(rng, 4, 16, 5e5 if prec == "f64" else 2e6)
        return {"kind": kind, "prec": prec, "L": L, "Ls": Ls, "npf": rng.choice((1, 2, 4))}
    if kind == "filter":
        L, Ls = _lattice(rng, 4, 16, 1e6)
        return {"kind": kind, "prec": "f32", "L": L, "Ls": Ls, "nrhs": rng.choice((1, 2, 4)), "order": rng.randrange(10, 61), "mf": mf}
    if kind == "vcycle":
        L = "x".join(str(4 * rng.choice((2, 3, 4))) for _ in range(4))
        return {"kind": kind, "L": L, "Ls": rng.choice((8, 16)), "block": 4, "nb": rng.choice((16, 24, 32)),
                "smooth": rng.randrange(8, 41), "coarse_iters": 24, "mf": mf}
    L = "x".join(str(2 * rng.choice((2, 4, 6) if m == 0 else (2, 3, 4, 6))) for m in range(4))
    return {"kind": kind, "prec": rng.choice(("tf32", "f32")), "L": L, "Ls": 4, "block": 2, "nb": 32,
            "nrhs": rng.choice((16, 32, 64)), "mf": mf}


# ---------------------------------------------------------------------- inputs
def _dims(case):
    return tuple(int(v) for v in case["L"].split("x"))


def _generator(seed, part):
    return torch.Generator(device="cuda").manual_seed(1000003 * int(seed) + part)


def _gaussian(gen, *shape):
    return torch.randn(*shape, dtype=torch.float64, device="cuda", generator=gen)


def _gauge(L, seed):
    """(T, Z, Y, X, mu, 3, 3) complex128 links."""
    base, times = list(L), [1, 1, 1, 1]
    for m in range(4):
        while base[m] > 16 and base[m] % 4 == 0:
            base[m], times[m] = base[m] // 2, times[m] * 2
    w = _gaussian(_generator(seed, 1), base[3], base[2], base[1], base[0], 4, 8) / 2
    H = torch.zeros(*w.shape[:-1], 3, 3, dtype=torch.complex128, device="cuda")
    for k, (a, b) in enumerate(((0, 1), (0, 2), (1, 2))):
        H[..., a, b] = torch.complex(w[..., 2 * k], -w[..., 2 * k + 1])
        H[..., b, a] = torch.complex(w[..., 2 * k], w[..., 2 * k + 1])
    d3, d8 = w[..., 6], w[..., 7] / math.sqrt(3)
    for a, v in enumerate((d3 + d8, -d3 + d8, -2 * d8)):
        H[..., a, a] = v.to(torch.complex128)
    U = torch.matrix_exp(1j * EPS * H)
    return U.repeat(times[3], times[2], times[1], times[0], 1, 1, 1).contiguous()


def _field(case, seed, parities, n, part=2, prec="f64"):
    """n Gaussian fields of one (half) or two parities as the library stores them: interleaved reals."""
    V = math.prod(_dims(case)) // 2 * parities
    return _gaussian(_generator(seed, part), n * V * 12 * case["Ls"] * 2).to(REAL[prec])


def _blocked_basis(case, seed):
    """nb orthonormal block vectors of definite Gamma_5 chirality as full FP32 fields: on every block Gaussian
    vectors orthonormalised in order, (1 + Gamma_5)/2 of the first half and (1 - Gamma_5)/2 of the rest."""
    L, Ls, nb, b = _dims(case), case["Ls"], case["nb"], case["block"]
    g = _gaussian(_generator(seed, 3), nb, math.prod(L), 12, Ls, 2)
    v = torch.view_as_complex(g)
    g5 = _gamma5(v.flatten(0, 1)).reshape(v.shape)
    sign = torch.where(torch.arange(nb, device="cuda") < nb // 2, 1.0, -1.0).reshape(nb, 1, 1, 1)
    v = (v + sign * g5) / 2
    blocks = _to_blocks(v, L, b)  # (nc, nb, dim)
    q = [torch.linalg.solve_triangular(torch.linalg.cholesky(h @ h.mH), h, upper=False)
         for h in (blocks[:, : nb // 2], blocks[:, nb // 2:])]
    return _from_blocks(torch.cat(q, 1), L, b, 12 * Ls)


def prepare(case, seed):
    L, kind = _dims(case), case["kind"]
    ctx = ops.Context(L, case["Ls"], M5, _gauge(L, seed))
    s = {"case": case, "ctx": ctx}
    if kind == "op":
        full = case["op"] in ("ddw", "hdw")
        s["in"] = _field(case, seed, 2 if full else 1, case["nrhs"], prec=case["prec"])
        s["out"] = torch.zeros_like(s["in"])
        if case["tuned"]:
            ops.dwf_autotune(ctx, PREC[case["prec"]], 10)
    elif kind == "solve":
        s["b"] = _field(case, seed, 2, 1)
        s["x"] = torch.zeros_like(s["b"])
    elif kind == "batch":
        s["b"] = _field(case, seed, 1, case["npf"])
        s["x"] = torch.zeros_like(s["b"])
    elif kind == "force":
        s["X"] = _field(case, seed, 1, case["npf"], prec=case["prec"])
        s["force"] = torch.zeros(L[3], L[2], L[1], L[0], 4, 3, 3, dtype=torch.complex128, device="cuda")
    elif kind == "filter":
        s["in"] = _field(case, seed, 2, case["nrhs"], prec="f32")
        s["out"] = torch.zeros_like(s["in"])
    elif kind == "vcycle":
        p = ops.mg_params((case["block"],) * 4, case["nb"], case["mf"], lambda_lo=0.5, lambda_max=80.0, filter_order=16,
                          smooth=(0.5, 80.0, case["smooth"]), coarse_tol=1e-12, coarse_maxiter=case["coarse_iters"],
                          coarse_solver=COARSE_CG)
        s["mg"] = ops.MG(ctx, p, _field(case, seed, 2, case["nb"]))
        s["in"] = _field(case, seed, 2, 1, part=4, prec="f32")
        s["out"] = torch.zeros_like(s["in"])
    elif kind == "coarse":
        basis = torch.view_as_real(_to_library(_blocked_basis(case, seed), L)).to(torch.float32).flatten()
        s["coarse"] = ops.coarse_build(ctx, basis, case["nb"], case["nb"] // 2, (case["block"],) * 4, case["mf"])
        s["in"] = _coarse_input(case, seed)
        s["out"] = torch.zeros_like(s["in"])
    return s


def _coarse_input(case, seed):
    nc = math.prod(_dims(case)) // case["block"] ** 4
    return _gaussian(_generator(seed, 5), nc * case["nb"] * case["nrhs"] * 2).to(torch.float32)


def run(s):
    case, ctx = s["case"], s["ctx"]
    kind = case["kind"]
    if kind == "op":
        op, dag, n = case["op"], int(case["dagger"]), case["nrhs"]
        if op == "dhop":
            return ops.dwf_dhop(ctx, s["out"], s["in"], 0, dag, n)
        if op == "mpc":
            return ops.dwf_mpc(ctx, s["out"], s["in"], case["mf"], dag, n)
        if op == "mpcdag":
            return ops.dwf_mpcdag_mpc(ctx, s["out"], s["in"], case["mf"], n)
        if op == "ddw":
            return ops.dwf_ddw(ctx, s["out"], s["in"], case["mf"], dag, n)
        return ops.dwf_hdw(ctx, s["out"], s["in"], case["mf"], n)
    if kind == "solve":
        ops.rbcg_solve(ctx, s["x"], s["b"], case["mf"], case["tol"], policy=SOLVE_MIXED_F32)
        return s["x"]
    if kind == "batch":
        ops.rbcg_normal_solve_batch(ctx, s["x"], s["b"], MASSES[: case["npf"]], case["tol"], policy=SOLVE_MIXED_F32)
        return s["x"]
    if kind == "force":
        s["force"].zero_()  # dwf_force adds to what is there
        ops.dwf_force(ctx, s["force"], s["X"], MASSES[: case["npf"]])
        # momenta of a single-precision trajectory take the force of FP32 fields in single precision
        return s["force"] if case["prec"] == "f64" else s["force"].to(torch.complex64)
    if kind == "filter":
        return ops.cheby_filter(ctx, s["out"], s["in"], case["nrhs"], 1.0, 80.0, case["order"], case["mf"])
    if kind == "vcycle":
        return ops.mg_precondition(s["mg"], s["out"], s["in"])
    return ops.coarse_apply(s["coarse"], s["out"], s["in"], case["nrhs"], TF32 if case["prec"] == "tf32" else F32)


# ---------------------------------------------------------------------- work
# Each distinct array that a pass needs is counted once per operator application that needs it: a solver of n
# iterations reads its operator's links and vectors n times, an operator writes its result once.  Nothing
# between the operator's own hopping terms is counted.
HOP_FLOPS = 1320                                  # per 5D output site
CG_ITERS = {"solve": 440, "batch": 330}           # iterations these solves take, about (batch: mean over the masses)


def _half(case, n, w):
    """Bytes of n half fields and of the links of both parities, w bytes a complex number."""
    Vh = math.prod(_dims(case)) // 2
    return n * Vh * 12 * case["Ls"] * w, 2 * Vh * 72 * (16 if w == 16 else 8)


def work(case):
    kind = case["kind"]
    sites = math.prod(_dims(case)) // 2 * case["Ls"]  # 5D sites of one parity
    if kind == "op":
        n = case["nrhs"]
        hops = {"dhop": 1, "mpc": 2, "mpcdag": 4, "ddw": 2, "hdw": 2}[case["op"]]
        f, u = _half(case, n * (4 if case["op"] in ("ddw", "hdw") else 2), BYTES[case["prec"]])
        return {"bytes": f + (u / 2 if hops == 1 else u), "flops": hops * n * sites * (HOP_FLOPS + 48)}
    if kind in ("solve", "batch"):
        n = case.get("npf", 1)
        f, u = _half(case, 9 * n, 8)  # p in, x, r, p in and out, A p folded into r, once more p
        return {"bytes": CG_ITERS[kind] * (f + u), "flops": CG_ITERS[kind] * 4 * n * sites * (HOP_FLOPS + 48)}
    if kind == "force":
        f, u = _half(case, case["npf"], BYTES[case["prec"]])
        V = math.prod(_dims(case))
        return {"bytes": f + u + 2 * V * 36 * 16, "flops": case["npf"] * sites * (4 * HOP_FLOPS + 2 * 8 * 9 * 2 * 8)}
    if kind == "filter":
        f, u = _half(case, 8 * case["nrhs"], 8)  # T_k, T_k-1 in, T_k+1 out, D T_k between
        return {"bytes": case["order"] * (f + u), "flops": case["order"] * 4 * case["nrhs"] * sites * (HOP_FLOPS + 48)}
    if kind == "vcycle":
        f, u = _half(case, 10, 8)
        basis = _half(case, 2 * 2 * case["nb"], 8)[0]
        nc = math.prod(_dims(case)) // case["block"] ** 4
        stencil = nc * 9 * case["nb"] ** 2 * 8
        hsq = 2 * case["smooth"]
        return {"bytes": hsq * (f + u) + basis + stencil,
                "flops": hsq * 4 * sites * (HOP_FLOPS + 48) + 2 * case["coarse_iters"] * nc * 9 * case["nb"] ** 2 * 8}
    nc = math.prod(_dims(case)) // case["block"] ** 4
    return {"bytes": nc * case["nb"] * (9 * case["nb"] + 2 * case["nrhs"]) * 8,
            "flops": nc * 9 * case["nb"] ** 2 * case["nrhs"] * 8}


# ---------------------------------------------------------------------- the same in 64 bits, in plain torch
# Fields here are (V, 12, Ls) complex128 in lexicographic site order, 12 = spin * 3 + colour.
_SHIFT_AXIS = (3, 2, 1, 0)


def _parity(L):
    i = torch.arange(math.prod(L), device="cuda")
    x, i = i % L[0], i // L[0]
    y, i = i % L[1], i // L[1]
    z, t = i % L[2], i // L[2]
    return (x + y + z + t) % 2


def _from_half(h, L, p):
    out = torch.zeros(math.prod(L), *h.shape[1:], dtype=h.dtype, device=h.device)
    out[_parity(L) == p] = h
    return out


def _to_library(v, L):
    """(..., V, 12, Ls) -> (..., 2, Vh, 12, Ls), even parity first."""
    par = _parity(L)
    return torch.stack([v[..., par == 0, :, :], v[..., par == 1, :, :]], dim=-4)


def _complex(t, *shape):
    return torch.view_as_complex(t.double().reshape(*shape, 2))


def _gamma(mu, v):
    """gamma_mu v in the chiral basis, v (V, 12, Ls)."""
    p = v.reshape(v.shape[0], 4, 3, v.shape[2])
    a, b, c, d = (p[:, k] for k in range(4))
    rows = ((-1j * d, -1j * c, 1j * b, 1j * a), (-d, c, b, -a), (-1j * c, 1j * d, 1j * a, -1j * b), (c, d, a, b))[mu]
    return torch.stack(rows, 1).reshape(v.shape)


def _gamma5(v):
    """Gamma_5 = gamma_5 with s reversed."""
    w = v.flip(-1).clone()
    w[:, 6:] *= -1
    return w


def _shift(v, L, mu, step):
    """v(x + step mu)."""
    return v.reshape(L[3], L[2], L[1], L[0], *v.shape[1:]).roll(-step, _SHIFT_AXIS[mu]).reshape(v.shape)


def _colour(U, v):
    """U (V, 3, 3) on the colour index of v (V, 12, Ls)."""
    p = v.reshape(v.shape[0], 4, 3, v.shape[2])
    out = torch.zeros_like(p)
    for a in range(3):
        for b in range(3):
            out[:, :, a] += U[:, a, b, None, None] * p[:, :, b]
    return out.reshape(v.shape)


class _Exact:
    def __init__(self, case, seed):
        self.L, self.Ls = _dims(case), case["Ls"]
        self.V = math.prod(self.L)
        self.U = _gauge(self.L, seed).reshape(self.V, 4, 3, 3)
        self.even = (_parity(self.L) == 0)[:, None, None]

    def field(self, case, seed, parities, n, **k):
        """The n input fields, each as (V, 12, Ls): halves are even fields."""
        h = _complex(_field(case, seed, parities, n, **k), n, parities, self.V // 2, 12, self.Ls)
        if parities == 1:
            return [_from_half(v[0], self.L, 0) for v in h]
        return [_from_half(v[0], self.L, 0) + _from_half(v[1], self.L, 1) for v in h]

    def back(self, vs, parities):
        """The reals of n fields as the library stores them."""
        h = [_to_library(v, self.L)[:parities] for v in vs]
        return torch.view_as_real(torch.stack(h)).flatten()

    def dhop(self, v, dag=False):
        out, s = torch.zeros_like(v), -1.0 if dag else 1.0
        for mu in range(4):
            f = _colour(self.U[:, mu], _shift(v, self.L, mu, 1))
            out += f - s * _gamma(mu, f)
            b = _shift(_colour(self.U[:, mu].mH, v), self.L, mu, -1)
            out += b + s * _gamma(mu, b)
        return out

    def fifth(self, mf, dag):
        """The Ls x Ls matrices of the site-local part on spins 0, 1 and on spins 2, 3."""
        M = torch.diag(torch.full((self.Ls,), 5.0 - M5, dtype=torch.float64, device="cuda"))
        for k in range(self.Ls):
            M[k, k - 1] += -1.0 if k else mf
        return (M.T, M) if dag else (M, M.T)

    def site(self, v, mf, dag=False, inverse=False):
        w = torch.empty_like(v)
        for half, M in zip((slice(0, 6), slice(6, 12)), self.fifth(mf, dag)):
            M = torch.linalg.inv(M) if inverse else M
            w[:, half] = v[:, half] @ M.T.to(torch.complex128)
        return w

    def ddw(self, v, mf, dag=False):
        return self.site(v, mf, dag) - 0.5 * self.dhop(v, dag)

    def hdw(self, v, mf):
        return _gamma5(self.ddw(v, mf))

    def mpc(self, v, mf, dag=False):
        o = self.site(self.dhop(v, dag), mf, dag, True)
        return (self.site(v, mf, dag) - 0.25 * self.dhop(o, dag)) * self.even

    def normal(self, v, mf):
        return self.mpc(self.mpc(v, mf), mf, True)

    def cg(self, rhs, mf, tol):
        x, r, p = torch.zeros_like(rhs), rhs.clone(), rhs.clone()
        rr = stop = float(torch.linalg.vector_norm(r)) ** 2
        for _ in range(2000):
            if rr <= tol * tol * stop:
                break
            q = self.normal(p, mf)
            a = rr / float(torch.vdot(p.flatten(), q.flatten()).real)
            x += a * p
            r -= a * q
            new = float(torch.linalg.vector_norm(r)) ** 2
            p = r + (new / rr) * p
            rr = new
        return x


def _force_exact(E, Xs, masses):
    G = torch.zeros(E.V, 4, 3, 3, dtype=torch.complex128, device="cuda")
    eye = torch.eye(3, dtype=torch.complex128, device="cuda")
    for X, mf in zip(Xs, masses):
        Y = E.mpc(X, mf)
        Xf = X - 0.5 * E.site(E.dhop(X), mf, False, True)
        Yf = Y - 0.5 * E.site(E.dhop(Y, True), mf, True, True)
        for mu in range(4):
            Xp, Yp = _shift(Xf, E.L, mu, 1), _shift(Yf, E.L, mu, 1)
            l, r = Xp - _gamma(mu, Xp), Xf + _gamma(mu, Xf)
            five = lambda f: f.reshape(E.V, 4, 3, E.Ls).transpose(1, 2).reshape(E.V, 3, 4 * E.Ls)
            A, B = five(l) @ five(Yf).mH, five(r) @ five(Yp).mH
            Z = E.U[:, mu] @ A - B @ E.U[:, mu].mH
            Z = (Z - Z.mH) / 2
            G[:, mu] += Z - Z.diagonal(dim1=1, dim2=2).sum(1)[:, None, None] / 3 * eye
    return G.reshape(E.L[3], E.L[2], E.L[1], E.L[0], 4, 3, 3)


def _to_blocks(v, L, b):
    """(n, V, 12, Ls) -> (nc, n, b^4 * 12 * Ls), coarse sites lexicographic."""
    n, c = v.shape[0], [m // b for m in L]
    w = v.reshape(n, c[3], b, c[2], b, c[1], b, c[0], b, -1)
    return w.permute(1, 3, 5, 7, 0, 2, 4, 6, 8, 9).reshape(math.prod(c), n, -1)


def _from_blocks(w, L, b, inner):
    n, c = w.shape[1], [m // b for m in L]
    w = w.reshape(c[3], c[2], c[1], c[0], n, b, b, b, b, inner)
    return w.permute(4, 0, 5, 1, 6, 2, 7, 3, 8, 9).reshape(n, math.prod(L), 12, inner // 12)


def _coarse_exact(case, seed):
    """P^dag H_DW P of the input: what the 9-point stencil is."""
    E, L, b, n = _Exact(case, seed), _dims(case), case["block"], case["nrhs"]
    P = _to_blocks(_blocked_basis(case, seed).to(torch.complex64).to(torch.complex128), L, b)  # (nc, nb, dim)
    v = _complex(_coarse_input(case, seed), P.shape[0], case["nb"], n)
    fine = _from_blocks(torch.einsum("ckd,ckr->crd", P, v), L, b, 12 * case["Ls"])
    h = torch.stack([E.hdw(f, case["mf"]) for f in fine])
    out = torch.einsum("ckd,crd->ckr", P.conj(), _to_blocks(h, L, b))
    return torch.view_as_real(out.contiguous()).flatten()


def exact(case, seed):
    kind = case["kind"]
    sites = math.prod(_dims(case)) * case["Ls"]
    if kind == "vcycle" or kind in ("solve", "batch") and sites > 1.5e5:
        return None  # minutes in plain torch
    if kind == "coarse":
        return _coarse_exact(case, seed)
    E = _Exact(case, seed)
    if kind == "op":
        parities, mf, dag = 2 if case["op"] in ("ddw", "hdw") else 1, case["mf"], case["dagger"]
        vs = E.field(case, seed, parities, case["nrhs"], prec=case["prec"])
        if case["op"] == "dhop":  # the input is of odd parity
            vs = [_from_half(v[_parity(E.L) == 0], E.L, 1) for v in vs]
        f = {"dhop": lambda v: E.dhop(v, dag), "mpc": lambda v: E.mpc(v, mf, dag), "mpcdag": lambda v: E.normal(v, mf),
             "ddw": lambda v: E.ddw(v, mf, dag), "hdw": lambda v: E.hdw(v, mf)}[case["op"]]
        return E.back([f(v) for v in vs], parities)
    if kind == "solve":
        b, mf = E.field(case, seed, 2, 1)[0], case["mf"]
        be = (b * E.even) + 0.5 * E.dhop(E.site(b * ~E.even, mf, False, True)) * E.even
        xe = E.cg(E.mpc(be, mf, True), mf, 1e-14)
        return E.back([xe + E.site(b * ~E.even + 0.5 * E.dhop(xe), mf, False, True)], 2)
    if kind == "batch":
        return E.back([E.cg(v, m, 1e-14) for v, m in zip(E.field(case, seed, 1, case["npf"]), MASSES)], 1)
    if kind == "force":
        return _force_exact(E, E.field(case, seed, 1, case["npf"], prec=case["prec"]), MASSES)
    a, c = 2.0 / 79.0, -81.0 / 79.0  # the interval [1, 80] to [-1, 1]
    out = []
    for v in E.field(case, seed, 2, case["nrhs"], prec="f32"):
        step = lambda w: a * E.ddw(E.ddw(w, case["mf"]), case["mf"], True) + c * w
        old, new = v, step(v)
        for _ in range(case["order"] - 1):
            old, new = new, 2 * step(new) - old
        out.append(new)
    return E.back(out, 2)
