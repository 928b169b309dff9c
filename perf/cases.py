"""Performance cases of the library: the calls a user makes, at the sizes they are made at.

One steady solve is a nested Newton iteration (Algorithm 3) whose steps are a
residual (Eq. 10 / 20), a finite-difference Jacobian (Eq. 12-13) and a few
multigrid V-cycles (Algorithm 2). Each of these is a call of its own, and most
of the cases are these single calls, in 1D and 2D, FP64 and mixed precision;
the others are whole solves: one alone, and batches of equal and of uneven
problems.

Inputs are the seeded channels, bumps and wedges of the package's `inputs`
module with the sizes of its tests and benchmark; the iterates handed to the
single calls are smooth flows with small-scale noise, as in the middle of a
Newton iteration. The Jacobians handed to the V-cycles are formed here, by the
plain torch restatement of the discretisation below, which also gives the
64-bit values of `exact`.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2505_10857_gb300 import inputs as I
from paper_2505_10857_gb300 import nswe

F64, F32 = torch.float64, torch.float32
DEVICE = "cuda" if torch.cuda.is_available() else "cpu"  # (the restatement below also runs without a GPU)


# ---------------------------------------------------------------------------------------------- cases

def listed():
    return [
        # the smallest call: the convergence check of one N = 200 channel; launch latency is all of it
        {"name": "residual-1d-200", "do": "residual1d", "N": 200, "levels": 4},
        # the residual and J3 of one very long channel: the throughput of the 1D Jacobian
        {"name": "jacobian-1d-j3-1m", "do": "jacobian1d", "N": 1 << 20, "levels": 14, "nb": 3, "precision": "fp64"},
        # one linear solve step of the 4096-cell channel for a caller with a Newton loop of its own
        {"name": "vcycle-1d-4096", "do": "vcycle1d", "N": 4096, "levels": 8, "nb": 3, "precision": "fp64"},
        # the residual of the 512 x 256 wedge: every Newton step's stopping test
        {"name": "residual-2d-512x256", "do": "residual2d", "Nx": 512, "Ny": 256, "levels": 7, "flow": "wedge"},
        # its simplified Jacobian under the frozen linearisation, with which the wedge converges
        {"name": "jacobian-2d-j9-512x256", "do": "jacobian2d", "Nx": 512, "Ny": 256, "levels": 7, "flow": "wedge",
         "nb": 9, "frozen": True, "precision": "fp64"},
        # the full Jacobian of Eq. 12 on a small bump channel whose sides are no powers of two
        {"name": "jacobian-2d-j21-96x40", "do": "jacobian2d", "Nx": 96, "Ny": 40, "levels": 4, "flow": "bump",
         "nb": 21, "frozen": False, "precision": "fp64"},
        # one FP64 V-cycle of the wedge (nu = 20), three of which make a Newton step
        {"name": "vcycle-2d-512x256", "do": "vcycle2d", "Nx": 512, "Ny": 256, "levels": 7, "flow": "wedge",
         "nb": 9, "precision": "fp64"},
        # the FP32 V-cycle of a mixed-precision step on a serving-sized bump channel
        {"name": "vcycle-2d-f32-128x64", "do": "vcycle2d", "Nx": 128, "Ny": 64, "levels": 5, "flow": "bump",
         "nb": 9, "precision": "mixed"},
        # one FP64 solve, as fast as it can be had: the latency form on a cluster of 16 blocks
        {"name": "solve-1d-4096", "do": "solve1d", "N": 4096, "levels": 8, "ctas": 16, "precision": "fp64"},
        # the benchmark's step: 608 channels of 4096 cells in FP64 to res < 1e-10, one launch
        {"name": "batch-1d-608x4096", "do": "batch1d", "count": 608, "N": 4096, "uneven": False,
         "precision": "fp64"},
        # a serving launch: 304 mixed-precision solves of uneven size, parameters per problem
        {"name": "batch-1d-304-uneven", "do": "batch1d", "count": 304, "N": 8192, "uneven": True,
         "precision": "mixed"},
        # a lockstep batch of four 2D bump channels of 64 x 32 and 32 x 16 cells, mixed precision
        {"name": "batch-2d-4x64x32", "do": "batch2d", "count": 4, "Nx": 64, "Ny": 32, "levels": 4,
         "precision": "mixed"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _nested_size(n):
    """(N, levels): about n cells, nested down to a coarsest grid of [32, 64) cells, as a serving request."""
    levels = max(1, int(math.floor(math.log2(n / 32.0))) + 1)
    m = 1 << (levels - 1)
    return max(32 * m, int(round(n / m)) * m), levels


def _grid(rng, most):
    """(Nx, Ny, levels): a nested 2D grid of at most `most` cells over a coarsest one of 8-11 x 4-6 cells."""
    while True:
        cx, cy, levels = rng.randint(8, 11), rng.randint(4, 6), rng.randint(2, 7)
        Nx, Ny = cx << (levels - 1), cy << (levels - 1)
        if Nx * Ny <= most:
            return Nx, Ny, levels


def draw(rng):
    do = rng.choice(["residual1d", "jacobian1d", "vcycle1d", "residual2d", "jacobian2d", "vcycle2d", "solve1d",
                     "batch1d", "batch2d"])
    prec = rng.choice(["fp64", "mixed"])
    if do in ("residual1d", "jacobian1d"):
        N, levels = _nested_size(_log_int(rng, 100, 1 << 20))
        return {"do": do, "N": N, "levels": levels} if do == "residual1d" else \
            {"do": do, "N": N, "levels": levels, "nb": rng.choice([3, 5]), "precision": prec}
    if do == "vcycle1d":
        N, levels = _nested_size(_log_int(rng, 200, 1 << 16))
        return {"do": do, "N": N, "levels": levels, "nb": rng.choice([3, 5]), "precision": prec}
    if do in ("residual2d", "jacobian2d", "vcycle2d"):
        flow = rng.choice(["wedge", "bump"])
        nb = rng.choice([9, 9, 21])
        Nx, Ny, levels = _grid(rng, 131072 if nb == 9 else 32768)
        c = {"do": do, "Nx": Nx, "Ny": Ny, "levels": levels, "flow": flow}
        if do != "residual2d":
            c.update(nb=nb, precision=prec)
        if do == "jacobian2d":
            c.update(frozen=prec == "fp64" and rng.random() < 0.5)
        return c
    if do == "solve1d":
        N, levels = _nested_size(_log_int(rng, 256, 8192))
        return {"do": do, "N": N, "levels": levels, "ctas": rng.choice([1, 4, 8, 16]), "precision": prec}
    if do == "batch1d":
        uneven = rng.random() < 0.5
        N = _log_int(rng, 512, 8192) if uneven else _nested_size(_log_int(rng, 256, 4096))[0]
        return {"do": do, "count": rng.randint(32, 400), "N": N, "uneven": uneven, "precision": prec}
    Nx, Ny, levels = rng.choice([(32, 16, 3), (40, 24, 3), (64, 32, 4)])
    return {"do": do, "count": rng.randint(2, 6), "Nx": Nx, "Ny": Ny, "levels": levels, "precision": prec}


# ---------------------------------------------------------------------------------------------- inputs

def _gen(seed):
    return np.random.default_rng(1_000_003 + int(seed))


def _dev(a, dtype=F64):
    return torch.as_tensor(np.ascontiguousarray(a)).to(DEVICE).to(dtype).contiguous()


def _channel(k, N, levels):
    """A seeded 1D channel: the sinusoidal-width one of the benchmark, the constant-width one below 256 cells."""
    if N < 256:
        return I.channel_small(k, N=N, levels=levels)
    return I.channel_irregular(k, N=N, levels=levels, start_level=max(0, levels - 4))


def _state1d(inp, seed):
    """An iterate: the lake-at-rest guess's depth and discharge with a wave and grid-scale noise on them."""
    rng, x = _gen(seed), inp.centres()
    h = 2.0 - inp.b_fn(x)
    ph = rng.uniform(0, 2 * np.pi, 2)
    H = inp.sig_fn(x) * h * (1 + 0.02 * np.sin(0.5 * x + ph[0])) + 1e-3 * rng.standard_normal(inp.N)
    Q = 4.42 * (1 + 0.01 * np.cos(0.4 * x + ph[1])) + 1e-3 * rng.standard_normal(inp.N)
    return np.stack([H, Q])


def _flow2d(case, k):
    Nx, Ny, levels = case["Nx"], case["Ny"], case["levels"]
    if case.get("flow", "bump") == "wedge":
        return I.wedge_serving_2d(k, Nx, Ny, levels, start_level=max(0, levels - 2))
    return I.gauss_bump_channel_2d(k, Nx, Ny, levels)


def _state2d(inp, seed):
    """An iterate: the inflow state with a wave and grid-scale noise on it."""
    rng = _gen(seed)
    X, Y = inp.centres()
    lx, ly = 2 * np.pi / (inp.x1 - inp.x0), 2 * np.pi / (inp.y1 - inp.y0)
    ph = rng.uniform(0, 2 * np.pi, 3)
    q = float(inp.bc_state[0][1]) or 1.0
    noise = lambda: 1e-3 * rng.standard_normal(X.shape)  # noqa: E731
    h = 1.0 + 0.1 * np.sin(lx * X + ph[0]) * np.cos(ly * Y) + noise()
    hu = q * (1 + 0.03 * np.cos(lx * X + ph[1])) + noise()
    hv = float(inp.bc_state[0][2]) + 0.05 * np.sin(ly * Y + ph[2]) + noise()
    return np.stack([h.ravel(), hu.ravel(), hv.ravel()])


def _inputs(case, seed):
    """(problem inputs, the host arrays of the call) of one case; no call into the library."""
    if case["do"] in ("residual1d", "jacobian1d", "vcycle1d"):
        inp = _channel(seed, case["N"], case["levels"])
        return inp, _state1d(inp, seed)
    inp = _flow2d(case, seed)
    return inp, _state2d(inp, seed)


def _system(case, seed):
    """The linear system of a Newton step in the V-cycle's precision: (problem inputs, J, R)."""
    inp, U = _inputs(case, seed)
    dt = F32 if case["precision"] == "mixed" else F64
    if case["do"] == "vcycle1d":
        m = Ref1D(inp)
        R, J = m.jacobian(_dev(U), case["nb"], I.eps_channel(case["N"]), 3.0)
    else:
        m = Ref2D(inp)
        R, J = m.jacobian(_dev(U), case["nb"], 1e-6, 3.0, frozen=case["flow"] == "wedge")
    return inp, J.to(dt).contiguous(), R.to(dt).contiguous()


def _uneven_sizes(case):
    """`count` sizes spread over the logarithm of [256, N], in a mixed order."""
    n, step = case["count"], math.log(max(300, case["N"]) / 256.0) / case["count"]
    return [_nested_size(256.0 * math.exp((k + 0.5) * step)) for k in np.random.default_rng(n).permutation(n)]


def _prec(case):
    return nswe.PREC_MIXED if case["precision"] == "mixed" else nswe.PREC_FP64


def _mg_params(case):
    if case["do"] == "vcycle1d":
        return nswe.params(case["N"], case["levels"], omega=0.7, nu1=2, nu2=2, nu3=1, precision=_prec(case))
    return nswe.params(96, case["levels"], omega=0.1, nu1=20, nu2=20, nu3=1, precision=_prec(case))


def prepare(case, seed):
    do = case["do"]
    ctx = nswe.Context(0)
    st = {"case": case, "ctx": ctx}
    if do in ("residual1d", "jacobian1d", "residual2d", "jacobian2d"):
        inp, U = _inputs(case, seed)
        two = do.endswith("2d")
        st["prob"] = (nswe.Problem2D if two else nswe.Problem1D).from_inputs(ctx, inp)
        st["U"] = _dev(U)
        st["R"] = torch.zeros_like(st["U"])
        st["res"] = torch.zeros((), dtype=F64, device="cuda")
        if do.startswith("jacobian"):
            nb, comps = case["nb"], 3 if two else 2
            dt = F32 if case["precision"] == "mixed" else F64
            st["J"] = torch.zeros((nb, comps * comps, st["U"].shape[1]), dtype=dt, device="cuda")
            st["eps"] = 1e-6 if two else I.eps_channel(case["N"])
    elif do in ("vcycle1d", "vcycle2d"):
        inp, J, R = _system(case, seed)
        st["prob"] = (nswe.Problem2D if do == "vcycle2d" else nswe.Problem1D).from_inputs(ctx, inp)
        st["J"], st["R"], st["dU"] = J, R, torch.zeros_like(R)
        st["prm"] = _mg_params(case)
    elif do == "solve1d":
        inp = _channel(seed, case["N"], case["levels"])
        st["prob"] = nswe.Problem1D.from_inputs(ctx, inp)
        nswe.nswe_ctx_set_solve_cluster(ctx, case["ctas"])
        q = nswe.params_from(I.Params1D.for_problem(inp, tol=3e-13, n_max=800))
        q.precision = _prec(case)
        st["prm"], st["U0"] = q, _dev(inp.U0_start)
        st["U"] = torch.zeros((2, inp.N), dtype=F64, device="cuda")
    elif do == "batch1d":
        sizes = _uneven_sizes(case) if case["uneven"] else [_nested_size(case["N"])] * case["count"]
        inps = [_channel(1000 * seed + k, N, L) for k, (N, L) in enumerate(sizes)]
        # the benchmark's stopping test for its equal problems, the serving comparison's for uneven ones
        tol = 3e-13 if case["uneven"] or case["precision"] == "mixed" else 1e-10
        prms = [nswe.params_from(I.Params1D.for_problem(p, tol=tol, n_max=800)) for p in inps]
        for q in prms:
            q.precision = _prec(case)
        if case["precision"] == "fp64":
            nswe.nswe_ctx_set_solve_shape(ctx, nswe.PREC_FP64, nswe.solve_shapes().index((128, 4)))
        st["probs"] = [nswe.Problem1D.from_inputs(ctx, p) for p in inps]
        st["prms"] = prms
        st["U0s"] = [_dev(p.U0_start) for p in inps]
        st["U"] = torch.zeros(2 * sum(p.N for p in inps), dtype=F64, device="cuda")
        st["Us"] = [u.view(2, -1) for u in torch.split(st["U"], [2 * p.N for p in inps])]
    else:  # batch2d
        inps, prms = [], []
        for k in range(case["count"]):
            # seeds of this family converge at these sizes in both precisions
            half = int(k % 3 == 2 and case["levels"] > 3)  # every third channel on the next coarser grid
            p = I.bump_channel_2d(1000 * seed + k, case["Nx"] >> half, case["Ny"] >> half, case["levels"] - half)
            inps.append(p)
            q = nswe.params2d_from(I.Params2D(levels=p.levels, nu1=[20], nu2=[20], tol=1e-11, n_max=400))
            q.precision = _prec(case)
            prms.append(q)
        st["probs"] = [nswe.Problem2D.from_inputs(ctx, p) for p in inps]
        st["prms"] = prms
        st["U0s"] = [_dev(p.U0_start) for p in inps]
        st["Us"] = [torch.zeros((3, p.Nx * p.Ny), dtype=F64, device="cuda") for p in inps]
    torch.cuda.synchronize()
    return st


def run(st):
    case, ctx = st["case"], st["ctx"]
    do = case["do"]
    if do in ("residual1d", "residual2d"):
        nswe.nswe_residual(ctx, st["prob"], 0, st["U"], st["R"], st["res"])
        return {"R": st["R"], "res": st["res"]}
    if do in ("jacobian1d", "jacobian2d"):
        a = (ctx, st["prob"], 0)
        b = (st["U"], st["eps"], 3.0, st["R"], st["J"], st["res"])
        if case["precision"] == "mixed":
            nswe.nswe_jacobian_f32(*a, case["nb"], *b)
        elif case.get("frozen"):
            nswe.nswe_jacobian_frozen(*a, case["nb"], *b)
        elif case["nb"] in (5, 21):
            nswe.nswe_jacobian_full(*a, *b)
        else:
            nswe.nswe_jacobian_simplified(*a, *b)
        return {"R": st["R"], "J": st["J"], "res": st["res"]}
    if do in ("vcycle1d", "vcycle2d"):
        st["dU"].zero_()  # a Newton step's first V-cycle starts from a zero correction
        f = nswe.nswe_mg_vcycle_f32 if case["precision"] == "mixed" else nswe.nswe_mg_vcycle
        f(ctx, st["prob"], 0, case["nb"], st["J"], st["R"], st["dU"], st["prm"])
        return {"dU": st["dU"]}
    if do == "solve1d":
        nswe.nswe_newton_solve(ctx, st["prob"], st["U0"], st["U"], st["prm"])
        return {"U": st["U"]}
    if do == "batch1d":
        if case["uneven"]:
            nswe.nswe_newton_solve_batch_each(ctx, st["probs"], st["U0s"], st["Us"], st["prms"])
        else:
            nswe.nswe_newton_solve_batch(ctx, st["probs"], st["U0s"], st["Us"], st["prms"][0], want_info=False)
        return {"U": st["U"]}
    nswe.nswe_newton_solve_batch_each(ctx, st["probs"], st["U0s"], st["Us"], st["prms"])
    return {"U": torch.cat([u.reshape(-1) for u in st["Us"]])}


# ---------------------------------------------------------------------------------------------- work

# Flops per cell of the steps, each quantity formed once (a division or square root is one): 1D, WENO of
# one component 38, an HLL face with its two states 40, the source 36, a block product pair 8; 2D, one
# characteristic reconstruction 140 (two sides of two faces), an LLF face with two Gauss points 120.
_RES1, _RES2 = 2 * 38 + 40 + 36 + 4, 4 * 140 + 2 * 120 + 60


def _jac1(nb):
    return 8 * 38 + 8 * 10 + 6 * 3 + 9 * 20 + (nb + 1) * 36 + 18 * nb + 12


def _jac2(nb):
    return 10 * 4 * 140 + (50 if nb == 9 else 74) * 2 * 60 + 3 * nb * 20


# Updates of a cell in one smoothing (2 steps in 1D, 20 in 2D; a colour visited twice in a row counts once).
_VISITS1, _VISITS2 = {3: 2.5, 5: 3.0}, {9: 161 / 3, 21: 641 / 9, "p5": 81 / 2, "p9": 241 / 4}


def _vcycle1(N, nb):
    return N * (2 * _VISITS1[nb] * (8 * (nb - 1) + 14) + 2 * 2.5 * 30 + 60)


def _vcycle2(n, nb):
    p, k = ("p5", 4) if nb == 9 else ("p9", 8)
    return n * (2 * _VISITS2[nb] * (18 * (nb - 1) + 24) + 2 / 3 * _VISITS2[p] * (18 * k + 24))


def work(case):
    do = case["do"]
    if do in ("residual1d", "jacobian1d", "vcycle1d"):
        N, w = case["N"], 4 if case.get("precision") == "mixed" else 8
        if do == "residual1d":
            return {"bytes": 8.0 * N * (2 + 2 + 7), "flops": float(N * _RES1)}
        nb = case["nb"]
        if do == "jacobian1d":
            return {"bytes": N * (8.0 * (2 + 2 + 7) + w * 4 * nb), "flops": float(N * _jac1(nb))}
        return {"bytes": N * w * (4.0 * nb + 2 + 4), "flops": float(_vcycle1(N, nb))}
    if do in ("residual2d", "jacobian2d", "vcycle2d"):
        n, w = case["Nx"] * case["Ny"], 4 if case.get("precision") == "mixed" else 8
        if do == "residual2d":
            return {"bytes": 8.0 * n * (3 + 3 + 8), "flops": float(n * _RES2)}
        nb = case["nb"]
        if do == "jacobian2d":
            return {"bytes": n * (8.0 * (3 + 3 + 8) + w * 9 * nb), "flops": float(n * _jac2(nb))}
        return {"bytes": n * w * (9.0 * nb + 3 + 6), "flops": float(_vcycle2(n, nb))}
    # whole solves: the Newton steps of all levels come to about 60 on the finest one at res < 1e-10, 100 at
    # res < 3e-13, and in 2D 40
    if do in ("solve1d", "batch1d"):
        cells = case["N"]
        if do == "batch1d":
            lo, hi = math.log(256), math.log(max(300, case["N"]))
            cells = case["count"] * ((math.exp(hi) - math.exp(lo)) / (hi - lo) if case["uneven"] else case["N"])
        step = _jac1(3) + 2 * _vcycle1(1, 3)
        return {"bytes": 8.0 * cells * (7 + 2 + 2), "flops": float(cells * (60 if do == "batch1d" and not case["uneven"] else 100) * step)}
    cells = case["count"] * case["Nx"] * case["Ny"]
    return {"bytes": 8.0 * cells * (8 + 3 + 3), "flops": float(cells * 40 * (_jac2(9) + 3 * _vcycle2(1, 9)))}


# ---------------------------------------------------------------------------------------------- 64-bit values

def exact(case, seed):
    do = case["do"]
    if do in ("residual1d", "jacobian1d", "residual2d", "jacobian2d"):
        inp, U = _inputs(case, seed)
        U = _dev(U)
        m = Ref2D(inp) if do.endswith("2d") else Ref1D(inp)
        if do.startswith("residual"):
            R = m.residual(U)
            return {"R": R, "res": R.abs().sum() / R.shape[1]}
        if do == "jacobian1d":
            R, J = m.jacobian(U, case["nb"], I.eps_channel(case["N"]), 3.0)
        else:
            R, J = m.jacobian(U, case["nb"], 1e-6, 3.0, frozen=case["frozen"])
        return {"R": R, "J": J, "res": R.abs().sum() / R.shape[1]}
    if do in ("vcycle1d", "vcycle2d"):
        inp, J, R = _system(case, seed)
        prm = _mg_params(case)
        m = Ref2D(inp) if do == "vcycle2d" else Ref1D(inp)
        return {"dU": m.vcycle(J.to(F64), R.to(F64), case["nb"], prm.nu1, prm.nu2, prm.omega)}
    return None  # a whole solve in plain torch takes minutes


ZETA, GS = 1e-6, 1.0 / (2.0 * math.sqrt(3.0))
# the cubic through t = -3/2, -1/2, 1/2, 3/2 at t = -/+ GS
LAG = [[np.prod([(t - b) / (a - b) for b in (-1.5, -0.5, 0.5, 1.5) if b != a]) for a in (-1.5, -0.5, 0.5, 1.5)]
       for t in (-GS, GS)]


def _weno(a, b, c, frozen=None):
    """WENO3 values at the left and right interface of the middle cell; weights from `frozen` if given."""
    a0, b0, c0 = frozen or (a, b, c)
    s0, s1 = (ZETA + (c0 - b0) ** 2) ** 2, (ZETA + (b0 - a0) ** 2) ** 2
    up = (s1 * (1.5 * b - 0.5 * c) + 2 * s0 * (0.5 * a + 0.5 * b)) / (s1 + 2 * s0)
    um = (2 * s1 * (0.5 * b + 0.5 * c) + s0 * (1.5 * b - 0.5 * a)) / (2 * s1 + s0)
    return up, um


class Ref1D:
    """The quasi-1D discretisation and V-cycle (Sections 2-3) in plain 64-bit torch."""

    def __init__(self, inp):
        self.inp, self.N, self.g, self.dx = inp, inp.N, inp.g, (inp.x1 - inp.x0) / inp.N
        self.sf, self.gq = _dev(inp.sig_face), _dev(inp.gq[0])

    def _pad(self, U):
        def ghost(bc, s, e):
            kind, h, q = bc
            H = e[0] if kind in (I.BC_DISCHARGE, I.BC_EXTRAP) else e[0] * 0 + s * h
            Q = e[1] if kind in (I.BC_DEPTH, I.BC_EXTRAP) else e[1] * 0 + q
            return torch.stack([H, Q]).view(2, 1).expand(2, 2)
        return torch.cat([ghost(self.inp.bcl, self.sf[0], U[:, 0]), U, ghost(self.inp.bcr, self.sf[-1], U[:, -1])], 1)

    def residual(self, U):
        P, g, sf = self._pad(U), self.g, self.sf
        up, um = _weno(P[:, :-2], P[:, 1:-1], P[:, 2:])  # cells -1 .. N

        def state(V):
            H, Q = V
            return H, Q, Q / H, torch.sqrt(g * H / sf), Q * Q / H + g * H * H / (2 * sf)
        HL, QL, uL, cL, FL = state(um[:, :-1])
        HR, QR, uR, cR, FR = state(up[:, 1:])
        SL, SR = torch.minimum(uL - cL, uR - cR), torch.maximum(uL + cL, uR + cR)
        F0 = (SR * QL - SL * QR + SL * SR * (HR - HL)) / (SR - SL)
        F1 = (SR * FL - SL * FR + SL * SR * (QR - QL)) / (SR - SL)
        F0 = torch.where(SL >= 0, QL, torch.where(SR <= 0, QR, F0))
        F1 = torch.where(SL >= 0, FL, torch.where(SR <= 0, FR, F1))
        v = [up[0, :-2], up[0, 1:-1], um[0, 1:-1], um[0, 2:]]
        S = 0
        for q in range(2):
            Hh = sum(LAG[q][i] * v[i] for i in range(4))
            sig, sx, bx = self.gq[0, q], self.gq[1, q], self.gq[2, q]
            S = S + 0.5 * g * (Hh / sig) ** 2 * sx - g * Hh * bx
        return torch.stack([F0[1:] - F0[:-1], F1[1:] - F1[:-1] - 0.5 * self.dx * S])

    def jacobian(self, U, nb, eps, alpha):
        N, hw = self.N, (nb - 1) // 2
        R = self.residual(U)
        J = torch.zeros((nb, 2, 2, N), dtype=F64, device=U.device)
        j = torch.arange(N, device=U.device)
        for a in range(5):
            for m in range(2):
                V = U.clone()
                V[m, a::5] += eps
                D = (self.residual(V) - R) / eps
                for k in range(nb):
                    on = ((j + k - hw) % 5 == a) & (j + k - hw >= 0) & (j + k - hw < N)
                    J[k, :, m] = torch.where(on, D, J[k, :, m])
        reg = alpha * R.abs().sum(0)
        J[hw, 0, 0] += reg
        J[hw, 1, 1] += reg
        return R, J.view(nb, 4, N)

    def vcycle(self, J, R, nb, nu1, nu2, omega, level=0):
        N, hw = J.shape[2], (nb - 1) // 2
        B = J.view(nb, 2, 2, N).permute(3, 0, 1, 2)  # cell, block, row, column
        if level == self.inp.levels - 1:
            A = torch.zeros((N, 2, N + 2 * hw, 2), dtype=F64, device=J.device)
            c = torch.arange(N, device=J.device)
            for k in range(nb):
                A[c, :, c + k] = B[:, k]
            A = A[:, :, hw:hw + N].reshape(2 * N, 2 * N)
            return torch.linalg.solve(A, -R.t().reshape(-1)).view(N, 2).t().contiguous()
        Di, C = torch.linalg.inv(B[:, hw]), hw + 1
        x = torch.zeros((N + 2 * hw, 2), dtype=F64, device=J.device)

        def smooth(steps):
            for _ in range(steps):
                for col in list(range(C)) + list(range(C - 1, -1, -1)):
                    c = torch.arange(col, N, C, device=J.device)
                    r = R[:, c].t()
                    for k in range(nb):
                        if k != hw:
                            r = r + (B[c, k] @ x[c + k].unsqueeze(2)).squeeze(2)
                    x[c + hw] = (1 - omega) * x[c + hw] - omega * (Di[c] @ r.unsqueeze(2)).squeeze(2)
        smooth(nu1)
        c = torch.arange(N, device=J.device)
        d = R.t() + sum((B[:, k] @ x[c + k].unsqueeze(2)).squeeze(2) for k in range(nb))
        Bc = torch.zeros((N // 2, 3, 2, 2), dtype=F64, device=J.device)
        for a in range(2):
            for k in range(nb):
                Bc[:, (a + k - hw) // 2 + 1] += B[a::2, k]
        Jc = Bc.permute(1, 2, 3, 0).reshape(3, 4, N // 2)
        e = self.vcycle(Jc, (d[0::2] + d[1::2]).t(), 3, nu1, nu2, omega, level + 1)
        x[hw:hw + N] += e.t().repeat_interleave(2, 0)
        smooth(nu2)
        return x[hw:hw + N].t().contiguous()


J9 = [(0, -2), (0, -1), (-2, 0), (-1, 0), (0, 0), (1, 0), (2, 0), (0, 1), (0, 2)]
J21 = sorted(((x, y) for x in range(-2, 3) for y in range(-2, 3) if abs(x) + abs(y) < 4), key=lambda o: (o[1], o[0]))
P5 = [(0, -1), (-1, 0), (0, 0), (1, 0), (0, 1)]
P9 = [(x, y) for y in (-1, 0, 1) for x in (-1, 0, 1)]


class Ref2D:
    """The 2D discretisation and V-cycle (Section 4) in plain 64-bit torch."""

    def __init__(self, inp):
        self.inp, self.Nx, self.Ny, self.g = inp, inp.Nx, inp.Ny, inp.g
        self.dx, self.dy = (inp.x1 - inp.x0) / inp.Nx, (inp.y1 - inp.y0) / inp.Ny
        self.gq = _dev(inp.gq[0]).view(2, 4, inp.Ny, inp.Nx)
        # every cell of the padded grid is an interior cell's state, scaled and shifted: x rule, then y rule
        Nx, Ny, kinds, st = inp.Nx, inp.Ny, inp.bc_kind[0], inp.bc_state
        src = np.zeros((Ny + 4, Nx + 4), np.int64)
        mul, add = np.ones((3, Ny + 4, Nx + 4)), np.zeros((3, Ny + 4, Nx + 4))

        def post(kind, s, normal, m, a):
            if kind == I.BC2_REFLECT:
                m[normal], a[normal] = -m[normal], -a[normal]
            elif kind == I.BC2_DISCHARGE:
                m[1:], a[1:] = 0, s[1:]
            elif kind == I.BC2_DEPTH:
                m[0], a[0] = 0, s[0]
        jj, ii = np.mgrid[0:Ny, 0:Nx]
        src[2:-2, 2:-2] = jj * Nx + ii
        ghosts = [(i, j) for j in range(-2, Ny + 2) for i in range(-2, Nx + 2)
                  if not (0 <= j < Ny and 0 <= i < Nx)] if Nx * Ny < 64 else \
            [(i, j) for j in (-2, -1, Ny, Ny + 1) for i in range(-2, Nx + 2)] + \
            [(i, j) for j in range(Ny) for i in (-2, -1, Nx, Nx + 1)]
        for gi, gj in ghosts:
            i, j, xk, m, a = gi, gj, 0, np.ones(3), np.zeros(3)
            at = (slice(None), gj + 2, gi + 2)
            if i < 0 or i >= Nx:
                xs = 0 if i < 0 else 1
                xk = kinds[xs * Ny + min(max(j, 0), Ny - 1)]
                if xk == I.BC2_INFLOW:
                    mul[at], add[at] = 0, st[xs]
                    continue
                i = (-1 - i if i < 0 else 2 * Nx - 1 - i) if xk == I.BC2_REFLECT else (0 if i < 0 else Nx - 1)
            if j < 0 or j >= Ny:
                ys = 2 if j < 0 else 3
                yk = kinds[2 * Ny + (ys - 2) * Nx + i]
                if yk == I.BC2_INFLOW:
                    m[:], a[:], j = 0, st[ys], 0
                else:
                    j = (-1 - j if j < 0 else 2 * Ny - 1 - j) if yk == I.BC2_REFLECT else (0 if j < 0 else Ny - 1)
                    post(yk, st[ys], 2, m, a)
            if xk:
                post(xk, st[xs], 1, m, a)
            src[gj + 2, gi + 2] = j * Nx + i
            mul[at], add[at] = m, a
        self.src, self.mul, self.add = torch.as_tensor(src).to(DEVICE), _dev(mul), _dev(add)

    def _pad(self, U):
        return self.mul * U[:, self.src.view(-1)].view(3, *self.src.shape) + self.add

    def _interfaces(self, P, B, d):
        """U^- and U^+ at the interfaces between cells k and k + 1 of direction d of the padded grid P, each
        where it has its three cells: L[k], k = 1.., and R[k], k = 0..; weights and eigenvectors from B."""
        n, t = (1, 2) if d == 0 else (2, 1)
        sh = (lambda A, a, b: A[:, :, a:b]) if d == 0 else (lambda A, a, b: A[:, a:b])
        M = P.shape[2 - d]

        def rec(s, lo):  # cells lo..lo+2 relative to the first interface's cells; side s (0: minus, 1: plus)
            cnt = M - 2
            f0 = 1 if s == 0 else 0  # interface index = left cell index
            a, b = sh(B, f0, f0 + cnt), sh(B, f0 + 1, f0 + 1 + cnt)
            h = 0.5 * (a[0] + b[0])
            un, ut = 0.5 * (a[n] + b[n]) / h, 0.5 * (a[t] + b[t]) / h
            c = torch.sqrt(self.g * h)

            def char(v):
                return [((un + c) * v[0] - v[n]) / (2 * c), v[t] - ut * v[0], (v[n] - (un - c) * v[0]) / (2 * c)]
            W = [char(sh(P, lo + i, lo + i + cnt)) for i in range(3)]
            Z = W if B is P else [char(sh(B, lo + i, lo + i + cnt)) for i in range(3)]
            w = [_weno(W[0][f], W[1][f], W[2][f], (Z[0][f], Z[1][f], Z[2][f]))[1 - s] for f in range(3)]
            o = [None, None, None]
            o[0], o[n], o[t] = w[0] + w[2], (un - c) * w[0] + (un + c) * w[2], ut * (w[0] + w[2]) + w[1]
            return torch.stack(o)
        return rec(0, 0), rec(1, 0)

    def _direction(self, P, B, d):
        """(flux difference, source part) of direction d."""
        L, R = self._interfaces(P, B, d)  # interface k + 1/2 of the padded grid: L[k-1], R[k]
        if d == 1:
            L, R = L.transpose(1, 2), R.transpose(1, 2)
        N, T = (self.Nx, self.Ny) if d == 0 else (self.Ny, self.Nx)
        n, t, g = (1, 2, self.g) if d == 0 else (2, 1, self.g)
        flux, acc = 0, 0
        for q, s in ((0, -1.0), (1, 1.0)):
            gp = lambda V: V[:, 2:2 + T] + s / (4 * math.sqrt(3.0)) * (V[:, 3:3 + T] - V[:, 1:1 + T])  # noqa: E731
            l, r = gp(L), gp(R)
            # faces -1/2 .. N-1/2 of the interior lie between padded cells 1|2 .. N+1|N+2
            A, C = l[:, :, 0:N + 1], r[:, :, 1:N + 2]

            def phys(V):
                F = [V[n], V[n] * V[1] / V[0], V[n] * V[2] / V[0]]
                F[n] = F[n] + 0.5 * g * V[0] ** 2
                return torch.stack(F)
            a = torch.maximum((A[n] / A[0]).abs() + torch.sqrt(g * A[0]), (C[n] / C[0]).abs() + torch.sqrt(g * C[0]))
            F = 0.5 * (phys(A) + phys(C)) - 0.5 * a * (C - A)
            flux = flux + 0.5 * (F[:, :, 1:] - F[:, :, :-1])
            v = [r[0, :, 0:N], r[0, :, 1:N + 1], l[0, :, 1:N + 1], l[0, :, 2:N + 2]]
            for p in range(2):
                z = self.gq[d, 2 * q + p] if d == 0 else self.gq[d, 2 * p + q].t()
                acc = acc + g * sum(LAG[p][i] * v[i] for i in range(4)) * z
        S = -0.25 * acc
        return (flux, S) if d == 0 else (flux.transpose(1, 2), S.t())

    def residual(self, U, base=None):
        P = self._pad(U)
        B = P if base is None else self._pad(base)
        (fx, sx), (fy, sy) = self._direction(P, B, 0), self._direction(P, B, 1)
        R = fx / self.dx + fy / self.dy
        return torch.stack([R[0], R[1] - sx, R[2] - sy]).reshape(3, -1)

    def jacobian(self, U, nb, eps, alpha, frozen=False):
        Nx, Ny = self.Nx, self.Ny
        offs = J9 if nb == 9 else J21
        R = self.residual(U)
        J = torch.zeros((nb, 3, 3, Ny * Nx), dtype=F64, device=U.device)
        c = torch.arange(Nx * Ny, device=U.device)
        i, j = c % Nx, c // Nx
        for b in range(5):
            for a in range(5):
                hit = (i % 5 == a) & (j % 5 == b)
                for m in range(3):
                    V = U.clone()
                    V[m] += eps * hit
                    D = (self.residual(V, U if frozen else None) - R) / eps
                    for k, (ox, oy) in enumerate(offs):
                        p, q = i + ox, j + oy
                        on = (p % 5 == a) & (q % 5 == b) & (p >= 0) & (p < Nx) & (q >= 0) & (q < Ny)
                        J[k, :, m] = torch.where(on, D, J[k, :, m])
        for m in range(3):
            J[offs.index((0, 0)), m, m] += alpha * R.abs().sum(0)
        return R, J.view(nb, 9, Ny * Nx)

    def vcycle(self, J, R, nb, nu1, nu2, omega):
        return self._level(J, R, J9 if nb == 9 else J21, self.Nx, self.Ny, nu1, nu2, omega, 0)

    def _level(self, J, R, offs, Nx, Ny, nu1, nu2, omega, level):
        n, W = Nx * Ny, Nx + 4
        B = J.reshape(len(offs), 3, 3, n).permute(3, 0, 1, 2).contiguous()
        c = torch.arange(n, device=J.device)
        i, j = c % Nx, c // Nx
        pos = (j + 2) * W + i + 2  # in the padded correction
        kc = offs.index((0, 0))
        if level == self.inp.levels - 1:
            A = torch.zeros((n, 3, (Ny + 4) * W, 3), dtype=F64, device=J.device)
            for k, (ox, oy) in enumerate(offs):
                A[c, :, pos + oy * W + ox] = B[:, k]
            A = A[:, :, pos].reshape(3 * n, 3 * n)
            return torch.linalg.solve(A, -R.t().reshape(-1)).view(n, 3).t().contiguous()
        cross = len(offs) in (5, 9) and offs is not P9
        if cross:
            C = 3 if offs is J9 else 2
            colour = (i + j) % C
        else:
            C, s = (9, 3) if offs is J21 else (4, 2)
            colour = i % s + s * (j % s)
        x = torch.zeros(((Ny + 4) * W, 3), dtype=F64, device=J.device)
        Di = torch.linalg.inv(B[:, kc])
        Rt, ks = R.t().contiguous(), [k for k in range(len(offs)) if k != kc]
        sets = []
        for col in range(C):
            z = c[colour == col]
            near = torch.stack([pos[z] + offs[k][1] * W + offs[k][0] for k in ks], 1)
            G = B[z][:, ks].permute(0, 2, 1, 3).reshape(len(z), 3, -1).contiguous()
            sets.append((pos[z], near, G, Di[z], Rt[z]))

        def smooth(steps):
            for _ in range(steps):
                for col in (list(range(C)) + list(range(C - 1, -1, -1))) * 2:
                    p, near, G, D, r = sets[col]
                    r = r + (G @ x[near].reshape(len(p), -1, 1)).squeeze(2)
                    x[p] = (1 - omega) * x[p] - omega * (D @ r.unsqueeze(2)).squeeze(2)
        smooth(nu1)
        d = Rt + sum((B[:, k] @ x[pos + oy * W + ox].unsqueeze(2)).squeeze(2) for k, (ox, oy) in enumerate(offs))
        sub = P5 if cross else P9
        Bc = torch.zeros((Ny // 2, Nx // 2, len(sub), 3, 3), dtype=F64, device=J.device)
        Bf = B.view(Ny, Nx, len(offs), 3, 3)
        for b in range(2):
            for a in range(2):
                for k, (ox, oy) in enumerate(offs):
                    Bc[:, :, sub.index(((a + ox) // 2, (b + oy) // 2))] += Bf[b::2, a::2, k]
        Jc = Bc.view(-1, len(sub), 3, 3).permute(1, 2, 3, 0).reshape(len(sub), 9, -1)
        Rc = d.view(Ny // 2, 2, Nx // 2, 2, 3).sum((1, 3)).view(-1, 3).t()
        e = self._level(Jc, Rc, sub, Nx // 2, Ny // 2, nu1, nu2, omega, level + 1)
        e = e.t().view(Ny // 2, Nx // 2, 3).repeat_interleave(2, 0).repeat_interleave(2, 1)
        x[pos] += e.reshape(-1, 3)
        smooth(nu2)
        return x[pos].t().contiguous()
