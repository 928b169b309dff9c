"""1D V-cycles and residuals at the edges of their tiles: levels of one tile
(16 pairs), of two that just overlap, of one more than a cluster takes, legs of
one and two smoothing steps, and what goes pass by pass (J5, other steps); the
residual at 31- and 254-cell tiles, around 16 tiles (one cluster) and where the
large tiles begin. Against the CPU oracle with the bounds of the other tests of
these calls: V-cycles 1e-12 relative in FP64 and 1e-5 in FP32, residuals 1e-12
of the flux scale."""
import numpy as np
import pytest

import oracle
from gpu_util import flux_scale
from paper_2505_10857_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nswe():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2505_10857_gb300 import nswe as N
    oracle.build()
    return N


@pytest.fixture(scope="module")
def ctx(nswe):
    return nswe.Context(0)


def state(inp, seed):
    rng, x = np.random.default_rng(seed), inp.centres()
    H = inp.sig_fn(x) * 2.0 * (1 + 0.05 * np.sin(3 * x)) + 0.01 * rng.standard_normal(inp.N)
    return np.ascontiguousarray(np.stack([H, 4.42 + 0.05 * rng.standard_normal(inp.N)]))


def dev(a, dtype=torch.float64):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda().to(dtype)


@pytest.mark.parametrize("N,levels", [(8, 2), (32, 2), (34, 2), (52, 2), (54, 2), (128, 6), (616, 4), (1280, 5),
                                      (1296, 5), (6016, 7)])
@pytest.mark.parametrize("nb,nu1,nu2", [(3, 2, 2), (3, 1, 2), (3, 2, 1), (3, 3, 2), (3, 0, 1), (5, 2, 2)])
def test_vcycle_at_tile_edges(nswe, ctx, N, levels, nb, nu1, nu2):
    inp = I.channel_small(7, N=N, levels=levels)
    prob = nswe.Problem1D.from_inputs(ctx, inp)
    J, R, _ = oracle.jacobian1d(oracle.problem_levels(inp)[0], state(inp, 1), I.eps_for_n(N), 3.0, nb)
    J, R = (a.astype(np.float32).astype(np.float64) for a in (J, R))
    dU0 = (1e-3 * np.random.default_rng(2).standard_normal((2, N))).astype(np.float32).astype(np.float64)
    ref = oracle.vcycle1d(J, R, dU0, nb, levels, 0.7, nu1, nu2)
    prm = nswe.params(N, levels, omega=0.7, nu1=nu1, nu2=nu2)
    both = ((torch.float64, nswe.nswe_mg_vcycle, 1e-12), (torch.float32, nswe.nswe_mg_vcycle_f32, 1e-5))
    # (on the larger noisy systems a cycle diverges, |dU| up to 1e11, and FP32 loses digits whatever the kernel)
    for dt, f, bound in both[:2 if N <= 616 else 1]:
        x = dev(dU0, dt)
        f(ctx, prob, 0, nb, dev(J, dt), dev(R, dt), x, prm)
        err = np.abs(x.cpu().numpy() - ref).max() / np.abs(ref).max()
        assert err <= bound, (dt, err)
    prob.close()


@pytest.mark.parametrize("N,levels", [(4, 1), (31, 1), (32, 1), (62, 1), (64, 1), (128, 1), (496, 3), (500, 3),
                                      (18688, 9), (18944, 9), (25344, 9), (299008, 13)])
def test_residual_at_tile_edges(nswe, ctx, N, levels):
    inp = I.make_problem_1d(N, levels, 0.0, 25.0, 9.81, I.bottom_gaussian(0.1, 10.0, 2.0),
                            I.width_sine(1.0, 1, 25.0), (I.BC_DISCHARGE, 0.0, 4.42), (I.BC_DEPTH, 2.0, 0.0),
                            h_init=2.0, q_init=4.42)
    prob = nswe.Problem1D.from_inputs(ctx, inp)
    U = state(inp, 3)
    Rref, resref = oracle.residual1d(oracle.problem_levels(inp)[0], U)
    dR = torch.zeros((2, N), dtype=torch.float64, device="cuda")
    res = torch.zeros((), dtype=torch.float64, device="cuda")
    nswe.nswe_residual(ctx, prob, 0, dev(U), dR, res)
    sc = flux_scale(U, inp.g)
    assert np.abs(dR.cpu().numpy() - Rref).max() <= 1e-12 * sc
    assert abs(float(res) - resref) <= 1e-12 * max(resref, sc * 1e-3)
    prob.close()


@pytest.mark.parametrize("precision,bound", [(0, 1e-13), (1, 1e-8)])
@pytest.mark.parametrize("count", [304, 305])
def test_batches_around_two_problems_per_sm(nswe, ctx, precision, bound, count):
    """The default launch shape's two register budgets: the same solve, to the
    compiler's choice of fused multiply-adds (bounds of the cluster form's test)."""
    inps = [I.channel_small(k % 3, N=128, levels=3) for k in range(count)]
    prm = nswe.params_from(I.Params1D.for_problem(inps[0], tol=1e-10, n_max=500))
    prm.precision = precision
    probs = [nswe.Problem1D.from_inputs(ctx, p) for p in inps]
    U0s = [dev(p.U0_start) for p in inps]
    Us = [torch.zeros((2, 128), dtype=torch.float64, device="cuda") for _ in inps]
    infos = nswe.nswe_newton_solve_batch(ctx, probs, U0s, Us, prm)
    one = torch.zeros_like(Us[0])
    for k in range(3):
        info = nswe.nswe_newton_solve(ctx, probs[k], U0s[k], one, prm)
        assert info["status"] == 0 and all(infos[i]["status"] == 0 for i in range(k, count, 3))
        for i in range(k, count, 3):
            assert float((Us[i] - one).abs().max()) <= bound * float(one.abs().max())
    for p in probs:
        p.close()
