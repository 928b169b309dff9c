"""The levels that lie beyond a cluster: 2D levels swept by grid-wide colour
passes (alone and in lockstep batches, colour-major and not) and 1D levels whose
legs are launches over the chip. The tail's default threshold puts the grids of
the other tests on the cluster, so the threshold is lowered here. Bounds of the
other tests of these calls: the same bits for another path of one computation,
1e-12 relative in FP64 and 1e-5 in FP32 against the CPU oracle."""
import numpy as np
import pytest

import oracle
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


def dev(a, dtype=torch.float64):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda().to(dtype)


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("tail,colour_major", [(16, -1), (16, 256), (128, 256)])
def test_lockstep_batches_with_grid_wide_levels_equal_single_solves(nswe, precision, tail, colour_major):
    """Problems whose V-cycles have different numbers of levels off the
    cluster: a wedge under the frozen linearisation, bumps with J9 and J21."""
    inps = [I.wedge(32, 16, 3, start_level=1), I.bump_channel_2d(1, 32, 16, 3), I.bump_channel_2d(2, 64, 32, 4),
            I.bump_channel_2d(3, 32, 16, 3)]
    kw = [dict(nest_start=1, omega=0.1, frozen=True), {}, {}, dict(st=1)]
    prms = [nswe.params2d_from(I.Params2D(levels=p.levels, nu1=[20], nu2=[20], tol=1e-10, n_max=400, **k))
            for p, k in zip(inps, kw)]
    ctx, ref = nswe.Context(0), nswe.Context(0)  # ref: the defaults, every level of these on the cluster
    nswe.nswe_ctx_set_tail_2d(ctx, precision, tail)
    nswe.nswe_ctx_set_colour_major_2d(ctx, colour_major)
    nswe.nswe_ctx_set_batch_2d(ctx, nswe.BATCH2D_LOCKSTEP)
    probs = [nswe.Problem2D.from_inputs(ctx, p) for p in inps]
    rprobs = [nswe.Problem2D.from_inputs(ref, p) for p in inps]
    U0s = [dev(p.U0_start) for p in inps]
    for q in prms:
        q.precision = precision
    try:
        alone = []
        for c, ps in ((ref, rprobs), (ctx, probs)):
            for pr, u0, p, q in zip(ps, U0s, inps, prms):
                U = torch.zeros((3, p.Nx * p.Ny), dtype=torch.float64, device="cuda")
                info = nswe.nswe_newton_solve(c, pr, u0, U, q)
                alone.append((U.cpu().numpy(), info))
        Us = [torch.zeros((3, p.Nx * p.Ny), dtype=torch.float64, device="cuda") for p in inps]
        infos = nswe.nswe_newton_solve_batch_each(ctx, probs, U0s, Us, prms)
        Us = [u.cpu().numpy() for u in Us]
    finally:
        for p in probs + rprobs:
            p.close()
    for k in range(len(inps)):
        for U, info in (alone[len(inps) + k], (Us[k], infos[k])):
            assert info["status"] == 0 and info["iters"] == alone[k][1]["iters"], k
            assert np.array_equal(U, alone[k][0]), k


@pytest.mark.parametrize("grid", [(32, 16, 3), (40, 24, 3), (64, 32, 4)])
@pytest.mark.parametrize("precision", [0, 1])
def test_a_v_cycle_copied_colour_major_gives_the_same_bits(nswe, grid, precision):
    Nx, Ny, levels = grid
    n = Nx * Ny
    rng = np.random.default_rng(n)
    J = 0.03 * rng.standard_normal((9, 9, n))
    c = np.arange(n)
    for k, (ox, oy) in enumerate(oracle.stencil2d(0)):
        i, j = c % Nx + ox, c // Nx + oy
        J[k][:, (i < 0) | (i >= Nx) | (j < 0) | (j >= Ny)] = 0
        if (ox, oy) == (0, 0):
            J[k][[0, 4, 8]] += 1 + rng.random((3, n))
    R, x = rng.standard_normal((3, n)), 0.1 * rng.standard_normal((3, n))
    dt, f, bound = ((torch.float64, nswe.nswe_mg_vcycle, 1e-12), (torch.float32, nswe.nswe_mg_vcycle_f32, 1e-5))[precision]
    ref = oracle.vcycle2d(J, R, x, Nx, Ny, 0, levels, 0.3, 3, 2)
    ref = ref if isinstance(ref, np.ndarray) else ref[0]
    ctx = nswe.Context(0)
    nswe.nswe_ctx_set_tail_2d(ctx, precision, 16)
    prob = nswe.Problem2D.from_inputs(ctx, I.gauss_bump_channel_2d(3, Nx, Ny, levels))
    prm = nswe.params(96, levels, omega=0.3, nu1=3, nu2=2, nu3=1)
    got, Jd = [], dev(J, dt)
    for min_cells in (-1, 1):
        nswe.nswe_ctx_set_colour_major_2d(ctx, min_cells)
        d = dev(x, dt)
        f(ctx, prob, 0, 9, Jd, dev(R, dt), d, prm)
        got.append(d.cpu().numpy())
    prob.close()
    assert np.array_equal(Jd.cpu().numpy(), J.astype(got[0].dtype))  # the caller's operator is left as it was
    assert np.array_equal(got[0], got[1])
    assert np.abs(got[0] - ref).max() <= bound * np.abs(ref).max()


@pytest.mark.parametrize("N,levels", [(6016, 7), (10368, 8), (20736, 9), (41472, 10)])
@pytest.mark.parametrize("nu1,nu2", [(2, 2), (1, 2)])
def test_legs_over_the_chip_in_both_precisions(nswe, N, levels, nu1, nu2):
    """One level of more tiles than a cluster takes, two in a row and three, on
    a diagonally dominant system, whose cycle converges."""
    rng = np.random.default_rng(N)
    J = 0.1 * rng.standard_normal((3, 4, N))
    J[1][[0, 3]] += 1 + rng.random((2, N))
    J[0][:, 0] = J[2][:, -1] = 0
    R, dU0 = rng.standard_normal((2, N)), 0.1 * rng.standard_normal((2, N))
    J, R, dU0 = (a.astype(np.float32).astype(np.float64) for a in (J, R, dU0))
    ref = oracle.vcycle1d(J, R, dU0, 3, levels, 0.7, nu1, nu2)
    ctx = nswe.Context(0)
    prob = nswe.Problem1D.from_inputs(ctx, I.channel_small(7, N=N, levels=levels))
    prm = nswe.params(N, levels, omega=0.7, nu1=nu1, nu2=nu2)
    errs = []
    for dt, f, bound in ((torch.float64, nswe.nswe_mg_vcycle, 1e-12), (torch.float32, nswe.nswe_mg_vcycle_f32, 1e-5)):
        x = dev(dU0, dt)
        f(ctx, prob, 0, 3, dev(J, dt), dev(R, dt), x, prm)
        errs.append((np.abs(x.cpu().numpy() - ref).max() / np.abs(ref).max(), bound))
    prob.close()
    assert all(e <= b for e, b in errs), errs
