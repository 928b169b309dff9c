"""The tile kernels of the 2D residual and Jacobian at the sizes where a tile
can go wrong: grids of four cells, sides that no tile divides, one row of
tiles, walls and inflow meeting in corners; against the CPU oracle, with the
bounds of the other 2D parity tests (1e-12 of the flux scale, and for the
Jacobian the finite-difference allowance 16 u scale / eps)."""
import numpy as np
import pytest

import oracle
from paper_2505_10857_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from gpu_util import EPS64  # noqa: E402

BUMPS = I.bottom2d_gaussians([(0.1, 1.2, 0.8, 0.6), (-0.05, 2.0, 1.5, 0.4)])


def problem(kind, Nx, Ny):
    """One level; every boundary kind, changing along a side, with walls in the corners or open ones."""
    if kind == "open":
        sides = (I.BC2_INFLOW, I.BC2_OUTFLOW, lambda x: I.BC2_OUTFLOW if x < 1.5 else I.BC2_REFLECT, I.BC2_DEPTH)
        st = np.array([[1.6, 2.2, 0.3], [0, 0, 0], [0, 0, 0], [1.4, 0.0, 0.0]])
    else:
        sides = (I.BC2_REFLECT, lambda y: I.BC2_DISCHARGE if y < 1 else I.BC2_REFLECT,
                 lambda x: I.BC2_INFLOW if x < 1 else I.BC2_REFLECT, I.BC2_REFLECT)
        st = np.array([[1.6, 2.2, 0.3], [0, 1.0, 0.2], [1.1, 0.3, 0.4], [1.4, 0.0, 0.0]])
    return I.make_problem_2d(Nx, Ny, 1, 0.0, 3.0, 0.0, 2.0, 9.81, BUMPS, sides, st, lambda X, Y: (1.5, 2.0, 0.1))


def state(n, seed):
    rng = np.random.default_rng(seed)
    return np.stack([1.3 + 0.3 * rng.random(n), 1.0 + 0.3 * rng.random(n), 0.2 * rng.standard_normal(n)])


def scale(U, inp):
    d = min((inp.x1 - inp.x0) / inp.Nx, (inp.y1 - inp.y0) / inp.Ny)
    m = np.abs(U[1:]).max()
    return (m * m / U[0].min() + 0.5 * inp.g * U[0].max() ** 2 + m) / d


@pytest.fixture(scope="module")
def nswe():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2505_10857_gb300 import nswe as N
    oracle.build()
    return N


@pytest.mark.parametrize("kind", ["open", "walls"])
@pytest.mark.parametrize("grid", [(4, 4), (5, 7), (13, 9), (33, 5), (6, 47), (21, 23)])
def test_tiles_match_the_oracle(nswe, kind, grid):
    inp = problem(kind, *grid)
    n = inp.Nx * inp.Ny
    U = state(n, n)
    ctx = nswe.Context(0)
    prob = nswe.Problem2D.from_inputs(ctx, inp)
    ref = oracle.problem_levels2d(inp)[0]
    sc, eps = scale(U, inp), 1e-4
    Ud = torch.from_numpy(U).cuda()
    R, res = torch.full_like(Ud, float("nan")), torch.zeros((), dtype=torch.float64, device="cuda")
    nswe.nswe_residual(ctx, prob, 0, Ud, R, res)
    Rr, rr = oracle.residual2d(ref, U)
    assert np.abs(R.cpu().numpy() - Rr).max() <= 1e-12 * sc
    assert abs(res.item() - rr) <= 1e-12 * sc
    for nb in (9, 21):
        for frozen in (False, True):
            J = torch.full((nb, 9, n), float("nan"), dtype=torch.float64, device="cuda")
            if frozen:
                nswe.nswe_jacobian_frozen(ctx, prob, 0, nb, Ud, eps, 3.0, R, J)
            else:
                f = nswe.nswe_jacobian_simplified if nb == 9 else nswe.nswe_jacobian_full
                f(ctx, prob, 0, Ud, eps, 3.0, R, J)
            Jr = oracle.jacobian2d(ref, U, eps, 3.0, 1 if nb == 21 else 0, frozen=frozen)[0]
            J = J.cpu().numpy()
            tol = 1e-12 * np.abs(Jr).max() + 16 * EPS64 * sc / eps
            assert np.abs(J - Jr).max() <= tol, (nb, frozen)
            i, j = np.arange(n) % inp.Nx, np.arange(n) // inp.Nx
            for k, (ox, oy) in enumerate(oracle.stencil2d(1 if nb == 21 else 0)):
                out = (i + ox < 0) | (i + ox >= inp.Nx) | (j + oy < 0) | (j + oy >= inp.Ny)
                assert (J[k][:, out] == 0).all()


def test_a_cell_that_is_not_a_number_reaches_the_cells_that_read_it_and_no_other(nswe):
    inp = problem("open", 21, 23)
    n = inp.Nx * inp.Ny
    U = state(n, 5)
    U[0, 11 * inp.Nx + 10] = np.nan
    ctx = nswe.Context(0)
    prob = nswe.Problem2D.from_inputs(ctx, inp)
    R = torch.zeros((3, n), dtype=torch.float64, device="cuda")
    res = torch.zeros((), dtype=torch.float64, device="cuda")
    nswe.nswe_residual(ctx, prob, 0, torch.from_numpy(U).cuda(), R, res)
    Rr, rr = oracle.residual2d(oracle.problem_levels2d(inp)[0], U)
    assert np.array_equal(np.isnan(R.cpu().numpy()), np.isnan(Rr)) and np.isnan(Rr).any() and not np.isnan(Rr).all()
    assert np.isnan(res.item()) and np.isnan(rr)
