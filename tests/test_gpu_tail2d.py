"""The cluster launch of a 2D V-cycle's lower levels at the sizes where a band
of rows can go wrong (row pairs that the CTAs share unevenly, fewer pairs than
CTAs, widths that no colour divides, one smoothed level), in both precisions,
against the CPU oracle with the bounds of the other V-cycle tests (1e-12
relative in FP64, 1e-5 in FP32); levels on and off the cluster give the same
bits."""
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


@pytest.mark.parametrize("grid", [(8, 8, 2), (16, 40, 3), (20, 24, 3), (10, 36, 2), (88, 48, 4)])
@pytest.mark.parametrize("nb,colours", [(9, 0), (9, 4), (21, 0)])
def test_vcycles_match_the_oracle_on_and_off_the_cluster(nswe, grid, nb, colours):
    Nx, Ny, levels = grid
    inp = I.gauss_bump_channel_2d(3, Nx, Ny, levels)
    n, st = Nx * Ny, 1 if nb == 21 else 0
    rng = np.random.default_rng(n)
    J = 0.03 * rng.standard_normal((nb, 9, n))
    c = np.arange(n)
    for k, (ox, oy) in enumerate(oracle.stencil2d(st)):
        i, j = c % Nx + ox, c // Nx + oy
        J[k][:, (i < 0) | (i >= Nx) | (j < 0) | (j >= Ny)] = 0
        if (ox, oy) == (0, 0):
            J[k][[0, 4, 8]] += 1 + rng.random((3, n))
    R, x = rng.standard_normal((3, n)), 0.1 * rng.standard_normal((3, n))
    ref = oracle.vcycle2d(J, R, x, Nx, Ny, st, levels, 0.3, 3, 2, colours=colours)
    ref = ref if isinstance(ref, np.ndarray) else ref[0]
    ctx = nswe.Context(0)
    prob = nswe.Problem2D.from_inputs(ctx, inp)
    prm = nswe.params(96, levels, omega=0.3, nu1=3, nu2=2, nu3=1, colours2d=colours)
    for dt, f, bound in ((torch.float64, nswe.nswe_mg_vcycle, 1e-12), (torch.float32, nswe.nswe_mg_vcycle_f32, 1e-5)):
        got = []
        for tail in (1 << 30, n // 4, 0):  # all levels on the cluster, all but the finest, none
            nswe.nswe_ctx_set_tail_2d(ctx, 1 if dt == torch.float32 else 0, tail)
            dU = torch.from_numpy(x).cuda().to(dt)
            f(ctx, prob, 0, nb, torch.from_numpy(J).cuda().to(dt), torch.from_numpy(R).cuda().to(dt), dU, prm)
            got.append(dU.cpu().numpy())
            assert np.abs(got[-1] - ref).max() <= bound * np.abs(ref).max(), (dt, tail)
        assert np.array_equal(got[0], got[1]) and np.array_equal(got[0], got[2])
