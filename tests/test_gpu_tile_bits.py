"""The 2D Jacobian's unperturbed fluxes round as the residual's: where a
perturbation cannot reach a component (the momentum along a face, two cells
across it, moves neither the depth's nor the normal momentum's flux), the
perturbed residual less the residual is exactly zero, so the block entry is.
One rounding apart it would be some 1e-10 of the flux scale. (The frozen
linearisation takes its weighted means in another order than the residual.)"""
import numpy as np
import pytest

import oracle
from paper_2505_10857_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("grid", [(21, 23), (64, 32), (96, 40)])
@pytest.mark.parametrize("nb", [9, 21])
def test_entries_that_a_perturbation_cannot_reach_are_zero(grid, nb):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2505_10857_gb300 import nswe
    Nx, Ny = grid
    sides = (I.BC2_INFLOW, I.BC2_OUTFLOW, lambda x: I.BC2_OUTFLOW if x < 1.5 else I.BC2_REFLECT, I.BC2_DEPTH)
    st = np.array([[1.6, 2.2, 0.3], [0, 0, 0], [0, 0, 0], [1.4, 0.0, 0.0]])
    bumps = I.bottom2d_gaussians([(0.1, 1.2, 0.8, 0.6), (-0.05, 2.0, 1.5, 0.4)])
    inp = I.make_problem_2d(Nx, Ny, 1, 0.0, 3.0, 0.0, 2.0, 9.81, bumps, sides, st, lambda X, Y: (1.5, 2.0, 0.1)) \
        if Nx * Ny <= 512 else I.bump_channel_2d(1, Nx, Ny, 4)
    n = Nx * Ny
    rng = np.random.default_rng(n)
    U = np.stack([1.3 + 0.3 * rng.random(n), 1.0 + 0.3 * rng.random(n), 0.2 * rng.standard_normal(n)])
    Ud = torch.from_numpy(U).cuda()
    ctx = nswe.Context(0)
    prob = nswe.Problem2D.from_inputs(ctx, inp)
    R = torch.zeros_like(Ud)
    J = torch.full((nb, 9, n), float("nan"), dtype=torch.float64, device="cuda")
    f = nswe.nswe_jacobian_simplified if nb == 9 else nswe.nswe_jacobian_full
    f(ctx, prob, 0, Ud, 1e-6, 3.0, R, J)
    J = J.cpu().numpy()
    prob.close()
    for k, (ox, oy) in enumerate(oracle.stencil2d(1 if nb == 21 else 0)):
        for across, m, rows in ((ox, 2, (0, 1)), (oy, 1, (0, 2))):
            if abs(across) == 2:
                for l in rows:
                    assert (J[k, l * 3 + m] == 0).all(), (ox, oy, l, m, np.abs(J[k, l * 3 + m]).max())
