"""A device that holds smaller clusters than 16 CTAs (fewer free SMs in a GPC):
the calls that run on a cluster take the largest it does hold. Levels see the
same arithmetic whatever the cluster, so V-cycles, residuals and solves give the
bits they give on 16 CTAs (res, a sum in another order, to rounding)."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

import oracle
from paper_2505_10857_gb300 import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

HERE = os.path.dirname(os.path.abspath(__file__))
CTAS = (16, 8, 4, 2, 1)


@pytest.fixture(scope="module")
def nswe():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2505_10857_gb300 import nswe as N
    oracle.build()
    return N


@pytest.fixture(scope="module")
def internals(tmp_path_factory, nswe):
    from paper_2505_10857_gb300 import build
    so = str(tmp_path_factory.mktemp("internals") / "libinternals.so")
    subprocess.run([build.nvcc()] + build.ARCH + build.FLAGS + ["-shared", os.path.join(HERE, "internals.cu"), "-o", so],
                   check=True)
    lib = ctypes.CDLL(so)
    lib.get_max_cluster.argtypes = [ctypes.c_void_p]
    lib.set_max_cluster.argtypes = [ctypes.c_void_p, ctypes.c_int]
    return lib


def dev(a, dtype=torch.float64):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda().to(dtype)


def test_the_device_is_asked(nswe, internals):
    assert internals.get_max_cluster(nswe.Context(0).h) in CTAS


@pytest.mark.parametrize("N,levels,nb,nu", [(128, 6, 3, 2), (1280, 5, 3, 2), (6016, 7, 3, 2), (616, 4, 5, 2),
                                            (616, 4, 3, 3)])
def test_1d_calls(nswe, internals, N, levels, nb, nu):
    inp = I.channel_small(7, N=N, levels=levels)
    ctx = nswe.Context(0)
    prob = nswe.Problem1D.from_inputs(ctx, inp)
    rng, x = np.random.default_rng(N), inp.centres()
    U = np.stack([inp.sig_fn(x) * 2.0 * (1 + 0.05 * np.sin(3 * x)), 4.42 + 0.05 * np.cos(x)])
    J, R, _ = oracle.jacobian1d(oracle.problem_levels(inp)[0], U, I.eps_for_n(N), 3.0, nb)
    dU0 = 1e-3 * rng.standard_normal((2, N))
    prm = nswe.params(N, levels, omega=0.7, nu1=nu, nu2=nu)
    got = []
    for ctas in CTAS:
        internals.set_max_cluster(ctx.h, ctas)
        out = []
        for dt, f in ((torch.float64, nswe.nswe_mg_vcycle), (torch.float32, nswe.nswe_mg_vcycle_f32)):
            d = dev(dU0, dt)
            f(ctx, prob, 0, nb, dev(J, dt), dev(R, dt), d, prm)
            out.append(d.cpu().numpy())
        Rg, res = torch.zeros((2, N), dtype=torch.float64, device="cuda"), torch.zeros((), dtype=torch.float64, device="cuda")
        nswe.nswe_residual(ctx, prob, 0, dev(U), Rg, res)
        got.append(out + [Rg.cpu().numpy(), float(res)])
    prob.close()
    for g in got:
        assert np.isfinite(g[0]).all() and g[0].any()
        assert all(np.array_equal(a, b) for a, b in zip(g[:3], got[0][:3]))
        assert abs(g[3] - got[0][3]) <= 1e-13 * got[0][3]


@pytest.mark.parametrize("precision", [0, 1])
def test_2d_calls(nswe, internals, precision):
    inps = [I.bump_channel_2d(2, 64, 32, 4), I.bump_channel_2d(1, 32, 16, 3)]
    ctx = nswe.Context(0)
    probs = [nswe.Problem2D.from_inputs(ctx, p) for p in inps]
    prms = [nswe.params2d_from(I.Params2D(levels=p.levels, nu1=[20], nu2=[20], tol=1e-10, n_max=400)) for p in inps]
    for q in prms:
        q.precision = precision
    U0s = [dev(p.U0_start) for p in inps]
    got = []
    for ctas in CTAS:
        internals.set_max_cluster(ctx.h, ctas)
        one = torch.zeros((3, 64 * 32), dtype=torch.float64, device="cuda")
        info = nswe.nswe_newton_solve(ctx, probs[0], U0s[0], one, prms[0])
        Us = [torch.zeros((3, p.Nx * p.Ny), dtype=torch.float64, device="cuda") for p in inps]
        infos = nswe.nswe_newton_solve_batch_each(ctx, probs, U0s, Us, prms)
        got.append(([one.cpu().numpy()] + [u.cpu().numpy() for u in Us], [info["status"]] + [i["status"] for i in infos]))
    for p in probs:
        p.close()
    for U, status in got:
        assert status == [0, 0, 0]
        assert np.array_equal(U[0], U[1])
        assert all(np.array_equal(a, b) for a, b in zip(U, got[0][0]))
