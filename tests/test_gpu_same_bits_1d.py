"""A 1D solve's bits do not depend on the launch it runs in: the solve kernel
is compiled for several register budgets (launch shapes), and its roundings are
written out, so that every shape, a batch of any size (the default shape
follows the batch's size) and the server's launches give the bits of the
problem solved alone, in both precisions."""
import time

import numpy as np
import pytest

from paper_2505_10857_gb300 import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

MANY = 305  # one more than two problems per SM


@pytest.fixture(scope="module")
def nswe():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2505_10857_gb300 import nswe as N
    N.lib()
    return N


def params(nswe, inp, precision, **kw):
    q = nswe.params_from(I.Params1D.for_problem(inp, tol=1e-10, n_max=500, **kw))
    q.precision = precision
    return q


def solve(nswe, ctx, inps, prms):
    probs = [nswe.Problem1D.from_inputs(ctx, p) for p in inps]
    U0s = [torch.from_numpy(p.U0_start).cuda() for p in inps]
    Us = [torch.zeros((2, p.N), dtype=torch.float64, device="cuda") for p in inps]
    infos = nswe.nswe_newton_solve_batch_each(ctx, probs, U0s, Us, prms)
    out = [u.cpu().numpy() for u in Us]
    for p in probs:
        p.close()
    return out, infos


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("nb", [3, 5])
def test_every_shape_gives_the_same_bits(nswe, precision, nb):
    inps = [I.channel_irregular(k, N=1024, levels=6, start_level=2) for k in range(3)] + [I.channel_small(1)]
    prms = [params(nswe, p, precision, nb=nb) for p in inps]
    ctx = nswe.Context(0)
    ref, infos = solve(nswe, ctx, inps, prms)  # the default
    assert all(i["status"] == 0 for i in infos)
    for shape in range(len(nswe.solve_shapes())):
        nswe.nswe_ctx_set_solve_shape(ctx, precision, shape)
        U, inf = solve(nswe, ctx, inps, prms)
        assert [i["iters"] for i in inf] == [i["iters"] for i in infos], shape
        assert all(np.array_equal(a, b) for a, b in zip(U, ref)), shape


@pytest.mark.parametrize("precision", [0, 1])
def test_a_large_batch_gives_the_bits_of_the_problem_alone(nswe, precision):
    inps = [I.channel_small(k % 3, N=128, levels=3) for k in range(MANY)]
    prms = [params(nswe, p, precision) for p in inps]
    ctx = nswe.Context(0)
    alone = [solve(nswe, ctx, [p], [q])[0][0] for p, q in zip(inps[:3], prms)]
    U, infos = solve(nswe, ctx, inps, prms)
    for k in range(MANY):
        assert infos[k]["status"] == 0 and np.array_equal(U[k], alone[k % 3]), k


@pytest.mark.parametrize("precision", [0, 1])
def test_a_large_server_launch_gives_the_bits_of_the_solve_alone(nswe, precision):
    inps = [I.channel_small(k % 3, N=128, levels=3) for k in range(MANY)]
    prms = [params(nswe, p, precision) for p in inps]
    ctx = nswe.Context(0)
    alone = [solve(nswe, ctx, [p], [q])[0][0] for p, q in zip(inps[:3], prms)]
    sv = nswe.Server(0, device_bytes=256 << 20, host_bytes=64 << 20, streams=1, max_batch=MANY, batch_window_s=10.0)
    try:
        tickets = [sv.submit(p, q) for p, q in zip(inps, prms)]
        out, t0 = {}, time.time()
        while len(out) < MANY:
            assert time.time() - t0 < 120.0
            sv.wait(1, 1.0)
            for t in sv.poll():
                out[t] = sv.take(t)
        assert sv.stats()["launches"] == 1
    finally:
        sv.close()
    for k, t in enumerate(tickets):
        assert out[t][1]["status"] == 0 and np.array_equal(out[t][0], alone[k % 3]), k


@pytest.mark.parametrize("precision", [0, 1])
def test_a_solve_that_stalls_on_its_coarse_levels_ends_alike_whatever_is_launched_with_it(nswe, precision):
    """Two nested levels of this request stall at the cap of 800 steps, where
    the last bits decide how the next level starts; its finer levels converge."""
    inp = I.serving_instance(733)
    prm = nswe.params_from(I.Params1D.for_problem(inp, tol=3e-13, n_max=800))
    prm.precision = precision
    small = [I.channel_small(0, N=128, levels=3)] * (MANY - 1)
    ctx = nswe.Context(0)
    (U,), (info,) = solve(nswe, ctx, [inp], [prm])
    Us, infos = solve(nswe, ctx, [inp] + small, [prm] + [params(nswe, small[0], precision)] * (MANY - 1))
    for i in (info, infos[0]):
        assert i["status"] == 0 and i["res"][0] < 3e-13 and i["iters"][3:5] == [800, 800], i
    assert infos[0]["iters"] == info["iters"] and np.array_equal(Us[0], U)
