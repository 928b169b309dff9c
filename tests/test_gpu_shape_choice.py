"""A launch shape that the caller sets is the one that runs, and the autotuner
times every shape itself: on a batch of at most two problems per SM the build
for four blocks per SM (64 registers a thread, with spills) takes about 1.4
times the one for two (128 registers), so the two cannot be one kernel."""
import pytest

from paper_2505_10857_gb300 import inputs as I

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def test_an_explicit_shape_runs_and_the_autotuner_times_it():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2505_10857_gb300 import nswe
    ctx = nswe.Context(0)
    inps = [I.channel_irregular(k, N=1024, levels=6, start_level=2) for k in range(152)]
    prm = nswe.params_from(I.Params1D.for_problem(inps[0], tol=1e-10, n_max=500))
    prm.precision = 1
    probs = [nswe.Problem1D.from_inputs(ctx, p) for p in inps]
    U0s = [torch.from_numpy(p.U0_start).cuda() for p in inps]
    Us = [torch.zeros((2, p.N), dtype=torch.float64, device="cuda") for p in inps]
    shapes = nswe.solve_shapes()
    four, two = shapes.index((256, 4)), shapes.index((256, 2))

    def ms():
        best = 1e9
        for _ in range(4):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            nswe.nswe_newton_solve_batch(ctx, probs, U0s, Us, prm, want_info=False)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b))
        return best

    try:
        default = ms()
        assert nswe.nswe_ctx_get_solve_shape(ctx, 1) == 0
        t = {}
        for shape in (four, two):
            nswe.nswe_ctx_set_solve_shape(ctx, 1, shape)
            assert nswe.nswe_ctx_get_solve_shape(ctx, 1) == shape
            t[shape] = ms()
        assert t[four] > 1.15 * t[two] and t[four] > 1.15 * default
        tuned, best = nswe.nswe_autotune_solve_batch(ctx, probs, U0s, Us, prm, reps=3)
        assert tuned[four] > 1.15 * tuned[two] and best != four
        assert nswe.nswe_ctx_get_solve_shape(ctx, 1) == best
    finally:
        for p in probs:
            p.close()
