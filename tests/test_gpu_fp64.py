"""The FP64 reciprocal, square root, reciprocal square root and division of
csrc/nswe_fp64.cuh against CUDA's own and, for the reciprocal square root,
against extended precision. Derived bounds: before its last rounding the
reciprocal and the square root are within 2^-57, the division (whose residual an
FMA forms exactly) far within, so each is within one ulp of the correctly
rounded value and seldom beside it; the reciprocal square root is within 1.3
2^-54 (its cut-off term and the rounding of x y), 1.15 ulp with the last
rounding where the mantissa is near two. Zeros, subnormal numbers, infinities, NaN and
negative arguments give exactly what the ordinary operation gives."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

HERE = os.path.dirname(os.path.abspath(__file__))
RCP, SQRT, RSQRT, DIV = range(4)
TINY, SUB, BIG = 2.0 ** -1022, 2.0 ** -1074, np.finfo(np.float64).max
EDGES = np.array([0.0, SUB, 3 * SUB, 2.0 ** -1040, 2.0 ** -1024, 2.0 ** -1023, np.nextafter(TINY, 0), TINY, 2 * TINY,
                  2.0 ** -1020, 2.0 ** -896, 2.0 ** -895, 2.0 ** -894, 2.0 ** -960, 1.0, 2.0, 3.0, 2.0 ** 896,
                  2.0 ** 897, 2.0 ** 898, 2.0 ** 1018, 2.0 ** 1019, 2.0 ** 1020, 2.0 ** 1022, 2.0 ** 1023, BIG,
                  np.inf, np.nan])


@pytest.fixture(scope="module")
def call(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2505_10857_gb300 import build
    so = str(tmp_path_factory.mktemp("fp64") / "libfp64.so")
    subprocess.run([build.nvcc()] + build.ARCH + build.FLAGS + ["-shared", os.path.join(HERE, "fp64_functions.cu"), "-o", so],
                   check=True)
    f = ctypes.CDLL(so).fp64_apply
    f.argtypes = [ctypes.c_int, ctypes.c_long] + [ctypes.c_void_p] * 3

    def run(op, a, b=None):
        a = torch.from_numpy(np.ascontiguousarray(a)).cuda()
        b = a if b is None else torch.from_numpy(np.ascontiguousarray(b)).cuda()
        out = torch.empty_like(a)
        assert f(op, a.numel(), a.data_ptr(), b.data_ptr(), out.data_ptr()) == 0
        return out.cpu().numpy()

    return run


def ulps(a, b):
    """Distance in units of the last place (finite values of one sign)."""
    return np.abs(a.view(np.int64) - b.view(np.int64))


def random(n, seed, lo, hi):
    rng = np.random.default_rng(seed)
    return np.ldexp(rng.uniform(1.0, 2.0, n), rng.integers(lo, hi, n))


@pytest.mark.parametrize("lo,hi", [(-8, 8), (-1022, 1023)])
@pytest.mark.parametrize("op", [RCP, SQRT, DIV])
def test_within_one_ulp_of_the_rounded_operation(call, op, lo, hi):
    n = 1 << 21
    sign = 1.0 if op == SQRT else np.where(np.random.default_rng(1).random(n) < 0.5, -1.0, 1.0)
    a, b = sign * random(n, 2 + op, lo, hi), random(n, 7, lo, hi)
    got, ref = call(op, a, b), call(op + 4, a, b)
    fin = np.isfinite(ref) & (np.abs(ref) >= TINY)
    assert np.array_equal(got[~fin], ref[~fin])
    d = ulps(got[fin], ref[fin])
    print(f"operation {op}, exponents {lo}..{hi}: {(d > 0).mean():.2e} of the results one ulp off")
    assert d.max() <= 1 and (d > 0).mean() <= 0.01, (d.max(), (d > 0).mean())


@pytest.mark.parametrize("lo,hi", [(-8, 8), (-1022, 1023)])
def test_reciprocal_square_root(call, lo, hi):
    a = random(1 << 19, 11, lo, hi)
    got = call(RSQRT, a)
    exact = 1 / np.sqrt(a.astype(np.longdouble))
    err = np.abs((got.astype(np.longdouble) - exact) / np.spacing(exact.astype(np.float64)))
    print(f"reciprocal square root, exponents {lo}..{hi}: {float(err.max()):.3f} ulp at most")
    assert err.max() <= 1.2, err.max()


@pytest.mark.parametrize("op", [RCP, SQRT, RSQRT])
def test_edges_of_the_range(call, op):
    a = np.concatenate([EDGES, -EDGES])
    got, ref = call(op, a), call(op + 4, a)
    same = (got.view(np.int64) == ref.view(np.int64)) | (np.isnan(got) & np.isnan(ref))
    ordinary = ~np.isfinite(ref) | (np.abs(ref) < TINY) | (np.abs(a) < TINY) | (a < 0) & (op != RCP)
    assert same[ordinary].all(), a[ordinary & ~same]
    assert (ulps(got[~ordinary], ref[~ordinary]) <= (2 if op == RSQRT else 1)).all()


def test_quotients_at_the_edges_of_the_range(call):
    e = np.concatenate([EDGES, -EDGES])
    a, b = (x.ravel() for x in np.meshgrid(e, e))
    got, ref = call(DIV, a, b), call(DIV + 4, a, b)
    same = (got.view(np.int64) == ref.view(np.int64)) | (np.isnan(got) & np.isnan(ref))
    ordinary = ~np.isfinite(ref) | (np.abs(ref) < TINY)
    assert same[ordinary].all(), list(zip(a[ordinary & ~same], b[ordinary & ~same]))[:8]
    assert (ulps(got[~ordinary], ref[~ordinary]) <= 1).all()
