"""The FP64 reciprocal, quotient, square root and limited slope of the Euler sub-steps against
IEEE division and square root (numpy's), over every exponent and at the ends of the range.

Each is an approximation of 2^-20 taken to 2^-60 or below by a step whose last operation rounds
once, so it is within an ulp of the exact value and within an ulp of the rounded one.  The
slope a (b / (a + b)) adds the roundings of the sum and the product: 3 ulp.  Outside
2^-1021 .. 2^1021 the reciprocal and the root are the compiler's; the slope is zero for sums
beyond it.  The sub-step scalars (cfl, k) are plain IEEE."""
import numpy as np
import pytest

from paper_1212_0204_gb300 import dvm
from paper_1212_0204_gb300 import workloads as W
from tests.helpers import conserved

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)


def device(which, a, b=None):
    a = torch.from_numpy(np.ascontiguousarray(a)).cuda()
    b = a if b is None else torch.from_numpy(np.ascontiguousarray(b)).cuda()
    return dvm.selftest_fp64(which, a, b).cpu().numpy()


def mantissas(rng, n):
    """uniform ones, and ones a few ulp from 1 and 2"""
    m = 1.0 + rng.random(n)
    m[::7] = 1.0 + rng.integers(0, 8, m[::7].size) * 2.0 ** -52
    m[3::7] = 2.0 - rng.integers(1, 9, m[3::7].size) * 2.0 ** -52
    return m


def ulps(got, want):
    return np.abs(got - want) / np.spacing(np.abs(want))


def test_reciprocal_and_root_over_all_exponents():
    rng = np.random.default_rng(3)
    e = np.repeat(np.arange(-1074, 1024), 64)
    x = np.ldexp(mantissas(rng, e.size), e)
    with np.errstate(over="ignore"):
        want = 1.0 / x
    s = np.where(rng.random(x.size) < 0.5, -1.0, 1.0)
    got = device(dvm.SELFTEST_RCP, s * x)
    fin = np.isfinite(want)
    assert np.array_equal(got[~fin], (s * want)[~fin])
    assert ulps(got[fin], (s * want)[fin]).max() <= 1.0
    assert ulps(device(dvm.SELFTEST_SQRT, x), np.sqrt(x)).max() <= 1.0
    ends = np.array([0.0, -0.0, np.inf, -np.inf])
    assert np.array_equal(device(dvm.SELFTEST_RCP, ends), np.array([np.inf, -np.inf, 0.0, -0.0]))
    assert np.isnan(device(dvm.SELFTEST_RCP, np.array([np.nan]))[0])
    assert np.array_equal(device(dvm.SELFTEST_SQRT, np.array([0.0, np.inf])), np.array([0.0, np.inf]))


def test_quotient():
    rng = np.random.default_rng(4)
    n = 1 << 20
    d = np.ldexp(mantissas(rng, n), rng.integers(-1020, 1020, n))
    # quotients whose residual (2^-53 of the numerator) is normal too
    q = np.ldexp(mantissas(rng, n), np.clip(rng.integers(-1000, 1000, n), -950 - np.frexp(d)[1], 1000 - np.frexp(d)[1]))
    q = np.clip(q, 2.0 ** -960, 2.0 ** 1000)
    num = q * d * np.where(rng.random(n) < 0.5, -1.0, 1.0)
    ok = np.isfinite(num) & (np.abs(num) > 2.0 ** -960)
    num, d = num[ok], d[ok]
    assert num.size > n // 2
    assert ulps(device(dvm.SELFTEST_QUOT, num, d), num / d).max() <= 1.0


def test_half_slope():
    rng = np.random.default_rng(5)
    n = 1 << 20
    e = rng.integers(-960, 1018, n)
    a = np.ldexp(mantissas(rng, n), e)
    b = np.ldexp(mantissas(rng, n), np.clip(e + rng.integers(-40, 41, n), -960, 1018))
    s = np.where(rng.random(n) < 0.5, -1.0, 1.0)
    want = s * (a * (b / (a + b)))
    assert ulps(device(dvm.SELFTEST_HALF_SLOPE, s * a, s * b), want).max() <= 3.0
    assert not device(dvm.SELFTEST_HALF_SLOPE, a, -b).any()
    z = np.array([0.0, -0.0, 1.0, 0.0, 1e-320, np.nan, 1.0])
    w = np.array([0.0, 0.0, 0.0, -1.0, 1e-320, 1.0, np.nan])
    assert not device(dvm.SELFTEST_HALF_SLOPE, z, w).any()


@pytest.mark.parametrize("d", [1, 2])
def test_sub_step_count_where_the_step_is_a_whole_number_of_them(d):
    """alpha dt / (dx / 2) = 4 exactly (rest, sqrt(gamma theta) a power of two): the quotient
    decides between 4 and 5 sub-steps."""
    n, nv, cs = 64, 12, 2.0
    dx = 1.0 / n
    dv = dx / (4 * 0.5 * dx / (d * cs))  # dt = dx / dv = 4 dx / (2 alpha), alpha = d cs
    theta = cs * cs / (1.0 + 2.0 / d)
    c = W.Case("rest", d, (n,) * d, dx, (nv,) * d, (-(nv // 2),) * d, dv, 1, (W.PERIODIC,) * d, 1e-3, np.ones(n ** d),
               np.zeros((d, n ** d)), np.full(n ** d, theta), 2, dvm.HOFKS)
    import oracle
    from tests.helpers import grid
    orc = oracle.Scheme(grid(c), tau=c.tau)
    orc.set_moments(conserved(c))
    s = dvm.Solver.from_case(c, precision=dvm.F64)
    s.set_moments(conserved(c))
    for _ in range(2):
        s.step(1)
        orc.step(1)
        assert s.info()["m"] == orc.info()["m"]


@pytest.mark.parametrize("d", [1, 2])
def test_densities_far_from_one(d):
    """A run scales with the density: at 2^-400 and 2^400 times it the velocities, and so the
    limited slopes, are those at 1 (the product of two differences leaves the normal range)."""
    n, nv = 40, 12
    x = (np.arange(n ** d) % n + 0.5) / n
    base = 1.0 + 0.3 * np.sin(2 * np.pi * x)

    def run(scale):
        c = W.Case("scale", d, (n,) * d, 1.0 / n, (nv,) * d, (-(nv // 2),) * d, 0.9, 1, (W.PERIODIC,) * d, 1e-2, scale * base,
                   np.full((d, n ** d), 0.2), 1.0 + 0.1 * np.cos(2 * np.pi * x), 3, dvm.HOFKS)
        s = dvm.Solver.from_case(c, precision=dvm.F64)
        s.set_moments(conserved(c))
        s.step(c.steps)
        return s.moments()

    U = run(1.0)
    for e in (-600, -400, 400, 600):
        assert np.abs(np.ldexp(run(2.0 ** e), -e) - U).max() <= 1e-13 * np.abs(U).max()
