"""f^0 = E[U^0] of the FP32 tier right after the moments are set, against the FP64 oracle.

The parameters of E[U^0] are FP64 (as the oracle's), so f^0 differs from the exact one by
the rounding of a value (at most 2^-24 = 6e-8, 3.4e-8 rms) and by that of the exponent
L - h |v - u|^2, L = log2 of the Maxwellian's prefactor: half an ulp of |L| < 4 (1D) is 1.2e-7,
7e-8 rms, times ln 2; of |L| < 8 (2D, 3D) twice that.  Cells differ, so in the norm over a state the parts add
to 6e-8 in 1D and 1.05e-7 in 2D and 3D: bounds 1e-7 and 2e-7.  The moments of a cell add
N_v^(1/d) correlated roundings of the exponent (1.6e-7 in 1D at most): 2.5e-7 of the moment
scale.  The total mass averages them over hundreds of cells: 1e-7.
"""
import numpy as np
import pytest

import oracle
from paper_1212_0204_gb300 import workloads as W
from tests.helpers import conserved, grid, velocities

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1212_0204_gb300 import dvm  # noqa: E402


def noisy_case(nx, nv, half, tl, tr, seed):
    """Two states (density 1 and 1/8, temperatures tl and tr) along x, densities of every cell
    1 % apart, velocities from -half to half."""
    d, rng = len(nx), np.random.default_rng(seed)
    nc = int(np.prod(nx))
    x = (np.arange(nc) % nx[0] + 0.5) / nx[0]
    rho = np.where(x < 0.5, 1.0, 0.125) * (1.0 + 0.01 * rng.uniform(-1, 1, nc))
    u = 0.2 * rng.uniform(-1, 1, (d, nc))
    return W.Case("initial", d, tuple(nx), 1.0 / nx[0], (nv,) * d, (-(nv // 2),) * d, 2.0 * half / nv, 1,
                  (W.OUTFLOW,) * d, 1e-3, rho, u, np.where(x < 0.5, tl, tr), 1, dvm.HOFKS)


CASES = [
    ((300,), 24, 6.4, 1.0, 0.8),
    ((300,), 64, 6.4, 1.0, 0.8),
    ((300,), 100, 6.4, 1.0, 0.8),
    ((517,), 128, 6.0, 0.9, 0.35),
    ((40, 30), 20, 6.4, 1.0, 0.8),
    ((33, 29), 33, 6.0, 1.0, 0.9),
    ((12, 10, 9), 13, 6.0, 1.0, 1.1),
]


def check(case, U0, f):
    orc = oracle.Scheme(grid(case), tau=case.tau)
    orc.set_moments(U0)
    fo = orc.f().reshape(f.shape)
    assert np.linalg.norm(f - fo) <= (1e-7 if case.d == 1 else 2e-7) * np.linalg.norm(fo)
    v = velocities(grid(case))[:case.d]
    m = np.concatenate([np.ones((1, v.shape[1])), v, 0.5 * (v ** 2).sum(0)[None]]) * case.dv ** case.d
    U = m @ f.reshape(v.shape[1], -1)
    scale = np.maximum(np.abs(U0).max(axis=1), np.abs(U0[0]).max())
    assert (np.abs(U - U0).max(axis=1) / scale).max() <= 2.5e-7
    assert abs(U[0].sum() - U0[0].sum()) <= 1e-7 * U0[0].sum()


@pytest.mark.parametrize("scheme", [dvm.HOFKS, dvm.FKS], ids=["hofks", "fks"])
@pytest.mark.parametrize("form", CASES)
def test_initial_f_of_the_fp32_tier(form, scheme):
    case = noisy_case(*form, seed=7)
    case.scheme = scheme
    U0 = conserved(case)
    s = dvm.Solver.from_case(case, precision=dvm.F32)
    s.set_moments(U0)
    check(case, U0, s.f())


def test_initial_f_of_an_fp32_batch():
    cases = [noisy_case(*form, seed=i) for i, form in enumerate(CASES) if len(form[0]) == 1]
    U0 = [conserved(c) for c in cases]
    b = dvm.Batch(cases, precision=dvm.F32)
    b.set_moments(b.pack(U0))
    for i, c in enumerate(cases):
        check(c, U0[i], np.asarray(b.f(i)))


@pytest.mark.parametrize("form", [CASES[0], CASES[4], CASES[6]])
def test_initial_f_below_the_normal_range(form):
    """Densities of 2^-122: most values are subnormal.  The exponent, -120 to -135, is rounded to
    half of 2^-17 or 2^-16: 2.6e-6 or 5.3e-6 of a value at most, and values to 2^-150."""
    case = noisy_case(*form, seed=7)
    U0 = np.ldexp(conserved(case), -122)
    orc = oracle.Scheme(grid(case), tau=case.tau)
    orc.set_moments(U0)
    s = dvm.Solver.from_case(case, precision=dvm.F32)
    s.set_moments(U0)
    f = s.f()
    fo = orc.f().reshape(f.shape)
    assert np.linalg.norm(f - fo) <= 5.3e-6 * np.linalg.norm(fo) + 2.0 ** -150 * np.sqrt(f.size)
