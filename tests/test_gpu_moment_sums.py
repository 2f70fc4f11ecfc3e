"""The moment sums of the FP32 kinetic pass, alone: with tau = inf (lambda = 1) f is
transported unchanged, so after a step the moments are the sums of the stored values and
differ from FP64 sums of these, with v_k = k dv rounded to FP32 once (the velocities of the FP32
tier), only by the pass's own summation.

Rounding a sequential FP32 sum of n like terms is off by 0.23 sqrt(n) u rms (u = 2^-24; n
roundings of partial sums that grow to the total); such sums of N independent parts added in
FP64 by that over sqrt(N).  Here rows of 4 and runs of 8 of them, 8 or more runs: 0.25 u, and as
much again for the products with v and |v|^2.  Bound 0.5 u of sum |m f|, rms over the cells.
One FP32 sum over a split's 32 or more runs is off by 1 u and more, and k times the rounded dv
by 2 u of the energy (dv lies half an ulp from its float)."""
import numpy as np
import pytest

from paper_1212_0204_gb300 import workloads as W
from tests.helpers import conserved, grid, velocities

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1212_0204_gb300 import dvm  # noqa: E402


@pytest.mark.parametrize("scheme", [dvm.FKS, dvm.HOFKS], ids=["fks", "hofks"])
@pytest.mark.parametrize("nx,nv,bc", [
    ((400, 384), (127, 4), W.PERIODIC),      # 2D, a long x axis of velocities
    ((400, 384), (64, 4), W.OUTFLOW),
    ((38, 32, 128), (5, 4, 48), W.PERIODIC),  # 3D, many kz planes
    ((38, 32, 128), (4, 4, 48), W.PERIODIC),
])
def test_sums_of_transported_values(nx, nv, bc, scheme):
    d, rng = len(nx), np.random.default_rng(5)
    nc = int(np.prod(nx))
    dv = 1.0 + 0.97 * 2.0 ** -24
    T = (max(nv) / 8.0) ** 2  # velocities to four thermal widths along the longest axis
    u = np.full((d, nc), 0.3)
    case = W.Case("sums", d, tuple(nx), 1.0, tuple(nv), tuple(-(n // 2) for n in nv), dv, 1, (bc,) * d, np.inf,
                  1.0 + 0.3 * rng.uniform(-1, 1, nc), u, np.full(nc, T), 2, scheme)
    s = dvm.Solver.from_case(case, precision=dvm.F32)
    s.set_moments(conserved(case))
    s.step(case.steps)
    U, f = s.moments(), s.f()
    s.close()
    v = velocities(grid(case))[:d].astype(np.float32).astype(np.float64)
    m = np.concatenate([np.ones((1, v.shape[1])), v, 0.5 * (v ** 2).sum(0)[None]]) * dv ** d
    off = U - m @ f
    scale = np.abs(m) @ np.abs(f)
    rms = np.sqrt(((off / scale) ** 2).mean(axis=1))
    assert rms.max() <= 0.5 * 2.0 ** -24, rms * 2.0 ** 24
