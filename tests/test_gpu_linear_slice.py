"""3D HOFKS on the shared rows, on both sides of the 2^24 points from which it takes the
single-quadratic form with the linear term's moments from three passes of their own: against
the FP64 oracle, at density 1 and at 2^-112 (see test_gpu_low_density.py).  Bounds: FP32 1e-5
of the moment scale and of max |f| (f is rounded once per step, 6e-8 relative); BF16 storage
a few rounding units of 2^-9."""
import numpy as np
import pytest

import oracle
from paper_1212_0204_gb300 import workloads as W
from tests.helpers import conserved, grid
from tests.test_gpu_shared_pass import case_of, moment_err

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1212_0204_gb300 import dvm  # noqa: E402

P = W.PERIODIC


@pytest.mark.parametrize("nv,launches,precision,power,tol", [
    ((10, 10, 9), 4, dvm.F32, 0, 1e-5),
    ((10, 10, 9), 4, dvm.BF16S, 0, 8 * 2.0 ** -9),
    ((11, 10, 10), 7, dvm.F32, 0, 1e-5),
    ((11, 10, 10), 7, dvm.F32, -112, 1e-5),
    ((11, 10, 10), 7, dvm.BF16S, 0, 8 * 2.0 ** -9),
], ids=["15M_f32", "15M_bf16", "19M_f32", "19M_f32_thin", "19M_bf16"])
def test_both_forms_match_the_oracle(nv, launches, precision, power, tol):
    case = case_of((33, 32, 16), nv, 1.0, (P, P, P), 1, dvm.HOFKS_UNLIMITED if power else dvm.HOFKS, True)
    U0 = np.ldexp(conserved(case), power)
    s = dvm.Solver.from_case(case, precision=precision)
    assert s.kinetic_route()[0] == "shared"
    s.set_moments(U0)
    s.step(2)
    assert s.launches_per_step() == launches
    orc = oracle.Scheme(grid(case), tau=case.tau)
    orc.set_moments(U0)
    orc.step(2)
    assert moment_err(s.moments(), orc.moments()) <= tol
    f, fo = s.f(), orc.f()
    assert np.abs(f - fo).max() <= tol * np.abs(fo).max()
