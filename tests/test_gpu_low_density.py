"""The FP32 shared-row pass at densities of 2^-112, against the FP64 oracle: the values of f
beyond 14 powers of two below their peak are subnormal and count for 1e-3 of the moments.
A subnormal value is rounded to 2^-150, which is 2^-38 of the peak, so the tier's bound of
1e-5 of the moment scale stands.  (The limited Euler slopes multiply two differences and are
zero at such densities in FP32; the forms run FKS and unlimited HOFKS.)"""
import numpy as np
import pytest

import oracle
from paper_1212_0204_gb300 import workloads as W
from tests.helpers import conserved, grid
from tests.test_gpu_shared_pass import FORMS, case_of, moment_err

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1212_0204_gb300 import dvm  # noqa: E402


@pytest.mark.parametrize("scheme", [dvm.FKS, dvm.HOFKS_UNLIMITED], ids=["fks", "unlimited"])
@pytest.mark.parametrize("form", [FORMS[i] for i in (0, 3, 4, 6, 8)],
                         ids=["periodic", "outflow", "mixed_p3", "3d", "3d_outflow_p2"])
def test_moments_of_a_thin_gas(form, scheme):
    case = case_of(*form[:5], scheme, form[5])
    U0 = np.ldexp(conserved(case), -112)
    s = dvm.Solver.from_case(case, precision=dvm.F32)
    assert s.kinetic_route()[0] == "shared"
    s.set_moments(U0)
    s.step(case.steps)
    orc = oracle.Scheme(grid(case), tau=case.tau)
    orc.set_moments(U0)
    orc.step(case.steps)
    assert moment_err(s.moments(), orc.moments()) <= 1e-5
