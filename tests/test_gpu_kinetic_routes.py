"""Paths of the kinetic pass that the other tests do not take, each with the kernel it runs
asserted, against the FP64 oracle: the shared source rows in FP64 over their forms (3D,
outflow, p > 1) and beside the limit of shared memory, shift denominators beyond the velocity counts, and the learned path switched
on and off where it changes the kernel.  Bounds as in test_gpu_shared_pass.py: 1e-12 in
FP64, 1e-5 in FP32."""
import numpy as np
import pytest

import oracle
from paper_1212_0204_gb300 import workloads as W
from tests.helpers import conserved, grid
from tests.test_gpu_shared_pass import FORMS, case_of, moment_err
from tests.test_oracle_learned import blocky_flags

from paper_1212_0204_gb300 import dvm

pytestmark = pytest.mark.gpu

P, O = W.PERIODIC, W.OUTFLOW


def compare(case, precision, tol, route):
    orc = oracle.Scheme(grid(case), tau=case.tau)
    orc.set_moments(conserved(case))
    orc.step(case.steps)
    s = dvm.Solver.from_case(case, precision=precision)
    assert s.kinetic_route()[0] == route
    s.set_moments(conserved(case))
    s.step(case.steps)
    assert moment_err(s.moments(), orc.moments()) <= tol
    fo = orc.f()
    assert np.abs(s.f() - fo).max() <= tol * np.abs(fo).max()
    s.close()


@pytest.mark.parametrize("scheme", [dvm.HOFKS, dvm.FKS], ids=["hofks", "fks"])
@pytest.mark.parametrize("form", FORMS)
def test_fp64_shared_rows_match_oracle(form, scheme):
    nx, nv, dv, bc, p, field = form
    compare(case_of(nx, nv, dv, bc, p, scheme, field), dvm.F64, 1e-12, "shared")


@pytest.mark.parametrize("precision,tol", [(dvm.F64, 1e-12), (dvm.F32, 1e-5)], ids=["f64", "f32"])
@pytest.mark.parametrize("p", [257, 200_000_000])
def test_shift_denominators_beyond_the_velocity_count(p, precision, tol):
    compare(case_of((24, 20), (9, 10), 0.95, (P, O), p, dvm.HOFKS, False), precision, tol, "shared")


EDGES = [
    # nx, ky, tier, folded rows (0: the per-cell pass)
    ((40, 32), 108, dvm.F64, 36),
    ((40, 32), 109, dvm.F64, 32),
    ((40, 16), 185, dvm.F64, 32),
    ((1, 512), 32, dvm.F64, 24),
    ((1, 512), 33, dvm.F64, 0),
    ((1, 512), 128, dvm.F32, 24),
    ((1, 512), 129, dvm.F32, 0),
]


@pytest.mark.parametrize("nx,nky,precision,rows", EDGES)
def test_rows_beside_the_limit_of_shared_memory(nx, nky, precision, rows):
    case = case_of(nx, (39, nky), 0.24, (P, P), 1, dvm.HOFKS, False)
    s = dvm.Solver.from_case(case, precision=precision)
    assert s.kinetic_route()[1] == rows
    s.close()
    compare(case, precision, 1e-12 if precision == dvm.F64 else 1e-5, "shared" if rows else "cell")


LEARNED = [
    # nx, nv, bc, p, tier, kernel without and with the learned path
    ((40, 32, 16), (8, 8, 6), (P, P, P), 1, dvm.F32, "shared", "window"),
    ((40, 36), (12, 13), (O, P), 2, dvm.F32, "shared", "shared"),
    ((40, 36), (12, 13), (O, O), 2, dvm.F64, "shared", "shared"),
]


@pytest.mark.parametrize("nx,nv,bc,p,precision,off,on", LEARNED)
def test_learned_path_switched_on_and_off(nx, nv, bc, p, precision, off, on):
    case = case_of(nx, nv, 0.9, bc, p, dvm.HOFKS, True)
    rng, tol = np.random.default_rng(17), 1e-12 if precision == dvm.F64 else 1e-5
    U0 = conserved(case)
    orc = oracle.Scheme(grid(case), tau=case.tau)
    orc.set_moments(U0)
    s = dvm.Solver.from_case(case, precision=precision)
    s.set_moments(U0)

    def same():
        assert moment_err(s.moments(), orc.moments()) <= tol
        fo = orc.f()
        assert np.abs(s.f() - fo).max() <= tol * np.abs(fo).max()

    for plain, flagged in ((1, 2), (2, 1), (1, 0)):
        assert s.kinetic_route()[0] == off
        s.step(plain)
        orc.step(plain)
        same()
        if not flagged:
            break
        s.learn_enable(dvm.LEARN_GIVEN)
        assert s.kinetic_route()[0] == on
        for _ in range(flagged):
            fl = blocky_flags(rng, case.nx, 0.6, 4)
            s.learn_set_flags(fl)
            s.step(1)
            orc.step_flagged(fl)
        assert moment_err(s.moments(), orc.moments()) <= tol
        s.learn_disable()
    s.close()
