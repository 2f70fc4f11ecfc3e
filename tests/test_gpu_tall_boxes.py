"""3D HOFKS in boxes so long in z (or y) that the linear-term passes of the single-quadratic
form reach their launch limits (65535 / 17 z planes): the last length within them and the
first beyond, in FP32 and BF16, against the oracle.  Bounds as in test_gpu_shared_pass.py."""
import numpy as np
import pytest

import oracle
from paper_1212_0204_gb300 import workloads as W
from tests.helpers import conserved, grid

from paper_1212_0204_gb300 import dvm

VELOCITIES = (8, 8, 6)


def case_of(nx, steps=2):
    dx, dv = 1.0 / max(nx), 0.75  # (velocities to 3 thermal widths: mu'' is 1e-2 of the moments)
    ax = [(np.arange(n) + 0.5) / n for n in nx]
    Z, Y, X = np.meshgrid(*ax[::-1], indexing="ij")
    wave = (np.sin(2 * np.pi * (X + 0.1)) * np.sin(2 * np.pi * Y) * np.sin(2 * np.pi * (Z + 0.2))).ravel()
    u = np.zeros((3, wave.size))
    u[0], u[2] = 0.3, -0.2
    return W.Case("tall", 3, tuple(nx), dx, VELOCITIES, tuple(-(n // 2) for n in VELOCITIES), dv, 1, (W.PERIODIC,) * 3,
                  dx / dv / np.log(2.0), 1.0 + 0.2 * wave, u, 1.0 + 0.1 * wave, steps, dvm.HOFKS)


@pytest.mark.parametrize("precision", [dvm.F32, dvm.BF16S], ids=["f32", "bf16"])
def test_plan_of_tall_boxes(precision):
    """(host only) beyond the limit of the linear-term passes no windowed pass is chosen"""
    from paper_1212_0204_gb300 import build
    build.build()
    for nx, kind in [((4, 8, 1000), "window"), ((4, 8, 3004), "window"), ((4, 8, 3855), "window"), ((4, 8, 3856), "generic"),
                     ((4, 65535, 2), "window"), ((4, 65536, 2), "window")]:
        cfg, keep = dvm.make_config(3, nx, 1.0, VELOCITIES, (-4, -4, -3), 1.0, tau=1.0, scheme=dvm.HOFKS, precision=precision)
        assert dvm.plan(cfg)[0] == kind, nx


@pytest.mark.gpu
@pytest.mark.parametrize("nx", [(4, 8, 1640), (4, 8, 3004), (4, 8, 3856), (2, 65536, 1)])
def test_tall_boxes_match_oracle(nx):
    case = case_of(nx)
    orc = oracle.Scheme(grid(case), tau=case.tau)
    orc.set_moments(conserved(case))
    orc.step(case.steps)
    Uo, fo = orc.moments(), orc.f()
    scale = np.maximum(np.abs(Uo).max(axis=1), np.abs(Uo[0]).max())
    for precision, tol in ((dvm.F32, 1e-5), (dvm.BF16S, 8 * 2.0 ** -9)):
        s = dvm.Solver.from_case(case, precision=precision)
        s.set_moments(conserved(case))
        s.step(case.steps)
        assert (np.abs(s.moments() - Uo).max(axis=1) / scale).max() <= tol
        assert np.abs(s.f() - fo).max() <= tol * np.abs(fo).max()
        s.close()
