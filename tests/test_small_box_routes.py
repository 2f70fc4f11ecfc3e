"""Which kernel of the kinetic pass small boxes take, on both sides of each line of the rule
(host only): planes that leave most threads of the shared rows' CTAs without a cell run one
thread per cell."""
import pytest

from paper_1212_0204_gb300 import dvm

P, O = dvm.PERIODIC, dvm.OUTFLOW
F64, F32, BF16 = dvm.F64, dvm.F32, dvm.BF16S


@pytest.mark.parametrize("nx,nv,bc,p,scheme,precision,want", [
    # 2D: first-order outflow below 1000 cells
    ((31, 32), 21, (O, O), 1, dvm.FKS, F32, "cell"),
    ((32, 32), 21, (O, O), 1, dvm.FKS, F32, "shared"),
    ((25, 25), 21, (P, O), 3, dvm.FKS, BF16, "cell"),
    ((25, 25), 21, (O, O), 1, dvm.HOFKS, F32, "shared"),
    ((25, 25), 21, (O, O), 1, dvm.FKS, F64, "shared"),
    ((25, 25), 21, (P, P), 1, dvm.FKS, F32, "shared"),
    # 2D where the windows can run too: by the useful rows
    ((2048, 17), 24, (P, P), 1, dvm.FKS, F32, "window"),
    ((2048, 28), 24, (P, P), 1, dvm.FKS, F32, "shared"),
    ((200, 200), 24, (P, P), 1, dvm.FKS, F32, "shared"),
    # 3D: below 0.35 of the threads (12 x 12 of 32 x 16: 0.28; 18 x 10: 0.352)
    ((12, 12, 12), 13, (P, P, P), 1, dvm.FKS, F32, "cell"),
    ((12, 12, 12), 9, (O, P, O), 2, dvm.HOFKS, BF16, "cell"),
    ((12, 12, 12), 9, (P, P, P), 1, dvm.HOFKS, F64, "cell"),
    ((12, 12, 12), 12, (P, P, P), 1, dvm.FKS, F32, "window"),
    ((18, 10, 7), 10, (O, P, O), 2, dvm.HOFKS, F32, "shared"),
    ((14, 14, 14), 13, (P, P, P), 1, dvm.FKS, F32, "shared"),
    # outflow, 4096 cells or more than 100 velocity pairs: below 0.56 (24 x 24 of 64 x 16: 0.5625)
    ((14, 14, 14), 11, (O, P, P), 1, dvm.HOFKS, F32, "cell"),
    ((14, 14, 14), 10, (O, P, P), 1, dvm.HOFKS, F32, "shared"),
    ((14, 14, 21), 10, (O, P, P), 1, dvm.HOFKS, F32, "cell"),    # 4116 cells
    ((14, 14, 20), 10, (O, P, P), 1, dvm.HOFKS, F32, "shared"),  # 3920
    ((24, 24, 24), 11, (O, P, P), 1, dvm.HOFKS, F32, "shared"),
    # FP64, likewise: below a half (16 x 16 of 32 x 16)
    ((14, 14, 14), 11, (P, P, P), 1, dvm.HOFKS, F64, "cell"),
    ((14, 14, 14), 10, (P, P, P), 1, dvm.HOFKS, F64, "shared"),
    ((16, 16, 16), 11, (O, O, O), 1, dvm.HOFKS, F64, "shared"),
])
def test_kernel_of_small_boxes(nx, nv, bc, p, scheme, precision, want):
    d = len(nx)
    cfg, keep = dvm.make_config(d, nx, 1.0, (nv,) * d, (-(nv // 2),) * d, 1.0, p=p, bc=bc, tau=1.0, scheme=scheme,
                                precision=precision)
    assert dvm.plan_route(cfg)[0] == want
