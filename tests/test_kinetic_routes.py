"""Which kinetic-pass kernel a configuration takes and how many folded source rows it gets,
host side (dvm_plan_route): the limit of shared memory from both sides and the fallbacks."""
import pytest

from paper_1212_0204_gb300 import build, dvm

P, O = dvm.PERIODIC, dvm.OUTFLOW


@pytest.fixture(scope="module", autouse=True)
def library():
    build.build()


def route(nx, nv, precision, scheme, bc=None, p=1):
    cfg, keep = dvm.make_config(len(nx), nx, 1.0, nv, tuple(-(n // 2) for n in nv), 1.0, p=p, bc=bc, tau=1.0,
                                scheme=scheme, precision=precision)
    return dvm.plan_route(cfg)


@pytest.mark.parametrize("nx,nky,scheme,precision,want", [
    # two CTAs per SM: 36 (FP64) or 40 rows where slots, staged f and tables fit 113 KB
    ((40, 32), 108, dvm.HOFKS, dvm.F64, ("shared", 36)),
    ((40, 32), 109, dvm.HOFKS, dvm.F64, ("shared", 32)),
    ((40, 32), 109, dvm.FKS, dvm.F64, ("shared", 36)),
    ((33, 17), 255, dvm.HOFKS, dvm.F32, ("shared", 40)),
    # a box one cell wide: 32 columns reach 32 blocks, whose tables leave no room for 24 rows
    ((1, 512), 32, dvm.HOFKS, dvm.F64, ("shared", 24)),
    ((1, 512), 33, dvm.HOFKS, dvm.F64, ("cell", 0)),
    ((1, 512), 128, dvm.HOFKS, dvm.F32, ("shared", 24)),
    ((1, 512), 129, dvm.HOFKS, dvm.F32, ("cell", 0)),
    # a 16-row column less than half full
    ((40, 7), 20, dvm.FKS, dvm.F64, ("cell", 0)),
    ((40, 8), 20, dvm.FKS, dvm.F64, ("shared", 36)),
])
def test_rows_beside_the_limit(nx, nky, scheme, precision, want):
    assert route(nx, (39, nky), precision, scheme) == want


def test_kernels_of_the_storage_tiers():
    for precision in (dvm.F64, dvm.F32, dvm.BF16S):
        assert route((100,), (32,), precision, dvm.HOFKS) == ("cell", 0)
        for bc, p in (((O, O), 1), ((P, O), 2), ((O, P), 3)):
            assert route((40, 36), (16, 16), precision, dvm.HOFKS, bc, p)[0] == "shared"
    assert route((40, 36), (16, 16), dvm.F64, dvm.HOFKS)[0] == "shared"
    assert route((40, 36), (16, 16), dvm.F32, dvm.HOFKS) == ("window", 0)
    assert route((40, 36), (16, 16), dvm.F32, dvm.FKS)[0] == "shared"
    assert route((64, 64, 64), (24, 24, 24), dvm.F32, dvm.HOFKS) == ("tile", 0)
    assert route((64, 64, 64), (24, 24, 24), dvm.BF16S, dvm.HOFKS) == ("window", 0)
    assert route((4, 8, 3856), (8, 8, 6), dvm.F32, dvm.HOFKS) == ("cell", 0)


@pytest.mark.parametrize("n,nv,scheme,precision,want", [
    # where both kernels can run in 3D: by the share of useful lanes of either
    (40, 16, dvm.HOFKS, dvm.F32, "shared"),
    (60, 20, dvm.HOFKS, dvm.F32, "window"),
    (60, 20, dvm.FKS, dvm.F32, "window"),
    (90, 24, dvm.FKS, dvm.BF16S, "window"),
    (100, 12, dvm.FKS, dvm.F32, "shared"),
    (64, 12, dvm.FKS, dvm.F32, "shared"),
    (64, 12, dvm.FKS, dvm.BF16S, "window"),
    (64, 12, dvm.HOFKS, dvm.F32, "window"),
    (64, 16, dvm.HOFKS, dvm.F32, "shared"),
    (24, 12, dvm.FKS, dvm.F32, "window"),
    (48, 16, dvm.HOFKS, dvm.BF16S, "window"),
])
def test_kernels_of_3d_boxes(n, nv, scheme, precision, want):
    assert route((n,) * 3, (nv,) * 3, precision, scheme)[0] == want
