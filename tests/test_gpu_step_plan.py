"""lks_step_plan: what lks_step launches.  A pass is one launch, three steps in a fused pass, all steps of a resident
lattice in one up to 16384."""
import ctypes

import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lks():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2112_13930_gb300 import build, lks as mod
    build.build()
    mod.load()
    return mod


def _plan(lks, nx, ny, storage, n, closure="link", coupling="maxwell", fx=2e-5, inplace=False):
    lat = lks.Lattice(nx, ny, 0.7, 0.9, 0.02, fx, closure, storage, coupling=coupling, inplace=inplace)
    try:
        return lat.step_plan(n)
    finally:
        lat.close()


def test_counts(lks):
    assert _plan(lks, 1024, 1024, "f32", 20, "moment") == (8, 8)        # 6 fused passes and 2 steps
    assert _plan(lks, 2048, 2048, "f64", 20) == (20, 20)
    assert _plan(lks, 4, 65, "f64", 1) == (1, 1) and _plan(lks, 4, 65, "f64", 0) == (0, 0)
    L = lks.load()
    n = ctypes.c_int64()
    assert L.lks_step_plan(None, 2, ctypes.byref(n), None) == lks.LKS_EINVAL
    lat = lks.Lattice(4, 65, 0.7, 0.9, 0.02, inplace=True)
    assert L.lks_step_plan(lat._h, 3, ctypes.byref(n), None) == lks.LKS_EINVAL
    assert L.lks_step_plan(lat._h, -2, ctypes.byref(n), None) == lks.LKS_EINVAL
    assert L.lks_step_plan(lat._h, 2, None, None) == 0
    lat.close()
