"""lks_step_plan: what lks_step launches.  The lattices that other tests take through the fused rows and the resident
kernel do take them (their comparisons with single steps would pass without), and the counts are those of the rules:
a pass is one launch, three steps in a fused pass, all steps of a resident lattice in one up to 16384."""
import ctypes

import numpy as np
import pytest

from test_gpu_resident import SIZES as RESIDENT
from test_gpu_rows import SIZES as ROWS

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


@pytest.mark.parametrize("storage", ["f32", "bf16", "f16"])
@pytest.mark.parametrize("closure", ["link", "moment"])
@pytest.mark.parametrize("coupling,fx", [("maxwell", 2e-5), ("maxwell", 0.0), ("lorentz", 2e-5)])
def test_lattices_of_the_rows_test_are_fused(lks, storage, closure, coupling, fx):
    for nx, ny in ROWS[storage]:
        assert _plan(lks, nx, ny, storage, 10, closure, coupling, fx) == (4, 4), (nx, ny)  # 3 + 3 + 3 + 1


# The fewest steps that a resident lattice takes in its cluster: 4 + N^2 / 1e5 for N nodes in FP64, 12 + N^2 / 1e6 in FP32,
# 12 + N^2 / 4e6 in 16 bits.
def _least(storage, nodes):
    return 4 + nodes ** 2 // 100000 if storage == "f64" else 12 + nodes ** 2 // (10 ** 6 if storage == "f32" else 4 * 10 ** 6)


@pytest.mark.parametrize("coupling", ["maxwell", "lorentz"])
@pytest.mark.parametrize("storage", ["f64", "f32", "bf16", "f16"])
def test_lattices_of_the_resident_test_are_resident(lks, storage, coupling):
    for nx, ny in RESIDENT[storage]:
        n = _least(storage, nx * ny)
        even = n + n % 2
        if (storage, nx, ny) == ("f64", 7, 289):  # 133 nodes a CTA
            assert _plan(lks, nx, ny, storage, even, coupling=coupling) == (even, even)
            continue
        assert _plan(lks, nx, ny, storage, n, coupling=coupling) == (1, 1), (nx, ny)
        assert _plan(lks, nx, ny, storage, n - 1, coupling=coupling) == (n - 1, n - 1), (nx, ny)
        assert _plan(lks, nx, ny, storage, even, coupling=coupling, inplace=True) == (1, 1), (nx, ny)
        assert _plan(lks, nx, ny, storage, even - 2, coupling=coupling, inplace=True) == (even - 2, even - 2), (nx, ny)
        assert _plan(lks, nx, ny, storage, 16385, coupling=coupling) == (2, 2)  # a launch and a single step
        assert _plan(lks, nx, ny, storage, 2 * 16384 + 2, coupling=coupling) == (3, 3)


@pytest.mark.parametrize("storage", ["f64", "f32", "bf16", "f16"])
@pytest.mark.parametrize("closure", ["link", "moment"])
@pytest.mark.parametrize("coupling,fx", [("maxwell", 2e-5), ("maxwell", 0.0), ("lorentz", 2e-5)])
def test_calls_above_the_least_equal_single_steps_bitwise(lks, storage, closure, coupling, fx):
    """As tests/test_gpu_resident.py, with calls long enough for the cluster."""
    for nx, ny in RESIDENT[storage] + ([(8, 256)] if storage == "f64" else []):
        kw = dict(seed=5, perturb_amp=1e-2, coupling=coupling)
        lats = [lks.Lattice(nx, ny, 0.7, 0.9, 0.02, fx, closure, storage, inplace=i, **kw) for i in (False, False, True)]
        for lat in lats:
            lat.set_walls(0.4, 3.0, 0.02, -0.04)
        a, b, c = lats
        least = _least(storage, nx * ny)
        for n in (least, least + 1):
            a.step(n)
        for _ in range(2 * least + 1):
            b.step(1)
        assert all(np.array_equal(x, y) for x, y in zip(a.get_state(), b.get_state())), (nx, ny)
        c.step(2 * least + 2)
        b.step(1)
        assert all(np.array_equal(x, y) for x, y in zip(c.get_state(), b.get_state())), (nx, ny, "in place")
        for lat in lats:
            lat.close()


@pytest.mark.parametrize("closure", ["link", "moment"])
@pytest.mark.parametrize("coupling", ["maxwell", "lorentz"])
def test_fp64_ctas_hold_at_most_128_nodes(lks, closure, coupling):
    """128 nodes a CTA are resident, bit for bit with single steps; one row or column more is not, nor are lattices of
    few wide rows, whose CTAs are few."""
    for nx, ny in [(8, 256), (128, 16), (128, 8), (128, 3)]:
        a, b = (lks.Lattice(nx, ny, 0.7, 0.9, 0.02, 2e-5, closure, "f64", seed=5, perturb_amp=1e-2, coupling=coupling)
                for _ in range(2))
        for lat in (a, b):
            lat.set_walls(0.4, 3.0, 0.02, -0.04)
        n = 46
        assert a.step_plan(n) == ((1, 1) if ny > 3 else (n, n))
        a.step(n)
        for _ in range(n):
            b.step(1)
        assert all(np.array_equal(x, y) for x, y in zip(a.get_state(), b.get_state())), (nx, ny)
        a.close()
        b.close()
    for nx, ny in [(129, 8), (43, 44), (160, 3), (200, 8), (20, 100)]:
        assert _plan(lks, nx, ny, "f64", 46, closure, coupling) == (46, 46), (nx, ny)


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
