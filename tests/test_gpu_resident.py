"""Small lattices stepped in one cluster's shared memory (lks_resident.cu) against single steps, bit for bit:
step(n) with n > 1 takes one resident launch, n calls of step(1) the step kernels (in place: pairs, against the
two-buffer lattice).  Sizes: fewer rows than CTAs, uneven bands, one band per row, FP64 with one group of four
warps a CTA, two, and none, and the largest of each storage type."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SIZES = {"f64": [(1, 3), (4, 65), (3, 101), (5, 97), (4, 257), (7, 289)],
         "f32": [(1, 3), (4, 65), (130, 17), (4, 1025), (64, 128)],
         "bf16": [(2, 3), (4, 65), (37, 40), (8, 1500)]}
SIZES["f16"] = SIZES["bf16"]


@pytest.fixture(scope="module")
def lks():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2112_13930_gb300 import build, lks as mod
    build.build()
    mod.load()
    return mod


@pytest.mark.parametrize("storage", ["f64", "f32", "bf16", "f16"])
@pytest.mark.parametrize("closure", ["link", "moment"])
@pytest.mark.parametrize("coupling", ["maxwell", "lorentz"])
@pytest.mark.parametrize("fx", [2e-5, 0.0])
def test_resident_steps_equal_single_steps_bitwise(lks, storage, closure, coupling, fx):
    for nx, ny in SIZES[storage]:
        lats = [lks.Lattice(nx, ny, 0.7, 0.9, 0.02, fx, closure, storage, seed=5, perturb_amp=1e-2, coupling=coupling,
                            inplace=inplace) for inplace in (False, False, True)]
        for lat in lats:
            lat.set_walls(0.4, 3.0, 0.02, -0.04)
        a, b, c = lats
        for n in (2, 7, 12):
            a.step(n)
            for _ in range(n):
                b.step(1)
            fa, ga = a.get_state()
            fb, gb = b.get_state()
            assert a.steps == b.steps
            assert np.array_equal(fa, fb) and np.array_equal(ga, gb), (nx, ny, n)
        b.step(1)              # 22 steps
        c.step(22)
        fb, gb = b.get_state()
        fc, gc = c.get_state()
        assert np.array_equal(fb, fc) and np.array_equal(gb, gc), (nx, ny, "in place")
        for lat in lats:
            lat.close()
