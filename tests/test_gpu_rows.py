"""Three fused steps per pass over memory (lks_step_rows.cu) against single steps, bit for bit: step(n)
takes n // 3 fused passes and n % 3 single steps, n calls of step(1) only single ones.  Sizes: the
narrowest row (one block wraps around it), one block's width and one column more (two strips), a
ragged last strip, and chunks of eight rows, the fewest that take the fused kernel, up to many.  Where half of a
block's columns are idle, the lattice is larger than L2, as the fused kernel asks."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# nx (columns of one node for FP32, of two for 16-bit storage), ny: 760 FP32 or 608 16-bit blocks are resident
SIZES = {"f32": [(64, 40000), (128, 6000), (129, 20000), (1001, 1300)],
         "bf16": [(128, 40000), (256, 4900), (258, 20000), (1034, 1200)]}
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


@pytest.mark.parametrize("storage", ["f32", "bf16", "f16"])
@pytest.mark.parametrize("closure", ["link", "moment"])
@pytest.mark.parametrize("coupling,fx", [("maxwell", 2e-5), ("maxwell", 0.0), ("lorentz", 2e-5)])
def test_fused_steps_equal_single_steps_bitwise(lks, storage, closure, coupling, fx):
    for nx, ny in SIZES[storage]:
        kw = dict(closure=closure, storage=storage, coupling=coupling, seed=5, perturb_amp=1e-2)
        a = lks.Lattice(nx, ny, 0.7, 0.9, 0.02, fx, **kw)
        b = lks.Lattice(nx, ny, 0.7, 0.9, 0.02, fx, **kw)
        for lat in (a, b):
            lat.set_walls(0.4, 3.0, 0.02, -0.04)
        for n in (3, 10):      # one pass; a graph of two, one pass and a single step
            a.step(n)
            for _ in range(n):
                b.step(1)
            assert a.steps == b.steps
            assert np.array_equal(a.get_state_raw(), b.get_state_raw()), (nx, ny, n)
        a.close()
        b.close()


@pytest.mark.parametrize("closure", ["link", "moment"])
@pytest.mark.parametrize("coupling", ["maxwell", "lorentz"])
def test_fused_steps_in_place_equal_two_buffer_single_steps_bitwise(lks, closure, coupling):
    """One buffer (FP32, larger than L2): fused passes come in twos (6 steps), the rest in AA pairs.  (124, 14000) is one
    strip whose halo columns wrap onto itself, (247, 7100) two strips, (1001, 2600) a ragged last strip, (1001, 2527) a
    last chunk of one row, (2056, 900) the shortest chunks."""
    storage = "f32"
    for nx, ny in [(124, 14000), (247, 7100), (1001, 2640), (1001, 2563), (2056, 900)]:
        kw = dict(closure=closure, storage=storage, coupling=coupling, seed=5, perturb_amp=1e-2)
        a = lks.Lattice(nx, ny, 0.7, 0.9, 0.02, 2e-5, inplace=True, **kw)
        b = lks.Lattice(nx, ny, 0.7, 0.9, 0.02, 2e-5, **kw)
        for lat in (a, b):
            lat.set_walls(0.4, 3.0, 0.02, -0.04)
        for n in (6, 14):      # one graph of two passes; two of them and a pair
            a.step(n)
            for _ in range(n):
                b.step(1)
            assert a.steps == b.steps
            fa, ga = a.get_state()
            fb, gb = b.get_state()
            assert np.array_equal(fa, fb) and np.array_equal(ga, gb), (nx, ny, n)
        a.close()
        b.close()
