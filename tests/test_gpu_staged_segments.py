"""The staged 16-bit kernels over rows of one to five segments, bit for bit: a lattice tiled from a narrower one that
is not staged, with two buffers and in place.  Segments of 13, 15 and 16 items for 15 consumer warps, full and ragged
last segments, and more rows than blocks."""
import numpy as np
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


@pytest.mark.parametrize("storage,closure,coupling", [("bf16", "moment", "maxwell"), ("f16", "link", "maxwell"),
                                                      ("bf16", "link", "lorentz")])
@pytest.mark.parametrize("base,k,ny", [
    (512, 2, 200),  # 1024: one segment of 16 items
    (960, 2, 40),   # 1920: two of 15
    (742, 4, 60),   # 2968: three of 16, the last ragged
    (513, 8, 33),   # 4104: five of 13
    (637, 8, 40),   # 5096: five of 16
])
def test_segments_equal_a_narrower_lattice_bitwise(lks, storage, closure, coupling, base, k, ny):
    lats = [lks.Lattice(nx, ny, 0.7, 0.9, 0.02, 2e-5, closure, storage, seed=8, perturb_amp=1e-2, coupling=coupling,
                        inplace=inplace) for nx, inplace in ((base, False), (base * k, False), (base * k, True))]
    for lat in lats:
        lat.set_walls(0.4, 3.0, 0.02, -0.04)
    a, b, c = lats
    f, g = a.get_state()
    for lat in (b, c):
        lat.set_state(np.concatenate([f] * k, axis=-1), np.concatenate([g] * k, axis=-1))
    for n in (2, 4):
        for lat in lats:
            lat.step(n)
        f, g = a.get_state()
        for lat in (b, c):
            fl, gl = lat.get_state()
            assert np.array_equal(fl, np.concatenate([f] * k, axis=-1))
            assert np.array_equal(gl, np.concatenate([g] * k, axis=-1))
