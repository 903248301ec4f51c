"""The staged 16-bit step at widths whose segments have fewer items than there are consumer warps, so that warps pass
tasks they have no item in: bit for bit against a lattice tiled from a narrower one that is not staged.  Two buffers
take steps one and two at a time, which only single-step launches can do."""
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


@pytest.mark.parametrize("storage,closure", [("bf16", "moment"), ("f16", "link")])
@pytest.mark.parametrize("base,k,ny", [
    (516, 2, 1500),  # 1032: two segments of 9 items, about 20 tasks a block
    (708, 2, 1500),  # 1416: two of 12
    (514, 4, 1000),  # 2056: three of 11
    (516, 4, 900),   # 2064: three of 11, the last segment ragged by other words
    (896, 2, 1200),  # 1792: two of 14
])
def test_passed_tasks_bitwise(lks, storage, closure, base, k, ny):
    lats = [lks.Lattice(nx, ny, 0.7, 0.9, 0.02, 2e-5, closure, storage, seed=8, perturb_amp=1e-2, inplace=inplace)
            for nx, inplace in ((base, False), (base * k, False), (base * k, True))]
    for lat in lats:
        lat.set_walls(0.4, 3.0, 0.02, -0.04)
    a, b, c = lats
    f, g = a.get_state()
    for lat in (b, c):
        lat.set_state(np.concatenate([f] * k, axis=-1), np.concatenate([g] * k, axis=-1))
    for _ in range(2):
        a.step(2)
        b.step(2)
        c.step(2)
    for _ in range(2):
        a.step(1)
        b.step(1)
    c.step(2)
    f, g = a.get_state()
    for lat in (b, c):
        fl, gl = lat.get_state()
        assert np.array_equal(fl, np.concatenate([f] * k, axis=-1))
        assert np.array_equal(gl, np.concatenate([g] * k, axis=-1))
        lat.close()
    a.close()
