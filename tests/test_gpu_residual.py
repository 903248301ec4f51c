"""The residual reduction where its blocks and its loads per thread run out: against the same sums in numpy over
the lattice's own node moments.  Both add the same non-negative FP64 terms in other orders, a thread at most nine in
a row and a tree over the rest, so the totals agree to some tens of roundings: 1e-13 of the value, taken as 1e-12."""
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


@pytest.mark.parametrize("storage", ["f64", "f32", "bf16"])
@pytest.mark.parametrize("nx,ny", [
    (1, 3),        # one block, most threads without a node
    (32, 64),      # one block, full
    (683, 3),      # 2049 nodes: two blocks
    (257, 41),     # six blocks, a ragged last pass
    (2001, 1251),  # the largest grid and one node more than its threads take at eight each, for some of them
])
def test_residual_against_numpy(lks, storage, nx, ny):
    lat = lks.Lattice(nx, ny, 0.8, 0.9, 0.02, 2e-5, "link", storage, seed=3, perturb_amp=1e-2)
    lat.set_walls(0.5, 0.5, 0.01, 0.02)
    lat.residual()
    before = np.asarray(lat.moments(), dtype=np.float64).reshape(5, -1)
    lat.step(2)
    got = lat.residual()
    after = np.asarray(lat.moments(), dtype=np.float64).reshape(5, -1)
    for r, k in zip(got, (1, 3)):
        want = np.sqrt(np.sum((after[k] - before[k]) ** 2) / np.sum(after[k] ** 2))
        assert abs(r - want) <= 1e-12 * want
    assert lat.residual() == (0.0, 0.0)
