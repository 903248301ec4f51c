"""lks_step on a stream under capture, bit for bit with the same steps outside: its launches become nodes of the caller's
graph, a cluster launch for a long call on a small lattice, single steps or fused passes otherwise."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,storage,inplace", [
    (4, 65, "f64", False), (64, 64, "f32", False), (100, 100, "f32", True), (37, 40, "bf16", False),  # resident
    (7, 289, "f64", False), (160, 3, "f64", True),         # FP64 with more nodes a CTA than the cluster takes
    (256, 257, "f32", False), (300, 200, "f16", True), (1032, 100, "bf16", False), (1032, 100, "bf16", True),
    (1001, 1300, "f32", False),                            # fused passes
    (1001, 2640, "f32", True),                             # fused in place, with a workspace
])
@pytest.mark.parametrize("n", [1, 2, 4, 14, 132])
def test_captured_steps_replay(nx, ny, storage, inplace, n):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2112_13930_gb300 import build, lks
    build.build()
    if inplace:
        n += n % 2
    stream = torch.cuda.Stream()
    a, b = (lks.Lattice(nx, ny, 0.7, 0.9, 0.02, 2e-5, "link", storage, seed=5, perturb_amp=1e-2, stream=stream,
                        inplace=inplace, workspace=w) for w in (True, False))
    for lat in (a, b):
        lat.set_walls(0.4, 3.0, 0.02, -0.04)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        a.step(n)
    assert a.steps == n
    replays = 1 if n % 2 else 3  # an odd call ends in the other buffer
    for _ in range(replays):
        graph.replay()
    torch.cuda.synchronize()
    for _ in range(n * replays // (2 if inplace else 1)):
        b.step(2 if inplace else 1)
    for x, y in zip(a.get_state(), b.get_state()):
        assert np.array_equal(x, y)
    a.step(6)                    # the handle's own graphs again
    for _ in range(3):
        b.step(2)
    for x, y in zip(a.get_state(), b.get_state()):
        assert np.array_equal(x, y)
    a.close()
    b.close()
