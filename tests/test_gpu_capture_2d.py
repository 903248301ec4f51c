"""lks_step of small lattices on a stream under capture: calls too short for the cluster otherwise are captured as one
cluster launch, and replays take the same steps bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,storage,inplace", [(4, 65, "f64", False), (64, 64, "f32", False), (100, 100, "f32", True),
                                                   (37, 40, "bf16", False)])
@pytest.mark.parametrize("n", [1, 2, 4, 200])
def test_captured_steps_replay(nx, ny, storage, inplace, n):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2112_13930_gb300 import build, lks
    build.build()
    if inplace and n % 2:
        pytest.skip("an in-place lattice steps in pairs")
    stream = torch.cuda.Stream()
    a, b = (lks.Lattice(nx, ny, 0.7, 0.9, 0.02, 2e-5, "link", storage, seed=5, perturb_amp=1e-2, stream=stream,
                        inplace=inplace) for _ in range(2))
    for lat in (a, b):
        lat.set_walls(0.4, 3.0, 0.02, -0.04)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        assert a.step_plan(n) == (1, 1)
        a.step(n)
    replays = 1 if n % 2 else 3  # an odd call ends in the other buffer
    for _ in range(replays):
        graph.replay()
    torch.cuda.synchronize()
    for _ in range(n * replays // (2 if inplace else 1)):
        b.step(2 if inplace else 1)
    for x, y in zip(a.get_state(), b.get_state()):
        assert np.array_equal(x, y)
