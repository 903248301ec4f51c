"""lks3_step on a stream under capture: its launches become nodes of the caller's graph, with the kernels' early start
between them, and replays take the same steps bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage,nx", [("f32", 36), ("bf16", 24), ("f64", 5)])
def test_captured_3d_steps_replay(storage, nx):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2112_13930_gb300 import build, lks3d
    build.build()
    stream = torch.cuda.Stream()
    lats = [lks3d.Lattice3D(nx, 9, 6, 0.7, 0.9, 0.02, 2e-5, storage, stream=stream) for _ in range(2)]
    for lat in lats:
        lat.set_walls(0.4, 3.0, 0.02, -0.04)
    a, b = lats
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        a.step(6)
    graph.replay()
    graph.replay()
    torch.cuda.synchronize()
    b.step(12)
    for x, y in zip(a.get_state(), b.get_state()):
        assert np.array_equal(x, y)
