"""The workspace of in-place FP32 lattices (lks_set_workspace): a handle takes no device memory beyond its footprint on
its own; with a workspace it steps in fused passes, without one in pairs, and the state is the two-buffer lattice's bit for
bit in either case and across the change.  (124, 15000) is one strip whose halo columns wrap onto itself, (247, 7500) two
strips, (1001, 2640) a ragged last strip, (1001, 2563) a last chunk of one row, (2056, 900) the shortest chunks."""
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


def test_handle_keeps_to_its_footprint(lks):
    import torch
    nx, ny = 2056, 1500  # its workspace would take 52 MB
    lks.Lattice(nx, ny, 0.7, 0.9, 0.02, storage="f32", inplace=True).close()  # loads the kernels
    buf = torch.empty(lks.footprint_bytes(nx, ny, storage="f32", inplace=True), dtype=torch.uint8, device="cuda")
    p = lks.make_params(nx, ny, 0.7, 0.9, 0.02, storage="f32", inplace=True, dev_buffer=buf.data_ptr(),
                        dev_buffer_bytes=buf.numel())
    import ctypes
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    h = ctypes.c_void_p()
    assert lks.load().lks_create(ctypes.byref(p), ctypes.byref(h)) == 0
    assert before - torch.cuda.mem_get_info()[0] < 16 << 20
    assert lks.load().lks_workspace_bytes(h) > 16 << 20
    assert lks.load().lks_step(h, 12) == 0 and lks.load().lks_sync(h) == 0
    lks.load().lks_destroy(h)
    lat = lks.Lattice(nx, ny, 0.7, 0.9, 0.02, storage="f32", inplace=True)
    assert lat.nbytes == buf.numel()
    lat.close()


@pytest.mark.parametrize("closure", ["link", "moment"])
@pytest.mark.parametrize("coupling", ["maxwell", "lorentz"])
def test_steps_with_and_without_workspace_bitwise(lks, closure, coupling):
    for nx, ny in [(124, 15000), (247, 7500), (1001, 2640), (1001, 2563), (2056, 900)]:
        kw = dict(closure=closure, storage="f32", coupling=coupling, seed=5, perturb_amp=1e-2)
        a = lks.Lattice(nx, ny, 0.7, 0.9, 0.02, 2e-5, inplace=True, workspace=True, **kw)
        b = lks.Lattice(nx, ny, 0.7, 0.9, 0.02, 2e-5, **kw)
        for lat in (a, b):
            lat.set_walls(0.4, 3.0, 0.02, -0.04)
        n_work = a.nbytes - lks.footprint_bytes(nx, ny, closure, "f32", inplace=True)
        assert 0 < n_work <= 0.4 * 19 * 4 * nx * ny
        for n, work in ((6, True), (14, True), (8, False), (20, True)):
            assert lks.load().lks_set_workspace(a._h, a._work.data_ptr() if work else None,
                                                a._work.numel() if work else 0) == 0
            # fused passes come in twos, each after a launch that saves the blocks' edges; the rest is single steps
            fused, single = (n // 6 * 2, n % 6) if work else (0, n)
            assert a.step_plan(n) == (fused + single, 2 * fused + single)
            a.step(n)
            for _ in range(n):
                b.step(1)
            assert a.steps == b.steps
            for x, y in zip(a.get_state(), b.get_state()):
                assert np.array_equal(x, y), (nx, ny, n)
        a.close()
        b.close()


def test_arguments(lks):
    import torch
    L = lks.load()
    for kw in (dict(nx=4096, ny=1024), dict(nx=64, ny=64, inplace=True), dict(nx=4096, ny=1024, inplace=True, st="bf16")):
        lat = lks.Lattice(kw["nx"], kw["ny"], 0.7, 0.9, 0.02, storage=kw.get("st", "f32"),
                          inplace=kw.get("inplace", False), workspace=True)
        assert L.lks_workspace_bytes(lat._h) == 0 and lat._work is None
        t = torch.empty(1 << 20, dtype=torch.uint8, device="cuda")
        assert L.lks_set_workspace(lat._h, t.data_ptr(), t.numel()) == lks.LKS_EINVAL
        assert L.lks_set_workspace(lat._h, None, 0) == 0
        lat.close()
    lat = lks.Lattice(4096, 1024, 0.7, 0.9, 0.02, storage="f32", inplace=True, workspace=True)
    n = lat._work.numel()
    assert L.lks_workspace_bytes(lat._h) == n
    assert L.lks_set_workspace(lat._h, lat._work.data_ptr(), n - 1) == lks.LKS_EINVAL
    assert L.lks_set_workspace(lat._h, lat._work.data_ptr() + 4, n) == lks.LKS_EINVAL
    assert L.lks_set_workspace(lat._h, None, n) == lks.LKS_EINVAL
    assert lat.step_plan(6) == (2, 4)
    lat.close()
