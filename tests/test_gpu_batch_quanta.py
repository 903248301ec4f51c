"""Batches on clusters by the length of their launches: long quanta hold the instances in shared memory, short ones and
those with frequent checks do not.  The state and the residuals are the same bit for bit however the steps are cut, also
where one batch goes back and forth between the two."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SIZES = [(4, 33), (5, 97), (16, 64), (33, 40), (64, 64)]


@pytest.fixture(scope="module")
def batch():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2112_13930_gb300 import batch as mod, build
    build.build()
    return mod


@pytest.mark.parametrize("storage", ["f32", "bf16", "f16"])
@pytest.mark.parametrize("coupling", ["maxwell", "lorentz"])
@pytest.mark.parametrize("inplace", [False, True])
def test_cuts_of_the_same_steps_are_equal_bitwise(batch, storage, coupling, inplace):
    def solve(quanta, check_every):
        b = batch.Batch(storage, max_instances=8, pool_bytes=64 << 20, threads_per_group=128, cluster_ctas=8,
                        coupling=coupling, inplace=inplace)
        slots = [b.add(batch.make_desc(nx, ny, ("link", "moment")[k % 2], 0.7, 0.9, 0.02, 2e-5, 0.4, 3.0, 0.02, -0.04,
                                       seed=k, perturb_amp=1e-2, tol=1e-30, check_every=check_every, max_steps=10**6,
                                       coupling=coupling)) for k, (nx, ny) in enumerate(SIZES)]
        for q in quanta:
            b.run(q)
        out = [b.get_state(s) + b.result(s) for s in slots]
        b.close()
        return out

    # 16 steps and more to the next check or the end of the launch are held in shared memory
    for check_every in (100, 16, 14):
        want = solve([2] * 120, check_every)
        for quanta in ([240], [16, 14, 40, 2, 68, 100]):
            for w, g in zip(want, solve(quanta, check_every)):
                assert np.array_equal(w[0], g[0]) and np.array_equal(w[1], g[1]) and w[2:] == g[2:], (check_every, quanta)


def test_more_shapes_than_kept_graphs(batch):
    """A batch keeps the graphs of eight shapes: twelve in turn, twice, give the states of one shape bit for bit."""
    descs = [batch.make_desc(nx, ny, "link", 0.7, 0.9, 0.02, 2e-5, 0.4, 3.0, seed=k, perturb_amp=1e-2, tol=1e-30,
                             check_every=100, max_steps=10**6) for k, (nx, ny) in enumerate(SIZES)]
    shapes = [(T, 1, C) for T in (32, 64, 128, 256) for C in (1, 4, 8)]
    a, b = (batch.Batch("f32", max_instances=8, pool_bytes=64 << 20, threads_per_group=128, cluster_ctas=8)
            for _ in range(2))
    sa, sb = [a.add(d) for d in descs], [b.add(d) for d in descs]
    for shape in shapes + shapes[::-1] + shapes[:2] * 2:
        a.set_shape(*shape)
        a.run(20)
        b.run(20)
    for x, y in zip(sa, sb):
        assert a.result(x)[:2] == b.result(y)[:2] == (batch.INST_RUNNING, 20 * 28)
        assert all(np.array_equal(p, q) for p, q in zip(a.get_state(x), b.get_state(y)))
    a.close()
    b.close()
