"""The reciprocal of the FP64 collisions (lks::recip, and 3/rho as collide_pairs forms it) against CUDA's division.

recip_seed reads the upper 32 bits of its argument, so all 2^20 upper mantissas with the lower word at either end are
every case of [1, 2); other binades differ by an exact power of two.  |e| = |1 - rho r| < 2^-19 there leaves e^3 < 2^-57 after
the iteration r + r (e + e^2), and the other roundings before the last are below 2^-71: the result is within
0.5 + 2^-57 / 2^-53 = 0.5625 units in the last place of 1/rho, so at most one from the correctly rounded quotient.  For
3/rho the seed's 21 bits times 3 are exact, and the same bound holds."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = r"""
#include "lks_device.cuh"
__global__ void k(const double* x, long n, double* e, double* r, double* r3, double* d, double* d3) {
    const long i = blockIdx.x * (long)blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double v = x[i], s = lks::recip_seed(v), t = lks::ffma(-v, s, 1.0), s3 = lks::fmul(3.0, s);
    e[i] = t;
    r[i] = lks::recip(v);
    r3[i] = lks::ffma(s3, lks::ffma(t, t, t), s3);
    d[i] = 1.0 / v;
    d3[i] = 3.0 / v;
}
extern "C" int run(const double* x, long n, double* e, double* r, double* r3, double* d, double* d3) {
    k<<<(unsigned)((n + 255) / 256), 256>>>(x, n, e, r, r3, d, d3);
    return (int)cudaDeviceSynchronize();
}
"""


def _values():
    upper = np.arange(1 << 20, dtype=np.uint64) << np.uint64(32)
    one = np.uint64(0x3FF) << np.uint64(52)
    ends = [(one | upper | np.uint64(low)).view(np.float64) for low in (0, 0xFFFFFFFF)]
    rng = np.random.default_rng(7)
    near_one = (one + np.arange(-4096, 4096).astype(np.int64).view(np.uint64)).view(np.float64)
    return np.concatenate(ends + [0.5 * ends[0], 2.0 * ends[1], near_one, np.exp2(np.arange(-40.0, 41.0)),
                                  1.0 + rng.uniform(-0.3, 0.3, 1 << 20), np.exp2(rng.uniform(-8, 8, 1 << 20))])


def test_recip_is_within_one_unit_of_the_quotient(tmp_path):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2112_13930_gb300 import build
    (tmp_path / "recip.cu").write_text(SOURCE)
    lib = str(tmp_path / "recip.so")
    subprocess.run([build._nvcc()] + build.ARCH + build.FLAGS + ["-I", build.CSRC, "-shared", "-cudart", "shared", "-o", lib,
                                                                 str(tmp_path / "recip.cu")], check=True)
    x = torch.tensor(_values(), device="cuda")
    out = [torch.empty_like(x) for _ in range(5)]
    assert ctypes.CDLL(lib).run(ctypes.c_void_p(x.data_ptr()), ctypes.c_long(x.numel()),
                                *[ctypes.c_void_p(o.data_ptr()) for o in out]) == 0
    e, r, r3, d, d3 = (o.cpu().numpy() for o in out)
    print("|e| <= 2^%.3f" % np.log2(np.max(np.abs(e))))
    assert np.max(np.abs(e)) < 2.0 ** -19
    for got, want in ((r, d), (r3, d3)):
        off = np.abs(got.view(np.int64) - want.view(np.int64))
        print("differ by a unit: %.4f" % np.mean(off != 0))
        assert np.max(off) <= 1
