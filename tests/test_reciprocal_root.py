"""The FP64 reciprocal and square root of the pointwise physics against CUDA's 1/x and sqrt(x), which are
correctly rounded.

Both end in one rounding of a value that is off by the remainder of a third-order step on a seed of
relative error d, measured at 2^-19.9: d^3 and 5/2 d^3, at most 2^-6.7 and 2^-5.4 units in the last place.
So they differ from the correctly rounded result by at most one unit, and only where the exact value lies
that close to a tie, for at most that share of uniform arguments: 2^-5. A root that keeps half of an
intermediate rounding misses about one in eight."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

from paper_2401_06132_gb300 import build as B

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

SRC = r"""
#include "fr_physics.cuh"
__global__ void k(const double *x, double *o, long long n)
{
    const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (i >= n) return;
    o[i] = fr_inv(x[i]);
    o[n + i] = 1.0 / x[i];
    o[2 * n + i] = fr_sqrt(x[i]);
    o[3 * n + i] = sqrt(x[i]);
}
extern "C" int run(const double *x, double *o, long long n)
{
    k<<<(unsigned)((n + 255) / 256), 256>>>(x, o, n);
    return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    d = tmp_path_factory.mktemp("root")
    src, lib = str(d / "r.cu"), str(d / "r.so")
    with open(src, "w") as f:
        f.write(SRC)
    subprocess.check_call([B.nvcc()] + B.NVCC_FLAGS + ["-I", B.CSRC, "-I", os.path.join(B.HERE, "..", "include"), "-shared", src, "-o", lib])
    L = C.CDLL(lib)

    def call(x):
        o = torch.empty(4, x.size, dtype=torch.float64, device="cuda")
        u = torch.from_numpy(x).cuda()
        torch.cuda.synchronize()
        assert L.run(C.c_void_p(u.data_ptr()), C.c_void_p(o.data_ptr()), C.c_longlong(x.size)) == 0
        return o.cpu().numpy()

    return call


@pytest.mark.parametrize("mantissa", ["uniform", "low", "high"])
def test_reciprocal_and_root_against_cuda(run, mantissa):
    n = 1 << 20
    rng = np.random.default_rng(5)
    m = rng.integers(0, 1 << 52, n, dtype=np.uint64)
    if mantissa != "uniform":   # mantissas next to powers of two
        m &= np.uint64(0xfff)
    if mantissa == "high":
        m ^= np.uint64((1 << 52) - 1)
    x = ((rng.integers(3, 2044, n, dtype=np.uint64) << np.uint64(52)) | m).view(np.float64)
    o = run(x)
    for mine, cuda in ((o[0], o[1]), (o[2], o[3])):
        d = np.abs(mine.view(np.int64) - cuda.view(np.int64))
        assert d.max() <= 1
        if mantissa == "uniform":
            assert np.count_nonzero(d) <= n / 32


def test_values_without_a_finite_result(run):
    o = run(np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 5e-324]))
    assert not np.isfinite(o[0]).any()
    assert not np.isfinite(o[2]).any()
    assert np.isnan(run(np.array([-1.0]))[2])
