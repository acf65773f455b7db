"""The FP64 kernels' reciprocal and square root are correctly rounded: every
result equals the host's IEEE division and root, over random significands at
every exponent, the neighbours of the exponent limits, and zeros, subnormals,
infinities, NaN and negative values."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_1902_02999_gb300 import build

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "maclab_kernels.cuh"
#include "maclab_march.cuh"
__global__ void functions(const double* a, double* r, double* s, long long n)
{
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        r[i] = maclab::Op<double>::rcp(a[i]);
        s[i] = maclab::Op<double>::sqrt(a[i]);
    }
}
extern "C" int run(const double* a, double* r, double* s, long long n)
{
    functions<<<512, 256>>>(a, r, s, n);
    return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def functions(tmp_path_factory):
    d = tmp_path_factory.mktemp("fp64")
    src, so = str(d / "functions.cu"), str(d / "functions.so")
    with open(src, "w") as f:
        f.write(SOURCE)
    subprocess.check_call([build.nvcc(), "-O3", "-std=c++17", build.ARCH, "-shared", "-Xcompiler", "-fPIC",
                           "-I" + build.INCLUDE, "-I" + build.CSRC, "-o", so, src])
    assert os.path.exists(so)
    return ctypes.CDLL(so)


def values():
    rng = np.random.default_rng(5)
    exponent = np.repeat(np.arange(2048, dtype=np.uint64), 512)
    bits = (exponent << np.uint64(52)) | rng.integers(0, 1 << 52, exponent.size, dtype=np.uint64)
    # both sides of every exponent's ends, and significands near one and two
    edge = (np.arange(2048, dtype=np.uint64) << np.uint64(52))[:, None] + np.arange(-4, 5).astype(np.uint64)[None, :]
    half = edge + np.uint64(1 << 51)
    bits = np.concatenate([bits, edge.reshape(-1), half.reshape(-1)])
    a = bits.view(np.float64)
    a = np.concatenate([a, -a, np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 5e-324, -5e-324])])
    # a few million ordinary depths and speeds squared
    return np.concatenate([a, rng.uniform(1e-6, 64.0, 1 << 21), 10.0 ** rng.uniform(-30, 3, 1 << 21)])


def test_reciprocal_and_root_are_correctly_rounded(functions):
    a = values()
    dev = torch.from_numpy(a).cuda()
    r, s = torch.empty_like(dev), torch.empty_like(dev)
    p = [ctypes.c_void_p(t.data_ptr()) for t in (dev, r, s)]
    torch.cuda.synchronize()
    assert functions.run(*p, ctypes.c_longlong(a.size)) == 0
    with np.errstate(all="ignore"):
        want_r, want_s = 1.0 / a, np.sqrt(a)
    for got, want in ((r.cpu().numpy(), want_r), (s.cpu().numpy(), want_s)):
        nan = np.isnan(want)
        assert np.array_equal(np.isnan(got), nan)
        assert np.array_equal(got[~nan].view(np.uint64), want[~nan].view(np.uint64))
