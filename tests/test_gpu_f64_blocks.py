"""The FP64 building blocks of ``csrc/dg_f64.cuh`` (reciprocal, square root, reciprocal
square root, power) against CUDA's own operations, over the whole range of the type: every
binade of the normal numbers, zero, infinities and NaN.  Subnormal operands count as zero
and subnormal results are zero, as the header says."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1305_5536_gb300", "csrc")
EPS = np.finfo(np.float64).eps

_SRC = r"""
#include "dg_f64.cuh"
using namespace dgk;
__global__ void blocks_kernel(const double* x, double z, double* o, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const size_t m = n;
  const double v = x[i];
  double w;
  o[i] = rcpv(v);
  o[m + i] = sqrt64(v);
  o[2 * m + i] = rsqrt64(v);
  o[3 * m + i] = pow_m1(v, z, w);
  o[4 * m + i] = w;
  o[5 * m + i] = 1.0 / v;
  o[6 * m + i] = sqrt(v);
  o[7 * m + i] = 1.0 / sqrt(v);
  o[8 * m + i] = expm1(z * log(v));
  o[9 * m + i] = pow(v, z);
}
extern "C" int blocks(const double* x, double z, double* o, int n) {
  blocks_kernel<<<(n + 127) / 128, 128>>>(x, z, o, n);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def blocks(tmp_path_factory):
    import torch

    d = tmp_path_factory.mktemp("blocks64")
    (d / "b.cu").write_text(_SRC)
    so = str(d / "libb.so")
    nvcc = "/usr/local/cuda/bin/nvcc" if os.path.exists("/usr/local/cuda/bin/nvcc") else "nvcc"
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17",
                    "--expt-relaxed-constexpr", "-Xcompiler", "-fPIC", "-shared", "-I", CSRC,
                    str(d / "b.cu"), "-o", so, "-lcudart"], check=True, capture_output=True)
    L = ctypes.CDLL(so)
    vp = ctypes.c_void_p
    L.blocks.argtypes = [vp, ctypes.c_double, vp, ctypes.c_int]

    def run(x, z=0.2):
        t = torch.from_numpy(np.ascontiguousarray(x)).cuda()
        o = torch.empty((10, len(x)), dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        assert L.blocks(t.data_ptr(), z, o.data_ptr(), len(x)) == 0
        return o.cpu().numpy()

    return run


def _values():
    """Positive normal numbers: 64 random and the two end mantissas of every binade."""
    rng = np.random.default_rng(4)
    m = np.concatenate([rng.uniform(1, 2, 64), [1.0, 2.0 - EPS]])
    return np.ldexp(m[None, :], np.arange(-1022, 1024)[:, None]).ravel()


@pytest.mark.parametrize("op", ["reciprocal", "sqrt", "rsqrt"])
def test_within_two_ulp_over_the_whole_range(blocks, op):
    k = ["reciprocal", "sqrt", "rsqrt"].index(op)
    x = _values()
    o = blocks(np.concatenate([x, -x]) if op == "reciprocal" else x)
    got, want = o[k], o[5 + k]
    small = np.abs(want) <= 2.0 ** -1022
    assert (np.abs(got[small]) <= 2.0 ** -1022).all()
    # one ulp of the result for the refinement, one where the two roundings of 1 / sqrt
    # differ from one
    assert (np.abs(got - want)[~small] <= 2 * np.spacing(np.abs(want[~small]))).all()


def test_special_values(blocks):
    x = np.array([0.0, -0.0, np.inf, -np.inf, np.nan])
    o = blocks(x)
    assert np.array_equal(o[0], o[5], equal_nan=True)
    assert np.array_equal(o[1][[0, 1, 2, 4]], o[6][[0, 1, 2, 4]], equal_nan=True)
    assert np.array_equal(o[2][[0, 1, 2, 4]], o[7][[0, 1, 2, 4]], equal_nan=True)
    # roots of negative numbers; subnormal operands as zero
    o = blocks(np.array([-1.0, -1e300, -1e-300]))
    assert np.isnan(o[1]).all() and np.isnan(o[2]).all()
    o = blocks(np.array([5e-324, 1e-310, 2.2e-308]))
    assert np.isinf(o[0]).all() and (o[1] < 2.0 ** -1022).all() and np.isinf(o[2]).all()


@pytest.mark.parametrize("z", [0.2, 1.0 / 7.0, 0.1 / 2.2, 0.45])
def test_power(blocks, z):
    rng = np.random.default_rng(5)
    x = np.concatenate([_values(), np.exp(rng.uniform(-30, 30, 200000)), rng.uniform(0.5, 2, 200000)])
    o = blocks(x, z)
    y = np.abs(z * np.log2(x))
    # z log2 x carries one rounding of its own size, the rest a few
    assert (np.abs(o[4] - o[9]) <= (3 + y) * EPS * o[9]).all()
    assert (np.abs(o[3] - o[8]) <= (3 + y) * EPS * np.maximum(1, o[9])).all()
    # near x = 1 the difference from one keeps its relative accuracy
    near = np.concatenate([1 + s * np.exp(rng.uniform(-36, -5.5, 50000)) for s in (1, -1)])
    o = blocks(near, z)
    assert (np.abs(o[3] - o[8]) <= 6 * EPS * np.abs(o[8])).all()
