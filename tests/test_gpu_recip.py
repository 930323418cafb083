"""The integer-pipe functions. The reciprocal, reciprocal square root and square root of csrc/dg_recip.cuh against extended
precision: within 0.51 ulp (square root 1 ulp) over the exponent range, at the ends of the binades where the FP32
start value rounds up or down, and CUDA's own results for arguments outside their range."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2306_12891_gb300 import build as B

pytestmark = pytest.mark.gpu
SRC = r"""
#include "dg_recip.cuh"
__global__ void k(const double *x, double *y, int n, int ref) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  y[i] = ref ? 1.0 / x[i] : rcp_int(x[i]);
  y[n + i] = ref ? rsqrt(x[i]) : rsq_int(x[i]);
  y[2 * n + i] = ref ? sqrt(x[i]) : sqr_int(x[i]);
}
extern "C" int run(const void *x, void *y, int n, int ref) {
  k<<<(n + 255) / 256, 256>>>((const double *)x, (double *)y, n, ref);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    import torch

    d = tmp_path_factory.mktemp("recip")
    src, lib = os.path.join(d, "t.cu"), os.path.join(d, "t.so")
    with open(src, "w") as f:
        f.write(SRC)
    subprocess.check_call([B.NVCC, *B.ARCH, "-O3", "-shared", "-Xcompiler", "-fPIC", "-I", B.CSRC, "-o", lib, src])
    L = ctypes.CDLL(lib)

    def go(x, ref=False):
        X = torch.from_numpy(np.ascontiguousarray(x)).cuda()
        Y = torch.empty(3 * X.numel(), dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        assert L.run(ctypes.c_void_p(X.data_ptr()), ctypes.c_void_p(Y.data_ptr()), X.numel(), int(ref)) == 0
        return Y.cpu().numpy().reshape(3, -1)

    return go


def test_within_half_an_ulp_and_a_hundredth(run):
    rng = np.random.default_rng(0)
    m = np.concatenate([rng.uniform(1, 2, 400000), 1 + 2.0 ** -rng.uniform(1, 52, 50000), 2 - 2.0 ** -rng.uniform(1, 51, 50000),
                        1 + (np.arange(50000) + rng.uniform(-1e-6, 1e-6, 50000)) * 2.0 ** -23])
    x = np.ldexp(m, rng.integers(-1020, 1020, m.size))
    got = run(x)
    X = x.astype(np.longdouble)
    for name, y, t, bound in (("rcp", got[0], 1 / X, 0.51), ("rsqrt", got[1], 1 / np.sqrt(X), 0.51), ("sqrt", got[2], np.sqrt(X), 1.0)):
        ulp = np.spacing(np.abs(t.astype(np.float64)))
        err = float((np.abs(y.astype(np.longdouble) - t) / ulp).max())
        print(f"RECIP {name}: {err:.4f} ulp")
        assert err <= bound


def test_arguments_out_of_range_give_cudas_results(run):
    x = np.array([0.0, -0.0, -1.0, -1e300, np.inf, -np.inf, np.nan, 5e-324, 1e-310, 2.2e-308, 1.7e308, 8.9e307, 4.4e307, -5e-324])
    np.testing.assert_array_equal(run(x).view(np.int64), run(x, ref=True).view(np.int64))


def test_log_for_sums(tmp_path):
    """log_int of csrc/dg_log.cuh against extended precision, and CUDA's values out of its range."""
    import torch

    src, lib = os.path.join(tmp_path, "l.cu"), os.path.join(tmp_path, "l.so")
    with open(src, "w") as f:
        f.write(r"""
#include "dg_log.cuh"
__global__ void k(const double *x, double *y, int n, const LogEntry *t) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) y[i] = log_int(x[i], t);
}
extern "C" int run(const void *x, void *y, int n) {
  LogEntry h[LOG_TABLE], *t;
  log_table(h);
  if (cudaMalloc(&t, sizeof(h)) || cudaMemcpy(t, h, sizeof(h), cudaMemcpyHostToDevice)) return 1;
  k<<<(n + 255) / 256, 256>>>((const double *)x, (double *)y, n, t);
  const int e = (int)cudaDeviceSynchronize();
  cudaFree(t);
  return e;
}
""")
    subprocess.check_call([B.NVCC, *B.ARCH, "-O3", "-shared", "-Xcompiler", "-fPIC", "-I", B.CSRC, "-o", lib, src])
    L = ctypes.CDLL(lib)
    rng = np.random.default_rng(1)
    m = np.concatenate([rng.uniform(1, 2, 200000), 1 + np.arange(129) / 128.0, np.nextafter(1 + np.arange(1, 129) / 128.0, 0)])
    ex = rng.integers(-1000, 1000, m.size)
    ex[:100000] = 0
    special = np.array([0.0, -1.0, np.inf, np.nan, 1e-310])
    x = np.concatenate([np.ldexp(m, ex), special])
    X = torch.from_numpy(x).cuda()
    Y = torch.empty_like(X)
    torch.cuda.synchronize()
    assert L.run(ctypes.c_void_p(X.data_ptr()), ctypes.c_void_p(Y.data_ptr()), X.numel()) == 0
    y = Y.cpu().numpy()
    xf = x[:-5]
    e = np.floor(np.log2(xf))
    err = np.abs(y[:-5].astype(np.longdouble) - np.log(xf.astype(np.longdouble))).astype(np.float64)
    # ln m in fixed point: 2^-58; its conversion to a double below 1: 2^-54; the rounded ln 2 (off by 2.32e-17) times
    # the exponent; the last sum's rounding: half an ulp of the result
    bound = 2.0 ** -58 + 2.0 ** -54 + 2.4e-17 * np.abs(e) + 0.5 * np.spacing(np.abs(y[:-5]))
    print(f"LOG worst error / bound {(err / bound).max():.3f}")
    assert (err <= bound).all()
    with np.errstate(all="ignore"):
        np.testing.assert_array_equal(y[-5:-1], np.log(special[:-1]))
    assert abs(y[-1] - np.log(special[-1])) <= 1e-12
