"""The float-pair sums of the block assembly (csrc/dg_pairs.cuh) have the bits of
the FP64 form they stand for: random rows, rows that cancel, sums at and beside
the boundary between two floats, and values at the ends of the range."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2002_04222_gb300", "csrc")

SOURCE = """
#include <cuda_runtime.h>
#include "dg_pairs.cuh"
template <int N>
__global__ void rows(const double* m, const float* x, long long n, float* pairs, float* fp64) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= n) return;
  float mh[N], ml[N];
  for (int k = 0; k < N; ++k) {
    mh[k] = (float)m[i * N + k];
    ml[k] = (float)(m[i * N + k] - (double)mh[k]);
  }
  pairs[2 * i] = dg::pair_row<N>(mh, ml, m + i * N, x + i * N, 1);
  fp64[2 * i] = dg::fp64_row<N>(m + i * N, x + i * N, 1);
  pairs[2 * i + 1] = dg::pair_scaled(mh[0], ml[0], m[i * N], x[i * N], i % 7 == 0 ? 1.0 : 0.0);
  fp64[2 * i + 1] = dg::fp64_scaled(m[i * N], x[i * N], i % 7 == 0 ? 1.0 : 0.0);
}
extern "C" int run(int N, const double* m, const float* x, long long n, float* p, float* f) {
  const int g = (int)((n + 255) / 256);
  if (N == 3) rows<3><<<g, 256>>>(m, x, n, p, f);
  else if (N == 4) rows<4><<<g, 256>>>(m, x, n, p, f);
  else if (N == 5) rows<5><<<g, 256>>>(m, x, n, p, f);
  else rows<7><<<g, 256>>>(m, x, n, p, f);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    from paper_2002_04222_gb300.build import ARCH, nvcc
    d = tmp_path_factory.mktemp("pairs")
    (d / "p.cu").write_text(SOURCE)
    subprocess.run([nvcc(), *ARCH, "-O3", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-I", CSRC,
                    str(d / "p.cu"), "-o", str(d / "p.so"), "-lcudart"], check=True)
    f = ctypes.CDLL(str(d / "p.so")).run
    f.argtypes = [ctypes.c_int, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_longlong,
                  ctypes.c_void_p, ctypes.c_void_p]
    return f


def inputs(N, kind, n, rng):
    m = rng.standard_normal((n, N)) * 10.0 ** rng.uniform(-2, 4, (n, N))
    x = rng.standard_normal((n, N)).astype(np.float32) * np.float32(10.0) ** rng.integers(-6, 6, (n, 1))
    if kind == "cancel":             # the last term takes away the others' sum, to 2^-j
        s = (m[:, :-1] * x[:, :-1]).sum(1)
        m[:, -1] = -s / x[:, -1] * (1 + 2.0 ** -rng.integers(1, 60, n).astype(float))
    elif kind == "boundary":         # the sum lies at half a unit of a float, give or take 2^-j of it
        s = (m[:, :-1] * x[:, :-1]).sum(1)
        a = rng.standard_normal(n).astype(np.float32) * np.float32(100.0)
        half = 0.5 * np.abs(np.spacing(a)).astype(float)
        t = a.astype(float) + half * (1 + rng.choice([-1, 0, 1], n) * 2.0 ** -rng.integers(2, 40, n).astype(float))
        x[:, -1] = 1.0
        m[:, -1] = t - s
    elif kind == "ends":             # zeros, ties, the smallest and largest values, what is not finite
        v = np.array([0.0, -0.0, 1.0, 2.0, 1 + 2.0 ** -23, 1e-38, 1e-45, 3e38, np.inf, np.nan], np.float32)
        x = v[rng.integers(0, len(v), (n, N))]
        w = np.array([0.0, 1.0, -1.0, 1 + 2.0 ** -24, 1 - 2.0 ** -25, 2.0 ** -24, 1e-30, -1e30])
        m = w[rng.integers(0, len(w), (n, N))]
    return m, x


@pytest.mark.parametrize("kind", ["random", "cancel", "boundary", "ends"])
@pytest.mark.parametrize("N", [3, 4, 5, 7])
def test_pairs_have_the_bits_of_fp64(run, N, kind):
    n = 500000
    m, x = inputs(N, kind, n, np.random.default_rng(N))
    md, xd = torch.from_numpy(np.ascontiguousarray(m)).cuda(), torch.from_numpy(np.ascontiguousarray(x)).cuda()
    p, f = (torch.zeros(2 * n, dtype=torch.float32, device="cuda") for _ in range(2))
    torch.cuda.synchronize()
    assert run(N, md.data_ptr(), xd.data_ptr(), n, p.data_ptr(), f.data_ptr()) == 0
    same = (p.view(torch.int32) == f.view(torch.int32)) | (torch.isnan(p) & torch.isnan(f)) \
        | ((p == 0) & (f == 0))
    assert bool(same.all()), int((~same).sum())
