"""The arithmetic that the kernels build for themselves, compiled into a small library of its own and
compared with what it stands for:

* exp_neg within 0.53 ulp of e^a (long double, 64 bits of mantissa or more: another 2^-10 ulp) for a in
  [-700, 0], 0 below -708;
* quotient(a, b, 1 / b): CUDA's a / b, bit for bit, for numerators above 2^-100;
* df_split_int: df_split, value for value, over the whole of FP64's range that FP32 holds, and zeros.
"""
import ctypes
import os
import subprocess

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "common.cuh"
#include "exp64.cuh"
using namespace pdd;
__global__ void k_exp(int n, const double *a, double *out) {
    __shared__ double2 tab[kExpTab];
    for (int q = threadIdx.x; q < kExpTab; q += blockDim.x) tab[q] = kExp2Tab[q];
    __syncthreads();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = exp_neg(a[i], tab);
}
__global__ void k_quot(int n, const float *a, const float *b, float *out, float *want) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    out[i] = quotient(a[i], b[i], 1.0f / b[i]);
    want[i] = a[i] / b[i];
}
__global__ void k_split(int n, const double *v, float2 *out, float2 *want) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    out[i] = df_split_int(v[i]);
    want[i] = df_split(v[i]);
}
extern "C" int run_exp(int n, const double *a, double *out) {
    k_exp<<<(n + 255) / 256, 256>>>(n, a, out);
    return (int)cudaDeviceSynchronize();
}
extern "C" int run_quot(int n, const float *a, const float *b, float *out, float *want) {
    k_quot<<<(n + 255) / 256, 256>>>(n, a, b, out, want);
    return (int)cudaDeviceSynchronize();
}
extern "C" int run_split(int n, const double *v, float2 *out, float2 *want) {
    k_split<<<(n + 255) / 256, 256>>>(n, v, out, want);
    return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    from paper_2311_08946_gb300 import build

    d = tmp_path_factory.mktemp("arith")
    src, so = str(d / "arith.cu"), str(d / "arith.so")
    with open(src, "w") as f:
        f.write(SOURCE)
    subprocess.run([build.nvcc(), *build.ARCH, *build.FLAGS, "-I", build.CSRC, "-shared", "-o", so, src], check=True,
                   capture_output=True)
    assert os.path.exists(so)
    return ctypes.CDLL(so)


def _ptr(t):
    return ctypes.c_void_p(t.data_ptr())


def test_exp_neg(lib):
    rng = np.random.default_rng(1)
    a = -np.concatenate([rng.uniform(0, 700, 200000), np.exp2(rng.uniform(-60, 9, 200000)), [0.0]])
    x = torch.tensor(a, device="cuda")
    out = torch.empty_like(x)
    assert lib.run_exp(x.numel(), _ptr(x), _ptr(out)) == 0
    want = np.exp(a.astype(np.longdouble))
    ulp = np.spacing(want.astype(np.float64)).astype(np.longdouble)
    assert (np.abs(out.cpu().numpy().astype(np.longdouble) - want) / ulp).max() <= 0.53 + 2.0 ** -10
    x = torch.tensor([-709.0, -745.0, -1e5, -1e300, -np.inf], dtype=torch.float64, device="cuda")
    out = torch.ones_like(x)
    assert lib.run_exp(x.numel(), _ptr(x), _ptr(out)) == 0 and not out.any()


def test_quotient(lib):
    rng = np.random.default_rng(2)
    n = 1 << 21
    mant = lambda: rng.integers(1 << 23, 1 << 24, n).astype(np.float64)
    b = mant() * np.exp2(rng.integers(-23, 20, n))
    q = np.where(rng.random(n) < 0.5, np.exp2(-rng.uniform(0, 90, n)), rng.uniform(0, 4, n) + 2.0 ** -90)
    a = b * q * rng.choice([-1.0, 1.0], n)
    # (reciprocals just above a power of 2)
    b[: n // 8] = (2.0 ** 24 - rng.integers(1, 64, n // 8)) * np.exp2(rng.integers(-50, 20, n // 8))
    a, b = (torch.tensor(v.astype(np.float32), device="cuda") for v in (a, b))
    out, want = torch.empty_like(a), torch.empty_like(a)
    assert lib.run_quot(n, _ptr(a), _ptr(b), _ptr(out), _ptr(want)) == 0
    assert torch.equal(out, want)


def test_df_split_int(lib):
    rng = np.random.default_rng(3)
    n = 1 << 21
    m = rng.integers(0, 1 << 52, n, dtype=np.uint64)
    tie = rng.random(n)
    m = np.where(tie < 0.1, (m & ~np.uint64(0x1FFFFFFF)) | np.uint64(0x10000000), m)            # ties
    m = np.where((tie > 0.1) & (tie < 0.2), m | np.uint64(0xFFFFFE0000000), m)                  # carries
    e = rng.integers(1023 - 160, 1023 + 127, n, dtype=np.uint64)
    s = rng.integers(0, 2, n, dtype=np.uint64)
    v = ((s << np.uint64(63)) | (e << np.uint64(52)) | m).view(np.float64)
    v = np.concatenate([v, [0.0, -0.0, 5e-324, -1e-310]])
    x = torch.tensor(v, device="cuda")
    out, want = (torch.empty(v.size, 2, dtype=torch.float32, device="cuda") for _ in range(2))
    assert lib.run_split(v.size, _ptr(x), _ptr(out), _ptr(want)) == 0
    assert torch.equal(out, want)                        # (-0 equals 0)
