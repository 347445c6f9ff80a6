"""The FP64 quotient and widening of the kernels against CUDA's own division and
conversion, over the exponent range and the values where they branch."""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCE = r"""
#include "kernels.cuh"
__global__ void ops(const double *a, const double *s, int n, double *out)
{
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= n) return;
    out[q] = sbp::quot64(a[q], s[q]);
    out[n + q] = a[q] / s[q];
    const double gam = 1e-3 + fmod(fabs(s[q]), 0.5);       // an absorbing node: old, increment, gamma
    out[2 * n + q] = sbp::sat_finish(a[q], 0.25 * a[q], gam);
    out[3 * n + q] = fma(1.0 - gam, a[q], 0.25 * a[q]) / (1.0 + gam);
}
__global__ void wide(const float *f, int n, double *out)
{
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= n) return;
    out[q] = sbp::to_double(f[q]);
    out[n + q] = sbp::widen<double>(f[q]);
}
extern "C" int run_ops(const double *a, const double *s, int n, double *out)
{
    ops<<<(n + 255) / 256, 256>>>(a, s, n, out);
    return (int)cudaDeviceSynchronize();
}
extern "C" int run_wide(const float *f, int n, double *out)
{
    wide<<<(n + 255) / 256, 256>>>(f, n, out);
    return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("arith")
    (d / "ops.cu").write_text(SOURCE)
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "-Xcompiler", "-fPIC",
                    "-shared", "-I", os.path.join(ROOT, "paper_2206_00638_gb300", "csrc"), "-o", str(d / "ops.so"),
                    str(d / "ops.cu")], check=True)
    return C.CDLL(str(d / "ops.so"))


def _ops(lib, a, s):
    ta, ts = torch.tensor(a, device="cuda"), torch.tensor(s, device="cuda")
    out = torch.empty((4, len(a)), dtype=torch.float64, device="cuda")
    assert lib.run_ops(C.c_void_p(ta.data_ptr()), C.c_void_p(ts.data_ptr()), len(a), C.c_void_p(out.data_ptr())) == 0
    return out.cpu().numpy()


def _ulps(x, ref):
    return np.abs(x - ref) / np.spacing(np.abs(ref))


def test_quotient(lib):
    """The quotient's error before its one rounding is below 2^-80 relative (the reciprocal's 2^-42
    squared), so it differs from the rounded quotient only next to a tie: never more than one ulp,
    and fewer than one in 2^20."""
    r = np.random.default_rng(3)
    n = 1 << 21
    a = r.uniform(1, 2, n) * 2.0 ** r.integers(-200, 200, n) * r.choice([-1, 1], n)
    s = r.uniform(1, 2, n) * 2.0 ** np.where(r.random(n) < 0.5, r.integers(-4, 12, n), r.integers(-130, 130, n))
    s[:4] = 2.0 ** np.array([-100, -101, 99, 100.0])
    s[4:8] = np.nextafter(s[:4], 0)
    q, q0, f, f0 = _ops(lib, a, s)
    for got, ref in ((q, q0), (f, f0)):
        u = _ulps(got, ref)
        assert u.max() <= 1 and np.count_nonzero(u) <= max(2, n >> 20), (u.max(), np.count_nonzero(u))


def test_special_values(lib):
    a = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 1e308, -1e308, 5e-324])
    s = np.full(len(a), 0.75)
    q, q0 = _ops(lib, a, s)[:2]
    assert np.array_equal(q[:-1], q0[:-1], equal_nan=True)
    assert abs(q[-1] - q0[-1]) <= 5e-324


def test_widening_is_exact(lib):
    r = np.random.default_rng(4)
    bits = np.concatenate([r.integers(0, 1 << 32, 1 << 20, dtype=np.uint32),
                           np.array([0, 1, 0x7fffff, 0x800000, 0x7f7fffff, 0x7f800000, 0x80000000, 0x80000001,
                                     0xff800000, 0x3f800000], dtype=np.uint32)])
    f = bits.view(np.float32)
    t = torch.tensor(f, device="cuda")
    out = torch.empty((2, len(f)), dtype=torch.float64, device="cuda")
    assert lib.run_wide(C.c_void_p(t.data_ptr()), len(f), C.c_void_p(out.data_ptr())) == 0
    any_value, normal = out.cpu().numpy()
    with np.errstate(invalid="ignore"):
        ref = f.astype(np.float64)
    assert np.array_equal(any_value, ref, equal_nan=True)
    plain = (f >= np.finfo(np.float32).tiny) & np.isfinite(f)
    assert np.array_equal(normal[plain], ref[plain])
