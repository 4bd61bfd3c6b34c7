"""The roots and quotients of csrc/fastmath.cuh that stand for IEEE expressions (fine_*, and the FP64 steps under them)
against exactly rounded references: an error no larger than that of the expression they stand for, every FP32
significand and FP64 samples, and the values past the FP32 estimates' range. A small kernel that includes the header is
built here with nvcc and run through ctypes."""
import ctypes
import subprocess

import numpy as np
import pytest

from paper_1401_0838_gb300 import build as B

pytestmark = pytest.mark.gpu

SRC = r"""
#include <cuda_runtime.h>
#include "fastmath.cuh"
using namespace picgb;

template <typename T>
__global__ void k_fine(const T* x, const T* u2, T* o, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const T v = x[i], q = u2[i], gp = T(1) + q, ign = fine_rsqrt(gp);
  T* r = o + 8 * (size_t)i;
  r[0] = fine_rsqrt(v);
  r[1] = T(1) / sqrt(v);
  r[2] = fine_recip(v);
  r[3] = T(1) / v;
  r[4] = fine_two_over(v);
  r[5] = T(2) / v;
  r[6] = fine_kinetic(q, gp, ign);
  r[7] = q / (sqrt(T(1) + q) + T(1));
}

template <typename T>
static int run(const T* x, const T* u2, T* out, int n) {
  T *dx = nullptr, *du = nullptr, *dout = nullptr;
  const size_t b = sizeof(T) * (size_t)n;
  int rc = cudaMalloc(&dx, b) || cudaMalloc(&du, b) || cudaMalloc(&dout, 8 * b);
  if (!rc) rc = cudaMemcpy(dx, x, b, cudaMemcpyHostToDevice) || cudaMemcpy(du, u2, b, cudaMemcpyHostToDevice);
  if (!rc) {
    k_fine<T><<<(n + 255) / 256, 256>>>(dx, du, dout, n);
    rc = cudaGetLastError() != cudaSuccess || cudaMemcpy(out, dout, 8 * b, cudaMemcpyDeviceToHost) != cudaSuccess;
  }
  cudaFree(dx);
  cudaFree(du);
  cudaFree(dout);
  return rc;
}
// 1 where a pair's values differ from the single ones
__global__ void k_pairs(const float* x, const float* u2, float* o, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int j = (i * 7 + 1) % n;
  const float2 v = make_float2(x[i], x[j]), q = make_float2(u2[i], u2[j]), gp = make_float2(1.f + q.x, 1.f + q.y);
  const float2 ign = fine_rsqrt(gp), r = fine_rsqrt(v), t = fine_two_over(v), k = fine_kinetic(q, gp, ign);
  auto same = [](float a, float b) { return __float_as_int(a) == __float_as_int(b) || (a != a && b != b); };
  auto one = [&](float a, float b, float g, float vr, float vt, float vk, float vi) {
    const float gi = fine_rsqrt(g);
    return same(fine_rsqrt(a), vr) && same(fine_two_over(a), vt) && same(fine_kinetic(b, g, gi), vk) && same(gi, vi);
  };
  o[i] = one(v.x, q.x, gp.x, r.x, t.x, k.x, ign.x) && one(v.y, q.y, gp.y, r.y, t.y, k.y, ign.y) ? 0.f : 1.f;
}
extern "C" int run_pairs(const float* x, const float* u2, float* out, int n) {
  float *dx = nullptr, *du = nullptr, *dout = nullptr;
  const size_t b = sizeof(float) * (size_t)n;
  int rc = cudaMalloc(&dx, b) || cudaMalloc(&du, b) || cudaMalloc(&dout, b);
  if (!rc) rc = cudaMemcpy(dx, x, b, cudaMemcpyHostToDevice) || cudaMemcpy(du, u2, b, cudaMemcpyHostToDevice);
  if (!rc) {
    k_pairs<<<(n + 255) / 256, 256>>>(dx, du, dout, n);
    rc = cudaGetLastError() != cudaSuccess || cudaMemcpy(out, dout, b, cudaMemcpyDeviceToHost) != cudaSuccess;
  }
  cudaFree(dx);
  cudaFree(du);
  cudaFree(dout);
  return rc;
}
extern "C" int run_f(const float* x, const float* u, float* o, int n) { return run(x, u, o, n); }
extern "C" int run_d(const double* x, const double* u, double* o, int n) { return run(x, u, o, n); }
"""


@pytest.fixture(scope="module")
def fine(tmp_path_factory):
    d = tmp_path_factory.mktemp("fine")
    src, so = d / "fine.cu", d / "libfine.so"
    src.write_text(SRC)
    r = subprocess.run([B.nvcc(), "-shared", "-Xcompiler", "-fPIC", "-O3", "-std=c++17", *B.ARCH, "-I", B.CSRC, "-o",
                        str(so), str(src), "-lcudart"], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    lib = ctypes.CDLL(str(so))

    def call(x, u2):
        out = np.empty((len(x), 8), x.dtype)
        f = lib.run_f if x.dtype == np.float32 else lib.run_d
        assert f(*(ctypes.c_void_p(a.ctypes.data) for a in (x, u2, out)), ctypes.c_int(len(x))) == 0
        return out

    call.lib = lib
    return call


def _ulps(got, exact):
    """Error of got in units of its own type's spacing at the exact value (which has more bits)."""
    return np.abs(got.astype(exact.dtype) - exact) / np.spacing(np.abs(exact).astype(got.dtype)).astype(exact.dtype)


def _check(r, x, u2, wide):
    X, U = x.astype(wide), u2.astype(wide)
    one = wide(1)
    exact = [one / np.sqrt(X), one / X, wide(2) / X, U / (np.sqrt(one + U) + one)]
    for k, e in enumerate(exact):
        fine, ieee = _ulps(r[:, 2 * k], e).max(), _ulps(r[:, 2 * k + 1], e).max()
        assert fine <= ieee * (1 + 1e-9), (k, fine, ieee)


def test_fp32_every_significand(fine):
    m = np.arange(1 << 23, dtype=np.uint32)
    rng = np.random.default_rng(1)
    for e in (0, 1):  # the root's two exponent classes
        x = (m + np.uint32((127 + e) << 23)).view(np.float32)
        u2 = (10.0 ** rng.uniform(-12, 10, len(m))).astype(np.float32)
        _check(fine(x, u2), x, u2, np.float64)


def test_fp64_samples(fine):
    rng = np.random.default_rng(2)
    n = 1 << 20
    x = np.ldexp(rng.uniform(1, 2, n), rng.integers(0, 60, n))
    u2 = 10.0 ** rng.uniform(-16, 12, n)
    r = fine(x, u2)
    if np.finfo(np.longdouble).nmant < 63:
        pytest.skip("no wider type for the reference")
    _check(r, x, u2, np.longdouble)


def test_pairs_equal_single_values(fine):
    rng = np.random.default_rng(3)
    n = 1 << 20
    x = np.ldexp(rng.uniform(1, 2, n), rng.integers(0, 128, n)).astype(np.float32)
    x[:4] = [np.inf, np.nan, 2.0 ** 126, 1.0]
    u2 = (10.0 ** rng.uniform(-12, 30, n)).astype(np.float32)
    out = np.empty(n, np.float32)
    assert fine.lib.run_pairs(*(ctypes.c_void_p(a.ctypes.data) for a in (x, u2, out)), ctypes.c_int(n)) == 0
    assert not out.any(), x[out != 0][:5]


@pytest.mark.parametrize("T", [np.float32, np.float64])
def test_range(fine, T):
    # past 2^126 (the FP32 reciprocal estimate's end) and, in FP64, past FP32's largest value; infinities and NaN
    x = np.array([2.0 ** 120, 2.0 ** 125, 2.0 ** 126, 1.5 * 2.0 ** 126, 2.0 ** 127, 3.4e38] +
                 ([1e40, 1e80, 1e300] if T is np.float64 else []) + [np.inf, np.nan], dtype=T)
    u2 = np.where(np.isfinite(x), x, T(1)).astype(T) if T is np.float64 else np.ones(len(x), T)
    r = fine(x, u2)
    for k in range(4):
        a, b = r[:, 2 * k], r[:, 2 * k + 1]
        ok = (a == b) | (np.isnan(a) & np.isnan(b)) | (np.abs(a - b) <= 2 * np.spacing(np.abs(b)))
        assert ok.all(), (k, x[~ok], a[~ok], b[~ok])


def test_kinetic_energy_over_momenta():
    # pic_energy's gamma - 1, from FP32 estimates refined in FP64, one particle at a time: no cancellation at small u,
    # the IEEE expression past the estimates' range
    from tests._pic import P, make_cfg, uniform_weight

    cfg = make_cfg(nx=8, nz=8, gamma=1.0, precision=1, ppc=1)
    h = P.pic_create(cfg)
    try:
        for u in [0.0, 1e-30, 1e-12, 1e-6, 1e-3, 0.1, 0.5, 1.0, 2.7, 130.0, 1e4, 1e9, 3e14, 1e16, 1e40, 1e150]:
            part = {"cell": np.zeros(1, np.int32), "species": np.zeros(1, np.int32), "id": np.zeros(1, np.uint32), "oy": None,
                    "w": None, "dux": np.full(1, u), "duy": np.zeros(1), "duz": np.zeros(1), "ox": np.full(1, 0.5),
                    "oz": np.full(1, 0.5)}
            P.pic_set_state(h, P.make_state(P.PIC_HOST, None, part))
            U = np.longdouble(u) ** 2
            want = np.longdouble(uniform_weight(cfg)) * (U / (np.sqrt(1 + U) + 1))
            assert abs(np.longdouble(P.pic_energy(h)["k"]) - want) <= 2.0 ** -50 * want, u
    finally:
        P.pic_destroy(h)
