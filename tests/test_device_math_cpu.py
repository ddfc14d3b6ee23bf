"""The kernels' arithmetic compiled for the host from the kernels' own headers,
against 64-bit (or exact) computations of the same."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2507_17175_gb300 import build_lib

SOURCE = r"""
#include "qpe_dft.cuh"
#include "qpe_fixed.cuh"
using namespace qpe;
// the same DFT with every twiddle product formed as a product and an FMA, twiddles
// rounded from the 64-bit values
template <typename C, int K> static void stages(C* x, const double2* w) {
  using R = typename real_of<C>::type;
  constexpr int N = 1 << K;
  for (int h = N / 2; h >= 1; h /= 2)
    for (int g = 0; g < N; g += 2 * h)
      for (int p = 0; p < h; ++p) {
        const C u = x[g + p], v = x[g + p + h], d = csub(u, v);
        const R c = (R)w[p * (16 / h)].x, s = (R)w[p * (16 / h)].y;
        x[g + p] = cadd(u, v);
        x[g + p + h] = p ? mk(fma(d.x, c, -(d.y * s)), fma(d.y, c, d.x * s)) : d;
      }
  for (int i = 0; i < N; ++i) {
    int r = 0;
    for (int b = 0; b < K; ++b) r |= ((i >> b) & 1) << (K - 1 - b);
    if (r > i) { const C t = x[i]; x[i] = x[r]; x[r] = t; }
  }
}
template <typename C, int K> static void dft(C* x, int64_t n, const double2* w, int ours) {
  for (int64_t t = 0; t < n; ++t, x += 1 << K) {
    if (ours) dft_k<C, K>(*reinterpret_cast<C(*)[1 << K]>(x));
    else stages<C, K>(x, w);
  }
}
template <typename C> static void any(C* x, int k, int64_t n, const double2* w, int ours) {
  switch (k) {
    case 1: dft<C, 1>(x, n, w, ours); break;
    case 2: dft<C, 2>(x, n, w, ours); break;
    case 3: dft<C, 3>(x, n, w, ours); break;
    case 4: dft<C, 4>(x, n, w, ours); break;
    default: dft<C, 5>(x, n, w, ours); break;
  }
}
extern "C" void dft32(float2* x, int k, int64_t n, const double2* w, int ours) { any(x, k, n, w, ours); }
// per row, per x 7 weight sums -> the sum of the squares of the fixed-point values
extern "C" int squares(const float* acc, int64_t rows, int per, double* out) {
  for (int64_t r = 0; r < rows; ++r) {
    OtSquares s;
    for (int i = 0; i < per; ++i) {
      uint32_t u[7];
      memcpy(u, acc + (r * per + i) * 7, sizeof u);
      s.add(ot_weights_fix(u[0], u[1], u[2], u[3], u[4], u[5], u[6]));
    }
    out[r] = s.value();
  }
  return kOtFix;
}
extern "C" void sums_of_squares(const long long* x, int64_t rows, int per, double* out) {
  for (int64_t r = 0; r < rows; ++r) {
    OtSquares s;
    for (int i = 0; i < per; ++i) s.add(x[r * per + i]);
    out[r] = s.value();
  }
}
extern "C" void dft64(double2* x, int k, int64_t n, const double2* w, int ours) { any(x, k, n, w, ours); }
"""


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    where = tmp_path_factory.mktemp("host")
    src, lib = where / "host.cu", where / "host.so"
    src.write_text(SOURCE)
    subprocess.run([build_lib.nvcc(), *build_lib.ARCH, "-O1", "-std=c++17", "-shared", "-Xcompiler", "-fPIC,-ffp-contract=off",
                    "-I", build_lib.CSRC, "-I", os.path.join(os.path.dirname(build_lib.HERE), "include"),
                    "-o", str(lib), str(src)], check=True)
    return ctypes.CDLL(str(lib))


def _p(a):
    return ctypes.c_void_p(a.ctypes.data)


@pytest.mark.parametrize("dtype", [np.complex64, np.complex128])
@pytest.mark.parametrize("k", [1, 2, 3, 4, 5])
def test_register_dft_is_as_accurate_as_products_and_fmas(host, k, dtype):
    """rms error against a transform in more bits, over 20,000 random inputs: no larger than
    with every twiddle product as a product and an FMA."""
    wide = np.complex128 if dtype is np.complex64 else np.clongdouble
    if dtype is np.complex128 and np.finfo(np.longdouble).nmant < 60:
        pytest.skip("no longer type than float64")
    rng = np.random.default_rng(3)
    n = 1 << k
    x = (rng.standard_normal((20000, n)) + 1j * rng.standard_normal((20000, n))).astype(dtype)
    real = np.finfo(wide).dtype.type
    ang = np.arange(n, dtype=real) * (np.arccos(real(-1)) / real(n // 2))
    W = np.cos(ang) - 1j * np.sin(ang)
    F = W[np.outer(np.arange(n), np.arange(n)) % n]
    want = x.astype(wide) @ F
    w = np.exp(-2j * np.pi * np.arange(32) / 32)
    err = []
    for ours in (1, 0):
        got = x.copy()
        (host.dft32 if dtype is np.complex64 else host.dft64)(_p(got), k, ctypes.c_int64(len(x)), _p(w), ours)
        err.append(float(np.sqrt(np.mean(np.abs(got.astype(wide) - want) ** 2))))
    assert err[0] <= err[1] * (1 + 1e-6), err


def nearest(got, want):
    """``got`` is the integer ``want`` rounded to 53 bits (a tie may go up)."""
    bits = want.bit_length()
    return abs(int(got) - want) <= (1 << (bits - 54) if bits > 53 else 0)


def test_squares_keep_every_bit_of_the_weight_sums_from_2_10(host):
    """Sums of |W|^2 from the accumulators' weight sums: every bit of floor(E / 2^10) counts,
    E = sum_w acc_w 2^(8 (6 - w))."""
    rng = np.random.default_rng(4)
    acc = np.zeros((1200, 8, 7), dtype=np.float32)
    for i, row in enumerate(acc):
        lead = i % 7  # the weights above are zero: small E count as well as large
        row[:, lead:] = rng.integers(-(1 << 21) + 1, 1 << 21, (8, 7 - lead))
        row[:, 0] = np.clip(row[:, 0], -(1 << 18), 1 << 18)
    out = np.empty(len(acc))
    unit = host.squares(_p(acc), ctypes.c_int64(len(acc)), 8, _p(out))
    for row, got in zip(acc, out):
        E = [sum(int(v) << (8 * (6 - w)) for w, v in enumerate(a)) for a in row]
        want = sum((e >> 10) ** 2 for e in E)
        assert nearest(got * 2.0 ** (2 * unit - 20), want)


def test_sums_of_squares_over_their_range(host):
    """Eight squares of even numbers of every magnitude up to the bound, exactly."""
    rng = np.random.default_rng(5)
    top = int(2 ** 61.6)
    edges = [0, 2, -2, 2 ** 31 - 2, 2 ** 31, -(2 ** 31), 2 ** 32 - 2, 2 ** 32, 2 ** 32 + 2 ** 31, 2 ** 54 + 2,
             (top - 2) & ~1, -((top - 2) & ~1), 2 ** 61 + 2 ** 31, 2 ** 61 - 2 ** 31]
    rows = [[e] + [0] * 7 for e in edges] + [[e] * 8 for e in edges]
    for bits in range(1, 62):
        rows += (rng.integers(-(1 << bits), 1 << bits, (40, 8)) & ~1).tolist()
    x = np.array(rows, dtype=np.int64)
    out = np.empty(len(x))
    host.sums_of_squares(_p(x), ctypes.c_int64(len(x)), 8, _p(out))
    for row, got in zip(rows, out):
        assert nearest(got, sum(int(v) ** 2 for v in row)), row
