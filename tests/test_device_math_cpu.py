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
