"""The 64-bit block fixed-point arithmetic of the FP64 transforms
(csrc/fft64.cuh), compiled for the host: against an FFT in extended precision
over lengths, spectra and exponents (CPU), and through the library (GPU)."""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

from _helpers import compare_uvh, gpu, turbulence

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SRC = r"""
#include "fft64.cuh"
using namespace lm;
template <int S> static void run(int L, double* d) {
  const int N = 1 << L, G = N / 8;
  std::vector<TwFx> tw(N);
  fft_twiddle_table_fx(L, tw.data());
  unsigned mx = 0, sum = 0;
  for (int i = 0; i < 2 * N; ++i) mx = std::max(mx, fx_abs_hi(d[i]));
  const int emax = std::max((int)(mx >> 20), FX_EMIN);
  std::vector<cfx> x(N), y(N);
  for (int j = 0; j < G; ++j) {
    unsigned ms = 0;
    for (int n = j; n < N; n += G) x[n] = cfx{fx_from_double(d[2 * n], emax, ms), fx_from_double(d[2 * n + 1], emax, ms)};
    sum += fx_sum_units(ms);
  }
  const int Dn = fx_sum_shift(sum);
  int drop = 0, lNs = 0;
  for (int p = 0; p < fft_num_passes(L); ++p) {
    const int l = fft_pass_lr(L, p), R = 1 << l, Ns = 1 << lNs;
    const int D = std::min(3 * p, Dn), sh = D - drop, half = (1 << sh) >> 1;
    drop = D;
    for (int j = 0; j < N / R; ++j) {
      const int k = j % Ns;
      cfx v[8];
      for (int r = 0; r < R; ++r) {
        v[r] = x[j + r * (N / R)];
        if (p) v[r] = r == 0 ? fx_shift(v[r], sh, half) : fx_twiddle<S>(v[r], tw[r * Ns + k - 1], sh, half);
      }
      if (R == 8) fdft_r<S, 8>(v);
      else if (R == 4) fdft_r<S, 4>(v);
      else fdft_r<S, 2>(v);
      for (int q = 0; q < R; ++q) y[(j - k) * R + k + q * Ns] = v[q];
    }
    x.swap(y);
    lNs += l;
  }
  for (int n = 0; n < N; ++n) {
    d[2 * n] = fx_to_double(x[n].x, emax + drop);
    d[2 * n + 1] = fx_to_double(x[n].y, emax + drop);
  }
}
extern "C" void fx_fft(int L, int sign, double* d) { sign < 0 ? run<-1>(L, d) : run<1>(L, d); }
"""


@pytest.fixture(scope="module")
def fx(tmp_path_factory):
    inc = "/usr/local/cuda/include"
    if shutil.which("g++") is None or not os.path.exists(os.path.join(inc, "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    d = tmp_path_factory.mktemp("fx")
    (d / "fx.cpp").write_text("#include <algorithm>\n" + SRC)
    so = str(d / "fx.so")
    subprocess.run(["g++", "-O1", "-std=c++17", "-fPIC", "-shared", "-I" + inc,
                    "-I" + os.path.join(ROOT, "paper_2208_02682_gb300", "csrc"), str(d / "fx.cpp"), "-o", so],
                   check=True)
    lib = C.CDLL(so)
    lib.fx_fft.argtypes = [C.c_int, C.c_int, C.POINTER(C.c_double)]
    return lib


def _inputs(N, rng, kind):
    z = rng.standard_normal(N) + 1j * rng.standard_normal(N)
    k = np.minimum(np.arange(N), N - np.arange(N))
    if kind == "steep":
        z *= (1.0 + k) ** -3.0
    elif kind == "spike":
        z = np.where(k == 3, z, 1e-3 * z)
    elif kind == "mode":
        z = np.where(np.arange(N) == N // 5, z, 0)
    elif kind == "scales":
        z = z.real + 1e-9j * z.imag
    return z


@pytest.mark.parametrize("L", range(4, 12))
@pytest.mark.parametrize("kind", ["white", "steep", "spike", "mode", "scales"])
def test_host_transform(fx, L, kind):
    """Relative 2-norm error below 2 units of FP64 (the bound of fft64.cuh's
    header plus the output rounding; FP64 butterflies reach 2e-16), at
    exponents from the smallest held to near the top of the range."""
    N = 1 << L
    rng = np.random.default_rng(17 + L)
    for scale in (1.0, 2.0 ** -880, 2.0 ** 900):
        for sign in (-1, 1):
            z = _inputs(N, rng, kind)
            ref = np.fft.fft(z.astype(np.clongdouble)) if sign < 0 else np.fft.ifft(z.astype(np.clongdouble)) * N
            d = np.ascontiguousarray(z * scale).view(np.float64)
            fx.fx_fft(L, sign, d.ctypes.data_as(C.POINTER(C.c_double)))
            got = d.view(np.complex128).astype(np.clongdouble) / scale
            err = np.sqrt(np.sum(np.abs(got - ref) ** 2) / np.sum(np.abs(ref) ** 2))
            assert err < 2.0 * 2.0 ** -53, (scale, sign, float(err))


def test_host_zeros(fx):
    d = np.zeros(64)
    fx.fx_fft(5, 1, d.ctypes.data_as(C.POINTER(C.c_double)))
    assert not d.any()


@pytest.mark.gpu
@pytest.mark.parametrize("N", [16, 32, 64, 256, 512, 2048])
@pytest.mark.parametrize("amp", [1.0, 1e-100])
def test_step_scales(N, amp):
    """One FP64 step against the oracle, also with tiny fields (linear flow)."""
    from oracle import SWOracle
    lm = gpu()
    u, v, h = turbulence(N)
    u, v, h = amp * u, amp * v, (h if amp == 1.0 else np.ones_like(h))
    o = SWOracle(N, 5e-3, u, v, h)
    o.step(1)
    g = lm.sw_create(lm.make_params(N, 5e-3, precision="f64"), np.ascontiguousarray(np.stack([u, v, h])))
    try:
        lm.sw_step(g, 1)
        out = np.zeros((3, N, N))
        lm.sw_get_fields(g, out)
    finally:
        lm.sw_destroy(g)
    e = compare_uvh(out, np.stack(o.fields()))
    assert e["u"] < 1e-12 and e["v"] < 1e-12 and (amp != 1.0 or e["h"] < 1e-12), e


@pytest.mark.gpu
@pytest.mark.parametrize("N", [64, 512])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_nonfinite_input(N, bad):
    """A non-finite value leaves no finite field behind, as in FP64 arithmetic."""
    lm = gpu()
    uvh = np.ascontiguousarray(np.stack(turbulence(N)))
    uvh[0, 3, 5] = bad
    g = lm.sw_create(lm.make_params(N, 5e-3, precision="f64"), uvh)
    try:
        lm.sw_step(g, 1)
        out = np.zeros((3, N, N))
        lm.sw_get_fields(g, out)
    finally:
        lm.sw_destroy(g)
    assert not np.isfinite(out).any()
