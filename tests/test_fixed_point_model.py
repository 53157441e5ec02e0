"""CPU model of the fixed-point transforms of fft64.cuh: the header compiled for
the host, with the stages of fft.cuh's plan around it (first stage converts on
the sequence's block exponent, shifts up between the stages as
stockham_stage64 does, last stage rounds), against long double.

Tolerance: 4 u log2 N of the output's 2-norm (u = 2^-53), a few times the
rounding of FP64 butterflies.  Worst amplitudes (every number at the end of its
block) fill the 62 bits and would show an overflow as an error of order 1."""
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA = "/usr/local/cuda/include"

SRC = r"""
#include <cmath>
#include <cstdio>
#include <vector>
#include "fft64.cuh"
using namespace epfft;
static int lg2(int n) { return n <= 1 ? 0 : 1 + lg2(n / 2); }
static Tw64 tw(long n, long d, int S) {
  const long double a = 2.0L * 3.141592653589793238462643383279502884L * (n % d) / d, sc = ldexpl(1.0L, S);
  i64 re = llrintl(cosl(a) * sc), im = llrintl(-sinl(a) * sc);
  if (bal_lo(re) == INT32_MIN) re += 1;
  if (bal_lo(im) == INT32_MIN) im += 1;
  return Tw64{bal_lo(re), bal_hi(re), bal_lo(im), bal_hi(im)};
}
template <int R, bool INV>
static void stage(std::vector<C2<i64>>& z, int NS, int& em) {
  const int N = (int)z.size(), NJ = N / R;
  constexpr int LR = R == 2 ? 1 : R == 4 ? 2 : R == 8 ? 3 : 4;
  int sh = 0;
  if (NS > 1 && lg2(NS) + LR >= (LR == 4 ? 6 : 7)) {
    unsigned mx = 0;
    for (auto& v : z)
      for (i64 x : {v.re, v.im}) {
        const int h = (int)(x >> 32);
        const unsigned m = (unsigned)(h ^ (h >> 31));
        mx = m > mx ? m : mx;
      }
    const int lz = mx ? __builtin_clz(mx) : 32;
    sh = lz > 2 ? lz - 2 : 0;
    em -= sh;
  }
  std::vector<C2<i64>> o(N);
  for (int j = 0; j < NJ; j++) {
    C2<i64> v[R];
    for (int r = 0; r < R; r++) {
      v[r] = z[j + r * NJ];
      v[r].re = (i64)((unsigned long long)v[r].re << sh);
      v[r].im = (i64)((unsigned long long)v[r].im << sh);
    }
    if (NS > 1) {
      v[0].re = rshift<LR>(v[0].re);
      v[0].im = rshift<LR>(v[0].im);
      for (int r = 1; r < R; r++) cmul_hi<INV>(v[r].re, v[r].im, tw((long)(j % NS) * r, (long)NS * R, 64 - LR));
    }
    Bfly64<R, INV>::run(v);
    for (int r = 0; r < R; r++) o[(j / NS) * NS * R + j % NS + r * NS] = v[r];
  }
  z = o;
}
template <int LG>
static double out(i64 v, int em) { return from_fixed<LG>(v, em); }
static double outn(int lg, i64 v, int em) {
  switch (lg) {
    case 2: return out<2>(v, em); case 3: return out<3>(v, em); case 4: return out<4>(v, em);
    case 5: return out<5>(v, em); case 6: return out<6>(v, em); case 7: return out<7>(v, em);
    case 8: return out<8>(v, em); case 9: return out<9>(v, em); case 10: return out<10>(v, em);
    case 11: return out<11>(v, em); default: return out<12>(v, em);
  }
}
template <int G>
static i64 in(double x, int em) { return to_fixed<G>(x, em); }
template <bool INV>
static void run(std::vector<double>& x, int RM) {
  const int N = (int)x.size() / 2, LG = lg2(N), LR = lg2(RM);
  const int L0 = LG % LR == 0 ? (N < RM ? LG : LR) : LG % LR;
  unsigned mx = 0;
  for (double v : x) {
    const unsigned h = (unsigned)hi_word(v) & 0x7fffffffu;
    mx = h > mx ? h : mx;
  }
  int em = block_exp(mx);
  std::vector<C2<i64>> z(N);
  const bool low = em < FIX_LOW;
  const int ec = low ? em + 64 : em;
  for (int i = 0; i < N; i++) {
    auto f = [&](double v) {
      if (low) v = lift64(v);
      return L0 == 1 ? in<1>(v, ec) : L0 == 2 ? in<2>(v, ec) : L0 == 3 ? in<3>(v, ec) : in<4>(v, ec);
    };
    z[i].re = f(x[2 * i]);
    z[i].im = f(x[2 * i + 1]);
  }
  int NS = 1;
  for (int l = L0; NS < N; l = LR) {
    if (l == 1) stage<2, INV>(z, NS, em);
    else if (l == 2) stage<4, INV>(z, NS, em);
    else if (l == 3) stage<8, INV>(z, NS, em);
    else stage<16, INV>(z, NS, em);
    NS <<= l;
  }
  for (int i = 0; i < N; i++) {
    x[2 * i] = outn(LG, z[i].re, em);
    x[2 * i + 1] = outn(LG, z[i].im, em);
  }
}
int main() {
  int h[4];  // N, RM, inverse, sequences
  while (fread(h, sizeof(int), 4, stdin) == 4) {
    for (int s = 0; s < h[3]; s++) {
      std::vector<double> x(2 * h[0]);
      if (fread(x.data(), 8, x.size(), stdin) != x.size()) return 1;
      if (h[2]) run<true>(x, h[1]);
      else run<false>(x, h[1]);
      fwrite(x.data(), 8, x.size(), stdout);
    }
  }
}
"""


@pytest.fixture(scope="module")
def model(tmp_path_factory):
    if not shutil.which("g++") or not os.path.isdir(CUDA):
        pytest.skip("needs g++ and the CUDA headers")
    d = tmp_path_factory.mktemp("fft64")
    (d / "m.cpp").write_text(SRC)
    exe = str(d / "m")
    subprocess.run(["g++", "-std=c++17", "-O2", "-I", os.path.join(ROOT, "paper_0802_2488_gb300", "csrc"), "-I", CUDA,
                    str(d / "m.cpp"), "-o", exe], check=True)

    def run(x, RM, inverse):
        n, N = x.shape
        head = np.array([N, RM, int(inverse), n], dtype=np.int32).tobytes()
        raw = np.ascontiguousarray(x, dtype=np.complex128).tobytes()
        out = subprocess.run([exe], input=head + raw, stdout=subprocess.PIPE, check=True).stdout
        return np.frombuffer(out, dtype=np.complex128).reshape(n, N)
    return run


def _dft(x, inverse):
    """Long double transform, radix 2 (error some 1e-19)."""
    x = x.astype(np.clongdouble)
    n, N = x.shape
    if N == 1:
        return x
    e, o = _dft(x[:, ::2], inverse), _dft(x[:, 1::2], inverse)
    a = 2 * np.longdouble("3.14159265358979323846264338327950288") * np.arange(N // 2).astype(np.longdouble) / N
    t = (np.cos(a) + (1j if inverse else -1j) * np.sin(a)) * o
    return np.concatenate([e + t, e - t], axis=1)


def _err(got, ref):
    s = np.abs(ref).max(axis=1, keepdims=True)
    return (np.linalg.norm(np.abs((got - ref) / s).astype(np.float64), axis=1)
            / np.linalg.norm(np.abs(ref / s).astype(np.float64), axis=1)).max()


@pytest.mark.parametrize("inverse", [False, True])
@pytest.mark.parametrize("N,RM", [(4, 4), (8, 4), (16, 4), (64, 4), (128, 8), (256, 4), (512, 8), (1024, 8),
                                  (2048, 16), (4096, 16)])
def test_transform_against_long_double(model, N, RM, inverse):
    rng = np.random.default_rng(N + RM)
    c = lambda *s: rng.standard_normal(s) + 1j * rng.standard_normal(s)
    white = c(2, N)
    mean = c(2, N) + 1e6
    pixel = np.zeros((2, N), complex)
    pixel[0, N // 3], pixel[1, 0] = 1 - 2j, 1.0
    top = np.nextafter(2.0, 1.0)
    amp = (rng.integers(0, 2, (4, N)) * 2 - 1) * top + 1j * (rng.integers(0, 2, (4, N)) * 2 - 1) * top
    amp[0] = top * (1 + 1j)
    tol = 4 * 2.0 ** -53 * np.log2(N)
    for name, x in (("white", white), ("mean", mean), ("pixel", pixel), ("amplitude", amp),
                    ("large", 1e300 * white), ("small", 1e-250 * white), ("smallest", 2.0 ** -1000 * white)):
        assert _err(model(x, RM, inverse), _dft(x, inverse)) < tol, name


def test_zeros_and_non_finite_numbers(model):
    x = np.zeros((1, 64), complex)
    assert not model(x, 4, False).any()
    for bad in (np.nan, np.inf, -np.inf):
        x = np.ones((1, 64), complex)
        x[0, 5] = bad
        y = model(x, 4, False)
        assert np.isnan(y.real).all() and np.isnan(y.imag).all()
