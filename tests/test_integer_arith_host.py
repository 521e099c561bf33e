"""The integer d-bar and the integer quotient (eik_exact.cuh), compiled for the
host: d-bar against bisection over its definition on 64-bit floats, the quotient
against the host's division.  The approximate FP32 functions that start them are
replaced by ones with random errors beyond the device's (a few 2^-23), on which
no result may depend; a Scaled kept over several evaluations of a cell gives what
a new one gives."""
import pytest

from . import device_fragments as frag

HEAD = r"""
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <random>
#include <utility>
#define __forceinline__ inline
#define __device__
#define EIK_HD
typedef unsigned long long u64;
static u64 bits(double x) { u64 u; std::memcpy(&u, &x, 8); return u; }
static double dbl(u64 u) { double x; std::memcpy(&x, &u, 8); return x; }
namespace eik { namespace ig {
static std::mt19937_64 noise(1);
inline float off(float x, float by) { return x * (1.0f + by * static_cast<float>(static_cast<int>(noise() % 2001) - 1000) / 1000.0f); }
inline float int_as_f(int i) { float f; std::memcpy(&f, &i, 4); return f; }
inline float sqrt_f(float x) { return off(std::sqrt(x), 1e-6f); }
inline float rcp_f(float x) { return off(1.0f / x, 3e-7f); }
inline float fma_f(float a, float b, float c) { return std::fma(a, b, c); }
inline float fabs_f(float a) { return std::fabs(a); }
inline float fmin_f(float a, float b) { return a < b ? a : b; }
inline int rint_i(float a) { return static_cast<int>(std::rint(a)); }
inline int ceil_i(float a) { return static_cast<int>(std::ceil(a)); }
inline u64 umulhi(u64 a, u64 b) { return static_cast<u64>((static_cast<unsigned __int128>(a) * b) >> 64); }
inline u64 shl64(u64 x, int n) { return x << n; }
inline u64 shr64(u64 x, int n) { return x >> n; }
inline u64 div_fallback(u64 a, u64 b) { return bits(dbl(a) / dbl(b)); }
}}
"""

DBAR = r"""
template <int D> double G(double t, const u64 *a) {
  double g = 0.0;
  for (int k = 0; k < D; ++k) {
    volatile double m = t - dbl(a[k]);
    if (!(m > 0.0)) m = 0.0;
    volatile double q = m * m, s = g + q;
    g = k ? s : q;
  }
  return g;
}
template <int D> u64 bisect(const u64 *a, double c) {
  u64 lo = a[0];
  for (int k = 1; k < D; ++k) lo = a[k] < lo ? a[k] : lo;
  u64 hi = bits(dbl(lo) + 3.0 * std::sqrt(c)) + 10;
  while (hi - lo > 1) {
    const u64 mid = lo + (hi - lo) / 2;
    if (G<D>(dbl(mid), a) >= c) hi = mid; else lo = mid;
  }
  return hi;
}
template <int D> void run(long n) {
  std::mt19937_64 R(7 + D);
  std::uniform_real_distribution<double> U(0, 1);
  long bad = 0, inside = 0, trials = 0;
  for (long i = 0; i < n; ++i) {
    const double ratio = std::exp(U(R) * std::log(i % 3 ? 5000.0 : 5e6) + 0.2);      // tau / r
    double r = std::exp((U(R) - 0.5) * 40);
    if (i % 5 == 0) r = std::ldexp(1.0, static_cast<int>(R() % 20) - 10);
    volatile double rr = r;
    const double c = rr * rr;
    eik::ig::Scaled<D> kept;
    for (int rep = 0; rep < 3; ++rep) {        // minima that fall, into lower binades too
      double s0 = ratio * r * (1.0 - 0.3 * rep);
      const double p2 = std::ldexp(1.0, static_cast<int>(std::floor(std::log2(s0))));
      if (i % 7 == 0) s0 = p2 * (1.0 - 1e-3 * U(R) * U(R) * U(R));
      if (i % 11 == 0) s0 = p2;
      u64 a[D];
      a[0] = bits(s0);
      for (int k = 1; k < D; ++k) {
        const double f = U(R);
        double b = s0 + r * 1.5 * f * f;
        if (R() % 17 == 0) b = s0;
        if (R() % 23 == 0) b = INFINITY;
        if (R() % 13 == 0) b = s0 + r * 0.7071 * (1 + 1e-7 * (U(R) - 0.5));
        if (R() % 29 == 0) b = s0 + r * (1 + 1e-9 * (U(R) - 0.5));
        a[k] = bits(b);
      }
      for (int k = D - 1; k > 0; --k) std::swap(a[k], a[R() % (k + 1)]);
      u64 got = 0;
      int m = eik::ig::dbar<D>(a, bits(c), got, kept);
      ++trials;
      if (m < 0) continue;                     // outside its range: the search is used
      ++inside;
      for (; m > 0 && G<D>(dbl(got), a) < c; --m) ++got;
      bad += got != bisect<D>(a, c);
    }
  }
  std::printf("dbar %d inside %d bad %ld\n", D, inside > trials / 2, bad);
}
int main(int, char **v) { const long n = std::atol(v[1]); run<2>(n); run<3>(n); }
"""

QUOTIENT = r"""
int main(int, char **v) {
  std::mt19937_64 Q(5);
  const u64 frac = (1ull << 52) - 1;
  const int ends[] = {0, 1, 2, 62, 63, 64, 65, 100, 123, 1023, 1924, 1999, 2000, 2001, 2045, 2046, 2047};
  long bad = 0;
  const long n = std::atol(v[1]);
  for (long i = 0; i < n; ++i) {
    u64 fa = Q() >> 12, fb = Q() >> 12;
    switch (Q() % 16) {                        // powers of two, all ones, neighbours, near ties
      case 0: fb = 0; break;
      case 1: fa = fb; break;
      case 2: fa = (fb + 1) & frac; break;
      case 3: fb = frac - Q() % 4; break;
      case 4: fa = Q() % 4; break;
      case 5: fb = Q() % 4; break;
      case 6: fa = frac - Q() % 4; break;
      case 7: fa = (fb - 1) & frac; break;
      case 8: fa = 0; break;
      case 9: {                                // a close to (q + 1/2) b
        const unsigned __int128 q2 = (static_cast<unsigned __int128>(1ull << 53) + (Q() >> 11)) | 1;
        u64 m = static_cast<u64>((q2 * ((1ull << 52) | fb)) >> 53);
        while (m >= (1ull << 53)) m >>= 1;
        fa = m & frac;
        break;
      }
    }
    u64 ea = 923 + Q() % 200, eb = 923 + Q() % 200;
    if (Q() % 8 == 0) ea = ends[Q() % 16];     // the ends of the integer range, subnormal
    if (Q() % 8 == 0) eb = ends[Q() % 17];     // and infinite divisors
    const u64 a = (ea << 52) | fa, b = (eb << 52) | (eb == 2047 ? 0 : fb);
    if (a == 0) continue;
    const u64 got = eik::ig::Divisor(b).quotient(a), want = bits(dbl(a) / dbl(b));
    bad += got != want;
  }
  std::printf("quotient bad %ld\n", bad);
}
"""


def _arithmetic() -> str:
    text = frag.source("eik_exact.cuh")
    start = text.index("#ifndef EIK_HD")
    end = text.rindex("#ifdef __CUDACC__", 0, text.index("double quotient(double a, double b)"))
    return HEAD + text[start:end] + "}\n}\n"


@pytest.mark.parametrize("main,n,want", [
    (DBAR, 300_000, "dbar 2 inside 1 bad 0\ndbar 3 inside 1 bad 0"),
    (QUOTIENT, 20_000_000, "quotient bad 0")], ids=["dbar", "quotient"])
def test_integer_arithmetic(tmp_path, main, n, want):
    out = frag.run(tmp_path, _arithmetic() + main, n)
    assert out.stdout.strip() == want, out
