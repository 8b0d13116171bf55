"""The fixed-point functions (fixed_math.cuh), compiled for the host, against
long double at random arguments and at both ends of their ranges.

Bounds: exp2_significand's truncations and constants sum to 4.0e-18 relative
(three truncated Horner steps of 2^-60 each, the series' end, two rounded
coefficients), 0.035 units in the last place of a double, so that a double
packed from it, and exp_fixed_bits, lie within 0.54 ulp; log2_fixed within
2^-54; fixed_to_double is the nearest double.
"""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")

PROGRAM = r"""
#include <cmath>
#include <cstdio>
#include <cstring>
#include <limits>
#include <random>

#include "fixed_math.cuh"

using namespace pj;

static uint64_t tab[256];
static LogEntry ltab[256];
static int bad = 0;

static double d(uint64_t b) { double x; std::memcpy(&x, &b, 8); return x; }
static uint64_t bits(double x) { uint64_t b; std::memcpy(&b, &x, 8); return b; }
// spacing of the doubles at |x| (subnormals and the top binade too)
static long double ulp(long double x) {
  int e;
  std::frexp(std::fabs(x), &e);
  return std::ldexp(1.0L, std::max(e - 53, -1074));
}
static void check(bool ok, const char* what, long double at) {
  if (ok) return;
  if (bad++ < 10) std::printf("%s at %.21Lg\n", what, at);
}

int main() {
  for (int j = 0; j < 256; j++) {
    tab[j] = (uint64_t)std::floor(std::exp2((long double)j / 256.0L) * 0x1p63L + 0.5L);
    ltab[j].r = (uint64_t)((32768 * 256 + 255 + j) / (256 + j));
    ltab[j].t = (uint64_t)std::floor(std::log2(32768.0L / (long double)ltab[j].r) * 0x1p62L + 0.5L);
  }
  std::mt19937_64 rng(5);

  // 2^(n + frac 2^-64) of any n: normal, both edges, subnormal, zero, infinity
  for (int n = -1100; n <= 1030; n++)
    for (int t = 0; t < 300; t++) {
      const uint64_t frac = t == 0 ? 0 : t == 1 ? ~0ull : t == 2 ? 1ull << 63 : rng();
      const long double want = std::ldexp(std::exp2((long double)frac * 0x1p-64L), n);
      const double got = d(pack_double_any(n, exp2_significand(frac, tab)));
      if (want >= 0x1.fffffffffffff8p1023L) check(std::isinf(got), "exp2 overflow", n + frac * 0x1p-64L);
      else check(std::isfinite(got) && std::fabs(got - want) <= 0.54L * ulp(want), "exp2", n + frac * 0x1p-64L);
    }

  // exp(x), |x| < 704
  for (int t = 0; t < 400000; t++) {
    std::uniform_real_distribution<double> u(-704.0, 704.0);
    double x = u(rng);
    if (t % 4 == 1) x /= 704.0;
    if (t % 4 == 2) x = std::ldexp(x, -(int)(rng() % 1080));
    if (t == 0) x = 0.0;
    if (t == 4) x = -0.0;
    const long double want = std::exp((long double)x);
    check(std::fabs(d(exp_fixed_bits(bits(x), tab)) - want) <= 0.54L * ulp(want), "exp", x);
  }

  // log2 of positive normal doubles
  for (int t = 0; t < 400000; t++) {
    uint64_t b = rng() & 0x7fffffffffffffffull;
    if (t % 3 == 1) b = bits(1.0) + (rng() >> 20) - (1ull << 43);
    if (t == 0) b = 0x0010000000000000ull;
    if (t == 3) b = 0x7fefffffffffffffull;
    if (b < 0x0010000000000000ull || b >= 0x7ff0000000000000ull) continue;
    int e;
    const uint64_t l = log2_fixed(b, e, ltab);
    // of the significand, so that the reference does not round at the size of e
    const long double want = std::log2(std::ldexp((long double)d(b), -e));
    check(std::fabs((long double)l * 0x1p-62L - want) <= 0x1p-54L, "log2", d(b));
  }

  // x 2^-s
  for (int t = 0; t < 400000; t++) {
    int64_t x = (int64_t)(rng() >> (rng() % 64));
    if (t & 1) x = -x;
    if (t == 0) x = std::numeric_limits<int64_t>::min();
    if (t == 2) x = std::numeric_limits<int64_t>::max();
    if (t == 4) x = 0;
    const int s = t % 3 == 0 ? 51 : t % 3 == 1 ? 59 : 0;
    const long double want = std::ldexp((long double)x, -s);
    check(std::fabs(d(fixed_to_double(x, s)) - want) <= 0.5L * ulp(want), "fixed_to_double", want);
  }

  // signed high product: short by at most 2
  for (int t = 0; t < 400000; t++) {
    const int64_t c = (int64_t)rng() >> (rng() % 32);
    const uint64_t b = rng() >> (rng() % 32);
    const int64_t exact = (int64_t)((__int128)c * (__int128)b >> 64);
    const int64_t got = mulhi_su(c, b);
    check(got <= exact && exact - got <= 2, "mulhi_su", (long double)c);
  }
  std::printf("bad %d\n", bad);
  return bad != 0;
}
"""


def test_fixed_point_functions(tmp_path):
    src, exe = tmp_path / "fixed.cpp", tmp_path / "fixed"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=gnu++17", "-O1", "-I", os.path.join(ROOT, "paper_1809_01029_gb300", "csrc"), "-I",
                    os.path.join(CUDA, "include"), str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout[-2000:]
