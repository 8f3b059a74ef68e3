"""Compensated FP32 sums on their way into the integer sums (csrc/fixsum.cuh), on
the host: the compensation is not lost."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_float_pairs_keep_their_compensation(tmp_path):
    if shutil.which("g++") is None:
        pytest.skip("no host compiler")
    src = tmp_path / "fxp.cpp"
    src.write_text(r'''
#include "fixsum.cuh"
#include <algorithm>
#include <cmath>
#include <cstring>
#include <random>
using namespace sem;
template <class U, class F> static U bits(F x) { U b; memcpy(&b, &x, sizeof b); return b; }
int main() {
  std::mt19937_64 g(1);
  for (int t = 0; t < 300000; ++t) {            // every finite float is the double's integer
    unsigned f = (unsigned)g();
    if (t % 5 == 0) f &= ~(0xFFu << 23);        // zero and subnormals
    float x;
    memcpy(&x, &f, 4);
    if (!std::isfinite(x)) continue;
    const int e = fx_expf(f) + (int)(g() % 70);
    if (fx_mantf(f, e) != fx_mant(bits<unsigned long long>((double)x), e + 896)) return 1;
  }
  for (int t = 0; t < 30000; ++t) {             // sums of Kahan pairs, as a warp makes them
    float s[32], c[32];
    long double want = 0, size = 0;
    int e = 1;
    for (int l = 0; l < 32; ++l) {
      s[l] = c[l] = 0.0f;
      for (int k = 0; k < 8; ++k) {
        const float v = std::ldexp((float)(g() >> 40) * 0x1p-24f - 0.4f, (int)(g() % 20));
        const float y = v - c[l], u = s[l] + y;
        c[l] = (u - s[l]) - y;
        s[l] = u;
      }
      want += (long double)s[l] - (long double)c[l];
      size = std::max(size, std::fabs((long double)s[l]));
      e = std::max({e, fx_expf(bits<unsigned>(s[l])), fx_expf(bits<unsigned>(c[l]))});
    }
    e += 1;
    long long m = 0;
    for (int l = 0; l < 32; ++l)
      m += fx_mantf(bits<unsigned>(s[l]), e) - fx_mantf(bits<unsigned>(c[l]), e);
    const double got = fx_round(m >> 32, (long long)(unsigned)m, e + 896);
    // one rounding, and two truncations a lane at 2^-56 of the largest value
    if (std::fabs((long double)got - want) > 0x1p-53L * std::fabs(want) + 64 * 0x1p-55L * size)
      return 2;
  }
  return 0;
}
''')
    exe = str(tmp_path / "fxp")
    csrc = os.path.join(ROOT, "paper_2107_01243_gb300", "csrc")
    subprocess.run(["g++", "-std=c++17", "-O1", "-ffp-contract=off", "-D__host__=",
                    "-D__device__=", "-I", csrc, str(src), "-o", exe], check=True)
    assert subprocess.run([exe]).returncode == 0


def test_sums_up_to_the_largest_double_and_beyond(tmp_path):
    """Sums whose terms reach 2^1023 are finite where the IEEE sum is, overflow to
    infinity where it does; +Inf and NaN come out as IEEE addition has them, -Inf as
    NaN."""
    if shutil.which("g++") is None:
        pytest.skip("no host compiler")
    src = tmp_path / "fxr.cpp"
    src.write_text(r'''
#include "fixsum.cuh"
#include <algorithm>
#include <cmath>
#include <cstring>
#include <limits>
#include <vector>
using namespace sem;
static unsigned long long bits(double x) { unsigned long long b; memcpy(&b, &x, 8); return b; }
// values -> one FxVal packed sh bits to the right, as a CTA hands it on -> total
static double total(const std::vector<double>& v, int sh) {
  int e = 1;
  for (double x : v) e = std::max(e, fx_exp(bits(x)));
  if (e >= kFxInf) return fx_round(0, 0, e);
  long long hi = 0, lo = 0;
  for (double x : v) {
    const long long m = fx_mant(bits(x), e);
    hi += m >> 32;
    lo += (long long)(unsigned)m;
  }
  const long long p = (hi << (32 - sh)) + (lo >> sh);
  return fx_round(p >> 32, (long long)(unsigned)p, e + sh);
}
int main() {
  const double inf = std::numeric_limits<double>::infinity(), big = 0x1p1022;
  for (int sh = 4; sh <= 5; ++sh) {
    if (total({big, big, big}, sh) != 3 * big) return 1;
    if (total({0x1.8p1023}, sh) != 0x1.8p1023) return 2;
    if (total({0x1.8p1023, -0x1p1023, 0x1p1020}, sh) != 0x1.4p1022) return 3;
    if (total({0x1p1023, 0x1p1023}, sh) != inf) return 4;
    if (total({-0x1p1023, -0x1p1023}, sh) != -inf) return 5;
    if (total({1.0, inf, 2.0}, sh) != inf || !std::isnan(total({-inf, 1.0}, sh))) return 6;
    if (!std::isnan(total({inf, -inf}, sh)) || !std::isnan(total({inf, NAN}, sh))) return 7;
    if (!std::isnan(total({NAN, 1.0}, sh)) || total({0.0, 0.0}, sh) != 0.0) return 8;
  }
  return 0;
}
''')
    exe = str(tmp_path / "fxr")
    csrc = os.path.join(ROOT, "paper_2107_01243_gb300", "csrc")
    subprocess.run(["g++", "-std=c++17", "-O1", "-D__host__=", "-D__device__=", "-I", csrc,
                    str(src), "-o", exe], check=True)
    assert subprocess.run([exe]).returncode == 0
