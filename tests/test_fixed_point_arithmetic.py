"""The fixed-point arithmetic of the FP64 transforms (csrc/mg_fixed.cuh) compiled
for the host: its roundings have no mean, and a block's scale depends on the
values that are in it only.  A mean error, however small beside the rounding
noise, is the same vector in every pass over the state and adds up.

Bounds.  Errors are in integer units and at most 4 each; over T = 40000 random
inputs the mean of an unbiased one stays within 5 * 1.1 / sqrt(T) = 0.03
(5 sigma at the largest root mean square, 1.1).  Truncation gives -1, a dropped
low bit 0.5 |m|, ties always up 0.5 at the first octave."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")

PROGRAM = r"""
#include <cmath>
#include <complex>
#include <cstdio>
#include <cstring>
#include <random>
#include "mg_fixed.cuh"
using namespace mgk;
typedef long double L;
typedef std::complex<L> C;
std::mt19937_64 rng(3);
const int T = 40000;
const double M61 = 2305843009213693952.0;
L uniform() { return (L)(long long)rng() / 9223372036854775808.0L; }
C val(I2 a) { return C((L)a.x, (L)a.y); }
// an FP64 value between 1 and 2, with sign, and its integers at 2^(62 - sh)
I2 words(L& exact, int sh) {
  double v = (1.0 + std::fabs((double)uniform())) * (rng() & 1 ? 1 : -1);
  long long b;
  std::memcpy(&b, &v, 8);
  b ^= (long long)(rng() & 15);
  std::memcpy(&v, &b, 8);
  exact = std::ldexp((L)v, 62 - sh);
  return I2{b, b};
}
I2 random_value(int bits) { return I2{(long long)(rng() >> 1) >> (63 - bits), -((long long)(rng() >> 1) >> (63 - bits))}; }
template <class F> void multiplier(const char* name, L scale, bool fresh, F f) {
  for (int m = 0; m < 6; ++m) {
    const double th = 0.3 + m;
    const int4 w = to_mult(double2{std::cos(th), std::sin(th)}, M61);
    const C ex(((L)w.x * 2147483648.0L + w.y) / (L)M61, ((L)w.z * 2147483648.0L + w.w) / (L)M61);
    C sum = 0;
    for (int t = 0; t < T; ++t) {
      I2 x = random_value(59);
      if (fresh) x = I2{x.x & ~1ll, x.y & ~1ll};
      sum += val(f(x, w)) - val(x) * ex * scale;
    }
    printf("%s%d %Lf\n", name, m, std::abs(sum / (L)T));
  }
}
template <int N, class F> void transform(const char* name, int shift, F f) {
  C sum[16];
  for (int t = 0; t < T; ++t) {
    I2 x[16];
    C ex[16];
    for (int i = 0; i < N; ++i) x[i] = random_value(57);
    for (int k = 0; k < N; ++k) {
      C a = 0;
      for (int i = 0; i < N; ++i) {
        const L th = -2 * 3.14159265358979323846264338327950288L * ((i * k) % N) / N;
        a += val(x[i]) * C(std::cos(th), std::sin(th));
      }
      ex[k] = a / (L)(1 << shift);
    }
    f(x);
    for (int k = 0; k < N; ++k) sum[k] += val(x[k]) - ex[k];
  }
  L worst = 0;
  for (int k = 0; k < N; ++k) worst = std::max(worst, std::abs(sum[k] / (L)T));
  printf("%s %Lf\n", name, worst);
}
int main() {
  for (int sh = 8; sh < 40; sh += sh < 14 ? 1 : 9) {
    L sum = 0, away = 0;
    for (int t = 0; t < T; ++t) {
      L ex;
      const I2 b = words(ex, sh);
      const int hi = hi32(b.x);
      const long long r = to_fixed(hi, (unsigned)b.x, ((hi >> 20) & 0x7ff) + sh, (int)(rng() & 1)) & ~1ll;
      sum += (L)r - ex;
      away += ((L)r - ex) * (ex > 0 ? 1 : -1);
    }
    printf("conversion%d %Lf\n", sh, std::fabs(sum / T));
    printf("conversion_away%d %Lf\n", sh, std::fabs(away / T));
  }
  multiplier("first", 1, true, [](I2 x, int4 w) { return cmul<false, true>(x, w); });
  multiplier("later", 1, false, [](I2 x, int4 w) { return cmul<false, true>(x, w, -1); });
  multiplier("halved", 0.5L, false, [](I2 x, int4 w) { return cmul_half(x, w, -1); });
  transform<8>("dft8_2", 1, [](I2* x) { IDft<false, 8, 1>::run(x); });
  transform<8>("dft8_4", 2, [](I2* x) { IDft<false, 8, 2>::run(x); });
  transform<8>("dft8_late_2", 1, [](I2* x) { idft8_late<false, 1>(x); });
  transform<8>("dft8_late_4", 2, [](I2* x) { idft8_late<false, 2>(x); });
  transform<12>("dft12_2", 1, [](I2* x) { IDft<false, 12, 1>::run(x); });
  transform<12>("dft12_4", 2, [](I2* x) { IDft<false, 12, 2>::run(x); });
  transform<16>("dft16_4", 2, [](I2* x) { IDft<false, 16, 2>::run(x); });
  // groups that are empty or next to it add no more than a unit to the squares
  // of a block, of which its largest value alone has 65536 and more
  const unsigned one = 0x3ff00000u, tiny = 0x00100000u;
  const int e = fx_exponent(one);
  printf("empty_groups %d\n", (int)fx_square(0, e) > 1);
  printf("tiny_groups %d\n", (int)fx_square(tiny, e) > 1);
  // a multiplier that is not finite gives words without an undefined shift
  const unsigned bad[2] = {0x7ff00000u, 0xfff80000u};
  for (unsigned b : bad) {
    const long long v = to_fixed((int)b, 0u, 1024, 0);
    printf("not_finite %d\n", v < -1 || v > 1);
  }
  return 0;
}
"""


def test_roundings_have_no_mean(tmp_path):
    gxx = shutil.which("g++")
    if not gxx or not os.path.exists(os.path.join(CUDA, "include", "cuda_runtime.h")):
        pytest.skip("no host compiler or CUDA headers")
    src, exe = tmp_path / "fixed.cpp", tmp_path / "fixed"
    src.write_text(PROGRAM)
    subprocess.run([gxx, "-O1", "-fwrapv", "-std=c++17", "-w", f"-I{CUDA}/include",
                    f"-I{ROOT}/paper_1909_06412_gb300/csrc", "-o", str(exe), str(src)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout
    rows = [line.split() for line in out.splitlines()]
    assert len(rows) > 40
    assert [r for r in rows if float(r[1]) > 0.03] == []
