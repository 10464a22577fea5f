"""quotient() of csrc/tp_quotient.h, which steps the absorbing layer, against the
division it replaces, bit for bit: random numerators of every exponent, around
2^-60 where the scaled branch begins, subnormal ones and subnormal results;
divisors 1 + a for layers of 1 to 64 cells and a from 1e-4 to 1000."""
import subprocess

from paper_2104_00794_gb300 import build

SOURCE = r"""
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <cmath>
#include <random>
#include "tp_quotient.h"
int main() {
  std::mt19937_64 g(1);
  for (int it = 0; it < 2000; ++it) {
    const int sw = 1 + (int)(g() % 64), d = (int)(g() % (sw + 1));
    float samax = std::pow(10.0, -4 + 4.3 * (double)(g() % 1000) / 1000.0);
    if (it % 7 == 0) samax *= 50;
    const float t = (float)(sw - d) / (float)sw, b = 1.0f + samax * t * t, inv = 1.0f / b;
    for (int k = 0; k < 10000; ++k) {
      uint32_t u = (uint32_t)g();
      if (k % 5 == 0) u = (u & 0x807fffffu) | (uint32_t)(g() % 70) << 23;                       // below 2^-57
      if (k % 50 == 1) u = (u & 0x807fffffu) | (uint32_t)(127 - 61 + (int)(g() % 3)) << 23;     // around 2^-60
      if (k % 97 == 0) u &= 0x807fffffu;                                                        // subnormal
      float n;
      memcpy(&n, &u, 4);
      if (std::isnan(n)) continue;
      const volatile float e = n / b;
      const float x = e, q = tp::quotient(n, b, inv);
      if (memcmp(&x, &q, 4) && !(x == 0.f && q == 0.f)) {
        printf("%a / %a: %a, not %a\n", n, b, q, x);
        return 1;
      }
    }
  }
  const float inf = INFINITY;
  return !(tp::quotient(inf, 1.5f, 1.f / 1.5f) == inf && tp::quotient(-inf, 1.5f, 1.f / 1.5f) == -inf &&
           std::isnan(tp::quotient(NAN, 1.5f, 1.f / 1.5f)) && tp::quotient(0.f, 1.5f, 1.f / 1.5f) == 0.f);
}
"""


def test_quotient_is_the_division(tmp_path):
    src, exe = tmp_path / "q.cpp", tmp_path / "q"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-I", build.CSRC, str(src), "-o", str(exe)], check=True)
    res = subprocess.run([str(exe)], capture_output=True, text=True)
    assert res.returncode == 0, res.stdout
