"""Rounding of the transforms' double butterfly (a, b) -> (a + w b, a - w b),
compiled for the host from the library's header.  Each output is two fused
operations: its error is at most half an ulp of the first one's result and
half an ulp of its own, whatever the other output is."""
import subprocess

PROGRAM = r"""
#include "sg_fft.cuh"
#include <cmath>
#include <cstdio>
#include <random>
int main() {
  std::mt19937_64 g(1);
  std::normal_distribution<double> nd;
  const long double u = ldexpl(1.0L, -53);
  int bad = 0;
  auto check = [&](double got, long double inner, long double exact, long double mag) {
    // long double: 2^-60 of the operands covers its own rounding here
    if (fabsl(got - exact) > (u * (fabsl(inner) + fabsl(exact)) + mag * ldexpl(1.0L, -60)) * 1.001L) ++bad;
  };
  for (int k = 0; k < 200000; ++k) {
    const double th = 6.283185307179586 * (k % 257) / 257, c = std::cos(th), s = std::sin(th);
    const sg::cplx<double> w{c, -s}, a{nd(g), nd(g)};
    sg::cplx<double> b{nd(g), nd(g)}, x0, x1;
    if (k & 1) {  // w b close to a or -a: one output nearly cancels
      const double e = std::ldexp(1.0, -(k % 50)), sg = k & 2 ? 1 : -1;
      b = {sg * (a.x * c - a.y * s) + e * b.x, sg * (a.y * c + a.x * s) + e * b.y};
    }
    sg::butterfly<double>(a, b, w, x0, x1);
    const long double px = (long double)b.x * w.x, qx = (long double)b.y * w.y, py = (long double)b.x * w.y,
                      qy = (long double)b.y * w.x;
    const long double mag = fabsl(a.x) + fabsl(a.y) + fabsl(b.x) + fabsl(b.y);
    check(x0.x, a.x + px, a.x + px - qx, mag);
    check(x0.y, a.y + py, a.y + py + qy, mag);
    check(x1.x, a.x - px, a.x - px + qx, mag);
    check(x1.y, a.y - py, a.y - py - qy, mag);
  }
  std::printf("%d\n", bad);
  return bad != 0;
}
"""


def test_each_output_is_rounded_twice(tmp_path):
    from paper_2008_09441_gb300 import build as b
    src = tmp_path / "butterfly.cu"
    src.write_text(PROGRAM)
    exe = tmp_path / "butterfly"
    subprocess.run([b.nvcc(), *b.ARCH, *b.FLAGS, "-I", b.CSRC, "-o", str(exe), str(src)], check=True)
    assert subprocess.run([str(exe)], capture_output=True, text=True).stdout.strip() == "0"
