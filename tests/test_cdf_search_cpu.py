"""The kernels' block-wise cdf search returns what the plain sequential search
does (CPU, no GPU).

csrc/sampling.cuh compiles as plain C++ on the host with the device's float
operations.  The plain search below is the definition (inversion, Poisson and
binomial); both run over uniforms next to every cdf entry and at both ends of
(0, 1), for n at the edges of the blocks (3, 4, 15, 16, 17), of the search's
cap (62 to 65) and of the float count-down (2^24).
"""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HEADER = os.path.join(ROOT, "paper_2402_13259_gb300", "csrc", "sampling.cuh")

SRC = r"""
#include <cstdio>
#include <cstdlib>
#include <cmath>
#include "%s"
using namespace eulernet;
static float rinv[64];
static int plain(bool binom, float u, float p0, float r, int n) {
  float pk = p0, F = p0;
  int k = 0;
  while (u > F) {
    if ((binom && k == n) || k == 63) break;
    pk = binom ? ((pk * (float)(n - k)) * r) * rinv[k + 1] : (pk * r) * rinv[k + 1];
    k = k + 1;
    const float Fn = F + pk;
    if (Fn == F) break;
    F = Fn;
  }
  return k;
}
static long bad = 0, checked = 0;
static void at(bool binom, float u, float p0, float r, int n) {
  if (!(u > 0.0f && u < 1.0f)) return;
  const int got = binom ? cdf_search<true>(u, p0, r, n, (float)n, rinv)
                        : cdf_search<false>(u, p0, r, 0, 0.0f, rinv);
  bad += got != plain(binom, u, p0, r, n);
  ++checked;
}
static void sweep(bool binom, float p0, float r, int n) {
  float pk = p0, F = p0;
  for (int k = 0; k < 63; ++k) {
    at(binom, nextafterf(F, 0.0f), p0, r, n);
    at(binom, F, p0, r, n);
    at(binom, nextafterf(F, 2.0f), p0, r, n);
    pk = binom ? (k < n ? ((pk * (float)(n - k)) * r) * rinv[k + 1] : 0.0f) : (pk * r) * rinv[k + 1];
    F = F + pk;
  }
  at(binom, 0x1p-24f, p0, r, n);
  at(binom, 1.0f - 0x1p-24f, p0, r, n);
  at(binom, 1.0f - 0x1.8p-23f, p0, r, n);
  for (int j = 0; j < 200; ++j) at(binom, (float)(2 * (rand() & 0x7fffff) + 1) * 0x1p-24f, p0, r, n);
}
int main() {
  for (int k = 1; k < 64; ++k) rinv[k] = 1.0f / (float)k;
  const int ns[] = {1, 2, 3, 4, 5, 7, 8, 11, 12, 13, 14, 15, 16, 17, 18, 31, 40, 61, 62, 63, 64, 65, 500, 4096,
                    (1 << 24) - 1, 1 << 24, (1 << 24) + 1, 1 << 30};
  const float means[] = {1e-9f, 1e-6f, 1e-3f, 0.05f, 0.5f, 1.0f, 2.7f, 5.0f, 8.5f, 9.999f};
  for (float m : means) {
    sweep(false, fm::exp_neg(-m), m, 0);
    for (int n : ns) {
      const float p = m / (float)n;
      if (!(p <= 0.5f) || !((float)n * p < 10.0f)) continue;
      const BinomConst c = binom_const(p);
      if (!(c.c0 > 0.0f)) continue;
      sweep(true, fm::exp_neg((float)n * c.lq), c.r, n);
    }
  }
  std::printf("%%ld %%ld\n", bad, checked);
  return bad != 0;
}
""" % HEADER


def test_block_search_equals_plain_search(tmp_path):
    src, exe = tmp_path / "search.cpp", tmp_path / "search"
    src.write_text(SRC)
    try:
        subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-fno-fast-math", str(src), "-o",
                        str(exe), "-lm"], check=True, capture_output=True, text=True)
    except FileNotFoundError:
        pytest.skip("no host C++ compiler")
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=600)
    bad, n = map(int, r.stdout.split())
    assert n > 50_000
    assert r.returncode == 0 and bad == 0, f"{bad} of {n} searches differ"
