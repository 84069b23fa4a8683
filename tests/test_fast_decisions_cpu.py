"""The rejection tests' fast log-probability ratios stay well inside the
tolerance within which a test is left to the exact functions (CPU, no GPU).

csrc/sampling.cuh compiles as plain C++ on the host.  Over the domain of the
fast path (np >= 10, standard deviation below 256, |k - mode| below 24 of them,
n < 2^24) the fast value may differ from the difference of the exact float
functions by at most a quarter of kFastTol + kFastRel |f|: three quarters are
left for the hardware's reciprocal and logarithm, whose stated errors (2 ulp;
2^-21.4 absolute near 1, 3 ulp elsewhere) enter multiplied by |k - mode| and by
k, where |f| grows with (k - mode)^2 / (2 np q).
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
static double U() { return (rand() + 0.5) / (RAND_MAX + 1.0); }
int main() {
  srand(7);
  double worst_b = 0.0, worst_p = 0.0;
  long nb = 0, np_ = 0;
  for (long it = 0; it < 6000000; ++it) {
    const float p = (float)(0.5 * pow(10.0, -6.0 * U() * U())), q = 1.0f - p;
    const double n_ = 10.0 * pow(13000.0, U()) / p;
    const double span = it %% 4 ? 14.0 : 47.9;
    const double dev = it %% 16 == 1 ? 0.0 : (U() - 0.5) * span;
    if (n_ < 16777216.0) {
      const int n = (int)n_;
      const float nf = (float)n, npf = nf * p, spq = sqrtf(npf * q);
      const int mode = (int)floorf((nf + 1.0f) * p);
      const int k = it %% 16 == 2 ? 2 : (int)floor(mode + spq * dev);
      if (npf >= 10.0f && spq < kFastMaxSd && k >= 2 && k <= n - 2 && fabsf((float)k - (float)mode) < kFastMaxDev * spq) {
        const float f = fast_log_ratio(fast_binom(nf, (float)mode, p, q), (float)k, nf - (float)k);
        const float se = stirling_err(nf);
        const double ex = (double)(log_binom_pmf(k, n, p, q, se) - log_binom_pmf(mode, n, p, q, se));
        worst_b = fmax(worst_b, fabs(f - ex) / (kFastTol + kFastRel * fabsf(f)));
        ++nb;
      }
    }
    const float lam = (float)(10.0 * pow(6500.0, U())), sl = sqrtf(lam);
    const int k = it %% 16 == 2 ? 2 : (int)floor(lam + sl * dev);
    if (sl < kFastMaxSd && k >= 2 && fabsf((float)k - lam) < kFastMaxDev * sl) {
      const float f = fast_log_pois((float)k, lam, fast_rcp(lam));
      worst_p = fmax(worst_p, fabs((double)f - (double)log_pois_pmf(k, lam)) / (kFastTol + kFastRel * fabsf(f)));
      ++np_;
    }
  }
  printf("%%g %%ld %%g %%ld\n", worst_b, nb, worst_p, np_);
  return 0;
}
""" % HEADER


def test_fast_ratio_is_within_a_quarter_of_the_tolerance(tmp_path):
    src, exe = tmp_path / "fast.cpp", tmp_path / "fast"
    src.write_text(SRC)
    try:
        subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-fno-fast-math", str(src), "-o",
                        str(exe), "-lm"], check=True, capture_output=True, text=True)
    except FileNotFoundError:
        pytest.skip("no host C++ compiler")
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=600, check=True)
    wb, nb, wp, npo = r.stdout.split()
    assert int(nb) > 3_000_000 and int(npo) > 3_000_000
    assert float(wb) <= 0.25, wb
    assert float(wp) <= 0.25, wp
