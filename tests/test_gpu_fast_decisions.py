"""The rejection tests' fast decisions with the device's own reciprocal and
logarithm (GPU): both sides of a test, evaluated fast and exactly on the device,
over the domain of the fast path.  A decision is safe while the two differences
lie less than the tolerance apart; by the stated errors of the hardware functions
(reciprocal 2 ulp; logarithm 2^-21.4 absolute near 1, 3 ulp elsewhere) times
|k - mode|, and the series' own quarter (test_fast_decisions_cpu.py), half of it
is expected at most.  Decided tests must agree with the exact ones without
exception.
"""
import os
import shutil
import subprocess

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HEADER = os.path.join(ROOT, "paper_2402_13259_gb300", "csrc", "sampling.cuh")

SRC = r"""
#include <cstdio>
#include <cmath>
#include <cuda_runtime.h>
#include "%s"
using namespace eulernet;

struct Worst { float binom, pois; unsigned long long nb, np, decided, wrong; };

__device__ void put(float* a, float v) { atomicMax(reinterpret_cast<int*>(a), __float_as_int(v)); }  // v >= 0

__device__ void weigh(float lv_fast, float f, float lv, float ex, float* worst, Worst* w) {
  const float tol = fmaf(kFastRel, fabsf(f), kFastTol);
  put(worst, (float)(fabs(((double)lv_fast - (double)f) - ((double)lv - (double)ex)) / (double)tol));
  const int dec = fast_decide(lv_fast, f);
  if (dec >= 0) {
    atomicAdd(&w->decided, 1ull);
    if ((dec == 1) != (lv <= ex)) atomicAdd(&w->wrong, 1ull);
  }
}

// Mode 0: k and v as the sampler draws them; 1: k spread over the fast path's
// range, v near the decision.
__global__ void probe(int mode, uint32_t seed, Worst* w) {
  const uint32_t id = blockIdx.x * blockDim.x + threadIdx.x;
  PhiloxStream st;
  st.init(seed, 5u, 0u, 0u, (uint32_t)mode, id);
  for (int it = 0; it < 64; ++it) {
    const float a1 = st.uniform(), a2 = st.uniform(), a3 = st.uniform(), a4 = st.uniform();
    float u, v;
    st.uniform2(u, v);
    u = u - 0.5f;
    const float us = 0.5f - fabsf(u);
    {  // binomial
      const float p = 0.5f * exp10f(-6.0f * a1 * a2), q = 1.0f - p;
      const double n_ = 10.0 * pow(13000.0, (double)a3) / p;
      if (n_ < 16777216.0) {
        const int n = (int)n_;
        const float nf = (float)n, np = nf * p, spq = sqrtf(np * q);
        const float b = 1.15f + 2.53f * spq, a = -0.0873f + 0.0248f * b + 0.01f * p;
        const float c = np + 0.5f, alpha = (2.83f + 5.1f / b) * spq;
        int md = (int)floorf((nf + 1.0f) * p);
        if (md > n) md = n;
        const FastBinom fb = fast_binom(nf, (float)md, p, q);
        const float kf = mode == 0 ? floorf((2.0f * a / us + b) * u + c)
                                   : floorf((float)md + (a4 - 0.5f) * 47.9f * spq);
        const int k = (int)kf;
        if (np >= 10.0f && spq < kFastMaxSd && kf >= 0.0f && kf <= nf && k >= 2 && k <= n - 2 &&
            fabsf(kf - fb.mf) < kFastMaxDev * spq) {
          const float f = fast_log_ratio(fb, kf, nf - kf);
          const float g = a / (us * us) + b;
          if (mode == 1) v = expf(f + 0.02f * (v - 0.5f)) * g / alpha;
          if (v >= 0x1p-24f && v < 1.0f) {  // a uniform
            const float se = stirling_err(nf);
            const float ex = log_binom_pmf(k, n, p, q, se) - log_binom_pmf(md, n, p, q, se);
            weigh(fast_log((v * alpha) * fast_rcp(fmaf(a, fast_rcp(us * us), b))), f,
                  fm::log_pos(v * alpha / g), ex, &w->binom, w);
            atomicAdd(&w->nb, 1ull);
          }
        }
      }
    }
    {  // Poisson
      const float lam = 10.0f * powf(6500.0f, a1), sl = sqrtf(lam);
      const float b = 0.931f + 2.53f * sl, a = -0.059f + 0.02483f * b, ia = 1.1239f + 1.1328f / (b - 3.4f);
      const float kf = mode == 0 ? floorf((2.0f * a / us + b) * u + lam + 0.43f)
                                 : floorf(lam + (a4 - 0.5f) * 47.9f * sl);
      const int k = (int)kf;
      if (kf >= 2.0f && sl < kFastMaxSd && fabsf(kf - lam) < kFastMaxDev * sl) {
        const float f = fast_log_pois(kf, lam, fast_rcp(lam));
        const float g = a / (us * us) + b;
        float V = a2;
        if (mode == 1) V = expf(f + 0.02f * (a2 - 0.5f)) * g / ia;
        if (V >= 0x1p-24f && V < 1.0f) {
          weigh(fast_log((V * ia) * fast_rcp(fmaf(a, fast_rcp(us * us), b))), f, fm::log_pos(V * ia / g),
                log_pois_pmf(k, lam), &w->pois, w);
          atomicAdd(&w->np, 1ull);
        }
      }
    }
  }
}

int main() {
  for (int mode = 0; mode < 2; ++mode) {
    Worst* w = nullptr;
    Worst h = {};
    if (cudaMalloc(&w, sizeof h) != cudaSuccess || cudaMemset(w, 0, sizeof h) != cudaSuccess) return 1;
    probe<<<1024, 128>>>(mode, 11u, w);
    if (cudaMemcpy(&h, w, sizeof h, cudaMemcpyDeviceToHost) != cudaSuccess) return 1;
    printf("%%g %%g %%llu %%llu %%llu %%llu\n", h.binom, h.pois, h.nb, h.np, h.decided, h.wrong);
    cudaFree(w);
  }
  return 0;
}
""" % HEADER


def test_device_decisions(tmp_path):
    import torch
    if not torch.cuda.is_available():
        pytest.fail("these tests need a CUDA GPU")
    nvcc = shutil.which(os.environ.get("NVCC", "nvcc")) or "/usr/local/cuda/bin/nvcc"
    src, exe = tmp_path / "fast.cu", tmp_path / "fast"
    src.write_text(SRC)
    from paper_2402_13259_gb300 import build as B
    r = subprocess.run([nvcc, *B.FLAGS, str(src), "-o", str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, (r.stdout, r.stderr)
    print(r.stdout)
    for line in r.stdout.splitlines():
        wb, wp, nb, npo, decided, wrong = line.split()
        assert int(nb) > 500_000 and int(npo) > 500_000 and int(decided) > 500_000
        assert float(wb) <= 0.5 and float(wp) <= 0.5, line
        assert int(wrong) == 0, line
