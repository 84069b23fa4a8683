"""The library's host code, run without a GPU on a stand-in for the CUDA
runtime (fake_cudart.cpp): what it allocates against what its launches address,
for calls of different sizes on one handle.  Each test is a child process that
preloads the stand-in; nothing runs on a device.
"""
import os
import shutil
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PRELUDE = r'''
import ctypes as C, os, sys
import numpy as np
from paper_2402_13259_gb300 import binding as Bd, workloads as W
F = C.CDLL(os.environ["LD_PRELOAD"])
F.fake_log.restype = C.c_char_p
F.fake_live_bytes.restype = C.c_longlong
F.fake_fail_malloc.argtypes = [C.c_longlong]
RT = C.CDLL(os.environ["LD_PRELOAD"])
L = Bd.lib()
def dev(nbytes):
    p = C.c_void_p()
    assert RT.cudaMalloc(C.byref(p), C.c_size_t(nbytes)) == 0
    return p
def log(clear=True):
    t = F.fake_log().decode()
    if clear:
        F.fake_clear()
    return t
def forms(t):
    """Kernels that ran: which form, without the repeats of a captured slot."""
    out = []
    for x in t.splitlines():
        k = x.split()[0]
        if not out or out[-1] != k:
            out.append(k)
    return out
def chain(n, skip=1, lam=12.0, m=9, every=3):
    edges = []
    for i in range(n - 1):
        edges.append((i, i + 1, 0.6))
        if skip > 1 and i + skip < n:
            edges.append((i, i + skip, 0.3))
    rp, col, prob = W.csr_from_edges(n, edges)
    w = np.zeros(n); w[::every] = lam
    return W.Network(n, rp, col, prob, np.full(n, m), np.full(n, 1.1),
                     W.Arrivals(kind=W.ARR_SINUSOID, w=w, a=1.0, b=0.2, period=3.0, phase=0.1))
def net(x):
    return Bd.EulerNet(x)
def simulate(h, scheme, R, dt=0.1, T=1.0):
    s = dev(8 * Bd.stats_len(h.n, R))
    rc = L.euler_net_simulate(h._h, scheme, dt, T, R, 1, 0, s, None)
    RT.cudaFree(s)
    return rc
def sojourn(h, scheme, R, S, dt=0.1, T=1.0):
    s, o = dev(8 * Bd.stats_len(h.n, R)), dev(4 * R * S)
    rc = L.euler_net_sojourn(h._h, scheme, dt, T, R, 1, 0, 0, 1, S, o, s, None)
    RT.cudaFree(s); RT.cudaFree(o)
    return rc
def grad(h, scheme, R, dt=0.1, T=1.0):
    g, v = dev(16 * (h.n + 3)), dev(16)
    rc = L.euler_net_grad(h._h, scheme, dt, T, R, 1, 0, g, v, None, None, None, None)
    RT.cudaFree(g); RT.cudaFree(v)
    return rc
'''


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    """run(code): the code after PRELUDE in a child process on the stand-in."""
    if shutil.which("g++") is None:
        pytest.skip("no host C++ compiler")
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    if not os.path.exists(os.path.join(cuda, "include", "cuda_runtime.h")):
        pytest.skip("no CUDA headers")
    from paper_2402_13259_gb300 import build as B
    B.build_library()
    so = str(tmp_path_factory.mktemp("fake") / "libfake_cudart.so")
    r = subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I", os.path.join(cuda, "include"),
                        os.path.join(ROOT, "tests", "fake_cudart.cpp"), "-o", so, "-ldl"],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]

    def run(code):
        r = subprocess.run([sys.executable, "-c", PRELUDE + code], capture_output=True, text=True, timeout=600,
                           cwd=ROOT, env=dict(os.environ, LD_PRELOAD=so, PYTHONPATH=ROOT))
        assert r.returncode == 0, (r.stdout[-3000:], r.stderr[-3000:])
        return r.stdout
    return run


@pytest.mark.parametrize("call", ["sojourn", "grad"])
@pytest.mark.parametrize("scheme", [0, 1])
def test_hbm_extra_state_after_a_larger_call(host, call, scheme):
    """The customers' and the score sums' arrays hold what the HBM form's
    kernels address after a larger call on the same handle, in one chunk and in
    several."""
    host(f'''
h = net(chain(40, 3))
h.set_option(Bd.OPT_FORM, 2)
for chunk in (-1, 96):
    h.set_option(Bd.OPT_HBM_CHUNK, -1)
    assert simulate(h, {scheme}, 600) == 0
    h.set_option(Bd.OPT_HBM_CHUNK, chunk)
    for R in (401, 33, 410, 1):
        assert {"sojourn(h, %d, R, 5)" % scheme if call == "sojourn" else "grad(h, %d, R)" % scheme} == 0
t = log()
assert "hbm_phase_kernel" in t
bad = sorted(set(x for x in t.splitlines() if "VIOLATION" in x))
assert not bad, bad[:6]
h.close()
''')
