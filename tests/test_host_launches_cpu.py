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
def dag(n, edges, every=4):
    rp, col, prob = W.csr_from_edges(n, edges)
    w = np.zeros(n); w[::every] = 6.0
    return W.Network(n, rp, col, prob, np.full(n, 9), np.full(n, 1.1),
                     W.Arrivals(kind=W.ARR_SINUSOID, w=w, a=1.0, b=0.2, period=3.0, phase=0.1))
def complete(n):
    return dag(n, [(i, j, 0.9 / (n - 1 - i)) for i in range(n) for j in range(i + 1, n)])
def two_wide(levels):  # two stations to a level, one edge from the first to the last
    e = [(2 * l + a, 2 * l + 2 + b, 0.4) for l in range(levels - 1) for a in range(2) for b in range(2)]
    return dag(2 * levels, e + [(0, 2 * levels - 1, 0.1)])
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


@pytest.mark.parametrize("call", ["simulate", "sojourn", "grad", "average"])
@pytest.mark.parametrize("form", [1, 2])
def test_calls_after_a_failed_allocation(host, call, form):
    """A call whose n-th allocation fails returns an error; the next, smaller
    call on the handle runs on allocations that hold what it addresses."""
    host(f'''
def average(h, scheme, R, T=1.0):
    a = dev(8 * Bd.stats_len(h.n, R))
    rc = L.euler_net_simulate_average(h._h, 0.1, T, R, 1, 0, a, None, None, None)
    RT.cudaFree(a)
    return rc
def go(h, R, T):
    call = {call!r}
    return (simulate(h, 0, R, T=T) if call == "simulate" else sojourn(h, 0, R, 5, T=T) if call == "sojourn" else
            grad(h, 0, R, T=T) if call == "grad" else average(h, 0, R, T=T))
real_dev = dev
def dev(n):  # the test's own buffers never fail
    F.fake_fail_malloc(0)
    p = real_dev(n)
    F.fake_fail_malloc(fail)
    return p
failed = 0
for fail_at in range(1, 12):
    h = net(chain(40, 3))
    h.set_servers_schedule(np.full((3, 40), 4, np.int32), 0.3)
    h.set_option(Bd.OPT_FORM, {form})
    fail = 0
    assert go(h, 300, 1.0) == 0
    fail = fail_at
    rc = go(h, 900, 2.0)
    fail = 0
    F.fake_fail_malloc(0)
    failed += rc != 0
    for R, T in ((200, 1.0), (900, 0.7), (100, 2.0), (900, 2.0)):
        assert go(h, R, T) == 0, (fail_at, R)
    h.close()
bad = sorted(set(x for x in log().splitlines() if "VIOLATION" in x))
assert not bad, bad[:6]
assert failed > 0
''')


def test_batch_after_a_failed_allocation(host):
    """A batch whose re-planning fails an allocation part way either reports it
    or runs on allocations that hold what it addresses."""
    host('''
for fail_at in range(0, 12):
    hs = [net(chain(n, 2)) for n in (3, 40, 120)]
    runs = (Bd._Run * 3)(*[Bd._Run(j % 2, 0.1, 1.0 + j, R, 5, 0) for j, R in enumerate((20000, 5000, 2000))])
    arr = (C.c_void_p * 3)(*[h._h for h in hs])
    b = C.c_void_p()
    assert L.euler_batch_create(C.byref(b), arr, runs, 3) == 0
    st = [dev(8 * Bd.stats_len(h.n, r.replications)) for h, r in zip(hs, runs)]
    ptr = (C.c_void_p * 3)(*[x.value for x in st])
    F.fake_fail_malloc(fail_at)
    L.euler_batch_autotune(b, None, None)
    F.fake_fail_malloc(0)
    L.euler_batch_run(b, ptr, None)
    L.euler_batch_destroy(b)
    for h in hs:
        h.close()
    for x in st:
        RT.cudaFree(x)
t = log()
assert "batch_kernel" in t
bad = sorted(set(x for x in t.splitlines() if "VIOLATION" in x))
assert not bad, bad[:6]
''')


def test_backward_tiles_hold_two_ring_slots(host):
    """A backward slot reads the slot before it only, so long edges take no
    replications from a backward tile; the bytes fit what the kernel addresses."""
    host("""
for make, least in ((lambda: complete(40), 33), (lambda: two_wide(100), 33), (lambda: chain(20, 19), 250)):
    h = net(make())
    h.set_option(Bd.OPT_FORM, 1)
    b, f = h.plan(0, 500_000), h.plan(1, 500_000)
    assert b["form"] == f["form"] == 1
    assert b["tile_reps"] >= least and b["tile_reps"] > 3 * f["tile_reps"], (b, f)
    assert b["smem"] <= 227 * 1024
    h.close()
""")


def test_form_rule(host):
    """The planner's form where a tile holds few units: per-step kernels for
    many waves of small tiles and for a few replications of a large network,
    the persistent form for one wave, for tiles of a few hundred units and for
    backward tiles of the same networks; batches follow for the networks they
    run by themselves."""
    host("""
def form(x, scheme, R):
    h = net(x); f = h.plan(scheme, R)["form"]; h.close(); return f
for x, R in ((complete(40), 10000), (complete(20), 40000), (two_wide(100), 1400), (two_wide(100), 10000)):
    assert form(x, 1, R) == 2 and form(x, 0, R) == 1, (x.n, R)
assert form(complete(12), 1, 40000) == 1 and form(two_wide(35), 1, 40000) == 1
assert form(chain(100), 0, 10000) == form(chain(100), 1, 10000) == 1
for n, R, want in ((3800, 1, 1), (3900, 1, 2), (3900, 6, 2), (3900, 7, 1), (3900, 60, 1), (9000, 4, 2), (2000, 1, 1)):
    assert form(chain(n), 0, R) == want, (n, R)
# tagged customers: as many as leave a tile one replication
h = net(chain(100)); h2 = net(two_wide(100))
for hh, R, S, want in ((h, 3000, 10000, "hbm_phase_kernel"), (h, 3000, 4, "persistent_kernel"),
                       (h, 3000, 5000, "persistent_kernel"), (h, 300, 10000, "persistent_kernel"),
                       (h2, 1400, 4, "hbm_phase_kernel"), (h2, 400, 4, "persistent_kernel")):
    log()
    assert sojourn(hh, 1, R, S) == 0
    assert want in forms(log()), (R, S)
log(); assert grad(h2, 1, 5000) == 0 and "hbm_phase_kernel" in forms(log())
assert grad(h2, 0, 5000) == 0 and "persistent_kernel" in forms(log())
# a caller's capture takes kernels, not the launch of another graph
for x, R in ((h2, 5000), (net(chain(4000)), 1)):
    for on, want in ((0, "hbm_phase_kernel"), (1, "persistent_kernel"), (0, "hbm_phase_kernel")):
        F.fake_capturing(on); log()
        assert simulate(x, 1, R) == 0 and want in forms(log())
h.close(); h2.close()
# in a batch: fewer than 2^18 units a step, but a tile beyond the shared launch's budget
hs = [net(chain(167, 155)), net(chain(3))]
for R, want in ((1500, "hbm_phase_kernel"), (300, "persistent_kernel")):
    runs = (Bd._Run * 2)(Bd._Run(1, 0.1, 1.0, R, 5, 0), Bd._Run(1, 0.1, 0.5, 80, 5, 0))
    b = C.c_void_p()
    assert L.euler_batch_create(C.byref(b), (C.c_void_p * 2)(*[x._h for x in hs]), runs, 2) == 0
    st = [dev(8 * Bd.stats_len(x.n, r.replications)) for x, r in zip(hs, runs)]
    log()
    assert L.euler_batch_run(b, (C.c_void_p * 2)(*[x.value for x in st]), None) == 0
    t = log()
    assert forms(t)[:2] == ["batch_kernel", want] and "VIOLATION" not in t, (R, forms(t))
    L.euler_batch_destroy(b)
""")


def test_options_that_no_longer_fit_the_tile(host):
    """A requested tile within the documented limit runs although the tile's
    lists and arrivals take more than the station sums did; a block for the
    persistent form does not stop a small call whose tile does not fit."""
    host("""
for n, Rt, want in ((450, 32, 16), (535, 32, 16), (545, 32, None), (400, 32, 32), (1611, 8, 4), (900, 16, 8),
                    (30, 512, 256), (23, 512, 512), (60, 512, None)):
    h = net(chain(n, every=1))
    h.set_option(Bd.OPT_FORM, 1)
    h.set_option(Bd.OPT_TILE_REPS, Rt)
    for scheme in (0, 1):
        fits = 256 + 48 * n + Rt * (32 + 4 * (n + 2 * (n - 1))) <= 227 * 1024
        assert fits == (want is not None), (n, Rt)
        try:
            p = h.plan(scheme, 1000)
            assert p["form"] == 1 and p["tile_reps"] == want and p["smem"] <= 227 * 1024, (n, Rt, p)
        except Bd.EulerError as e:
            assert e.code == -7 and not fits, (n, Rt, str(e))
    assert simulate(h, 0, 100) == (0 if fits else -7)
    h.close()
# a deep ring leaves no forward tile: the per-step kernels, at their own block
h = net(complete(60)); h.set_option(Bd.OPT_BLOCK, 512)
log(); assert sojourn(h, 1, 100, 4) == 0 and "hbm_phase_kernel" in forms(log())
h.set_option(Bd.OPT_FORM, 2); assert sojourn(h, 1, 100, 4) == -1
h.close()
h = net(chain(4000)); h.set_option(Bd.OPT_BLOCK, 512)
log(); assert grad(h, 0, 2) == 0
assert h.plan(0, 2)["form"] == 1
h.close()
""")


def test_launches_of_tiles(host):
    """A run beyond 2e10 updates is several launches of whole waves; one wave is
    one launch however long its horizon."""
    host("""
import re
for R, K in ((30000, 10000), (30000, 1000), (300000, 1000), (10000, 400000)):
    h = net(chain(100))
    p = h.plan(0, R)
    tiles = -(-R // p["tile_reps"])
    log()
    assert simulate(h, 0, R, dt=0.01, T=0.01 * K) == 0
    got = [int(x) for x in re.findall(r"tiles=([0-9]+)", log())]
    per = p["grid"] * max(1, int(2e10 / (100.0 * p["tile_reps"] * K * p["grid"])))
    assert sum(got) == tiles and max(got) <= per and len(got) == -(-tiles // per), (R, K, got, per)
    assert (len(got) > 1) == (R * K * 100 > 2e10 and tiles > p["grid"]), (R, K, got)
    h.close()
""")


def test_autotuner_times_step_kernels_where_they_run(host):
    """The per-step kernels' launch shape is chosen on networks that take them,
    and left alone where none does."""
    host("""
def tuned(x, R, scheme):
    hs = [net(x), net(chain(3))]
    runs = (Bd._Run * 2)(Bd._Run(scheme, 0.1, 20.0, R, 5, 0), Bd._Run(0, 0.1, 2.0, 80, 5, 0))
    b = C.c_void_p()
    assert L.euler_batch_create(C.byref(b), (C.c_void_p * 2)(*[x._h for x in hs]), runs, 2) == 0
    log()
    assert L.euler_batch_autotune(b, None, None) == 0
    blocks = set(y.split("block=")[1] for y in log().splitlines() if y.startswith("hbm_phase_kernel"))
    v = [C.c_int32() for _ in range(7)]; v[1] = C.c_int64()
    L.euler_batch_info(b, *[C.byref(y) for y in v])
    L.euler_batch_destroy(b)
    return blocks, v[5].value, v[6].value
for _ in range(4):  # the stand-in's times favour another shape each time
    assert tuned(chain(100), 10000, 0) == (set(), 256, 32)
assert tuned(two_wide(100), 5000, 1)[0] == {"128", "256"}
""")


def test_threads_on_different_networks(host):
    """Calls of several threads, each on its own handle, do not lower one
    another's shared-memory limits."""
    host("""
import threading
def work(n, R, scheme, out):
    h = net(chain(n))
    s = dev(8 * Bd.stats_len(n, R))
    for _ in range(150):
        rc = L.euler_net_simulate(h._h, scheme, 0.1, 1.0, R, 1, 0, s, None)
        if rc:
            out.append((n, rc, L.euler_net_last_error().decode()))
            break
    h.close()
for form_scheme in (0, 1):
    bad = []
    ts = [threading.Thread(target=work, args=(n, R, form_scheme, bad)) for n, R in ((100, 10000), (100, 4000), (90, 9000))]
    [t.start() for t in ts]; [t.join() for t in ts]
    assert not bad, bad
""")


def test_batch_tile_leaves_room_for_its_tables(host):
    """The largest shared-memory budget of the autotuner leaves room for the
    work item's tables, which are static memory of the batched kernel."""
    host("""
for n in (1887, 1890, 943, 944):  # 8 and 16 replications: 232,048 to 232,448 bytes
    hs = [net(chain(n))]
    runs = (Bd._Run * 1)(Bd._Run(0, 0.1, 1.0, 150, 5, 0))
    b = C.c_void_p()
    assert L.euler_batch_create(C.byref(b), (C.c_void_p * 1)(hs[0]._h), runs, 1) == 0
    st = (C.c_void_p * 1)(dev(8 * Bd.stats_len(n, 150)))
    for _ in range(6):  # the stand-in's times favour another shape each time
        assert L.euler_batch_autotune(b, None, None) == 0, L.euler_net_last_error()
        assert L.euler_batch_run(b, st, None) == 0, L.euler_net_last_error()
    L.euler_batch_destroy(b)
    hs[0].close()
""")
