"""The host side of libh4d over a CUDA runtime that needs no GPU (tests/host/fake_cudart.c,
preloaded in a child process): what several threads, several devices and failing calls do to it."""
import os
import subprocess
import sys

import pytest

from paper_2307_11447_gb300 import lib as h4d

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SETUP = """
import ctypes, sys
import numpy as np
from concurrent.futures import ThreadPoolExecutor
from paper_2307_11447_gb300 import lib as h4d, workloads as wl
rt = ctypes.CDLL(None)
cfg = wl.lj_config(100, 0.1, 10)

def context(R):
    rng = np.random.default_rng(1)
    reps = [dict(L=cfg["L"], n_pairs=50 - r, cap_pairs=60, x=rng.uniform(0, cfg["L"], (100 - 2 * r, 3)),
                 v=rng.normal(size=(100 - 2 * r, 3))) for r in range(R)]
    return h4d.Context(h4d.make_params(cfg), reps, seed=1), reps
"""


@pytest.fixture(scope="session")
def runtime(tmp_path_factory):
    h4d.lib()  # built before the children load it
    out = tmp_path_factory.mktemp("host") / "fake_cudart.so"
    inc = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
    subprocess.check_call(["gcc", "-O1", "-Wall", "-fexceptions", "-fPIC", "-shared", "-I", inc, "-o", str(out),
                           os.path.join(ROOT, "tests", "host", "fake_cudart.c"), "-lstdc++"])

    def run(code):
        env = dict(os.environ, LD_PRELOAD=str(out), PYTHONPATH=ROOT)
        r = subprocess.run([sys.executable, "-c", SETUP + code], env=env, cwd=ROOT, capture_output=True, text=True, timeout=120)
        assert r.returncode == 0 and r.stdout.endswith("ok\n"), (r.returncode, r.stdout, r.stderr)

    return run


def test_getters_from_several_threads_read_what_one_thread_reads(runtime):
    runtime("""
ctx, reps = context(8)
want = [ctx.h4d_get_state(r) for r in range(8)]
for r, rep in enumerate(reps):
    assert np.abs(want[r][0] - rep["x"]).max() < 1e-8 and np.abs(want[r][1] - rep["v"]).max() < 1e-6

def read(t):
    bad = 0
    for k in range(60):
        r = (t + k) % 8
        x, v = ctx.h4d_get_state(r)
        bad += not (np.array_equal(x, want[r][0]) and np.array_equal(v, want[r][1]))
        bad += ctx.h4d_get_counts(r)["n_pairs"] != 50 - r
    return bad

with ThreadPoolExecutor(8) as ex:
    bad = sum(ex.map(read, range(8)))
assert bad == 0, bad
ctx.close()
print("ok")
""")


def test_getters_work_from_another_current_device(runtime):
    runtime("""
ctx, reps = context(2)
x0, v0 = ctx.h4d_get_state(1)
c0 = ctx.h4d_get_counts(1)
rt.cudaSetDevice(1)
x1, v1 = ctx.h4d_get_state(1)
assert np.array_equal(x0, x1) and np.array_equal(v0, v1)
assert len(ctx.h4d_get_work(1, 4)) == 0 and ctx.h4d_get_counts(1) == c0
dev = ctypes.c_int(-1)
rt.cudaGetDevice(ctypes.byref(dev))
assert dev.value == 1
print("ok")
""")


def test_stateless_calls_keep_at_most_the_pool_bound(runtime):
    runtime("""
rt.fake_device_bytes.restype = ctypes.c_size_t
keep = 16 << 20
for n in (64, 60000):  # a gradient of 60000 records takes 53 MB of scratch
    h4d.h4d_proposal_grad(np.zeros(h4d.H4D_PROP_NW), np.zeros((n, 2, 96), np.float32), np.zeros((n, 2), np.float32))
    assert rt.fake_device_bytes() <= keep, (n, rt.fake_device_bytes())
h4d.h4d_proposal_grad(np.zeros(h4d.H4D_PROP_NW), np.zeros((64, 2, 96), np.float32), np.zeros((64, 2), np.float32))
context(2)[0].close()  # what the pool keeps goes back with a context
assert rt.fake_device_bytes() == 0
print("ok")
""")


def test_stateless_calls_work_after_a_device_reset(runtime):
    runtime("""
def grad():
    h4d.h4d_proposal_grad(np.zeros(h4d.H4D_PROP_NW), np.zeros((64, 2, 96), np.float32), np.zeros((64, 2), np.float32))

grad()
for _ in range(2):
    rt.cudaDeviceReset()
    grad()
    grad()
print("ok")
""")


def test_static_scratch_is_found_again_after_a_device_reset(runtime):
    runtime("""
x = np.random.default_rng(1).uniform(0, cfg["L"], (100, 3))
for _ in range(3):
    h4d.h4d_eval_forces_static(h4d.make_params(cfg), cfg["L"], x)
    rt.cudaDeviceReset()
print("ok")
""")


def test_no_exception_crosses_the_interface(runtime):
    runtime("""
L, p = cfg["L"], h4d.make_params(cfg)
x = np.random.default_rng(1).uniform(0, L, (100, 3))
w, f, t = np.zeros(h4d.H4D_PROP_NW), np.zeros((64, 2, 96), np.float32), np.zeros((64, 2), np.float32)
ctx, _ = context(2)
rt.fake_device_bytes.restype = ctypes.c_size_t

def out_of_memory(call, at_least):
    held, failed = rt.fake_device_bytes(), 0
    for k in range(60):
        rt.fake_fail_new(k)
        try:
            call()
        except h4d.H4DError as e:
            failed += 1
            assert e.code == h4d.H4D_ECUDA, e
            assert rt.fake_device_bytes() <= held, k  # (a failed context gives the pool back too)
        finally:
            rt.fake_fail_new(-1)
    assert failed >= at_least, failed

out_of_memory(lambda: h4d.h4d_proposal_grad(w, f, t), 1)  # first, while it makes the scratch pool
out_of_memory(lambda: h4d.h4d_eval_forces(p, L, x), 2)
out_of_memory(lambda: h4d.h4d_eval_forces_static(p, L, x), 1)
out_of_memory(lambda: context(2)[0].close(), 5)
rt.fake_fail_pinned(1)
ctx, _ = context(2)  # one without a pinned buffer yet
out_of_memory(lambda: ctx.h4d_get_state(0), 1)
out_of_memory(lambda: ctx.h4d_get_work(0, 4), 1)
print("ok")
""")
