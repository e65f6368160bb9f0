"""The scratch pool of the stateless calls: a program that resets the device goes on as before."""
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

CODE = """
import ctypes, os, sys
sys.path.insert(0, os.getcwd())
import numpy as np
from paper_2307_11447_gb300 import lib as h4d, workloads as wl

cfg = wl.lj_config(250, 0.2, 10)
L, p = cfg["L"], h4d.make_params(cfg)
x = wl.lj_positions(125, L, 3)
rng = np.random.default_rng(1)
w = rng.normal(size=h4d.H4D_PROP_NW) * 0.1
f, t = rng.random((64, 2, 96)).astype(np.float32), rng.random((64, 2)).astype(np.float32)

def calls():
    U, F = h4d.h4d_eval_forces(p, L, x)
    u, s, G = h4d.h4d_ewald_lr(p, L, x, 0.6, 5)
    l, g = h4d.h4d_proposal_grad(w, f, t)
    return [np.array([U, u, s, l]).tobytes(), F.tobytes(), G.tobytes(), g.tobytes()]

want = calls()
rt = ctypes.CDLL("libcudart.so.13")
for _ in range(2):
    assert rt.cudaDeviceReset() == 0
    assert calls() == want and calls() == want
print("ok")
"""


def test_stateless_calls_after_a_device_reset():
    r = subprocess.run([sys.executable, "-c", CODE], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout == "ok\n", (r.returncode, r.stdout, r.stderr)
