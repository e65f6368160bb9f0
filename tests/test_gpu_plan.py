"""Warps per replica of a launch with no more replicas than SMs: 16 below 300 atoms, 32 from there on,
with the bits of each replica alone (which has 16)."""
import numpy as np
import pytest

from paper_2307_11447_gb300 import lib as h4d
from paper_2307_11447_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def _run(cfg, reps):
    ctx = h4d.Context(h4d.make_params(cfg), reps, seed=5)
    ctx.h4d_run_md(25)
    ctx.h4d_run_trials(3, 5)
    out = [(ctx.h4d_get_state(r), ctx.h4d_get_work(r, 8), ctx.h4d_get_counts(r)["plan_warps"]) for r in range(len(reps))]
    ctx.close()
    return out


@pytest.mark.parametrize("n,warps", [(250, 16), (298, 16), (300, 32), (1000, 32)])
def test_small_replicas_keep_16_warps(n, warps):
    cfg = wl.lj_config(n, 0.2, 12, beta_mu=-8.7)
    reps = [dict(L=cfg["L"], n_pairs=n // 2, cap_pairs=n // 2 + 30, x=wl.lj_positions(n // 2, cfg["L"], s), key=s) for s in (3, 4)]
    both = _run(cfg, reps)
    for r in range(2):
        (x, v), rec, w = both[r]
        (xa, va), reca, wa = _run(cfg, [reps[r]])[0]
        assert (w, wa) == (warps, 16)
        assert np.array_equal(x, xa) and np.array_equal(v, va) and rec.tobytes() == reca.tobytes()
