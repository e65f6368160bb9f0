"""Getters of one context called by several threads at once: the bits that one thread reads."""
from concurrent.futures import ThreadPoolExecutor

import numpy as np
import pytest

from paper_2307_11447_gb300 import lib as h4d
from paper_2307_11447_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def test_getters_from_several_threads_read_what_one_thread_reads():
    n = [100, 250, 400, 1000] * 2
    cfg = wl.lj_config(250, 0.1, 5, beta_mu=-8.7)
    reps = [dict(L=wl.box_for(m, 0.1), n_pairs=m // 2, cap_pairs=m // 2 + 20, x=wl.lj_positions(m // 2, wl.box_for(m, 0.1), k))
            for k, m in enumerate(n)]
    ctx = h4d.Context(h4d.make_params(cfg), reps, seed=5)
    ctx.h4d_run_trials(12, 3)

    def read(r):
        x, v = ctx.h4d_get_state(r)
        return x.tobytes(), v.tobytes(), ctx.h4d_get_work(r, 8).tobytes(), ctx.h4d_get_counts(r)

    want = [read(r) for r in range(len(n))]
    with ThreadPoolExecutor(8) as ex:
        got = list(ex.map(lambda t: [read((t + k) % len(n)) == want[(t + k) % len(n)] for k in range(100)], range(8)))
    assert np.all(got)
    ctx.close()
