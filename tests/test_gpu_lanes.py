"""Paths whose results must be the same bits: four lanes taking several parts of a row against one
lane per part, at the sizes where the default number of parts changes and with rows that end in
any part; two replicas with 32 warps each against each alone with 16; records read in one piece
and across the end of the ring."""
import numpy as np
import pytest

from paper_2307_11447_gb300 import lib as h4d
from paper_2307_11447_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def _replica(n, rho, cap, seed):
    L = wl.box_for(n, rho)
    return dict(L=L, n_pairs=n // 2, cap_pairs=cap, x=wl.lj_positions(n // 2, L, seed))


def _run(cfg, reps, tpa=0):
    ctx = h4d.Context(h4d.make_params(cfg, threads_per_atom=tpa), reps, seed=5)
    ctx.h4d_run_md(25)
    ctx.h4d_run_trials(3, 5)
    out = [(ctx.h4d_get_state(r), ctx.h4d_get_work(r, 8)) for r in range(len(reps))]
    tpa = ctx.h4d_get_counts(0)["threads_per_atom"]
    ctx.close()
    return out, tpa


def _same(a, b):
    (xa, va), ra = a
    (xb, vb), rb = b
    return np.array_equal(xa, xb) and np.array_equal(va, vb) and ra.tobytes() == rb.tobytes()


@pytest.mark.parametrize("n,rho,cap", [(110, 0.1, 60), (250, 0.2, 255), (250, 0.2, 256), (300, 0.3, 160), (1000, 0.3, 510)])
def test_parts_of_a_row_on_fewer_lanes_give_the_same_bits(n, rho, cap):
    cfg = wl.lj_config(n, rho, 12, beta_mu=-8.7)
    reps = [_replica(n, rho, cap, 3)]
    a, tpa = _run(cfg, reps)
    assert tpa == (16 if 2 * cap < 512 else 8)
    b, _ = _run(cfg, reps, tpa)
    assert _same(a[0], b[0])


def test_few_replicas_on_wide_ctas_give_the_same_bits():
    cfg = wl.lj_config(250, 0.2, 12, beta_mu=-8.7)
    reps = [dict(_replica(250, 0.2, 150, s), key=s) for s in (3, 4)]
    both, _ = _run(cfg, reps)
    for r in range(2):
        alone, _ = _run(cfg, [reps[r]])
        assert _same(both[r], alone[0])


def test_records_across_the_end_of_the_ring():
    cfg = wl.lj_config(110, 0.1, 1, beta_mu=-8.7)
    ctx = h4d.Context(h4d.make_params(cfg), [_replica(110, 0.1, 80, 9)], seed=5)
    assert len(ctx.h4d_get_work(0, 4)) == 0 and len(ctx.h4d_get_work(0, 0)) == 0
    ctx.h4d_run_trials(1020, 0)
    early = ctx.h4d_get_work(0, 2000)
    assert len(early) == 1020
    ctx.h4d_run_trials(10, 0)  # the ring holds 1024
    late = ctx.h4d_get_work(0, 2000)
    assert len(late) == 1024 and late[:1014].tobytes() == early[6:].tobytes()
    for k in (1, 5, 6, 7, 10):
        assert ctx.h4d_get_work(0, k).tobytes() == late[1024 - k:].tobytes()
    assert np.all(late["n_before"][1:] == late["n_after"][:-1])
    ctx.close()
