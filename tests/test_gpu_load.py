"""What h4d_load keeps of the context it loads into (the training-record rings of every replica,
whichever of them was read last) and what it takes from the file (a row's parts and lanes)."""
import numpy as np
import pytest

from paper_2307_11447_gb300 import lib as h4d
from paper_2307_11447_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def _context(R=2, **kw):
    cfg = wl.lj_config(250, 0.2, 10, beta_mu=-8.7)
    reps = [dict(L=cfg["L"], n_pairs=125, cap_pairs=150, x=wl.lj_positions(125, cfg["L"], k)) for k in range(R)]
    return h4d.Context(h4d.make_params(cfg, **kw), reps, seed=3)


def test_training_records_of_every_replica_survive_a_load(tmp_path):
    path = str(tmp_path / "c")
    ctx = _context()
    ctx.h4d_proposal(h4d.H4D_PROPOSAL_UNIFORM, 1.0, records_per_replica=64)
    ctx.h4d_run_trials(6, 0)
    ctx.h4d_save(path)
    ctx.h4d_run_trials(4, 0)
    assert ctx.h4d_get_counts(0)["cycles"] == 10  # reads replica 0 alone
    ctx.h4d_load(path)
    assert [len(ctx.h4d_proposal_records(r)[1]) for r in range(2)] == [10, 10]
    assert [ctx.h4d_get_counts(r)["cycles"] for r in range(2)] == [6, 6]
    ctx.close()


def _layout(ctx, path):
    """parts and lanes of a row of replica 0, from the table entry that a checkpoint holds"""
    ctx.h4d_save(path)
    parts, lanes = np.fromfile(path, np.int32, 2, offset=32 + 56)
    assert parts == ctx.h4d_get_counts(0)["threads_per_atom"]
    return int(parts), int(lanes)


def test_lanes_of_a_row_come_with_its_parts(tmp_path):
    path = str(tmp_path / "a")
    a, b = _context(1), _context(1, threads_per_atom=1)
    assert _layout(a, path) == (16, 4) and _layout(b, str(tmp_path / "b")) == (1, 1)
    b.h4d_load(path)
    assert _layout(b, str(tmp_path / "b")) == (16, 4)
    a.h4d_run_trials(3, 5)
    b.h4d_run_trials(3, 5)
    assert all(np.array_equal(u, v) for u, v in zip(a.h4d_get_state(0), b.h4d_get_state(0)))
    # lanes that no kernel takes (a row has at most four parts to a lane) are not taken over
    raw = np.fromfile(path, np.int32)
    for bad in (0, 2, 3, 32):
        raw[(32 + 60) // 4] = bad
        raw.tofile(path)
        c = _context(1, threads_per_atom=1)
        c.h4d_load(path)
        assert _layout(c, str(tmp_path / "b")) == (16, 16)
        c.close()
    a.close()
    b.close()
