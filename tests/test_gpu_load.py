"""What h4d_load keeps of the context it loads into: the training-record rings of every replica,
whichever of them was read last."""
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
