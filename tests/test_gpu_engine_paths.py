"""The engine's own pair loops and energies against the oracle, through the entry points that run
them (h4d_eval_forces_static, h4d_get_energies; h4d_eval_forces has a kernel of its own), where the
other tests do not reach: aqueous rows with flyers and without the fitted erfcx, energies at the
edges of the Coulomb table, and h4d_eval_forces where it falls back to the engine's lists.

Tolerances as in the other force and energy tests: 1e-5 (|F| + F_rms) per atom plus the force jump of
pairs at a cut-off; 1e-13 (|U| + n) for electrolytes, 1e-10 |U| for water (sum |u| is some hundred
times |U|)."""
import numpy as np
import pytest

from oracle import oracle as orc
from paper_2307_11447_gb300 import lib as h4d
from paper_2307_11447_gb300 import workloads as wl

from .parity_util import force_bounds

pytestmark = pytest.mark.gpu

TWO32 = 4294967296.0


def quantize(x, L):
    return np.mod(np.rint(np.mod(x, L) / L * TWO32), TWO32) * (L / TWO32)


@pytest.mark.parametrize("alpha", [0.25, 0.319, 0.321, 0.36])  # erfcx fitted up to alpha rc = 3.2, table up to 3.55
@pytest.mark.parametrize("w_fly", [0.0, 1.75])
def test_aqueous_rows_match_oracle(alpha, w_fly):
    nw, n_pairs, L = 400, 10, 24.0
    cfg = wl.aq_config(nw, n_pairs, L, 20, alpha=alpha)
    x = quantize(wl.aqueous_positions(nw, n_pairs, L, 2), L)
    w, fly = np.zeros(len(x)), np.zeros(len(x), np.uint8)
    if w_fly:
        k = [3 * nw + 4, 3 * nw + 7]  # a cation and an anion
        w[k] = float(np.float32(w_fly))
        fly[k] = 1
    Uo, Fo = orc.energy_forces(orc.make_params(cfg), x, w, fly)
    Ug, Fg = h4d.h4d_eval_forces_static(h4d.make_params(cfg), L, x, w, n_water=nw)
    err, bound = np.linalg.norm(Fg - Fo, axis=1), force_bounds(cfg, x, Fo, w)
    keep = fly == 0  # a flyer's 3D force is never used
    assert np.all(err[keep] <= bound[keep]), (err[keep] / bound[keep]).max()
    assert Ug == pytest.approx(Uo, rel=1e-10)


@pytest.mark.parametrize("alpha", [0.0, 0.02, 0.3, 3.54 / 4.0, 3.56 / 4.0])
@pytest.mark.parametrize("n_ions,rho,rc_coul,w_fly", [(2, 0.002, 4.0, 0.0), (162, 0.2, 4.0, 0.0), (250, 0.2, 2.0, 0.0),
                                                      (1000, 0.3, 4.0, 1.7)])
def test_engine_energy_matches_oracle_over_the_table_range(alpha, n_ions, rho, rc_coul, w_fly):
    cfg = wl.lj_config(n_ions, rho, 100, alpha=alpha * 4.0 / rc_coul, rc_coul=rc_coul, kappa_sr=0.5)
    L = cfg["L"]
    x = quantize(wl.lj_positions(n_ions // 2, L, 11), L)
    if n_ions == 2:
        x = quantize(np.array([[0.1, 0.2, 0.3], [1.3, 0.2, 0.3]]), L)
    w, fly = np.zeros(n_ions), np.zeros(n_ions, np.uint8)
    if w_fly:
        w[[10, 33]] = float(np.float32(w_fly))
        fly[[10, 33]] = 1
    p = h4d.make_params(cfg)
    Uo, _ = orc.energy_forces(orc.make_params(cfg), x, w, fly)
    U = [h4d.h4d_eval_forces_static(p, L, x, w)[0]]
    if not w_fly:
        ctx = h4d.Context(p, [dict(L=L, n_pairs=n_ions // 2, cap_pairs=n_ions // 2, x=x)], seed=1)
        U.append(ctx.h4d_get_energies(0)[0])
        ctx.close()
    assert np.all(np.abs(np.array(U) - Uo) <= 1e-13 * (abs(Uo) + n_ions)), (U, Uo)


@pytest.mark.parametrize("n_ball", [128, 129, 130])
def test_rows_near_their_capacity_go_through_the_lists(n_ball):
    # rows of 128 entries, and a ball whose atoms are all in each other's rows: from 129 atoms on, the
    # single-point kernel's count (the atom itself included) sends the call through the lists,
    # where 129 atoms fit and 130 do not
    L = 40.0
    cfg = wl.lj_config(140, 140 / L**3, 10, max_nbr=128)
    g = np.arange(-10, 11) * 0.65
    x = np.stack(np.meshgrid(g, g, g, indexing="ij"), -1).reshape(-1, 3)
    r = np.sqrt((x**2).sum(1))
    k = np.argsort(r, kind="stable")[:n_ball]
    assert 2 * r[k].max() < cfg["rc_coul"] + cfg["skin"]
    far = np.stack([np.arange(140 - n_ball) * 1.1 - 6.0, np.zeros(140 - n_ball), np.full(140 - n_ball, 15.0)], 1)
    x = quantize(np.concatenate([x[k], far]) + L / 2, L)
    p = h4d.make_params(cfg)
    if n_ball == 130:
        with pytest.raises(h4d.H4DError) as e:
            h4d.h4d_eval_forces(p, L, x)
        assert e.value.code == h4d.H4D_ECAPACITY
        return
    Uo, Fo = orc.energy_forces(orc.make_params(cfg), x, np.zeros(140), np.zeros(140, np.uint8))
    Ug, Fg = h4d.h4d_eval_forces(p, L, x)
    assert np.all(np.linalg.norm(Fg - Fo, axis=1) <= force_bounds(cfg, x, Fo))
    assert abs(Ug - Uo) <= 1e-13 * (abs(Uo) + 140)


@pytest.mark.parametrize("alpha", [0.3, 0.9])  # Coulomb table, library erfc
def test_waters_in_an_lj_system_have_the_energy_of_their_types(alpha):
    cfg = wl.lj_config(250, 0.2, 10, alpha=alpha)
    x = quantize(wl.lj_positions(125, cfg["L"], 7), cfg["L"])
    p = h4d.make_params(cfg)
    Up, _ = h4d.h4d_eval_forces(p, cfg["L"], x, n_water=8)
    Ue, _ = h4d.h4d_eval_forces_static(p, cfg["L"], x, n_water=8)
    assert Up == pytest.approx(Ue, rel=1e-12)
    assert Up != pytest.approx(h4d.h4d_eval_forces(p, cfg["L"], x)[0], rel=1e-6)
