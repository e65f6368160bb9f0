"""The three forms of the LJ-electrolyte pair loop (erfc; polynomial Coulomb term with the LJ
cut-off inside the Coulomb one, and beyond it) against the oracle, in 3D and with a flying pair,
through the entry point that runs the engine's lists and force pass.  Tolerance as in the other
force tests: 1e-5 (|F| + F_rms) per atom plus the force jump of pairs at a cut-off."""
import numpy as np
import pytest

from oracle import oracle as orc
from paper_2307_11447_gb300 import lib as h4d
from paper_2307_11447_gb300 import workloads as wl

from .parity_util import force_bounds

pytestmark = pytest.mark.gpu

TWO32 = 4294967296.0


@pytest.mark.parametrize("alpha,rc_coul", [(0.5, 4.0), (0.3, 4.0), (0.3, 2.5), (0.3, 2.0)])
@pytest.mark.parametrize("n_ions,w_fly", [(250, 0.0), (162, 1.7)])
def test_force_forms_match_oracle(alpha, rc_coul, n_ions, w_fly):
    cfg = wl.lj_config(n_ions, 0.2, 100, alpha=alpha, rc_coul=rc_coul, kappa_sr=0.5)
    assert h4d.h4d_coulomb_poly(alpha, rc_coul)[1] == (alpha * rc_coul <= 1.3)
    L = cfg["L"]
    x = wl.lj_positions(n_ions // 2, L, 17)
    x = np.mod(np.rint(np.mod(x, L) / L * TWO32), TWO32) * (L / TWO32)
    w = np.zeros(n_ions)
    fly = np.zeros(n_ions, np.uint8)
    if w_fly:
        w[[10, 33]] = float(np.float32(w_fly))
        fly[[10, 33]] = 1
    _, Fo = orc.energy_forces(orc.make_params(cfg), x, w, fly)
    _, Fg = h4d.h4d_eval_forces_static(h4d.make_params(cfg), L, x, w)
    err, bound = np.linalg.norm(Fg - Fo, axis=1), force_bounds(cfg, x, Fo, w)
    keep = fly == 0  # a flyer's 3D force is never used
    assert np.all(err[keep] <= bound[keep]), (err[keep] / bound[keep]).max()
