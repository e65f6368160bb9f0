"""FP64 energies (table of erf(alpha r)/r, integer cut-off tests) against the oracle at the
edges of the table's range: no screening (one piece), the last alpha rc the table covers and
the first one that falls back to the library erfc, a Coulomb cut-off inside the LJ one, two
atoms, and rows that end inside a packet.

Tolerance: each pair term of either side is within 8 ulp (9e-16) of the exact one, so
the sums differ by less than 2e-15 sum |u|; sum |u| is below 50 |U| + 50 n for these
configurations (their charges cancel by less than that), hence 1e-13 (|U| + n).
"""
import numpy as np
import pytest

from oracle import oracle as orc
from paper_2307_11447_gb300 import lib as h4d
from paper_2307_11447_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

TWO32 = 4294967296.0


def quantize(x, L):
    return np.mod(np.rint(np.mod(x, L) / L * TWO32), TWO32) * (L / TWO32)


@pytest.mark.parametrize("alpha", [0.0, 0.02, 0.3, 3.54 / 4.0, 3.56 / 4.0])
@pytest.mark.parametrize("n_ions,rho,rc_coul,w_fly", [(2, 0.002, 4.0, 0.0), (162, 0.2, 4.0, 0.0), (250, 0.2, 2.0, 0.0),
                                                      (1000, 0.3, 4.0, 1.7)])
def test_energy_matches_oracle_over_the_table_range(alpha, n_ions, rho, rc_coul, w_fly):
    cfg = wl.lj_config(n_ions, rho, 100, alpha=alpha * 4.0 / rc_coul, rc_coul=rc_coul, kappa_sr=0.5)
    L = cfg["L"]
    x = quantize(wl.lj_positions(n_ions // 2, L, 11), L)
    if n_ions == 2:
        x = quantize(np.array([[0.1, 0.2, 0.3], [1.3, 0.2, 0.3]]), L)
    w = np.zeros(n_ions)
    fly = np.zeros(n_ions, np.uint8)
    if w_fly:
        w[[10, 33]] = float(np.float32(w_fly))
        fly[[10, 33]] = 1
    Uo, _ = orc.energy_forces(orc.make_params(cfg), x, w, fly)
    Ug, _ = h4d.h4d_eval_forces(h4d.make_params(cfg), L, x, w)
    assert abs(Ug - Uo) <= 1e-13 * (abs(Uo) + n_ions), (Ug, Uo)
