"""Two atoms on one grid point: the Coulomb energy of two like charges is infinite, not NaN."""
import numpy as np
import pytest

from paper_2307_11447_gb300 import lib as h4d
from paper_2307_11447_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("call", [h4d.h4d_eval_forces, h4d.h4d_eval_forces_static])
@pytest.mark.parametrize("alpha", [0.25, 0.36])  # table of erf(alpha r)/r, library erfc
def test_hydrogens_on_one_point_have_infinite_energy(call, alpha):
    L = 32.0
    cfg = wl.aq_config(2, 0, L, 10, alpha=alpha)
    d, h = cfg["d_oh"], cfg["d_hh"]
    y = np.sqrt(d * d - h * h / 4)
    # the second water mirrored at the first one's second hydrogen: only these two coincide
    a = np.array([[0, 0, 0], [-h / 2, y, 0], [h / 2, y, 0]]) + 16.0
    a = np.rint(a / L * 2.0**32) * (L / 2.0**32)
    x = np.concatenate([a, 2 * a[2] - a])
    U, _ = call(h4d.make_params(cfg), L, x, n_water=2)
    assert U == np.inf
