"""The largest systems that fit the static scratch array: the FP64 Coulomb table takes its place only
where there is room for it, and the results are those of h4d_eval_forces with and without it."""
import numpy as np
import pytest

from paper_2307_11447_gb300 import lib as h4d
from paper_2307_11447_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [6216, 6218, 6220, 6222])
def test_sizes_up_to_the_limit(n):
    cfg = wl.lj_config(n, 0.3, 10)
    L, p = cfg["L"], h4d.make_params(cfg)
    x = wl.lj_positions(n // 2, L, 4)
    w = np.zeros(n)
    w[[5, 40]] = 1.25
    Us, Fs = h4d.h4d_eval_forces_static(p, L, x, w)
    Ua, Fa = h4d.h4d_eval_forces(p, L, x, w)
    assert Us == pytest.approx(Ua, rel=1e-12)
    frms = np.sqrt((Fa**2).sum(1).mean())
    assert np.all(np.linalg.norm(Fs - Fa, axis=1) <= 1e-5 * (np.linalg.norm(Fa, axis=1) + frms))


def test_the_next_size_is_refused():
    cfg = wl.lj_config(6224, 0.3, 10)
    with pytest.raises(h4d.H4DError) as e:
        h4d.h4d_eval_forces_static(h4d.make_params(cfg), cfg["L"], wl.lj_positions(3112, cfg["L"], 4), np.zeros(6224))
    assert e.value.code == h4d.H4D_ECAPACITY
