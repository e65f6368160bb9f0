"""Neighbour lists at the edges of the build: boxes without cells, 3 to 8 cells per edge (where
the runs of z neighbours wrap), atom counts that leave partial home passes, masks and packets,
and clustered atoms (cells of many home passes next to empty ones).  Integers: bit-exact
against the fixed-point criterion evaluated in numpy."""
import numpy as np
import pytest

from paper_2307_11447_gb300 import lib as h4d

pytestmark = pytest.mark.gpu

TWO32 = 4294967296.0


def pairs_by_criterion(x, L, r_list):
    X = np.rint(np.mod(x, L) / L * TWO32).astype(np.uint64).astype(np.uint32)
    T = int((r_list / L * TWO32) ** 2)
    out = []
    for i in range(len(x) - 1):
        d = (X[i + 1:] - X[i]).astype(np.int32).astype(np.int64)  # wraps: the minimum image
        d2 = (d * d).astype(np.uint64).sum(1)
        out += [(i, i + 1 + int(k)) for k in np.nonzero(d2 <= np.uint64(T))[0]]
    return out


@pytest.mark.parametrize("n,cells,clustered", [(2, 0, False), (33, 0, False), (250, 0, False), (97, 3, False), (1000, 3, True),
                                               (1023, 4, False), (1500, 5, True), (2001, 8, False), (700, 11, True)])
def test_neighbor_pairs_bit_exact(n, cells, clustered):
    r_list = 2.0
    L = 5.0 if cells == 0 else r_list * (cells + 0.3)
    rng = np.random.default_rng(n)
    x = rng.random((n, 3)) * L
    if clustered:  # half of the atoms in one corner, across the periodic boundary
        x[: n // 2] = rng.normal(size=(n // 2, 3)) * 0.6
    x = np.mod(np.rint(np.mod(x, L) / L * TWO32), TWO32) * (L / TWO32)
    i, j = h4d.h4d_neighbor_pairs(L, x, r_list)
    assert list(zip(i.tolist(), j.tolist())) == pairs_by_criterion(x, L, r_list)
