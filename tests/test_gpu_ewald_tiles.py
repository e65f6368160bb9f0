"""Long-range Coulomb term at the edges of its tiles: atom counts around one stage (64 atoms) and
one chunk (512), and enough of them for several batches; k ranges around one tile of n_z values
(16) and of columns (32).  Reference: the half-space sum in complex128.

Tolerances as for the other sizes (U_recip 1e-6, forces 1e-5 (|F| + F_rms)): a term's two phases
are good to 1e-7 each and the FP32 sums are no longer than 64 terms, so the errors of the sums
are below 1e-6 of their root-mean-square size.
"""
import numpy as np
import pytest

from paper_2307_11447_gb300 import lib as h4d
from paper_2307_11447_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

TWO32 = 4294967296.0


def _reference(x, q, L, K, alpha, kmax):
    ph = 2.0 * np.pi * x / L
    m = np.arange(-kmax, kmax + 1)
    ey, ez = np.exp(1j * np.outer(m, ph[:, 1])), np.exp(1j * np.outer(m, ph[:, 2]))
    g, u, F = 2.0 * np.pi / L, 0.0, np.zeros_like(x)
    for nx in range(kmax + 1):
        a = np.exp(1j * nx * ph[:, 0]) * ey  # [n_y, atom]
        S = (a * q) @ ez.T
        k2 = g * g * (nx * nx + m[:, None] ** 2 + m[None, :] ** 2)
        keep = np.ones(k2.shape, bool)
        if nx == 0:
            keep = (m[:, None] > 0) | ((m[:, None] == 0) & (m[None, :] > 0))
        A = np.where(keep, np.exp(-k2 / (4.0 * alpha**2)) / np.where(k2 > 0, k2, 1.0), 0.0)
        u += float((A * np.abs(S) ** 2).sum())
        W = A * np.conj(S)
        T, Tz = W @ ez, (W * m[None, :]) @ ez
        F[:, 0] += nx * (a * T).imag.sum(0)
        F[:, 1] += (m[:, None] * (a * T).imag).sum(0)
        F[:, 2] += (a * Tz).imag.sum(0)
    V = L**3
    return 4.0 * np.pi * K / V * u, F * q[:, None] * (8.0 * np.pi * K / V * g)


@pytest.mark.parametrize("n,kmax", [(2, 1), (2, 15), (62, 3), (64, 16), (66, 5), (130, 17), (512, 2), (514, 14), (3586, 64)])
def test_tile_edges(n, kmax):
    cfg = dict(wl.CONFIGS["lj250"])
    L, alpha = cfg["L"], 0.6
    x = np.random.default_rng(n + kmax).uniform(0.0, L, (n, 3))
    x = np.mod(np.rint(x / L * TWO32), TWO32) * (L / TWO32)
    q = np.where(np.arange(n) % 2 == 0, cfg["q"][0], cfg["q"][1])
    uo, Fo = _reference(x, q, L, cfg["kcoul"], alpha, kmax)
    p = h4d.make_params(cfg)
    u, _, F = h4d.h4d_ewald_lr(p, L, x, alpha, kmax)
    assert abs(u - uo) <= 1e-6 * abs(uo)
    err, f = np.linalg.norm(F - Fo, axis=1), np.linalg.norm(Fo, axis=1)
    assert np.all(err <= 1e-5 * (f + np.sqrt((f**2).mean())))
    assert h4d.h4d_ewald_lr(p, L, x, alpha, kmax, forces=False)[0] == u
