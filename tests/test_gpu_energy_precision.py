"""FP64 energies against sums in extended precision: h4d_eval_forces and h4d_get_energies must be
as good as FP64 erfc, square roots and divisions per pair.

Electrolytes at random positions: a pair term carries a few independent roundings (the r^-12 term
six times those of r^2), so the error of the sum in units of 2^-53 (|U| + sqrt(sum u^2)) has an rms
of 1 to 2; an error shared by many pairs (a rounded unit, a rounded table constant) grows with
their number instead.  Bound: 3.5 over ten configurations.

Waters on a lattice: equal distances share their roundings, so each term's one rounding (2^-53 |u|,
half of it on average) only averages over the some hundred distinct distances.  Bound: 0.5 2^-53 sum |u|.
"""
import numpy as np
import pytest

from paper_2307_11447_gb300 import lib as h4d
from paper_2307_11447_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

TWO32 = 4294967296.0
LD = np.longdouble
PI = LD(np.pi) + LD(1.2246467991473532e-16)


def _erf_over_r(alpha, s):
    """erf(alpha r)/r, r^2 = s: 2 alpha/sqrt(pi) e^-v sum (2v)^k / (2k+1)!!, v = alpha^2 s"""
    v = LD(alpha) ** 2 * s
    t, tot, k = np.ones_like(s), np.zeros_like(s), 0
    while np.max(t / (tot + t)) > 1e-22:
        tot = tot + t
        k += 1
        t = t * (2 * v) / (2 * k + 1)
    return LD(alpha) * 2 / np.sqrt(PI) * np.exp(-v) * tot


def _reference(cfg, X, nw3):
    """U, sum |u| and sum u^2 of positions X on the 32-bit grid"""
    n, sc = len(X), LD(cfg["L"]) / LD(TWO32)
    a = np.arange(n)
    ty = np.where(a < nw3, np.where(a % 3 == 0, 2, 3), (a - nw3) & 1)
    q, sig, eps = (np.array(cfg[k], LD) for k in ("q", "sig", "eps"))
    rl2, rc2 = LD(cfg["rc_lj"]) ** 2, LD(cfg["rc_coul"]) ** 2
    shift = 1 / LD(cfg["rc_coul"]) - _erf_over_r(cfg["alpha"], np.array([rc2]))[0]
    U = A = Q = LD(0)
    for i in range(n - 1):
        d = (X[i + 1:] - X[i]).astype(np.int32).astype(np.int64)
        d2 = (d * d).astype(np.uint64).sum(1)
        near = d2.astype(float) * float(sc) ** 2 < 1.001 * float(max(rl2, rc2))
        if i < nw3:
            near[: i - i % 3 + 2 - i] = False  # the rest of its molecule
        j = np.nonzero(near)[0] + i + 1
        if len(j) == 0:
            continue
        s = d2[j - i - 1].astype(LD) * sc * sc
        e4, sg2 = 4 * np.sqrt(eps[ty[i]] * eps[ty[j]]), ((sig[ty[i]] + sig[ty[j]]) / 2) ** 2
        s6, c6 = (sg2 / s) ** 3, (sg2 / rl2) ** 3
        u = np.where(s < rl2, e4 * (s6 * s6 - s6 - c6 * c6 + c6), 0)
        u += np.where(s < rc2, LD(cfg["kcoul"]) * q[ty[i]] * q[ty[j]] * (1 / np.sqrt(s) - _erf_over_r(cfg["alpha"], s) - shift), 0)
        U, A, Q = U + u.sum(), A + np.abs(u).sum(), Q + (u * u).sum()
    return U, A, Q


def _energies(cfg, x, nw):
    L = cfg["L"]
    X = np.mod(np.rint(np.mod(x, L) / L * TWO32), TWO32).astype(np.uint64).astype(np.uint32)
    xq = X.astype(float) * (L / TWO32)
    p, n_pairs = h4d.make_params(cfg), (len(x) - 3 * nw) // 2
    point = h4d.h4d_eval_forces(p, L, xq, n_water=nw)[0]
    ctx = h4d.Context(p, [dict(L=L, n_pairs=n_pairs, cap_pairs=n_pairs, x=xq, n_water=nw)], seed=1)
    engine = ctx.h4d_get_energies(0)[0]
    ctx.close()
    return X, np.array([point, engine])


def test_electrolyte_energies_have_no_shared_error():
    rng = np.random.default_rng(1)
    z = []
    for k in range(10):
        cfg = wl.lj_config(1000, rng.uniform(0.15, 0.34), 10)
        X, u = _energies(cfg, wl.lj_positions(500, cfg["L"], 100 + k), 0)
        U, _, Q = _reference(cfg, X, 0)
        z.append((u - U) / (2.0**-53 * (abs(U) + np.sqrt(Q))))
    rms = np.sqrt((np.array(z, float) ** 2).mean(0))
    print("rms error (single point, engine):", rms)
    assert np.all(rms <= 3.5), rms


def test_water_lattice_energies_have_no_shared_error():
    L = (31.0 * 400 * 1.05) ** (1 / 3)  # (its square is not exact in FP64)
    cfg = wl.aq_config(400, 10, L, 10)
    X, u = _energies(cfg, wl.aqueous_positions(400, 10, L, 50), 400)
    U, A, _ = _reference(cfg, X, 1200)
    z = (u - U) / (2.0**-53 * A)
    print("error / (2^-53 sum |u|):", z.astype(float))
    assert np.all(np.abs(z) <= 0.5), z
