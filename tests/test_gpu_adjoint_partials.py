"""Entries of the FP64 adjoint that consist of one partial derivative of the
convection increment (Eq. 28): with a cotangent of single entries, far apart, the
entries upwind of one hold lam dM/df alone, no sum that would hide how
many digits the partial has.  Against the oracle's entries, relative to
each; one grid per tile height (2, 4 and 8 rows).

Tolerance 1e-11 relative: the oracle's own partials lose up to 2^-53 / v to
cancellation, v = |D| / (|D| + |Dp|) > 1e-4 in all but a few entries; those left out
below 1e-3 of the largest also cover directions nearly along a coordinate line,
whose Courant numbers are a cancelled cosine.
"""
import math

import numpy as np
import pytest

import oracle as O
from paper_1302_7104_gb300 import inputs as I
from paper_1302_7104_gb300 import pclb as P

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

GRIDS = [(64, 24), (64, 400), (64, 1000)]


def _adjoint(w, f, lam):
    with P.PCLB(w, precision="fp64") as g:
        out = g.adjoint_step(torch.as_tensor(f, device="cuda"), torch.as_tensor(lam, device="cuda"))
        return out.cpu().numpy(), g.status_flags()


def _state(w):
    f = O.set_state(w)
    return np.ascontiguousarray(f * (1.0 + 0.02 * np.random.default_rng(3).normal(size=f.shape)))


def _seeds(w):
    """(q, t, r) of single entries, at least 6 nodes apart, and their upwind
    offsets in r and theta."""
    n_t = min(w.n_theta, 96)
    out = []
    for j, (t, r) in enumerate((t, r) for t in range(3, n_t - 3, 6) for r in range(12, 52, 6)):
        q = 1 + (7 * j) % 32
        i = (q - 1) % 8
        th = (t + 1) * 2.0 * math.pi / w.n_theta
        a = 2.0 * math.pi * i / 8 - th
        out.append((q, t, r, -1 if math.cos(a) >= 0 else 1, -1 if math.sin(a) >= 0 else 1))
    return np.array(out).T


@pytest.mark.parametrize("n_r,n_t", GRIDS)
def test_partials_of_small_courant_numbers_keep_their_digits(n_r, n_t):
    w = I.random_smooth(n_r, n_t, seed=5, cfl=1e-10)
    f = _state(w)
    q, t, r, ur, ut = _seeds(w)
    lam = np.zeros_like(f)
    lam[q, t, r] = 1.0
    got, flags = _adjoint(w, f, lam)
    assert flags == 0
    for dr, dt in ((ur, 0 * ut), (2 * ur, 0 * ut), (0 * ur, ut), (0 * ur, 2 * ut)):
        tt, rr = (t + dt) % n_t, r + dr
        want = O.adjoint_entries(w, f, lam, q, tt, rr)
        keep = np.abs(want) > 1e-3 * np.abs(want).max()
        assert keep.sum() >= 5
        err = np.abs(got[q, tt, rr] - want)[keep] / np.abs(want)[keep]
        assert err.max() <= 1e-11, err.max()


@pytest.mark.parametrize("n_r,n_t", GRIDS)
def test_partials_of_a_small_difference_keep_their_digits(n_r, n_t):
    """D = 2^-20 f beside Dp = 0.3 f: M_Dp = -2 K v^2, K = |C_r| (1 - |C_r|), v = 3e-6,
    alone two nodes upwind; against that expression, which has no cancellation
    (the oracle differentiates the form with the switch S, which does)."""
    w = I.random_smooth(n_r, n_t, seed=5)
    f = _state(w)
    q, t, r, ur, _ = _seeds(w)
    f[q, t, r + ur] = f[q, t, r] * (1.0 - 2.0 ** -20)
    f[q, t, r + 2 * ur] = f[q, t, r + ur] - 0.3 * f[q, t, r]
    lam = np.zeros_like(f)
    lam[q, t, r] = 1.0
    got, flags = _adjoint(w, f, lam)
    assert flags == 0
    i, th = (q - 1) % 8, (t + 1) * 2.0 * math.pi / w.n_theta
    v = np.asarray(w.speeds)[1 + (q - 1) // 8] * np.cos(2.0 * math.pi * i / 8 - th)
    a = np.abs(v) * w.dt / ((w.r_out - w.r_in) / (n_r - 1))
    D, Dp = f[q, t, r] - f[q, t, r + ur], f[q, t, r + ur] - f[q, t, r + 2 * ur]
    want = -2.0 * a * (1.0 - a) * (D / (D + Dp)) ** 2
    keep = np.abs(np.cos(2.0 * math.pi * i / 8 - th)) > 0.05
    assert keep.sum() >= 5 and (D[keep] / Dp[keep] > 0).all()
    err = np.abs(got[q, t, r + 2 * ur] - want)[keep] / np.abs(want)[keep]
    assert err.max() <= 1e-11, err.max()
