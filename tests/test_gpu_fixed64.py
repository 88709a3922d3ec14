"""Rounding of the FP64 steps' 64-bit fixed point (fixed64.cuh), in the three
kernels that use it (grids of at most 19 tiles of 32 x 16 nodes, of at most 76,
and larger ones) and the 16-direction step.

The oracle works in double: its rounding errors have no preferred sign, so over
many entries the mean relative difference from it must vanish, and single
entries may differ by a few units in the last place of the terms they are made
of.
"""
import numpy as np
import pytest

import oracle as O
from paper_1302_7104_gb300 import inputs as I
from paper_1302_7104_gb300 import pclb as P

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

GRIDS = [(64, 24, 8), (64, 400, 8), (64, 1300, 8), (64, 24, 16)]   # n_r, n_theta, n_dirs


def _step(w, f):
    with P.PCLB(w, precision="fp64") as g:
        got = g.set_f(torch.as_tensor(f, device="cuda")).step(1).get_f().cpu().numpy()
        return got, g.status_flags()


def _noisy(w, seed=3, noise=0.01):
    f = O.set_state(w)
    return np.ascontiguousarray(f * (1.0 + noise * np.random.default_rng(seed).normal(size=f.shape)))


@pytest.mark.parametrize("n_r,n_t,n_dirs", GRIDS)
@pytest.mark.parametrize("scheme", [P.SCHEME_WB, P.SCHEME_LW, P.SCHEME_UPWIND2])
def test_rounding_has_no_preferred_sign(n_r, n_t, n_dirs, scheme):
    """Columns of thin gas (1/20) between columns of dense gas: the thin nodes'
    values lie four to five bits below the largest of their stencils.  The time
    step is small beside tau and the grid, so that the carried part d f - M_r - M_theta is nearly all of the result, and
    the scheme linear, so that no quotient enters.  An entry's error is then
    a sum of roundings of at most 2^-52 of it in standard deviation; six
    standard deviations of the mean of N entries."""
    w = I.random_smooth(n_r, n_t, seed=5, tau=1.0, cfl=0.02, n_dirs=n_dirs, n_f=n_dirs)
    cols = np.arange(n_r)
    thin = (cols >= 8) & (cols < n_r - 8) & (cols % 2 == 1)
    w.rho = np.where(thin, 0.05, 1.0) * np.ones_like(w.rho)
    w.scheme = scheme
    f = _noisy(w)
    got, flags = _step(w, f)
    want = O.run(w, f, 1)
    assert flags == 0
    g, x = got[:, :, thin], want[:, :, thin]
    keep = np.abs(x) > 0.25 * np.abs(f[:, :, thin])      # no entry that the differences all but cancel
    assert keep.mean() > 0.8
    rel = ((g - x) / x)[keep]
    assert abs(rel.mean()) <= 6.0 * 2.0 ** -52 / np.sqrt(rel.size), (rel.mean(), rel.std(), rel.size)


@pytest.mark.parametrize("n_r,n_t,n_dirs", GRIDS)
def test_cold_gas_beside_hot_gas_keeps_its_own_precision(n_r, n_t, n_dirs):
    """T falls from 3 to 1 and rho from 64 to 1 inside a tile: the fourth
    shell's values fall by ~2^13.  Cold nodes away from the jump, shell by shell:
    the largest error against eight roundings (2^-50) of the shell's own scale
    there, rho times the largest term of the polynomial F_k(T), which bounds what
    double arithmetic can resolve of it (F_k is a difference of such terms)."""
    w = I.random_smooth(n_r, n_t, seed=5, n_dirs=n_dirs, n_f=n_dirs, amp=0.1)
    hot = np.arange(n_r) < 16
    w.T = np.where(hot, 3.0, 1.0) * w.T
    w.rho = np.where(hot, 64.0, 1.0) * w.rho
    f = _noisy(w, noise=1e-3)
    got, flags = _step(w, f)
    want = O.run(w, f, 1)
    assert flags == 0
    cold = np.s_[:, 20:32]
    v2 = [s * s for s in w.speeds]
    T = w.T[cold].max()
    for k in range(1, 5):
        a, b, c = (v2[j] for j in range(1, 5) if j != k)
        den = v2[k] * (v2[k] - a) * (v2[k] - b) * (v2[k] - c)
        terms = (w.B[1] * a * b * c, w.B[2] * (a * b + b * c + c * a), w.B[3] * (a + b + c), w.B[4])
        scale = w.rho[cold].max() * max(abs(x / den) * T ** (n + 1) for n, x in enumerate(terms))
        q = slice(1 + (k - 1) * n_dirs, 1 + k * n_dirs)
        err = np.abs(got[q, :, 20:32] - want[q, :, 20:32]).max()
        assert err <= 2.0 ** -50 * scale, (k, err / scale)


@pytest.mark.parametrize("n_r,n_t,n_dirs", GRIDS)
def test_mass_drift_of_a_long_run_beside_dense_gas(n_r, n_t, n_dirs):
    """Columns of thin gas (1/20) beside dense gas at rest relative to one
    another, 100 steps of a tiny time step: every step multiplies the thin
    gas's f by d and adds (1 - d) f^eq, so an error with a preferred sign adds
    up linearly, one without as a square root.  The mean relative change of the
    thin columns' density against the oracle's run of the same steps: 100 steps
    of one rounding of 2^-53 each in one direction would give 1.1e-14; allowed
    is a tenth of that."""
    w = I.random_smooth(n_r, n_t, seed=5, tau=1.0, cfl=1e-5, n_dirs=n_dirs, n_f=n_dirs, amp=0.0)
    cols = np.arange(n_r)
    thin = (cols >= 8) & (cols < n_r - 8) & (cols % 2 == 1)
    w.rho = np.where(thin, 0.05, 1.0) * np.ones_like(w.rho)
    w.u_r, w.u_theta = 0.0 * w.u_r, 0.0 * w.u_theta
    f = _noisy(w, noise=0.001)
    with P.PCLB(w, precision="fp64") as g:
        got = g.set_f(torch.as_tensor(f, device="cuda")).step(100).get_f().cpu().numpy()
    want = O.run(w, f, 100)
    drift = (got[:, :, thin].sum(0) - want[:, :, thin].sum(0)) / want[:, :, thin].sum(0)
    assert abs(drift.mean()) <= 0.1 * 100 * 2.0 ** -53, drift.mean()
