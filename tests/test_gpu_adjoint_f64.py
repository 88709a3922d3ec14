"""The FP64 adjoint's partials formed in integers (fx_mwb_partials) and its two
tile heights, against the oracle's adjoint entries.

Tolerance: 1e-12 of max|lam|, as the other FP64 adjoint tests; scaling f by a
power of two changes no partial derivative, so scaled states use the same one.
"""
import numpy as np
import pytest

import oracle as O
from paper_1302_7104_gb300 import inputs as I
from paper_1302_7104_gb300 import pclb as P

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _state(w, seed=3, noise=0.02):
    f = O.set_state(w)
    return np.ascontiguousarray(f * (1.0 + noise * np.random.default_rng(seed).normal(size=f.shape)))


def _adjoint(w, f, lam):
    with P.PCLB(w, precision="fp64") as g:
        out = g.adjoint_step(torch.as_tensor(f, device="cuda"), torch.as_tensor(lam, device="cuda"))
        return out.cpu().numpy(), g.status_flags()


def _sample(w, seed, n=400):
    """Entries at the walls, the seam, tile edges and at random."""
    rng = np.random.default_rng(seed)
    r = np.concatenate([rng.choice([0, 1, 2, 30, 31, 32, 33, w.n_r - 3, w.n_r - 2, w.n_r - 1], n), rng.integers(0, w.n_r, n)])
    t = np.concatenate([rng.choice([0, 1, 2, 3, 4, 7, 8, 9, w.n_theta - 2, w.n_theta - 1], n), rng.integers(0, w.n_theta, n)])
    return rng.integers(0, 33, 2 * n), t, np.clip(r, 0, w.n_r - 1)


# 32 x 8-node tiles: up to 152 of them take tiles of 4 rows
@pytest.mark.parametrize("n_r,n_t", [(64, 608), (64, 609), (65, 405), (66, 408), (2432, 16), (2433, 16)])
def test_adjoint_matches_oracle_at_the_edges_of_the_tile_rule(n_r, n_t):
    w = I.random_smooth(n_r, n_t, seed=n_t, bc_kind=(I.BC_WALL | I.BC_NEQ, I.BC_EXTRAP))
    f = _state(w)
    lam = np.random.default_rng(4).normal(size=f.shape)
    got, flags = _adjoint(w, f, lam)
    q, t, r = _sample(w, n_r + n_t)
    want = O.adjoint_entries(w, f, lam, q, t, r)
    assert flags == 0
    assert np.max(np.abs(got[q, t, r] - want)) <= 1e-12 * np.max(np.abs(lam))


@pytest.mark.parametrize("scale", [2.0 ** -900, 2.0 ** -300, 2.0 ** 300])
def test_partials_do_not_depend_on_the_magnitude_of_f(scale):
    """h's derivatives are ratios of differences: scaling f leaves the
    convection part of the adjoint alone; the equilibrium part scales with the
    state's own terms, so both steps are compared with the oracle's entries of the
    unscaled state (Eq. 10 is linear in rho)."""
    w = I.random_smooth(40, 20, seed=5)
    f = _state(w)
    lam = np.random.default_rng(6).normal(size=f.shape)
    got, _ = _adjoint(w, f * scale, lam)
    q, t, r = _sample(w, 7)
    want = O.adjoint_entries(w, f, lam, q, t, r)
    assert np.max(np.abs(got[q, t, r] - want)) <= 1e-12 * np.max(np.abs(lam))


def test_equal_neighbours_and_one_sided_zeros():
    """Runs of equal values: D = 0, Dp = 0 and both, at planted nodes of a noisy
    state, where the derivative on the active branch is defined by sign(0) = 0."""
    w = I.random_smooth(70, 24, seed=8)
    f = _state(w)
    f[:, :, 10:13] = f[:, :, 10:11]       # radial runs of three
    f[:, :, 40] = f[:, :, 41]             # of two
    f[:, 5:8, 20:30] = f[:, 5:6, 20:30]   # azimuthal runs
    lam = np.random.default_rng(9).normal(size=f.shape)
    got, _ = _adjoint(w, f, lam)
    q, t, r = (a.ravel() for a in np.meshgrid(np.arange(33), np.arange(3, 11), np.arange(7, 45), indexing="ij"))
    want = O.adjoint_entries(w, f, lam, q, t, r)
    assert np.max(np.abs(got[q, t, r] - want)) <= 1e-12 * np.max(np.abs(lam))


def test_non_finite_values_stay_local_and_are_flagged():
    w = I.random_smooth(100, 24, seed=10)
    f = _state(w)
    f[7, 12, 50] = np.nan
    lam = np.random.default_rng(11).normal(size=f.shape)
    got, flags = _adjoint(w, f, lam)
    assert flags & P.FLAG_NONPHYS
    bad = ~np.isfinite(got)
    assert bad[7, 12, 50] and bad[7].sum() >= 5          # the stencils that read the value
    far = np.ones(f.shape, dtype=bool)
    far[:, 8:17, 46:55] = False
    assert not bad[far].any()


# the line between tiles of 4 and 8 rows: 228 tiles of 32 x 8
@pytest.mark.parametrize("n_r,n_t", [(32, 1824), (33, 905), (32, 1825)])
def test_adjoint_matches_oracle_beside_the_line_of_the_tile_rule(n_r, n_t):
    w = I.random_smooth(n_r, n_t, seed=n_t, bc_kind=(I.BC_WALL | I.BC_NEQ, I.BC_EXTRAP))
    f = _state(w)
    lam = np.random.default_rng(4).normal(size=f.shape)
    got, flags = _adjoint(w, f, lam)
    q, t, r = _sample(w, n_r + n_t)
    want = O.adjoint_entries(w, f, lam, q, t, r)
    assert flags == 0
    assert np.max(np.abs(got[q, t, r] - want)) <= 1e-12 * np.max(np.abs(lam))


# tiles of 2 rows up to 38 tiles of 32 x 8: both sides, last tiles of one row and of one to three columns
@pytest.mark.parametrize("n_r,n_t", [(32, 304), (32, 305), (33, 150), (34, 31), (35, 2), (3, 9), (99, 21)])
@pytest.mark.parametrize("bc", [(I.BC_EXTRAP, I.BC_EXTRAP), (I.BC_WALL | I.BC_NEQ, I.BC_DIRICHLET | I.BC_NEQ)])
def test_tiles_of_two_rows_match_oracle(n_r, n_t, bc):
    w = I.random_smooth(n_r, n_t, seed=n_r + n_t, bc_kind=bc, amp=0.02 if n_r < 8 else 0.2)
    f = _state(w)
    lam = np.random.default_rng(8).normal(size=f.shape)
    got, flags = _adjoint(w, f, lam)
    q, t, r = _sample(w, n_r + n_t)
    t = np.clip(t, 0, n_t - 1)
    want = O.adjoint_entries(w, f, lam, q, t, r)
    assert flags == 0
    assert np.max(np.abs(got[q, t, r] - want)) <= 1e-12 * np.max(np.abs(lam))
