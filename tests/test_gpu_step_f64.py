"""The FP64 step in fixed point (step_kernel_f64.cu): its tiles of 4 and 16
rows, the edges of its grid rule, and the states that leave fixed point
(thin gas beside dense gas in one tile, magnitudes near the ends of the double
range, NaN), against the oracle.

Tolerance: 1e-12 of max|f| per step, as the other FP64 parity tests; a state
scaled by a power of two scales the result exactly in the oracle, so scaled
cases use the same relative tolerance.
"""
import numpy as np
import pytest

import oracle as O
from paper_1302_7104_gb300 import inputs as I
from paper_1302_7104_gb300 import pclb as P

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _noisy(w, seed=3, noise=0.01):
    f = O.set_state(w)
    return np.ascontiguousarray(f * (1.0 + noise * np.random.default_rng(seed).normal(size=f.shape)))


def _step(w, f, n=1):
    with P.PCLB(w, precision="fp64") as g:
        got = g.set_f(torch.as_tensor(f, device="cuda")).step(n).get_f().cpu().numpy()
        return got, g.status_flags()


# 32 x 16-node tiles: up to 76 of them take tiles of 4 rows
@pytest.mark.parametrize("n_r,n_t", [(3, 2), (33, 4), (32, 5), (35, 17), (64, 608), (64, 609), (2432, 16), (2433, 17),
                                     (31, 1217)])
@pytest.mark.parametrize("bc", [(I.BC_EXTRAP, I.BC_EXTRAP), (I.BC_WALL | I.BC_NEQ, I.BC_DIRICHLET | I.BC_NEQ)])
def test_step_matches_oracle_at_the_edges_of_the_tile_rule(n_r, n_t, bc):
    w = I.random_smooth(n_r, n_t, seed=n_r + n_t, bc_kind=bc, amp=0.02 if n_r < 8 else 0.2)
    f = _noisy(w)
    got, _ = _step(w, f, 2)
    want = O.run(w, f, 2)
    assert np.max(np.abs(got - want)) <= 2e-12 * np.max(np.abs(want))


def _contrast(w, ratio):
    """Density falling by `ratio` across the middle of a 32-node tile."""
    w.rho = np.where(np.arange(w.n_r) < 16, 1.0, 1.0 / ratio) * np.ones_like(w.rho)
    return w


@pytest.mark.parametrize("n_t", [40, 1300])            # tiles of 4 and of 16 rows
@pytest.mark.parametrize("ratio", [200.0, 300.0, 1e6, 1e12])
def test_thin_gas_beside_dense_gas_keeps_its_own_precision(n_t, ratio):
    """Every node to 1e-12 of its own row's scale: the thin side (radial nodes
    20..31, four nodes off the jump) against the largest value there."""
    w = _contrast(I.random_smooth(64, n_t, seed=5), ratio)
    f = _noisy(w)
    got, _ = _step(w, f)
    want = O.run(w, f, 1)
    assert np.max(np.abs(got - want)) <= 1e-12 * np.max(np.abs(want))
    thin = np.s_[:, :, 20:32]
    assert np.max(np.abs(got[thin] - want[thin])) <= 1e-12 * np.max(np.abs(want[thin]))


@pytest.mark.parametrize("n_t", [24, 1300])
@pytest.mark.parametrize("scale", [2.0 ** -1000, 2.0 ** -880, 2.0 ** -300, 2.0 ** 300, 2.0 ** 860, 2.0 ** 1000])
def test_states_of_any_magnitude(n_t, scale):
    w = I.random_smooth(40, n_t, seed=6)
    f = _noisy(w)
    got, flags = _step(w, f * scale)
    want = O.run(w, f, 1)
    assert flags == 0
    assert np.max(np.abs(got / scale - want)) <= 1e-12 * np.max(np.abs(want))


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_non_finite_values_stay_local_and_are_flagged(bad):
    w = I.random_smooth(100, 40, seed=7)
    f = _noisy(w)
    f[5, 20, 50] = bad
    got, flags = _step(w, f)
    assert flags & P.FLAG_NONPHYS
    want = O.run(w, np.where(np.isfinite(f), f, 0.1), 1)
    far = np.ones(f.shape, dtype=bool)
    far[:, 18:23, 48:53] = False
    assert not np.isfinite(got[5, 20, 50])
    assert np.max(np.abs(got[far] - want[far])) <= 1e-12 * np.max(np.abs(want))


def test_zero_planes_and_equal_neighbours():
    """A shell that is exactly zero, and a uniform state (every difference 0)."""
    w = I.uniform(70, 24)
    f = O.set_state(w)
    f[9:17] = 0.0
    got, _ = _step(w, f)
    want = O.run(w, f, 1)
    assert np.max(np.abs(got - want)) <= 1e-12 * np.max(np.abs(want))


# Tiles of 2 rows on at most 19 tiles of 32 x 16, of 4 rows up to 76: both
# sides of that line, last tiles of one to three columns (the wall node or its
# neighbour in another tile's columns) and of one row
@pytest.mark.parametrize("n_r,n_t", [(32, 304), (32, 305), (608, 16), (609, 17), (33, 301), (34, 303), (35, 302), (3, 307)])
@pytest.mark.parametrize("bc", [(I.BC_EXTRAP, I.BC_EXTRAP), (I.BC_WALL | I.BC_NEQ, I.BC_DIRICHLET | I.BC_NEQ)])
def test_small_tiles_match_oracle(n_r, n_t, bc):
    w = I.random_smooth(n_r, n_t, seed=n_r + n_t, bc_kind=bc, amp=0.02 if n_r < 8 else 0.2)
    f = _noisy(w)
    got, _ = _step(w, f, 2)
    want = O.run(w, f, 2)
    assert np.max(np.abs(got - want)) <= 2e-12 * np.max(np.abs(want))


@pytest.mark.parametrize("ratio,scale", [(300.0, 2.0 ** -1000), (300.0, 1.0), (300.0, 2.0 ** 1000), (1e12, 1.0),
                                         (1e12, 2.0 ** 1000)])
def test_tiles_of_four_rows_outside_fixed_point(ratio, scale):
    w = _contrast(I.random_smooth(64, 400, seed=8), ratio)
    f = _noisy(w)
    got, flags = _step(w, f * scale)
    want = O.run(w, f, 1)
    assert flags == 0
    thin = np.s_[:, :, 20:32]
    got = got / scale
    assert np.max(np.abs(got - want)) <= 1e-12 * np.max(np.abs(want))
    assert np.max(np.abs(got[thin] - want[thin])) <= 1e-12 * np.max(np.abs(want[thin]))


# The compared schemes in fixed point, tiles of 2, 4 and 16 rows (6, 50 and
# 164 tiles of 32 x 16), and with magnitudes outside fixed point's range
@pytest.mark.parametrize("scheme", [P.SCHEME_WB, P.SCHEME_LW, P.SCHEME_UPWIND2])
@pytest.mark.parametrize("n_r,n_t", [(35, 33), (65, 259), (97, 643)])
@pytest.mark.parametrize("bc", [(I.BC_EXTRAP, I.BC_EXTRAP), (I.BC_WALL | I.BC_NEQ, I.BC_DIRICHLET | I.BC_NEQ)])
@pytest.mark.parametrize("relax", [P.RELAX_EXACT, P.RELAX_EULER])
def test_compared_schemes_match_oracle(scheme, n_r, n_t, bc, relax):
    w = I.random_smooth(n_r, n_t, seed=n_r, bc_kind=bc)
    w.scheme, w.relaxation = scheme, relax
    f = _noisy(w)
    got, flags = _step(w, f, 2)
    want = O.run(w, f, 2)
    assert flags == 0
    assert np.max(np.abs(got - want)) <= 2e-12 * np.max(np.abs(want))


@pytest.mark.parametrize("scheme", [P.SCHEME_WB, P.SCHEME_LW, P.SCHEME_UPWIND2])
@pytest.mark.parametrize("n_t", [40, 1300])
@pytest.mark.parametrize("scale", [2.0 ** -950, 2.0 ** 950])
def test_compared_schemes_of_any_magnitude(scheme, n_t, scale):
    w = I.random_smooth(64, n_t, seed=9)
    w.scheme = scheme
    f = _noisy(w)
    got, flags = _step(w, f * scale)
    want = O.run(w, f, 1)
    assert flags == 0
    assert np.max(np.abs(got / scale - want)) <= 1e-12 * np.max(np.abs(want))


# N_i = 16 and 24: blocks of 32 nodes of a row, four wall rows per ghost block
@pytest.mark.parametrize("n_dirs", [16, 24])
@pytest.mark.parametrize("scheme,relax", [(P.SCHEME_MWB, P.RELAX_EXACT), (P.SCHEME_WB, P.RELAX_EULER),
                                          (P.SCHEME_LW, P.RELAX_EXACT), (P.SCHEME_UPWIND2, P.RELAX_EULER)])
@pytest.mark.parametrize("n_r,n_t", [(3, 2), (32, 5), (33, 9), (66, 4)])
@pytest.mark.parametrize("bc", [(I.BC_EXTRAP, I.BC_EXTRAP), (I.BC_WALL | I.BC_NEQ, I.BC_DIRICHLET | I.BC_NEQ)])
def test_larger_sets_match_oracle(n_dirs, scheme, relax, n_r, n_t, bc):
    w = I.random_smooth(n_r, n_t, seed=n_r + n_t, bc_kind=bc, amp=0.02 if n_r < 8 else 0.2, tau=0.05,
                        n_dirs=n_dirs, n_f=n_dirs)
    w.scheme, w.relaxation = scheme, relax
    f = _noisy(w)
    got, _ = _step(w, f, 2)
    want = O.run(w, f, 2)
    assert np.max(np.abs(got - want)) <= 2e-12 * np.max(np.abs(want))


@pytest.mark.parametrize("n_dirs", [16, 24])
@pytest.mark.parametrize("scale", [2.0 ** -950, 2.0 ** 950])
def test_larger_sets_of_any_magnitude(n_dirs, scale):
    w = _contrast(I.random_smooth(64, 24, seed=10, n_dirs=n_dirs, n_f=n_dirs), 300.0)
    f = _noisy(w)
    got, flags = _step(w, f * scale)
    want = O.run(w, f, 1)
    assert flags == 0
    assert np.max(np.abs(got / scale - want)) <= 1e-12 * np.max(np.abs(want))
