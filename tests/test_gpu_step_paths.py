"""Every kernel of the octagon's step on the states and limits that take its
rarer paths: grids of at most 19 tiles of 32 x 16 nodes, of at most 76 and larger
ones (other kernels and tile heights), each with tiles at a wall and between
the walls.
"""
import ctypes

import numpy as np
import pytest

import oracle as O
from paper_1302_7104_gb300 import inputs as I
from paper_1302_7104_gb300 import pclb as P

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

GRIDS = [(130, 40), (130, 90), (130, 260)]          # FP64 tiles of 2, 4 and 16 rows
SCHEMES = [P.SCHEME_MWB, P.SCHEME_WB, P.SCHEME_LW, P.SCHEME_UPWIND2]


def _noisy(w, seed=3, noise=0.01):
    f = O.set_state(w)
    return np.ascontiguousarray(f * (1.0 + noise * np.random.default_rng(seed).normal(size=f.shape)))


def _step(w, f):
    with P.PCLB(w, precision="fp64") as g:
        got = g.set_f(torch.as_tensor(f, device="cuda")).step(1).get_f().cpu().numpy()
        return got, g.status_flags()


@pytest.mark.parametrize("n_r,n_t", GRIDS)
@pytest.mark.parametrize("r", [16, 50, 120])         # in a tile at the inner wall, between the walls, at the outer one
@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_non_finite_values_stay_local_and_are_flagged(n_r, n_t, r, bad):
    w = I.random_smooth(n_r, n_t, seed=7)
    f = _noisy(w)
    f[5, 20, r] = bad
    got, flags = _step(w, f)
    want = O.run(w, np.where(np.isfinite(f), f, 0.1), 1)
    far = np.ones(f.shape, dtype=bool)
    far[:, 18:23, r - 2:r + 3] = False
    assert flags & P.FLAG_NONPHYS
    assert not np.isfinite(got[5, 20, r])
    assert np.max(np.abs(got[far] - want[far])) <= 1e-12 * np.max(np.abs(want))


@pytest.mark.parametrize("n_r,n_t", GRIDS)
@pytest.mark.parametrize("r", [16, 50])
@pytest.mark.parametrize("what", ["density", "temperature"])
def test_non_physical_nodes_are_flagged_and_evaluated(n_r, n_t, r, what):
    """One node of negative density or temperature: the same finite expressions as
    everywhere else, and a flag."""
    w = I.random_smooth(n_r, n_t, seed=7)
    f = _noisy(w)
    if what == "density":
        f[:, 20, r] *= -1.0
    else:
        f[25, 20, r] -= 0.5                          # takes 5 from the energy
    got, flags = _step(w, f)
    want = O.run(w, f, 1)
    assert flags & P.FLAG_NONPHYS
    assert np.max(np.abs(got - want)) <= 1e-12 * np.max(np.abs(want))


@pytest.mark.parametrize("n_r,n_t", GRIDS)
@pytest.mark.parametrize("shell", [1, 4])
def test_a_shell_of_zeros(n_r, n_t, shell):
    w = I.uniform(n_r, n_t)
    f = O.set_state(w)
    f[1 + 8 * (shell - 1):1 + 8 * shell] = 0.0
    got, _ = _step(w, f)
    want = O.run(w, f, 1)
    assert np.max(np.abs(got - want)) <= 1e-12 * np.max(np.abs(want))


@pytest.mark.parametrize("n_r,n_t", GRIDS)
@pytest.mark.parametrize("scheme", SCHEMES)
@pytest.mark.parametrize("rho,T", [(30.0, 1.0), (300.0, 1.0), (1e9, 1.0), (64.0, 3.0), (1.0, 4.0)])
@pytest.mark.parametrize("bc", [(I.BC_EXTRAP, I.BC_EXTRAP), (I.BC_WALL | I.BC_NEQ, I.BC_DIRICHLET | I.BC_NEQ)])
def test_jumps_inside_tiles(n_r, n_t, scheme, rho, T, bc):
    """Jumps of density and temperature inside tiles of every kind: each
    column to 1e-12 of the largest value within its stencils."""
    w = I.random_smooth(n_r, n_t, seed=5, bc_kind=bc)
    col = np.arange(n_r)
    dense = (col < 12) | ((col >= 48) & (col < 80)) | (col >= 118)
    w.rho = np.where(dense, rho, 1.0) * w.rho
    w.T = np.where(dense, T, 1.0) * w.T
    w.scheme = scheme
    f = _noisy(w, noise=1e-3)
    got, _ = _step(w, f)
    want = O.run(w, f, 1)
    err, size = np.abs(got - want).max((0, 1)), np.abs(f).max((0, 1))
    near = np.array([size[max(c - 2, 0):c + 3].max() for c in col])
    assert (err <= 1e-12 * near).all(), (err / near).max()


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("n_r,n_t", GRIDS)
def test_window_wait_that_runs_out_on_small_grids(prec, n_r, n_t):
    """Limit 0: every tile is given up without waiting, the timeout is reported
    and the context steps a reloaded state like a fresh one."""
    w = I.random_smooth(n_r, n_t, seed=9)
    dtype = torch.float32 if prec == "fp32" else torch.float64
    f0 = torch.as_tensor(_noisy(w), dtype=dtype, device="cuda")
    with P.PCLB(w, precision=prec) as g:
        g.set_f(f0).set_wait_limit(0).step(3)
        flags = ctypes.c_uint32()
        assert P.lib().pclb_status_flags(g.ctx, ctypes.byref(flags), 1) == 5 and flags.value & P.FLAG_TIMEOUT
        got = g.set_wait_limit().set_f(f0).step(2).get_f()
        assert g.status_flags() == 0
    with P.PCLB(w, precision=prec) as h:
        want = h.set_f(f0).step(2).get_f()
    assert torch.equal(got, want)


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("n_r,n_t", [(130, 40), (130, 200), (130, 500)])     # FP64 tiles of 2, 4 and 8 rows
def test_adjoint_window_wait_that_runs_out_on_small_grids(prec, n_r, n_t):
    w = I.random_smooth(n_r, n_t, seed=9)
    dtype = torch.float32 if prec == "fp32" else torch.float64
    f0 = torch.as_tensor(_noisy(w), dtype=dtype, device="cuda")
    lam = torch.as_tensor(np.random.default_rng(4).normal(size=tuple(f0.shape)), dtype=dtype, device="cuda")
    with P.PCLB(w, precision=prec) as g:
        g.set_wait_limit(0)
        g.adjoint_step(f0, lam)
        flags = ctypes.c_uint32()
        assert P.lib().pclb_status_flags(g.ctx, ctypes.byref(flags), 1) == 5 and flags.value & P.FLAG_TIMEOUT
        g.set_wait_limit()
        got = g.adjoint_step(f0, lam)
        assert g.status_flags() == 0
    with P.PCLB(w, precision=prec) as h:
        want = h.adjoint_step(f0, lam)
        h.sync()
    assert torch.equal(got, want)
