"""The FP32 step at the edges of its grid rule (tiles of 4 rows on at most 76
tiles of 32 x 16, else of 16 rows), and the packed copies of the state at the
sizes and alignments where their vector paths change.

Tolerance of a step: 2e-6 of max|f|, as the other FP32 parity tests; copies are
exact.
"""
import numpy as np
import pytest

import oracle as O
from paper_1302_7104_gb300 import inputs as I
from paper_1302_7104_gb300 import pclb as P

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n_r,n_t", [(33, 4), (64, 608), (64, 609), (2432, 16), (2433, 17), (31, 1217), (32, 3)])
@pytest.mark.parametrize("scheme", [P.SCHEME_MWB, P.SCHEME_LW])
@pytest.mark.parametrize("bc", [(I.BC_EXTRAP, I.BC_EXTRAP), (I.BC_WALL | I.BC_NEQ, I.BC_DIRICHLET | I.BC_NEQ)])
def test_step_matches_oracle_at_the_edges_of_the_tile_rule(n_r, n_t, scheme, bc):
    w = I.random_smooth(n_r, n_t, seed=n_r + n_t, bc_kind=bc)
    w.scheme = scheme
    f = O.set_state(w)
    f = (f * (1.0 + 0.01 * np.random.default_rng(2).normal(size=f.shape))).astype(np.float32)
    want = O.run(w, np.ascontiguousarray(f.astype(np.float64)), 1)
    with P.PCLB(w, precision="fp32") as g:
        got = g.set_f(torch.as_tensor(f, device="cuda")).step(1).get_f().double().cpu().numpy()
    assert np.max(np.abs(got - want)) <= 2e-6 * np.max(np.abs(want))


@pytest.mark.parametrize("prec,dtype", [("fp32", torch.float32), ("fp64", torch.float64)])
@pytest.mark.parametrize("n_dirs", [8, 16])
@pytest.mark.parametrize("n_r,n_t", [(3, 2), (31, 3), (32, 2), (34, 5), (129, 4), (1029, 3)])
@pytest.mark.parametrize("shift", [0, 1, 2])
def test_packed_copies_are_exact(prec, dtype, n_dirs, n_r, n_t, shift):
    """f in and out again, from and to buffers `shift` elements off their alignment."""
    w = I.random_smooth(n_r, n_t, seed=1, amp=0.02, n_dirs=n_dirs, n_f=n_dirs)
    shape = (1 + 4 * n_dirs, n_t, n_r)
    n = int(np.prod(shape))
    gen = torch.Generator(device="cuda").manual_seed(n)
    f = torch.rand(n + shift, generator=gen, dtype=dtype, device="cuda")[shift:].view(shape)
    with P.PCLB(w, precision=prec) as g:
        out = torch.zeros(n + shift, dtype=dtype, device="cuda")[shift:].view(shape)
        assert torch.equal(g.set_f(f).get_f(out=out), f)
