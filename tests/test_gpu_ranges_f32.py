"""FP32 states of any magnitude: fields, integrals and initial states against the
same expressions in extended precision on the host, from the FP32 values
themselves.

Every one of these is defined by sums that the library forms to double
precision or better, so a float result may differ by its own rounding (2^-24)
and a double one by a few roundings of the sums.
"""
import math

import numpy as np
import pytest

import oracle as O
from paper_1302_7104_gb300 import inputs as I
from paper_1302_7104_gb300 import pclb as P

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

LD = np.longdouble
HALF_ULP = 2.0 ** -24 * (1.0 + 1e-5)


def _state(n_dirs, scale, n_r=70, n_t=30):
    w = I.random_smooth(n_r, n_t, seed=3, n_dirs=n_dirs, n_f=n_dirs)
    f = O.set_state(w) * (1.0 + 0.01 * np.random.default_rng(1).normal(size=(w.q, n_t, n_r)))
    return w, (f * scale).astype(np.float32)


def _moments(w, f):
    """rho, j_x, j_y, e and the sums of |terms| of j_x."""
    f = f.astype(LD)
    rho, jx, jy, e, size = f.sum(0), 0, 0, 0, 0
    for k in range(1, 5):
        for i in range(w.n_dirs):
            sgn, phi = (1.0 if i < w.n_dirs // 2 else -1.0), 2.0 * math.pi * (i % (w.n_dirs // 2)) / w.n_dirs
            q = 1 + (k - 1) * w.n_dirs + i
            vx, vy = LD(w.speeds[k] * sgn * math.cos(phi)), LD(w.speeds[k] * sgn * math.sin(phi))
            jx, jy, size = jx + vx * f[q], jy + vy * f[q], size + abs(vx * f[q])
            e = e + LD(0.5 * w.speeds[k] ** 2) * f[q]
    return rho, jx, jy, e, size


def _area(w):
    dr, dth = (w.r_out - w.r_in) / (w.n_r - 1), 2.0 * math.pi * w.n_f / (w.n_dirs * w.n_theta)
    return ((w.r_in + np.arange(w.n_r) * LD(dr)) * dr * dth)[None, :]


SCALES = [1.0, 2.0 ** -100, 2.0 ** -120, 2.0 ** 121, 2.0 ** 124]


@pytest.mark.parametrize("n_dirs", [16, 24])
@pytest.mark.parametrize("scale", SCALES)
def test_integrals_of_the_larger_sets_in_double(n_dirs, scale):
    """Tolerance: 16 roundings (2^-53) of the sums of the terms' sizes."""
    w, f = _state(n_dirs, scale)
    with P.PCLB(w, precision="fp32") as g:
        d = g.set_f(torch.as_tensor(f, device="cuda")).diagnostics()
        assert g.status_flags() == 0
    rho, jx, jy, e, size = _moments(w, f)
    a, T = _area(w), (e - (jx * jx + jy * jy) / (2 * rho)) / rho
    tol = 16.0 * 2.0 ** -53
    assert abs(d[0] - (a * rho).sum()) <= tol * (a * rho).sum()
    assert abs(d[1] - (a * jx).sum()) <= tol * (a * size).sum()
    assert abs(d[2] - (a * jy).sum()) <= tol * (a * size).sum()
    assert abs(d[3] - (a * e).sum()) <= tol * (a * e).sum()
    assert d[4] == float(rho.min()) or abs(d[4] - rho.min()) <= tol * rho.min()
    assert abs(d[5] - T.min()) <= tol * T.min()


@pytest.mark.parametrize("n_dirs", [16, 24])
@pytest.mark.parametrize("scale", SCALES)
def test_fields_of_the_larger_sets_round_once(n_dirs, scale):
    w, f = _state(n_dirs, scale)
    with P.PCLB(w, precision="fp32") as g:
        got = [x.cpu().numpy().astype(LD) for x in g.set_f(torch.as_tensor(f, device="cuda")).moments()]
        assert g.status_flags() == 0
    rho, jx, jy, e, size = _moments(w, f)
    th = (np.arange(1, w.n_theta + 1) * (2.0 * math.pi * w.n_f / (w.n_dirs * w.n_theta)))[:, None]
    c, s = np.cos(th), np.sin(th)
    want = [rho, (jx * c + jy * s) / rho, (jy * c - jx * s) / rho, (e - (jx * jx + jy * jy) / (2 * rho)) / rho]
    for x, y in zip(got, want):
        room = 32.0 * 2.0 ** -53 * (size / rho)      # roundings of the sums
        assert (abs(x - y) <= HALF_ULP * abs(y) + (room if y is not rho else 32.0 * 2.0 ** -53 * rho)).all()


@pytest.mark.parametrize("n_dirs", [16, 24])
@pytest.mark.parametrize("rho,T,u", [(1.0, 1.0, 0.3), (2.0 ** -100, 1.0, 0.3), (2.0 ** -124, 1.0, 0.3), (2.0 ** 100, 1.0, 0.3),
                                     (2.0 ** 120, 0.5, 0.3), (1.0, 2.0 ** -40, 0.0), (2.0 ** -60, 2.0 ** -60, 0.0),
                                     (1.0, 2.0 ** 25, 1.0), (1.0, 1e-3, 1.0)])
def test_initial_states_of_the_larger_sets_round_once(n_dirs, rho, T, u):
    """f^eq (Eqs. 10-11) of fields around (rho, T, u), label by label: half a
    unit in the last place (of the smallest normal number below it), and 64
    roundings of double on the shell's largest term."""
    w = I.random_smooth(40, 20, seed=3, n_dirs=n_dirs, n_f=n_dirs)
    rng = np.random.default_rng(2)
    fields = [(np.asarray(x) * (1.0 + 0.1 * rng.random(w.rho.shape))).astype(np.float32) for x in (rho, u, -0.5 * u, T)]
    with P.PCLB(w, precision="fp32") as g:
        got = g.set_state(*[torch.as_tensor(x, device="cuda") for x in fields]).get_f().cpu().numpy().astype(LD)
        assert g.status_flags() == 0
    R, ur, ut, E = (x.astype(LD) for x in fields)
    th = (np.arange(1, w.n_theta + 1) * (2.0 * math.pi * w.n_f / (w.n_dirs * w.n_theta)))[:, None]
    c, s = np.cos(th), np.sin(th)
    ux, uy = ur * c - ut * s, ur * s + ut * c
    z = (ux * ux + uy * uy) / E
    a1 = 1 - z / 2
    a0 = a1 + z * z / 8
    v2, Fs, sizes = [LD(v) ** 2 for v in w.speeds], 0, 0
    for k in range(4, -1, -1):
        if k:
            a, b, e = (v2[j] for j in range(1, 5) if j != k)
            den = v2[k] * (v2[k] - a) * (v2[k] - b) * (v2[k] - e)
            terms = [w.B[1] * a * b * e, w.B[2] * (a * b + b * e + e * a), w.B[3] * (a + b + e), w.B[4]]
            F = sum(t / den * E ** (n + 1) for n, t in enumerate(terms))
            size = sum(abs(t / den) * E ** (n + 1) for n, t in enumerate(terms))
            Fs, sizes = Fs + F, sizes + size
        else:
            F, size = 1 - w.B[0] * Fs, 1 + w.B[0] * sizes
        for i in range(w.n_dirs if k else 1):
            sgn, phi = (1.0 if i < w.n_dirs // 2 else -1.0), 2.0 * math.pi * (i % (w.n_dirs // 2)) / w.n_dirs
            x = (w.speeds[k] * sgn * math.cos(phi) * ux + w.speeds[k] * sgn * math.sin(phi) * uy) / E
            poly = a0 + x * (a1 + x * (a1 / 2 + x * (LD(1) / 6 + x / 24)))
            room = 64.0 * 2.0 ** -53 * R * size * (1 + z + z * z + abs(x) ** 4)
            want = R * F * poly
            q = 1 + (k - 1) * w.n_dirs + i if k else 0
            assert (abs(got[q] - want) <= np.maximum(HALF_ULP * abs(want), 2.0 ** -150) + room).all(), (k, i)


def test_manifestations_near_the_largest_float():
    """The octagon's central manifestations at a power-of-two scale at which the
    sums of Sec. IV, taken in float label by label, just stay finite: they are
    finite, and those of the unscaled state to the few roundings by which the node's
    velocity may differ (its reciprocal density has no room for a low part)."""
    w, f = _state(8, 1.0, n_r=41, n_t=12)
    with P.PCLB(w, precision="fp32") as g:
        base = g.set_f(torch.as_tensor(f, device="cuda")).noneq(P.NEQ_MSTAR | P.NEQ_DSTAR).cpu().numpy()
        rho, jx, jy, e, _ = _moments(w, f)
        ux, uy = (jx / rho).astype(np.float32), (jy / rho).astype(np.float32)
        peak, total, size = 0.0, np.zeros((12,) + f.shape[1:], np.float32), np.zeros((12,) + f.shape[1:])
        th = (np.arange(1, w.n_theta + 1) * (2.0 * math.pi * w.n_f / (w.n_dirs * w.n_theta)))[:, None].astype(np.float32)
        c, s = np.cos(th), np.sin(th)
        for q in range(w.q):
            k, i = (0, 0) if q == 0 else (1 + (q - 1) // 8, (q - 1) % 8)
            vx, vy = np.float32(w.speeds[k] * math.cos(math.pi * i / 4)), np.float32(w.speeds[k] * math.sin(math.pi * i / 4))
            cr, ct = (vx - ux) * c + (vy - uy) * s, (vy - uy) * c - (vx - ux) * s
            h = np.float32(0.5) * (cr * cr + ct * ct)
            for n, x in enumerate((cr * cr, cr * ct, ct * ct, cr ** 3, cr * cr * ct, cr * ct * ct, ct ** 3, h * cr, h * ct,
                                   h * cr * cr, h * cr * ct, h * ct * ct)):
                total[n] += f[q] * x
                size[n] += np.abs(f[q] * x)
            peak = max(peak, np.abs(total).max())
        scale = 2.0 ** (127 - math.floor(math.log2(1.02 * peak)))
        got = g.set_f(torch.as_tensor((f * np.float32(scale)), device="cuda")).noneq(P.NEQ_MSTAR | P.NEQ_DSTAR).cpu().numpy()
    assert np.isfinite(got).all()
    for g in (0, 1):   # 2^-20 of the terms' size
        assert (np.abs(got[g] / scale - base[g]) <= 2.0 ** -20 * size).all()


def test_integrals_near_the_largest_float():
    """The octagon's integrals where each node's moments are finite floats but a
    few of them together are not: those of the unscaled state, to the rounding of
    the sums (the grid is large enough for several rows per thread)."""
    w = I.random_smooth(1024, 1300, seed=3)
    with P.PCLB(w, precision="fp32") as g:
        f = g.set_state().get_f()
        base = g.diagnostics()
        scale = 2.0 ** 125
        got = g.set_f(f * scale).diagnostics()
        assert g.status_flags() == 0
    assert np.isfinite(got).all()
    assert np.abs(got[:6] / scale ** np.array([1, 1, 1, 1, 1, 0]) - base[:6]).max() <= 1e-6 * base[0]
