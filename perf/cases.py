"""What a user of this library has it do, as measurable cases.

Kinds of pass, each through the public binding (``pclb.PCLB``, ``autograd``):

* ``run``       set the state from fields, advance n steps, read the fields back (a simulation segment);
* ``restart``   load a distribution, advance n steps, read the distribution back (checkpoint and restart);
* ``analysis``  macroscopic fields, all non-equilibrium manifestations and the global integrals of a state;
* ``grad``      a differentiable rollout and its gradient with respect to the initial fields;
* ``host``      fields from page-locked host memory, n steps, fields back to the host.

The flows are those of the paper's sections and of ``inputs.py`` (rigid
rotation, rotating cylinders, shock tube, shocked interface, shear layer,
smooth random fields), their parameters drawn from the seed.  ``exact``
restates the step (Eqs. 2-5, 10-12, 18-19, 23-28, 37-40) in plain torch at 64
bits.
"""
import math
import random

import numpy as np
import torch

from paper_1302_7104_gb300 import autograd as A
from paper_1302_7104_gb300 import inputs as I
from paper_1302_7104_gb300 import pclb as P

_CASE = dict(kind="run", flow="smooth", n_r=64, n_theta=64, n_dirs=8, n_f=8, prec="fp32", scheme=0, relax=0, neq=0,
             steps=1, graph=False)


def _case(name=None, **kw):
    c = dict(_CASE, **kw)
    if "n_f" not in kw:
        c["n_f"] = c["n_dirs"]
    return c if name is None else dict(name=name, **c)


def listed():
    return [
        # the paper's small verification grids, stepped many times in a row: launches and latency
        _case("rot_32x64_f32_graph", flow="rot", n_r=32, n_theta=64, steps=20, graph=True),
        _case("couette_100x20_f64", flow="couette", n_r=100, n_theta=20, n_f=1, prec="fp64", neq=1, steps=20),
        _case("shock_2000x16_f32", flow="shock", n_r=2000, n_theta=16, steps=20),
        # production runs: the shocked interface and the shear layer at their stated sizes
        _case("rm_1024x2048_f32", flow="rm", n_r=1024, n_theta=2048, steps=10),
        _case("kh_4096x4096_f32", flow="kh", n_r=4096, n_theta=4096, steps=4),
        # the double-precision run that a single-precision one is checked against
        _case("rm_512x1024_f64", flow="rm", n_r=512, n_theta=1024, prec="fp64", steps=4),
        # checkpoint and restart on a grid no tile divides, with one of the compared schemes
        _case("restart_1999x1013_f32", kind="restart", n_r=1999, n_theta=1013, scheme=2, steps=3),
        # the larger velocity set
        _case("dvm16_1024x1024_f32", n_r=1024, n_theta=1024, n_dirs=16, steps=5),
        # output time of a production run: fields, departures from equilibrium, integrals
        _case("analysis_1024x2048_f32", kind="analysis", flow="rm", n_r=1024, n_theta=2048),
        # gradients with respect to the initial fields, at the size of the gradient configuration and, in double
        # precision, of its finite-difference copy; smooth flows (in the nearly uniform gas around a shock the limiter
        # sits on its kinks, and the gradient of single nodes is left to rounding)
        _case("grad_512x1024_f32", kind="grad", n_r=512, n_theta=1024, steps=16),
        _case("grad_64x128_f64", kind="grad", n_r=64, n_theta=128, prec="fp64", steps=9),
        # fields that live on the host, one step per call
        _case("host_4096x4096_f32", kind="host", flow="kh", n_r=4096, n_theta=4096, steps=1),
    ]


# ---------------------------------------------------------------------------
# Drawn cases
# ---------------------------------------------------------------------------
def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _seconds(c):
    """Rough time of a pass, to keep drawn cases below the largest listed one."""
    n = c["n_r"] * c["n_theta"] * (1 + 4 * c["n_dirs"])
    rate = 3e11 if c["prec"] == "fp32" else 1.3e10
    per = {"grad": 4.0, "analysis": 2.0}.get(c["kind"], 1.0)
    return n * (c["steps"] * per + 2) / rate


def draw(rng):
    kind = rng.choices(["run", "restart", "analysis", "grad", "host"], [10, 3, 2, 4, 1])[0]
    dirs = 8 if kind in ("grad", "host") else rng.choices([8, 16, 24], [7, 2, 1])[0]
    prec = rng.choices(["fp32", "fp64"], [3, 2])[0]
    flow = rng.choice(["smooth", "rm", "kh", "shock", "rot", "couette"])
    if kind == "grad":
        flow = "smooth"
    c = _case(kind=kind, flow=flow, n_dirs=dirs, prec=prec, n_r=_log_int(rng, 24, 4096), n_theta=_log_int(rng, 8, 4096))
    if kind == "grad":
        c["n_r"], c["n_theta"] = _log_int(rng, 24, 1024), _log_int(rng, 16, 1024)
    if flow == "couette" or rng.random() < 0.15:
        c["n_f"] = rng.choice([1, 2, 3])
    c["neq"] = int(rng.random() < 0.25)
    if kind in ("run", "restart"):
        c["scheme"] = rng.choices([0, 1, 2, 3], [7, 1, 1, 1])[0]
        c["relax"] = int(rng.random() < 0.15)
        c["graph"] = kind == "run" and rng.random() < 0.3
    c["steps"] = 0 if kind == "analysis" else rng.randint(2, 12) if kind == "grad" else _log_int(rng, 1, 20)
    while _seconds(c) > 0.005:
        if c["steps"] > 2:
            c["steps"] = max(2, c["steps"] // 2)
        elif c["n_r"] > c["n_theta"]:
            c["n_r"] = max(24, int(c["n_r"] * 0.7))
        else:
            c["n_theta"] = max(8, int(c["n_theta"] * 0.7))
    return c


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _device():
    return torch.device("cuda", torch.cuda.current_device())


def _problem(case, seed):
    """The workload (grid, velocity set, boundaries, time step) and its
    initial fields [4][n_theta][n_r] (rho, u_r, u_theta, T) in the case's type."""
    rng = random.Random(seed)
    n_r, n_t, nd, n_f, flow = (case[k] for k in ("n_r", "n_theta", "n_dirs", "n_f", "flow"))
    r_in, r_out, tau = {"rot": (0.5, 1.5, 1e-4), "couette": (1.0, 2.0, 0.05), "shock": (1.0, 3.0, 2e-5),
                        "smooth": (1.0, 2.0, 2e-3)}.get(flow, (1.0, 3.0, 1e-5))
    dt = I.dt_from_cfl(I.STABLE_CFL, n_r, n_t, r_in, r_out, nd, n_f)
    if flow == "couette":
        dt = min(dt, 1e-3)
    if case["kind"] == "grad":
        dt = min(dt, 5e-5)
    if case["relax"]:
        tau = max(tau, dt)
    dev = _device()
    r = torch.linspace(r_in, r_out, n_r, dtype=torch.float64, device=dev)[None, :]
    period = 2.0 * math.pi * n_f / nd
    th = (torch.arange(1, n_t + 1, dtype=torch.float64, device=dev) * (period / n_t))[:, None]
    dr = (r_out - r_in) / (n_r - 1)
    one = torch.ones(n_t, n_r, dtype=torch.float64, device=dev)
    kk = 2.0 * math.pi / period                    # lowest azimuthal wave number of the period
    bc, vals = [I.BC_EXTRAP, I.BC_EXTRAP], [None, None]

    def walls(rows):
        """Prescribed states of both walls' ghost layers: rows[side](r) -> (rho, u_r, u_theta, T)."""
        out = []
        for radii, fn in zip(I.ghost_radii(n_r, r_in, r_out), rows):
            v = np.zeros((2, 4, n_t))
            for layer, rg in enumerate(radii):
                v[layer] = np.asarray(fn(rg), dtype=np.float64)[:, None]
            out.append(v)
        return out

    def waves(base, amp):
        out = base * one
        x = (r - r_in) / (r_out - r_in)
        for m in (1, 2, 3):
            a, b, c = rng.uniform(-1, 1), rng.uniform(0, 6.28), rng.uniform(0, 1)
            out = out + amp / m * a * torch.cos(kk * m * th + b) * torch.cos(math.pi * (0.5 * m * x + c))
        return out

    if flow == "smooth":
        rho, T, ur, ut = waves(1.0, 0.15), waves(1.0, 0.15), waves(0.0, 0.2), waves(0.1, 0.2)
        bc = [I.BC_WALL, I.BC_DIRICHLET] if case["kind"] == "restart" else bc
        if case["kind"] == "restart":
            vals = walls([lambda g: (1.0, 0.0, 0.1, 1.0), lambda g: (1.05, 0.02, 0.05, 0.95)])
    elif flow == "rot":
        w = 0.2 * rng.uniform(0.8, 1.2)
        rho, T, ur, ut = torch.exp(0.5 * w * w * r * r) * one, one, 0.0 * one, w * r * one
        bc = [I.BC_DIRICHLET, I.BC_DIRICHLET]
        vals = walls([lambda g: (math.exp(0.5 * w * w * g * g), 0.0, w * g, 1.0)] * 2)
    elif flow == "couette":
        wi, wo, s = -0.1 * rng.uniform(0.8, 1.2), 0.1 * rng.uniform(0.8, 1.2), rng.uniform(0.2, 0.8)
        d = r_out ** 2 - r_in ** 2
        a, b = (wo * r_out ** 2 - wi * r_in ** 2) / d, r_in ** 2 * r_out ** 2 * (wi - wo) / d
        rho, T, ur, ut = one, one, 0.0 * one, s * (a * r + b / r) * one
        bc = [I.BC_WALL, I.BC_WALL]
        vals = walls([lambda g: (1.0, 0.0, wi * g, 1.0), lambda g: (1.0, 0.0, wo * g, 1.0)])
    elif flow == "shock":
        split, t_out = 2.0 + rng.uniform(-0.2, 0.2), 0.8 if seed % 2 else 0.4
        inner = (r < split) & (one > 0)
        rho, T, ur, ut = torch.where(inner, 1.0, 0.125 * one), torch.where(inner, 1.0, t_out * one), 0.0 * one, 0.0 * one
    elif flow == "rm":
        r_if = 2.0 + sum(rng.uniform(0.0, 0.01) * torch.cos(kk * k * th) for k in range(1, 17))
        chi = 0.5 * (1.0 - torch.tanh((r - r_if) / (2.0 * dr)))
        rho = 1.0 + 2.0 * chi
        rho_h, u_h, p_h, _ = I.hugoniot_from_mach(1.0, 0.0, 1.0, 2.0, direction=-1.0)
        post = (r >= 2.6) & (one > 0)
        m = waves(1.0, 2e-3)                       # a smooth background: nowhere exactly uniform
        rho, T = torch.where(post, rho_h, rho) * m, torch.where(post, p_h / rho_h, 1.0 / rho) * m
        ur, ut = torch.where(post, u_h, 0.0 * one), waves(0.0, 2e-3)
        bc, vals = [I.BC_EXTRAP, I.BC_DIRICHLET], [None, walls([lambda g: (rho_h, u_h, 0.0, p_h / rho_h)] * 2)[1]]
    else:   # kh
        u0, m = 0.5 * rng.uniform(0.8, 1.2), rng.choice([8, 12, 16])
        s = torch.tanh((r - 2.0) / 0.02)
        rho, ut = (1.5 + 0.5 * s) * one, u0 * s * one
        ur = 0.01 * torch.sin(kk * m * th + rng.uniform(0, 6.28)) * torch.exp(-((r - 2.0) / 0.05) ** 2)
        T = 1.0 / rho
    dtype = torch.float32 if case["prec"] == "fp32" else torch.float64
    fields = torch.stack([rho, ur, ut, T]).to(dtype)
    w = I.Workload(flow, n_r, n_t, r_in, r_out, tau, dt, case["steps"], None, None, None, None, n_dirs=nd, n_f=n_f,
                   B=I.TABLE1_B[nd], bc_kind=tuple(b | (I.BC_NEQ if case["neq"] else 0) for b in bc),
                   bc_values=tuple(vals), scheme=case["scheme"], relaxation=case["relax"])
    return w, fields


def _noisy_f(w, fields, seed):
    """A distribution off equilibrium: f^eq of the fields with 1% noise."""
    ref = _Reference(w)
    f = torch.stack(ref.equilibrium(*ref.cartesian(fields.double())))
    gen = torch.Generator(device=f.device)
    gen.manual_seed(seed)
    for plane in f:
        plane.mul_(1.0 + 0.01 * torch.randn(plane.shape, generator=gen, device=f.device, dtype=torch.float64))
    return f.to(fields.dtype)


def _cotangent(fields, seed):
    """The derivative of a scalar objective with respect to the final fields."""
    gen = torch.Generator(device=fields.device)
    gen.manual_seed(seed)
    return 1.0 + 0.1 * torch.randn(fields.shape, generator=gen, device=fields.device, dtype=fields.dtype)


def prepare(case, seed):
    w, fields = _problem(case, seed)
    kind = case["kind"]
    sim = P.PCLB(w, precision=case["prec"])
    s = {"case": case, "sim": sim, "fields": fields}
    if kind in ("run", "analysis"):
        s["out"] = torch.empty_like(fields)
    if kind in ("restart", "analysis"):
        s["f"] = _noisy_f(w, fields, seed)
        s["f_out"] = torch.empty_like(s["f"])
    if kind == "analysis":
        sim.set_f(s["f"])
        del s["f"], s["f_out"]
        s["noneq"] = torch.empty((4, 12) + tuple(fields.shape[1:]), dtype=fields.dtype, device=fields.device)
    if kind == "grad":
        s["g"] = _cotangent(fields, seed)
    if kind == "host":
        s["in"] = [torch.empty(f.shape, dtype=f.dtype, pin_memory=True).copy_(f) for f in fields]
        s["host_out"] = torch.empty(fields.shape, dtype=fields.dtype, pin_memory=True)
    return s


def run(s):
    c, sim = s["case"], s["sim"]
    if c["kind"] == "run":
        sim.set_state(*s["fields"])
        (sim.step_graph if c["graph"] else sim.step)(c["steps"])
        sim.moments(out=list(s["out"]))
        return s["out"]
    if c["kind"] == "restart":
        sim.set_f(s["f"])
        sim.step(c["steps"])
        return sim.get_f(out=s["f_out"])
    if c["kind"] == "analysis":
        sim.moments(out=list(s["out"]))
        sim.noneq(out=s["noneq"])
        return {"fields": s["out"], "noneq": s["noneq"], "integrals": sim.diagnostics()}
    if c["kind"] == "grad":
        x = s["fields"].detach().requires_grad_(True)
        out = torch.stack(A.rollout(sim, *x.unbind(0), n_steps=c["steps"]))
        (g,) = torch.autograd.grad(out, x, s["g"])
        return {"fields": out.detach(), "gradient": g}
    sim.run_host(*s["in"], n=c["steps"], outs=list(s["host_out"]))
    return s["host_out"]


def work(case):
    """Each field and each distribution the caller gives or gets once; per
    step one read and one write of the state; per adjoint step the state and
    the cotangent read, the new cotangent written, and the forward states
    formed once."""
    es = 4 if case["prec"] == "fp32" else 8
    cells, q = case["n_r"] * case["n_theta"], 1 + 4 * case["n_dirs"]
    f, fields, n = cells * q * es, 4 * cells * es, case["steps"]
    updates = cells * q
    if case["kind"] == "analysis":
        return {"bytes": f + fields + 48 * cells * es, "flops": updates * 40}
    if case["kind"] == "restart":
        return {"bytes": 2 * f * n + 2 * f, "flops": updates * 46 * n}
    if case["kind"] == "grad":
        return {"bytes": 2 * f * n + 3 * f * n + 4 * fields, "flops": updates * (46 + 100) * n}
    return {"bytes": 2 * f * n + 2 * fields, "flops": updates * (46 * n + 20)}


# ---------------------------------------------------------------------------
# The step restated in plain torch, 64 bits
# ---------------------------------------------------------------------------
class _Reference:
    def __init__(self, w):
        self.w, self.nd = w, w.n_dirs
        dev = _device()
        self.dr = (w.r_out - w.r_in) / (w.n_r - 1)
        self.dth = 2.0 * math.pi * w.n_f / (w.n_dirs * w.n_theta)
        self.r = torch.linspace(w.r_in, w.r_out, w.n_r, dtype=torch.float64, device=dev)[None, :]
        th = (torch.arange(1, w.n_theta + 1, dtype=torch.float64, device=dev) * self.dth)[:, None]
        self.cos, self.sin = torch.cos(th), torch.sin(th)
        self.vel, self.shell = [(0.0, 0.0)], [0]
        for k in range(1, 5):
            for i in range(self.nd):
                sgn, a = (1.0, i) if i < self.nd // 2 else (-1.0, i - self.nd // 2)
                phi = 2.0 * math.pi * a / self.nd
                self.vel.append((w.speeds[k] * sgn * math.cos(phi), w.speeds[k] * sgn * math.sin(phi)))
                self.shell.append(k)
        self.q = len(self.vel)
        self.decay = 1.0 - w.dt / w.tau if w.relaxation else math.exp(-w.dt / w.tau)

    def cartesian(self, fields):
        rho, ur, ut, T = fields
        return rho, ur * self.cos - ut * self.sin, ur * self.sin + ut * self.cos, T

    def moments(self, f):
        rho = sum(f[1:], f[0])
        jx = sum(v[0] * p for v, p in zip(self.vel, f) if v[0])
        jy = sum(v[1] * p for v, p in zip(self.vel, f) if v[1])
        e = sum(0.5 * self.w.speeds[k] ** 2 * p for k, p in zip(self.shell, f) if k)
        ux, uy = jx / rho, jy / rho
        return rho, ux, uy, (e - 0.5 * (jx * ux + jy * uy)) / rho

    def polar(self, f):
        rho, ux, uy, E = self.moments(f)
        return torch.stack([rho, ux * self.cos + uy * self.sin, uy * self.cos - ux * self.sin, E])

    def weights(self, E):
        v2, B, F = [s * s for s in self.w.speeds], self.w.B, [None]
        for k in range(1, 5):
            a, b, c = (v2[j] for j in range(1, 5) if j != k)
            den = v2[k] * (v2[k] - a) * (v2[k] - b) * (v2[k] - c)
            num = E * (B[1] * a * b * c + E * (B[2] * (a * b + b * c + c * a) + E * (B[3] * (a + b + c) + E * B[4])))
            F.append(num / den)
        F[0] = 1.0 - B[0] * (F[1] + F[2] + F[3] + F[4])
        return F

    def equilibrium(self, rho, ux, uy, E):
        wk = [rho * F for F in self.weights(E)]
        s = (ux * ux + uy * uy) / E
        a1 = 1.0 - 0.5 * s
        a0 = a1 + 0.125 * s * s
        out = []
        for (vx, vy), k in zip(self.vel, self.shell):
            x = (vx * ux + vy * uy) / E
            out.append(wk[k] * (a0 + x * (a1 + x * (0.5 * a1 + x * (1.0 / 6.0 + x / 24.0)))))
        return out

    def ghosts(self, side, f, m):
        """The two radial ghost layers of a wall, nearest first: planes [n_theta][1]."""
        a, b = (0, 1) if side == 0 else (-1, -2)
        at = lambda x, i: x[:, i:i + 1] if i != -1 else x[:, -1:]  # noqa: E731
        wall, nxt = [at(x, a) for x in m], [at(x, b) for x in m]
        kind = self.w.bc_kind[side] & ~I.BC_NEQ
        layers = []
        for layer in range(2):
            g = [(2 + layer) * p - (1 + layer) * n for p, n in zip(wall, nxt)]
            if kind != I.BC_EXTRAP:
                v = torch.as_tensor(self.w.bc_values[side][layer], dtype=torch.float64, device=f[0].device)[:, :, None]
                g[1], g[2] = v[1] * self.cos - v[2] * self.sin, v[1] * self.sin + v[2] * self.cos
                if kind == I.BC_DIRICHLET:
                    g[0], g[3] = v[0], v[3]
            layers.append(self.equilibrium(*g))
        if self.w.bc_kind[side] & I.BC_NEQ:
            eq = self.equilibrium(*wall)
            layers = [[g + at(p, a) - e for g, p, e in zip(lay, f, eq)] for lay in layers]
        return layers

    def rows(self, f, q):
        """Plane q with two azimuthal ghost rows on each side (Eq. 40)."""
        if q == 0:
            return torch.cat([f[0][-2:], f[0], f[0][:2]])
        base, j = 1 + (q - 1) // self.nd * self.nd, (q - 1) % self.nd
        lo, hi = base + (j + self.w.n_f) % self.nd, base + (j - self.w.n_f) % self.nd
        return torch.cat([f[lo][-2:], f[q], f[hi][:2]])

    def increment(self, C, at):
        """Convection increment of Sec. II B 3 with Courant number C; at(j) the values j cells away."""
        a, pos = C.abs(), C >= 0
        c = at(0)
        up1, up2 = torch.where(pos, at(-1), at(1)), torch.where(pos, at(-2), at(2))
        D, Dp, scheme = c - up1, up1 - up2, self.w.scheme
        if scheme == I.SCHEME_MWB:
            n = D.abs() + Dp.abs()
            ok = n > 0
            h = torch.where(ok, D.abs() * (D - Dp) / torch.where(ok, n, 1.0), 0.0)
            return a * D + a * (1.0 - a) * h
        if scheme == I.SCHEME_WB:
            return a * D + 0.5 * a * (1.0 - a) * (D - Dp)
        if scheme == I.SCHEME_LW:
            return a * D + 0.5 * a * (1.0 - a) * (torch.where(pos, at(1), at(-1)) - c - D)
        return a * D + 0.5 * a * (D - Dp)

    def step(self, f):
        w, n_r, n_t = self.w, self.w.n_r, self.w.n_theta
        m = self.moments(f)
        eq = self.equilibrium(*m)
        inner, outer = self.ghosts(0, f, m), self.ghosts(1, f, m)
        out = []
        for q, (vx, vy) in enumerate(self.vel):
            o = eq[q] + (f[q] - eq[q]) * self.decay
            if q:
                wide = torch.cat([inner[1][q], inner[0][q], f[q], outer[0][q], outer[1][q]], dim=1)
                tall = self.rows(f, q)
                cr = (vx * self.cos + vy * self.sin) * (w.dt / self.dr)
                ct = (vy * self.cos - vx * self.sin) * (w.dt / self.dth) / self.r
                o = o - self.increment(cr, lambda j: wide[:, 2 + j:2 + j + n_r])
                o = o - self.increment(ct, lambda j: tall[2 + j:2 + j + n_t])
            out.append(o)
        return out

    def manifestations(self, f):
        m = self.moments(f)
        eq = self.equilibrium(*m)
        ur, ut = m[1] * self.cos + m[2] * self.sin, m[2] * self.cos - m[1] * self.sin
        groups = []
        for central, departure in ((0, 0), (0, 1), (1, 0), (1, 1)):
            acc = [0.0] * 12
            for (vx, vy), p, e in zip(self.vel, f, eq):
                w = p - e if departure else p
                cr, ct = vx * self.cos + vy * self.sin - central * ur, vy * self.cos - vx * self.sin - central * ut
                h = 0.5 * (cr * cr + ct * ct)
                for i, x in enumerate((cr * cr, cr * ct, ct * ct, cr * cr * cr, cr * cr * ct, cr * ct * ct, ct * ct * ct,
                                       h * cr, h * ct, h * cr * cr, h * cr * ct, h * ct * ct)):
                    acc[i] = acc[i] + w * x
            groups.append(torch.stack(acc))
        return torch.stack(groups)

    def integrals(self, f):
        rho, ux, uy, E = self.moments(f)
        a = self.r * self.dr * self.dth
        out = [(a * x).sum() for x in (rho, rho * ux, rho * uy, rho * (E + 0.5 * (ux * ux + uy * uy)))]
        return np.array([float(x) for x in out + [rho.min(), E.min()]] + [float(rho.numel()), 0.0])


def exact(case, seed):
    w, fields = _problem(case, seed)
    ref, kind = _Reference(w), case["kind"]
    if kind in ("restart", "analysis"):
        f = list(_noisy_f(w, fields, seed).double().unbind(0))
        if kind == "analysis":
            return {"fields": ref.polar(f), "noneq": ref.manifestations(f), "integrals": ref.integrals(f)}
        for _ in range(case["steps"]):
            f = ref.step(f)
        return torch.stack(f)
    x = fields.double()
    if kind != "grad":
        f = ref.equilibrium(*ref.cartesian(x))
        for _ in range(case["steps"]):
            f = ref.step(f)
        out = ref.polar(f)
        return out.cpu() if kind == "host" else out
    # the gradient by plain torch differentiation, one step at a time
    g = _cotangent(fields, seed).double()
    states = [torch.stack(ref.equilibrium(*ref.cartesian(x)))]
    for _ in range(case["steps"]):
        states.append(torch.stack(ref.step(list(states[-1].unbind(0)))))

    def back(fn, at, cotangent):
        at = at.detach().requires_grad_(True)
        return torch.autograd.grad(fn(at), at, cotangent)[0]

    out = ref.polar(list(states[-1].unbind(0)))
    lam = back(lambda f: ref.polar(list(f.unbind(0))), states[-1], g)
    for f in reversed(states[:-1]):
        lam = back(lambda v: torch.stack(ref.step(list(v.unbind(0)))), f, lam)
    return {"fields": out, "gradient": back(lambda v: torch.stack(ref.equilibrium(*ref.cartesian(v))), x, lam)}
