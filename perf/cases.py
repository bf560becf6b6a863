"""Performance cases of the solver: what a program that uses it has it do.

A case is one pass through the public entry points of ``paper_2003_08746_gb300.jz``: load a
state, advance it a few Runge-Kutta steps and take it out (``step``), the same from and to host
arrays (``host``), one evaluation of the right-hand side (``residual``), a window of flow
statistics (``stats``), or the gradient of the observer functional by the discrete adjoint
(``adjoint``).  Sizes are the repository's own workloads, the paper's meshes and the ragged
shapes of the tests; ``draw`` spreads over the range between them.  ``exact`` evaluates the same
quantities in plain FP64 torch.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2003_08746_gb300 import jz
from paper_2003_08746_gb300 import workloads as W

FORMS = {"fp64": jz.JZ_PREC_FP64, "pair": jz.JZ_PREC_FP64PAIR, "fp32flux": jz.JZ_PREC_FP32FLUX}
R_OBS = 0.75                 # observer radius of the adjoint workload
EXACT_NODES = 20_000_000     # above this the plain evaluation takes too long


def _case(name, kind, topo, shape, form, steps, **kw):
    ni, nj, nk = shape
    c = dict(name=name, kind=kind, topo=topo, ni=ni, nj=nj, nk=nk, form=form, steps=steps, stretch=False, compact=False,
             stats=False, every=0)
    c.update(kw)
    return c


def listed():
    return [
        # the periodic box of the conservation checks, its ten steps with the monitor line: the
        # smallest run, where launches and latency count
        _case("box_32x24x16_pair", "step", "box", (32, 24, 16), "pair", 10, stats=True),
        # a coarse jet with odd extents, as used to try parameters before a long run
        _case("jet_70x33x18_pair", "step", "jet", (70, 33, 18), "pair", 10, stats=True),
        # the jet subsample in the FP32-flux form, between two exchanges of the state
        _case("jet_64x32x16_fp32flux", "step", "jet", (64, 32, 16), "fp32flux", 2),
        # the quick start: host arrays in, a block of steps with the monitor line, host arrays out
        _case("jet_256x128x64_pair_host", "host", "jet", (256, 128, 64), "pair", 50, stats=True),
        # the same jet in the FP32-flux form, two steps between exchanges of the state with a program
        _case("jet_256x128x64_fp32flux", "step", "jet", (256, 128, 64), "fp32flux", 2),
        # the default (all-FP64) form on the adjoint workload's jet
        _case("jet_128x96x64_fp64", "step", "jet", (128, 96, 64), "fp64", 5, stats=True),
        # the medium jet in the FP32-flux form
        _case("jet_512x256x128_fp32flux", "step", "jet", (512, 256, 128), "fp32flux", 2, stats=True),
        # the paper's mesh E in the headline form
        _case("jet_512x512x360_pair", "step", "jet", (512, 512, 360), "pair", 2, stretch=True),
        # the paper's mesh F on a compact grid, the form of the largest meshes
        _case("jet_1024x512x360_compact", "step", "jet", (1024, 512, 360), "fp32flux", 2, compact=True),
        # one right-hand side for a program with a time integrator of its own; ragged extents
        _case("residual_333x177x90_pair", "residual", "jet", (333, 177, 90), "pair", 0),
        # a window of the validation statistics
        _case("stats_256x128x64_pair", "stats", "jet", (256, 128, 64), "pair", 12, every=2),
        # gradient of the observer functional with respect to the entrance forcing
        _case("adjoint_128x96x64_pair", "adjoint", "jet", (128, 96, 64), "pair", 10, every=5),
    ]


def draw(rng):
    """One more case: kind and form by how often a program uses them, the node count spread over
    its logarithm, extents ragged; the steps bounded so that a pass stays under the largest
    listed one."""
    kind = rng.choice(["step", "step", "step", "step", "host", "residual", "stats", "adjoint"])
    if kind == "adjoint":
        lo, hi, form = 3.5e4, 6e5, rng.choice(["pair", "pair", "fp64"])
    elif kind == "stats":
        lo, hi, form = 2e4, 4e6, "pair"
    elif kind == "residual":
        lo, hi, form = 1e4, 2e7, rng.choice(["pair", "pair", "fp64"])
    elif kind == "host":
        lo, hi, form = 1e4, 4e6, rng.choice(["pair", "fp64"])
    else:
        form = rng.choice(["pair", "pair", "fp32flux", "fp32flux", "fp64"])
        lo, hi = {"pair": (8e3, 4e7), "fp32flux": (3e4, 1e8), "fp64": (8e3, 4e6)}[form]
    n = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    topo = "box" if kind in ("step", "residual") and form != "fp32flux" and rng.random() < 0.25 and n < 3e6 else "jet"
    # extents around the paper's proportions (axial : radial : azimuthal), each its own factor
    a, b, c = 2.0 * math.exp(rng.uniform(-0.4, 0.4)), math.exp(rng.uniform(-0.4, 0.4)), math.exp(rng.uniform(-0.5, 0.2))
    u = (n / (a * b * c)) ** (1.0 / 3.0)
    ni, nj, nk = max(12, round(a * u)), max(10, round(b * u)), max(8, 2 * round(c * u / 2))
    if topo == "box":
        nk += rng.randrange(2)
    if kind in ("step", "host"):
        steps = rng.randint(1, 3) if form == "fp32flux" else rng.randint(2, 12)
        if form == "pair" and ni * nj * nk > 1e7:
            steps = min(steps, 4)
    else:
        steps = {"residual": 0, "stats": rng.randint(4, 12), "adjoint": rng.randint(3, 9)}[kind]
    every = {"stats": rng.randint(1, 3), "adjoint": rng.randint(2, 5)}.get(kind, 0)
    c = _case("", kind, topo, (ni, nj, nk), form, steps, every=every, stats=rng.random() < 0.5,
              stretch=topo == "jet" and rng.random() < 0.3, compact=form == "fp32flux" and n > 5e6 and rng.random() < 0.5)
    del c["name"]
    return c


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _grid_xyz(case):
    if case["topo"] == "box":
        g = W.box_grid(case["ni"], case["nj"], case["nk"])
        return torch.as_tensor(g.xyz, device="cuda"), g.period
    return W.jet_grid_device(case["ni"], case["nj"], case["nk"], "cuda", axial_stretch=case["stretch"]), None


def _params(case, seed):
    return W.box_params() if case["topo"] == "box" else W.jet_params(seed=2 + seed % 1000)


def _initial(case, xyz, seed):
    """Box: Mach 0.5 flow with velocity noise.  Jet: the parallel tanh jet with a developing
    shear layer (helical modes and noise around r = 0.5, pressure and density noise)."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    shape = tuple(xyz.shape[1:])

    def noise(a):
        return a * torch.randn(shape, generator=gen, device="cuda", dtype=torch.float64)

    gamma = W.GAMMA
    q = torch.empty((5,) + shape, dtype=torch.float64, device="cuda")
    if case["topo"] == "box":
        rho, p = torch.ones(shape, dtype=torch.float64, device="cuda"), 1.0 / gamma
        vel = [0.5 + noise(1e-3), noise(1e-3), noise(1e-3)]
    else:
        r = torch.sqrt(xyz[1] * xyz[1] + xyz[2] * xyz[2])
        env = torch.exp(-((r - 0.5) / 0.2) ** 2) * (r > 0)
        th = torch.atan2(xyz[2], xyz[1])
        ph = torch.rand(4, generator=gen, device="cuda", dtype=torch.float64).cpu()
        wave = torch.zeros_like(r)
        for m in range(4):
            wave += torch.cos(m * th - (1.0 + 0.5 * m) * xyz[0] + 2.0 * math.pi * float(ph[m]))
        base = 0.7 * (1.0 + torch.tanh((0.5 - r) / 0.1))
        del r, th
        vel = [base + env * (0.02 * wave + noise(2e-3)), env * (0.01 * wave + noise(2e-3)), env * noise(2e-3)]
        del base, wave
        rho = 1.0 + env * noise(1e-3)
        p = (1.0 + env * noise(1e-3)) / gamma
        del env
    q[0] = rho
    for a in range(3):
        q[a + 1] = rho * vel[a]
    q[4] = p / (gamma - 1.0) + 0.5 * rho * (vel[0] * vel[0] + vel[1] * vel[1] + vel[2] * vel[2])
    return q


def prepare(case, seed):
    xyz, period = _grid_xyz(case)
    q = _initial(case, xyz, seed)
    topo = W.TOPO_PERIODIC if case["topo"] == "box" else W.TOPO_JET
    prm = _params(case, seed)
    grid = jz.Grid(case["ni"], case["nj"], case["nk"], xyz, topo, period)
    del xyz
    torch.cuda.empty_cache()     # the library allocates beside torch's pool
    if case["compact"]:
        grid.compact()
    s = jz.Solver(grid, prm, FORMS[case["form"]])
    state = {"case": case, "solver": s, "grid": grid, "prm": prm, "q": q}
    if case["kind"] == "host":
        state["q"] = q.cpu().numpy()
        state["out"] = np.empty_like(state["q"])
    elif case["kind"] == "adjoint":
        s.set_state(q, 0.0)
        state["amps"] = np.asarray(prm.forcing_amp)
    else:
        state["out"] = torch.empty_like(q)
    return state


def _stat_outputs(st):
    return {"t": st.t, "dt": st.dt, "res_l2": st.res_l2, "totals": np.array(list(st.totals)), "min_rho": st.min_rho,
            "min_p": st.min_p}


def run(state):
    c, s = state["case"], state["solver"]
    if c["kind"] == "adjoint":
        J, g = jz.jz_adjoint_step(s.h, state["amps"], c["steps"], c["every"], R_OBS)
        return {"J": J, "grad": g}
    if c["kind"] == "residual":
        return {"rhs": s.residual(state["q"], state["out"])}
    if c["kind"] == "stats":
        s.set_state(state["q"], 0.0)
        s.stats_begin(c["every"])
        s.step(c["steps"], False)
        mean, rms, _ = s.stats_read()
        return {"mean": mean, "rms": rms, "q": s.get_state(state["out"])}
    s.set_state(state["q"], 0.0)
    st = s.step(c["steps"], c["stats"])
    out = {"q": s.get_state(state["out"])}
    if c["stats"]:
        out.update(_stat_outputs(st))
    return out


def work(case):
    """Bytes: per point-stage Q^(l-1), Q^n (once at stage 1), the metrics and Q^(l) (192 bytes with
    FP64 metrics, 152 with FP32 ones), the state in and out; the adjoint adds a reverse stage that
    reads the stage state and metrics again and the adjoint state twice.  Flops: the FP64 form's
    operations per point-stage, a reverse stage about twice a forward one."""
    n = case["ni"] * case["nj"] * case["nk"]
    per = 152 if case["form"] == "fp32flux" else 192
    io = 2 * 40 * n
    if case["kind"] == "residual":
        return {"bytes": 160 * n, "flops": 600 * n}
    ps = 5 * case["steps"] * n
    if case["kind"] == "adjoint":
        return {"bytes": ps * (per + 240), "flops": ps * 600 * 3}
    extra = 48 * n * (case["steps"] // case["every"]) if case["kind"] == "stats" else 0
    return {"bytes": ps * per + io + extra, "flops": ps * 600}


# ---------------------------------------------------------------------------
# The same quantities in plain FP64 torch
# ---------------------------------------------------------------------------
ALPHA = (0.25, 1.0 / 6.0, 0.375, 0.5, 1.0)


def _root(x, e):
    """x^e for x >= 0 with value and derivative 0 at 0."""
    ok = x > 0
    return torch.where(ok, torch.where(ok, x, torch.ones_like(x)) ** e, torch.zeros_like(x))


class _Plain:
    """The scheme on arrays padded by two ghost layers ([nk+4][nj+4][ni+4])."""

    def __init__(self, case, prm):
        self.n = (case["nk"], case["nj"], case["ni"])
        self.jet = case["topo"] == "jet"
        self.prm = prm
        self.g = prm.gamma
        self.gm1 = prm.gamma - 1.0
        xyz, period = _grid_xyz(case)
        self.x1d = xyz[0, 0, 0].clone()
        self.y0, self.z0 = xyz[1, :, :, 0].clone(), xyz[2, :, :, 0].clone()
        self._metrics(self._pad_xyz(xyz, period))
        adv = torch.ones(self.n, dtype=torch.bool, device="cuda")
        if self.jet:
            adv[:, 0] = adv[:, -1] = False
            adv[:, :, 0] = adv[:, :, -1] = False
        self.adv = adv

    # -- ghosts --
    def pad(self, f):
        nk, nj, ni = self.n
        if self.jet:
            far = f[..., -1:, :]
            f = torch.cat([f[..., 2:3, :].roll(-(nk // 2), -3), f[..., 1:2, :].roll(-(nk // 2), -3), f, far, far], -2)
            i = torch.arange(-2, ni + 2, device="cuda").clamp(0, ni - 1)
        else:
            f = f[..., torch.arange(-2, nj + 2, device="cuda") % nj, :]
            i = torch.arange(-2, ni + 2, device="cuda") % ni
        return f[..., i][..., torch.arange(-2, nk + 2, device="cuda") % nk, :, :]

    def _pad_xyz(self, xyz, period):
        nk, nj, ni = self.n
        p = self.pad(xyz)
        if not self.jet:
            for axis, n, per in ((-1, ni, period[0]), (-2, nj, period[1]), (-3, nk, period[2])):
                wrap = torch.div(torch.arange(-2, n + 2, device="cuda"), n, rounding_mode="floor").double()
                wrap = wrap.reshape([-1 if a == axis else 1 for a in (-3, -2, -1)])
                for c in range(3):
                    p[c] += wrap * float(per[c])
            return p
        for m in (1, 2):
            p[:, :, nj + 1 + m] = (1 + m) * p[:, :, nj + 1] - m * p[:, :, nj]
        for m in (1, 2):
            p[..., 2 - m] = (1 + m) * p[..., 2] - m * p[..., 3]
            p[..., ni + 1 + m] = (1 + m) * p[..., ni + 1] - m * p[..., ni]
        return p

    def at(self, f, layers, axis=None, off=0):
        """View of a padded array on the nodes within `layers` of the real ones, shifted by `off`
        along `axis` (-1 i, -2 j, -3 k)."""
        pad = (f.shape[-1] - self.n[2]) // 2
        for a in (-3, -2, -1):
            o = off if a == axis else 0
            f = f.narrow(a, pad - layers + o, self.n[a] + 2 * layers)
        return f

    def diff(self, f, layers, axis):
        return 0.5 * (self.at(f, layers, axis, 1) - self.at(f, layers, axis, -1))

    def _metrics(self, X):
        def cross(a, b):
            return torch.stack([a[1] * b[2] - a[2] * b[1], a[2] * b[0] - a[0] * b[2], a[0] * b[1] - a[1] * b[0]])
        ax = (-1, -2, -3)
        r1 = self.at(X, 1)
        C = [cross(self.diff(X, 1, a), r1) for a in ax]
        S = [0.5 * (self.diff(C[1], 0, -3) - self.diff(C[2], 0, -2)), 0.5 * (self.diff(C[2], 0, -1) - self.diff(C[0], 0, -3)),
             0.5 * (self.diff(C[0], 0, -2) - self.diff(C[1], 0, -1))]
        d = [self.diff(X, 0, a) for a in ax]
        V = (d[0] * cross(d[1], d[2])).sum(0)
        self.V = V
        self.Sfar = S[1][:, :, -1].clone()
        self.S = self.pad(torch.stack(S))                      # [dir][component] padded
        Vp = self.pad(V)
        self.iV = torch.where(Vp > 0, 1.0 / torch.where(Vp > 0, Vp, torch.ones_like(Vp)), torch.zeros_like(Vp))
        self.Delta = _root(Vp, 1.0 / 3.0)
        self.Smag = torch.sqrt((self.S * self.S).sum(1))

    # -- one right-hand side --
    def prims(self, Q):
        u = Q[1:4] / Q[0]
        p = self.gm1 * (Q[4] - 0.5 * (Q[1:4] * u).sum(0))
        return u, p, self.g * p / Q[0]

    def radii(self, u, T, S, Smag):
        a = torch.sqrt(T)
        return [torch.abs((S[d] * u).sum(0)) + a * Smag[d] for d in range(3)]

    def rhs(self, Q):
        P = self.prm
        Qp = self.pad(Q)
        up, pp, Tp = self.prims(Qp)
        S1, iV1 = self.at(self.S, 1), self.at(self.iV, 1)
        Q1, u, p, T = self.at(Qp, 1), self.at(up, 1), self.at(pp, 1), self.at(Tp, 1)
        ax = (-1, -2, -3)
        f = torch.cat([up, Tp[None]])
        dd = [self.diff(f, 1, a) for a in ax]
        grad = [iV1 * (S1[0][j] * dd[0] + S1[1][j] * dd[1] + S1[2][j] * dd[2]) for j in range(3)]   # grad[j][n]
        del dd
        sij = [[0.5 * (grad[j][i] + grad[i][j]) for j in range(3)] for i in range(3)]
        div = sij[0][0] + sij[1][1] + sij[2][2]
        SS = sum(sij[i][j] * sij[i][j] for i in range(3) for j in range(3))
        sh = P.S1_K / P.T_ref_K
        mu = P.mach_ref / P.Re * T * torch.sqrt(T) * (1.0 + sh) / (T + sh)
        mus = Q1[0] * (P.C_s * self.at(self.Delta, 1)) ** 2 * _root(2.0 * SS, 0.5)
        cp = 1.0 / self.gm1
        kap = mu * cp / P.Pr + mus * cp / P.Pr_sgs
        tau = [[2.0 * (mu + mus) * (sij[i][j] - (div / 3.0 if i == j else 0.0)) for j in range(3)] for i in range(3)]
        F = [[tau[0][j], tau[1][j], tau[2][j],
              u[0] * tau[0][j] + u[1] * tau[1][j] + u[2] * tau[2][j] + kap * grad[j][3]] for j in range(3)]
        del grad, sij
        lam = self.radii(u, T, S1, self.at(self.Smag, 1))
        hi, lo = [_root(x, P.sigma) for x in lam], [_root(x, 1.0 - P.sigma) for x in lam]
        acc = torch.zeros_like(Q)
        for d in range(3):
            a = ax[d]
            U = (S1[d] * u).sum(0)
            H = [Q1[0] * U] + [Q1[m + 1] * U + p * S1[d][m] for m in range(3)] + [(Q1[4] + p) * U]
            for m in range(4):
                H[m + 1] = H[m + 1] - sum(S1[d][j] * F[j][m] for j in range(3))
            H = torch.stack(H)
            Lam = lam[d] + lo[d] * sum(hi[e] for e in range(3) if e != d)
            pm, pq = self.at(pp, 1, a, -1), self.at(pp, 1, a, 1)
            nu = torch.abs(pq - 2.0 * p + pm) / (pq + 2.0 * p + pm)
            # faces n + 1/2 for n = -1 .. N-1 along a, real nodes across
            n = self.n[a]

            def line(x, off):                       # nodes n + off of the faces
                lay = (x.shape[-1] - self.n[2]) // 2
                for b in (-3, -2, -1):
                    x = x.narrow(b, lay - 1 + off, n + 1) if b == a else x.narrow(b, lay, self.n[b])
                return x

            n0, n1 = line(nu, 0), line(nu, 1)
            e2 = P.kappa2 * torch.where(n0 >= n1, n0, n1)
            k4 = P.kappa4 - e2
            e4 = torch.where(k4 > 0, k4, torch.zeros_like(k4))
            L = 0.5 * (line(Lam, 0) + line(Lam, 1))
            q0, q1 = line(Qp, 0), line(Qp, 1)
            D = L * (e2 * (q1 - q0) - e4 * (line(Qp, 2) - 3.0 * q1 + 3.0 * q0 - line(Qp, -1)))
            G = 0.5 * (line(H, 0) + line(H, 1)) - D
            acc = acc + G.narrow(a, 1, n) - G.narrow(a, 0, n)
        return acc * self.at(self.iV, 0)

    # -- boundary conditions of the jet --
    def _cons(self, rho, u, p):
        return torch.cat([rho[None], rho * u, (p / self.gm1 + 0.5 * rho * (u * u).sum(0))[None]])

    def target(self, t, amp):
        P = self.prm
        y, z = self.y0[:, 1:], self.z0[:, 1:]
        r, th = torch.sqrt(y * y + z * z), torch.atan2(z, y)
        f = torch.zeros_like(r)
        for m in range(8):
            for q in range(4):
                s = torch.sin(2.0 * math.pi * P.strouhal[q] * P.jet_mach * t + float(P.forcing_psi[m, q]))
                f = f + amp[m, q] * s * torch.cos(m * th + float(P.forcing_phi[m, q]))
        return (0.5 * P.jet_mach * (1.0 + torch.tanh((0.5 - r) / (2.0 * P.theta_mom)))
                + P.jet_mach * torch.exp(-((r - 0.5) / 0.1) ** 2) * f)

    def bcs(self, Q, t, amp):
        g, gm1 = self.g, self.gm1
        # far field
        S = self.Sfar[:, :, 1:-1]
        nrm = S / torch.sqrt((S * S).sum(0))
        qi = Q[:, :, -2, 1:-1]
        u, p, T = self.prims(qi)
        un_i = (u * nrm).sum(0)
        Rp, Rm = un_i + 2.0 * torch.sqrt(T) / gm1, -2.0 / gm1
        un, ab = 0.5 * (Rp + Rm), 0.25 * gm1 * (Rp - Rm)
        o = un > 0
        s = torch.where(o, p / qi[0] ** g, torch.full_like(p, 1.0 / g))
        rho = (ab * ab / (g * s)) ** (1.0 / gm1)
        ut = torch.where(o, u - un_i * nrm, torch.zeros_like(u))
        far = self._cons(rho, ut + un * nrm, rho * ab * ab / g)
        Q = torch.cat([Q[:, :, :-1], torch.cat([Q[:, :, -1, :1], far, Q[:, :, -1, -1:]], -1)[:, :, None]], 2)
        # entrance
        ut = self.target(t, amp)
        u, p, T = self.prims(Q[:, :, 1:, 1])
        Rm, Rp = u[0] - 2.0 * torch.sqrt(T) / gm1, ut + 2.0 / gm1
        ub, ab = 0.5 * (Rp + Rm), 0.25 * gm1 * (Rp - Rm)
        rs = (ab * ab) ** (1.0 / gm1)
        sup = ut >= 1.0
        rho = torch.where(sup, torch.ones_like(rs), rs)
        p = torch.where(sup, torch.full_like(rs, 1.0 / g), rs * ab * ab / g)
        zero = torch.zeros_like(ub)
        ent = self._cons(rho, torch.stack([torch.where(sup, ut, ub), zero, zero]), p)
        # exit: ambient pressure, velocity and temperature of the node before
        u, p, T = self.prims(Q[:, :, 1:, -2])
        ex = self._cons(1.0 / T, u, torch.full_like(T, 1.0 / g))
        Q = torch.cat([Q[..., :1, :], torch.cat([ent[..., None], Q[..., 1:, 1:-1], ex[..., None]], -1)], -2)
        ring = Q[:, :, 1:2].mean(1, keepdim=True).expand(-1, self.n[0], -1, -1)
        return torch.cat([ring, Q[:, :, 1:]], 2)

    def rate(self, Q):
        u, _, T = self.prims(Q)
        lam = self.radii(u, T, self.at(self.S, 0), self.at(self.Smag, 0))
        return ((lam[0] + lam[1] + lam[2]) * self.at(self.iV, 0))[self.adv].max()

    def stage(self, Qn, Qs, a, dt, t, amp):
        R = self.rhs(Qs)
        Qs = torch.where(self.adv, Qn - a * dt * R, Qs)
        return (self.bcs(Qs, t + a * dt, amp) if self.jet else Qs), R

    def step(self, Q, t, dt, amp):
        Qs, R0 = Q, None
        for a in ALPHA:
            Qs, R = self.stage(Q, Qs, a, dt, t, amp)
            R0 = R if R0 is None else R0
        return Qs, R0

    def functional(self, Q):
        r = torch.sqrt(self.y0[0] ** 2 + self.z0[0] ** 2)
        j = int((r <= R_OBS).nonzero().max())
        b = float((R_OBS - r[j]) / (r[j + 1] - r[j]))
        x = self.x1d
        dx = torch.cat([x[1:2] - x[:1], x[2:] - x[:-2], x[-1:] - x[-2:-1]]) * 0.5
        pt = (1.0 - b) * self.prims(Q[:, :, j])[1] + b * self.prims(Q[:, :, j + 1])[1]
        return (R_OBS * (2.0 * math.pi / self.n[0]) * dx * (pt - 1.0 / self.g) ** 2).sum()


def exact(case, seed):
    n = case["ni"] * case["nj"] * case["nk"]
    if n > EXACT_NODES:
        return None
    xyz, _ = _grid_xyz(case)
    Q = _initial(case, xyz, seed)
    del xyz
    prm = _params(case, seed)
    with torch.no_grad():
        pl = _Plain(case, prm)
        amp = None if prm.forcing_amp is None else torch.as_tensor(np.asarray(prm.forcing_amp), device="cuda")
        t = torch.zeros((), dtype=torch.float64, device="cuda")
        if case["kind"] == "residual":
            R = pl.rhs(Q)
            return {"rhs": torch.where(pl.adv, R, torch.zeros_like(R))}
    if case["kind"] == "adjoint":
        return _exact_gradient(pl, Q, amp, case["steps"])
    with torch.no_grad():
        U, R = [], None
        for k in range(case["steps"]):
            dt = prm.cfl / pl.rate(Q)
            Q, R = pl.step(Q, t, dt, amp)
            t = t + dt
            if case["kind"] == "stats" and (k + 1) % case["every"] == 0:
                U.append(Q[1] / Q[0])
        if case["kind"] == "stats":
            U = torch.stack(U)
            m = U.mean(0)
            rms = torch.sqrt(((U - m) ** 2).mean(0))
            return {"mean": m.mean(0).cpu().numpy(), "rms": rms.mean(0).cpu().numpy(), "q": Q}
        out = {"q": Q.cpu().numpy() if case["kind"] == "host" else Q}
        if case["stats"]:
            p = pl.prims(Q)[1]
            out.update({"t": float(t), "dt": float(dt), "res_l2": float(torch.sqrt((R[0][pl.adv] ** 2).mean())),
                        "totals": (Q * pl.V).reshape(5, -1).sum(1).cpu().numpy(), "min_rho": float(Q[0].min()),
                        "min_p": float(p.min())})
        return out


def _exact_gradient(pl, Q, amp, steps):
    """J and dJ/dA by reverse-mode differentiation, one stage's graph at a time."""
    from torch.utils.checkpoint import checkpoint
    with torch.no_grad():
        dt = pl.prm.cfl / pl.rate(Q)
    A = amp.clone().requires_grad_(True)
    J = torch.zeros((), dtype=torch.float64, device="cuda")
    for n in range(steps):
        Qn = Qs = Q
        for a in ALPHA:
            Qs = checkpoint(lambda q0, q, am, a=a, t=n * dt: pl.stage(q0, q, a, dt, t, am)[0], Qn, Qs, A, use_reentrant=False)
        Q = Qs
        J = J + dt * pl.functional(Q)
    (g,) = torch.autograd.grad(J, A)
    return {"J": float(J.detach()), "grad": g.cpu().numpy()}
