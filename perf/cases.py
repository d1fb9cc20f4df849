"""Performance cases of the UGKS library: what a user of it has it do, through its public
entry points (`ugks.Solver`, `ugks.Batch`), and what each pass has to give in 64 bits.

A pass advances a channel flow that is under way by a few explicit steps and takes the whole
state (f and W) out to device buffers, as a program does between two residual checks or
checkpoints.  The configurations are those of `inputs.py`: the 2D pressure-driven channel, its
mesh-size and velocity-grid sweeps, the uneven batch and the serving requests.

The FP32-f form stores and transports f in FP32; a program that picks it keeps what it takes out
in FP32, so its outputs are FP32 tensors here.  The FP64 and DF64 (FP64-accurate) forms' are FP64.
"""
import math

import numpy as np
import torch

from paper_1810_08137_gb300 import inputs as I
from paper_1810_08137_gb300 import ugks

FORMS = {"fp32f": ugks.FP32F, "fp64": ugks.FP64, "df64": ugks.DF64}


# ---------------------------------------------------------------------------------------
# Cases
# ---------------------------------------------------------------------------------------
def solve(name, form, nx, ny, n_vel, kn, steps, vrange=4.0, rho_in=1.2, pr=1.0):
    """One instance: mesh, velocities per axis on [-vrange, vrange]^2, Kn, steps per pass."""
    return {"name": name, "kind": "solve", "form": form, "nx": nx, "ny": ny, "n_vel": n_vel, "kn": kn,
            "steps": steps, "vrange": vrange, "rho_in": rho_in, "pr": pr}


def batch(name, count, mix, scale, steps, tuned):
    """`count` uneven FP32-f instances in one batch, drawn with the integer `mix` as in the
    uneven batch (scale "full") or the serving requests (scale "small")."""
    return {"name": name, "kind": "batch", "count": count, "mix": mix, "scale": scale, "steps": steps,
            "tuned": tuned}


def listed():
    return [
        # the small channel of the first workload, to be run to steady state: many cheap steps,
        # where the launches and each kernel's latency count
        solve("small_40x20_v20", "fp32f", 40, 20, 20, 0.1, 40),
        # mesh sweep, smallest mesh: a few thousand cells, less work than the chip has room for
        solve("mesh_100x50_v28", "fp32f", 100, 50, 28, 0.05, 20),
        # ragged: an odd mesh, an odd velocity grid with nodes at u = 0 and v = 0, a rarefied gas
        solve("ragged_333x167_v37", "fp32f", 333, 167, 37, 0.5, 5, rho_in=1.5),
        # mesh sweep, largest mesh: the headline workload, f far larger than L2
        solve("mesh_800x400_v28", "fp32f", 800, 400, 28, 0.05, 5),
        # large velocity space (particle-like phase): few cells, many velocities
        solve("velocity_200x100_v101", "fp32f", 200, 100, 101, 0.01, 5, vrange=20.0, rho_in=1.05),
        # the Prandtl number of a monatomic gas: the Shakhov model
        solve("shakhov_200x100_v28", "fp32f", 200, 100, 28, 0.05, 5, pr=2.0 / 3.0),
        # serving: a dozen small requests in flight, the steps between two residual checks
        batch("serve_12_small", 12, 7, "small", 20, False),
        # uneven batch with tuned tiles: meshes 50x25 to 400x200, 16^2 to 64^2 velocities
        batch("batch_16_uneven", 16, 3, "full", 5, True),
        # FP64-accurate results at the second mesh of the sweep
        solve("df64_200x100_v28", "df64", 200, 100, 28, 0.05, 3),
        # the same on a wide velocity grid
        solve("df64_60x30_v101", "df64", 60, 30, 101, 0.01, 3, vrange=20.0, rho_in=1.05),
        # the plain FP64 form: reference runs on a small and a medium mesh
        solve("fp64_40x20_v20", "fp64", 40, 20, 20, 0.1, 10),
        solve("fp64_100x50_v28", "fp64", 100, 50, 28, 0.05, 3),
    ]


def draw(rng):
    def logint(lo, hi):
        return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))

    what = rng.choices(("fp32f", "batch", "df64", "fp64"), (6, 2, 2, 2))[0]
    if what == "batch":
        small = rng.random() < 0.5
        while True:
            case = batch("", rng.randint(4, 24) if small else rng.randint(3, 16), rng.randint(100, 99999),
                         "small" if small else "full", rng.randint(10, 20) if small else rng.randint(2, 5), not small)
            if work(case)["bytes"] <= 3e10:
                break
    else:
        # velocity-cells of the instance: up to the largest of the form's listed cases
        most = {"fp32f": 200e6, "df64": 20e6, "fp64": 5e6}[what]
        while True:
            nx, n_vel = logint(20, 800), logint(16, 201)
            ny = max(8, nx // 2 + rng.randint(-3, 3))
            if 1e5 <= nx * ny * n_vel * n_vel <= most:
                break
        vc = nx * ny * n_vel * n_vel
        steps = max(3, min(40, int(2e7 / vc))) if what == "fp32f" else 3
        wide = n_vel >= 51
        case = solve("", what, nx, ny, n_vel, round(math.exp(rng.uniform(math.log(1e-3), 0.0)), 6), steps,
                     vrange=20.0 if wide else 4.0, rho_in=round(rng.uniform(1.05, 1.5), 4),
                     pr=rng.choice((2.0 / 3.0, 0.72)) if what != "df64" and rng.random() < 0.15 else 1.0)
    del case["name"]
    return case


def configs(case):
    """The inputs.Config of every instance of the case."""
    if case["kind"] == "solve":
        c = I.channel_config(nx=case["nx"], ny=case["ny"], n_vel=case["n_vel"], vrange=case["vrange"],
                             kn=case["kn"], rho_in=case["rho_in"])
        return [c.replace(pr=case["pr"])]
    if case["scale"] == "full":
        return I.workload_batch(case["count"], seed=case["mix"])
    return I.workload_serving(case["count"], seed=case["mix"], scale="small")[0]


def form_of(case):
    return case["form"] if case["kind"] == "solve" else "fp32f"


def fields(cfg, seed, instance):
    """Primitive fields (rho, U, V, T) of a channel flow under way: density falling from the
    inlet to the outlet, a parabolic velocity profile, and noise of 1e-3 in every field."""
    r = np.random.default_rng([seed, instance])
    noise = 1e-3 * r.standard_normal((4, cfg.ny, cfg.nx))
    x = (np.arange(cfg.nx) + 0.5) / cfg.nx
    y = (np.arange(cfg.ny) + 0.5) / cfg.ny
    rin, rout = cfg.bc[I.SIDE_W].rho, cfg.bc[I.SIDE_E].rho
    rho = (rin + (rout - rin) * x)[None, :] * (1.0 + noise[0])
    U = 0.3 * (rin - rout) * (0.3 + 4.0 * y * (1.0 - y))[:, None] + noise[1]
    return [np.ascontiguousarray(a.reshape(-1)) for a in (rho, U, noise[2], 1.0 + noise[3])]


def prepare(case, seed):
    cfgs = configs(case)
    if case["kind"] == "solve":
        owner = ugks.Solver(cfgs[0], FORMS[case["form"]])
        solvers = [owner]
    else:
        owner = ugks.Batch(len(cfgs))
        slots = [owner.admit(c) for c in cfgs]
        solvers = [owner.instance(s) for s in slots]
        # the fields of every instance are set again after the tuner's own steps
        for k, (c, s) in enumerate(zip(cfgs, solvers)):
            s.init_maxwellian(*fields(c, seed, k))
        if case["tuned"]:
            owner.tune(1)
        else:
            owner.set_persistent(False)  # what serve.gpu_server picks for little work in flight
    for k, (c, s) in enumerate(zip(cfgs, solvers)):
        s.init_maxwellian(*fields(c, seed, k))
    out = [(torch.empty(c.nc, c.nq, 2, dtype=torch.float64, device="cuda"),
            torch.empty(4, c.nc, dtype=torch.float64, device="cuda")) for c in cfgs]
    return {"owner": owner, "solvers": solvers, "out": out, "steps": case["steps"],
            "fp32": form_of(case) == "fp32f"}


def run(state):
    state["owner"].step(state["steps"])
    got = {}
    for k, (s, (f, W)) in enumerate(zip(state["solvers"], state["out"])):
        s.get_state_device(f, W)
        got["f%d" % k], got["W%d" % k] = (f.float(), W.float()) if state["fp32"] else (f, W)
    return got


def work(case):
    """Each step has to read f once and write it once as the form stores it (8 bytes per cell and
    velocity in FP32-f, 16 in the others); the state goes out once.  Operations per cell and
    velocity: two limited slopes of two components (28), their moments (40), the micro flux of
    two faces (2 x 34) and the implicit update (34)."""
    vc = sum(c.nc * c.nq for c in configs(case))
    stored, taken = (8, 8) if form_of(case) == "fp32f" else (16, 16)
    return {"bytes": vc * (2.0 * stored * case["steps"] + stored + taken), "flops": 170.0 * vc * case["steps"]}


# ---------------------------------------------------------------------------------------
# The same steps in 64 bits, in plain torch: the scheme's definition face by face (Eqs. 1-4
# and S1-S8 of Liu, Hu & Li, arXiv:1810.08137), for channels with pressure ends and diffuse
# walls
# ---------------------------------------------------------------------------------------
def exact(case, seed):
    if sum(c.nc * c.nq for c in configs(case)) * case["steps"] > 1.5e9:
        return None
    got = {}
    for k, c in enumerate(configs(case)):
        s = Channel64(c)
        s.start(*fields(c, seed, k))
        for _ in range(case["steps"]):
            s.step()
        f, W = torch.stack((s.h, s.b), dim=-1).reshape(c.nc, c.nq, 2), s.W.reshape(4, c.nc)
        got["f%d" % k], got["W%d" % k] = f, W
    return got


class Channel64:
    def __init__(self, c):
        self.c = c
        self.dev = "cuda" if torch.cuda.is_available() else "cpu"
        self.K, self.dx, self.dy = c.K, c.lx / c.nx, c.ly / c.ny
        u, wu = self.axis(c.nu, c.umin, c.umax)
        v, wv = self.axis(c.nv, c.vmin, c.vmax)
        self.u, self.v = u.repeat(c.nv), v.repeat_interleave(c.nu)
        self.w = (wv[:, None] * wu[None, :]).reshape(-1)
        self.dt = c.cfl / (float(u.abs().max()) / self.dx + float(v.abs().max()) / self.dy)
        a, om = c.alpha, c.omega
        self.mu = 5 * (a + 1) * (a + 2) * math.sqrt(math.pi) / (4 * a * (5 - 2 * om) * (7 - 2 * om)) * c.kn

    def axis(self, n, lo, hi):
        d = (hi - lo) / (n - 1)
        x = 0.5 * (lo + hi) + (torch.arange(n, dtype=torch.float64) - 0.5 * (n - 1)) * d
        w = torch.full((n,), d, dtype=torch.float64)
        w[0] = w[-1] = 0.5 * d
        return x.to(self.dev), w.to(self.dev)

    def g(self, rho, U, V, lam):
        """Maxwellian at every velocity; the fields have any shape, velocities go last."""
        e = (self.u - U[..., None]).square_()
        e.add_((self.v - V[..., None]).square_()).mul_(-lam[..., None]).exp_()
        return e.mul_((rho * lam / math.pi)[..., None])

    def start(self, rho, U, V, T):
        shape = (self.c.ny, self.c.nx)
        rho, U, V, T = (torch.from_numpy(a).to(self.dev).reshape(shape) for a in (rho, U, V, T))
        self.h = self.g(rho, U, V, 1 / T)
        self.b = self.h * (self.K * T / 2)[..., None]
        self.W = torch.stack((rho, rho * U, rho * V, rho * (0.5 * (U * U + V * V) + (self.K + 2) * T / 4)))

    def prim(self, W):
        U, V = W[1] / W[0], W[2] / W[0]
        return W[0], U, V, (self.K + 2) * W[0] / (4 * (W[3] - 0.5 * W[0] * (U * U + V * V)))

    def tau(self, rho, lam):
        return self.mu * lam ** -self.c.omega * 2 * lam / rho

    def ghosts(self):
        """h, b and W with one ghost cell on each side (a wall's is a copy of its neighbour)."""
        ends = []
        for side, col in ((I.SIDE_W, 0), (I.SIDE_E, -1)):
            bc = self.c.bc[side]
            _, U, V, _ = self.prim(self.W[:, :, col])
            r, lam = torch.full_like(U, bc.rho), torch.full_like(U, 1 / bc.T)
            gh = self.g(r, U, V, lam)
            Wg = torch.stack((r, r * U, r * V, r * (0.5 * (U * U + V * V) + (self.K + 2) / (4 * lam))))
            ends.append((gh[:, None], gh[:, None] * (self.K / 2 * bc.T), Wg[:, :, None]))
        wide = [torch.cat((ends[0][k], a, ends[1][k]), dim=d)
                for k, (a, d) in enumerate(((self.h, 1), (self.b, 1), (self.W, 2)))]
        return [torch.cat((a.narrow(d, 0, 1), a, a.narrow(d, a.shape[d] - 1, 1)), dim=d)
                for a, d in zip(wide, (0, 0, 1))]

    @staticmethod
    def limited(a, d):
        """van Leer limited slope times the cell width along dimension d; 0 on the outer cells."""
        s = a.diff(dim=d)
        n = s.shape[d]
        s1, s2 = s.narrow(d, 0, n - 1), s.narrow(d, 1, n - 1)
        p = s1 * s2
        r = torch.where(p > 0, 2 * p / (s1 + s2), torch.zeros((), dtype=a.dtype, device=a.device))
        out = torch.zeros_like(a)
        out.narrow(d, 1, n - 1).copy_(r)
        return out

    def moments(self, h, b, un, ut, weight):
        """sum weight (1, un, ut, (un^2 + ut^2)/2) h + (0, 0, 0, 1/2) b over the velocities."""
        m = torch.stack((weight, weight * un, weight * ut, weight * 0.5 * (un * un + ut * ut)), dim=1)
        r = h @ m
        r[..., 3] += b @ (0.5 * weight)
        return r.movedim(-1, 0)

    @staticmethod
    def gauss(U, lam, top):
        """<x^n> of the normalised Gaussian over x > 0, x < 0 and all x, n = 0 .. top."""
        e = torch.exp(-lam * U * U) / (2 * torch.sqrt(math.pi * lam))
        rl = torch.sqrt(lam)
        out = []
        for m0, m1 in ((0.5 * torch.erfc(-rl * U), e), (0.5 * torch.erfc(rl * U), -e),
                       (torch.ones_like(U), torch.zeros_like(U))):
            m = [m0, U * m0 + m1]
            for n in range(top - 1):
                m.append(U * m[-1] + (n + 1) / (2 * lam) * m[-2])
            out.append(m)
        return out

    def slope(self, U, V, lam, s):
        """a of <psi (a . psi)> = s for the normalised Maxwellian."""
        q = (self.K + 2) / (4 * lam)
        a4 = lam / q * (2 * s[3] - 2 * (U * s[1] + V * s[2]) + s[0] * (U * U + V * V - 2 * q))
        a3 = 2 * lam * (s[2] - V * s[0]) - V * a4
        a2 = 2 * lam * (s[1] - U * s[0]) - U * a4
        return s[0] - U * a2 - V * a3 - a4 * (0.5 * (U * U + V * V) + q), a2, a3, a4

    @staticmethod
    def psi(mu, mv, X, a, b):
        """<un^a ut^b psi_i>, i = 0 .. 3, of moments mu, mv and <xi^n> = X[n]."""
        m = lambda p, q, x=0: mu[a + p] * mv[b + q] * X[x]  # noqa: E731
        return m(0, 0), m(1, 0), m(0, 1), 0.5 * (m(2, 0) + m(0, 2) + m(0, 0, 2))

    def apsi(self, mu, mv, X, a, b, c):
        """<un^a ut^b psi_i (c . psi)>."""
        def t(p, q, x):
            m = lambda i, j, y: mu[a + p + i] * mv[b + q + j] * X[x + y]  # noqa: E731
            return (c[0] * m(0, 0, 0) + c[1] * m(1, 0, 0) + c[2] * m(0, 1, 0)
                    + 0.5 * c[3] * (m(2, 0, 0) + m(0, 2, 0) + m(0, 0, 2)))
        return t(0, 0, 0), t(1, 0, 0), t(0, 1, 0), 0.5 * (t(2, 0, 0) + t(0, 2, 0) + t(0, 0, 2))

    def weights(self, tau):
        dt, x = self.dt, self.dt / tau
        xs = torch.where(x < 0.1, x, torch.full_like(x, 0.1))
        c = [torch.zeros_like(x) for _ in range(5)]
        for n in range(16):
            f1, f2 = math.factorial(n + 1), math.factorial(n + 2)
            t = (-xs) ** n
            c[3] += t / f1
            c[4] += (n + 1) * t / f2
            if n:
                c[0] -= t / f1
                c[2] -= t / f2
                c[1] += n * t / f2
        e, c4 = torch.exp(-x), -torch.expm1(-x) / x
        c1, c5 = 1 - c4, (c4 - e) / x
        big = (c1, c5 - c1 / x, 0.5 - c1 / x, c4, c5)
        return [torch.where(x < 0.1, s, y) * k for s, y, k in zip(c, big, (dt, dt * dt, dt * dt, dt, dt * dt))]

    def face(self, un, ut, left, right, WL, WR, delta):
        """Fluxes through the faces between `left` and `right` (each h, b, their normal and their
        tangential slopes), in the face frame: of W, and of h and b at every velocity."""
        H = torch.where(un > 0, 1.0, torch.where(un < 0, 0.0, 0.5)).to(torch.float64)
        fh, fb = (H * (l + 0.5 * sl) + (1 - H) * (r - 0.5 * sr)
                  for l, sl, r, sr in zip(left[0:2], left[2:4], right[0:2], right[2:4]))
        th, tb = (H * l + (1 - H) * r for l, r in zip(left[4:6], right[4:6]))
        dh, db = (un * (H * l + (1 - H) * r) / delta[0] + ut * t / delta[1]
                  for l, r, t in zip(left[2:4], right[2:4], (th, tb)))
        W0 = self.moments(fh, fb, un, ut, self.w)
        St = self.moments(th, tb, un, ut, self.w) / delta[1]
        rho, U, V, lam = self.prim(W0)
        X2 = self.K / (2 * lam)
        X = {0: torch.ones_like(lam), 2: X2, 4: (self.K + 2) * X2 / (2 * lam)}
        pos, neg, full = self.gauss(U, lam, 7)
        mv = self.gauss(V, lam, 7)[2]
        Mt = self.weights(self.tau(rho, lam))
        k = rho * delta[0] / 2
        aL, aR = self.slope(U, V, lam, (W0 - WL) / k), self.slope(U, V, lam, (WR - W0) / k)
        bt = self.slope(U, V, lam, St / rho)
        A = self.slope(U, V, lam, [-(x + y + z) for x, y, z in zip(
            self.apsi(pos, mv, X, 1, 0, aL), self.apsi(neg, mv, X, 1, 0, aR), self.apsi(full, mv, X, 0, 1, bt))])
        F = [rho * (Mt[0] * p + Mt[1] * (x + y + z) + Mt[2] * t) for p, x, y, z, t in zip(
            self.psi(full, mv, X, 1, 0), self.apsi(pos, mv, X, 2, 0, aL), self.apsi(neg, mv, X, 2, 0, aR),
            self.apsi(full, mv, X, 1, 1, bt), self.apsi(full, mv, X, 1, 0, A))]
        shk = None
        if self.c.pr != 1.0:
            shk = self.shakhov(rho, U, V, lam, self.heat(fh, fb, un, ut, U, V))
            for i, e in enumerate(self.shakhov_flux(shk, full, mv, X, U, V, lam)):
                F[i] = F[i] + rho * Mt[0] * e
        wu = self.w * un
        F = torch.stack(F) + Mt[3] * self.moments(fh, fb, un, ut, wu) - Mt[4] * self.moments(dh, db, un, ut, wu)
        # micro flux: (the equilibrium's polynomial) g + Mt4 f_up - Mt5 (u . slope)
        col = lambda a: a[..., None]  # noqa: E731
        g = torch.exp(-col(lam) * ((un - col(U)) ** 2 + (ut - col(V)) ** 2)) * col(rho * lam / math.pi)
        r2 = 0.5 * (un * un + ut * ut)

        def poly(a, x, y):  # (a . psi) times 1 (x = 0) or xi^2, over the internal variable
            return (col(a[0] * X[x]) + col(a[1] * X[x]) * un + col(a[2] * X[x]) * ut + col(a[3] * X[x]) * r2
                    + col(0.5 * a[3] * X[y]))
        out = []
        for x, y, f, d in ((0, 2, fh, dh), (2, 4, fb, db)):
            P = torch.where(un > 0, poly(aL, x, y), poly(aR, x, y)) * un * col(Mt[1])
            P += poly(bt, x, y) * ut * col(Mt[1])
            P += poly(A, x, y) * col(Mt[2])
            P += col(Mt[0] * X[x])
            if shk is not None:
                P += col(Mt[0]) * self.shakhov_at(shk, un, ut, U, V, lam, x)
            out.append(un * (P * g + col(Mt[3]) * f - col(Mt[4]) * d))
        return F, out[0], out[1]

    # Shakhov model: g+ = g [1 + alpha (c . q) (2 lam (|c|^2 + xi^2) - (K + 4))]
    def heat(self, h, b, un, ut, U, V):
        def m(i, j, a):
            return a @ (self.w * un ** i * ut ** j)
        def c(i, j, a):  # sum w (un - U)^i (ut - V)^j a
            return sum(math.comb(i, p) * math.comb(j, q) * (-U) ** (i - p) * (-V) ** (j - q) * m(p, q, a)
                       for p in range(i + 1) for q in range(j + 1))
        return 0.5 * (c(3, 0, h) + c(1, 2, h) + c(1, 0, b)), 0.5 * (c(2, 1, h) + c(0, 3, h) + c(0, 1, b))

    def shakhov(self, rho, U, V, lam, q):
        al = (1 - self.c.pr) * 4 * lam * lam / ((self.K + 4) * rho)
        return al * q[0], al * q[1]

    def shakhov_at(self, s, un, ut, U, V, lam, x):
        """The factor over the internal variable: S of h (x = 0), or <xi^2 S> of b (x = 2)."""
        col = lambda a: a[..., None]  # noqa: E731
        cu, cv = un - col(U), ut - col(V)
        r = 2 * col(lam) * (cu * cu + cv * cv) - (4 if x == 0 else 2)
        return (col(s[0]) * cu + col(s[1]) * cv) * r * (1 if x == 0 else col(self.K / (2 * lam)))

    def shakhov_flux(self, s, mu, mv, X, U, V, lam):
        """<un psi_i S> over the normalised Maxwellian: S expanded in un^p ut^q xi^x."""
        terms = {}
        lin = (((1, 0), s[0]), ((0, 1), s[1]), ((0, 0), -(s[0] * U + s[1] * V)))
        quad = (((2, 0, 0), 2 * lam), ((1, 0, 0), -4 * lam * U), ((0, 2, 0), 2 * lam), ((0, 1, 0), -4 * lam * V),
                ((0, 0, 2), 2 * lam), ((0, 0, 0), 2 * lam * (U * U + V * V) - (self.K + 4)))
        for (p, q), x in lin:
            for (i, j, y), z in quad:
                terms[p + i, q + j, y] = terms.get((p + i, q + j, y), 0) + x * z
        def t(a, b, x):
            return sum(z * mu[p + a + 1] * mv[q + b] * X[y + x] for (p, q, y), z in terms.items())
        return t(0, 0, 0), t(1, 0, 0), t(0, 1, 0), 0.5 * (t(2, 0, 0) + t(0, 2, 0) + t(0, 0, 2))

    def wall(self, side, h, b, sh, sb, F, fh, fb):
        """Replaces the fluxes of a y wall's faces: what arrives is the gas, what leaves is the
        wall's Maxwellian with no net mass flux, first order in time."""
        bc = self.c.bc[side]
        south = side == I.SIDE_S
        arrives = self.v < 0 if south else self.v > 0
        leaves = self.v > 0 if south else self.v < 0
        sg = -0.5 if south else 0.5
        one = torch.ones(1, dtype=torch.float64, device=self.dev)
        gw = self.g(one, one * bc.U, 0 * one, one / bc.T)[0] * leaves
        ih, ib = (h + sg * sh) * arrives, (b + sg * sb) * arrives
        rw = -(ih @ (self.w * self.v)) / (gw @ (self.w * self.v))
        ih, ib = ih + rw[:, None] * gw, ib + rw[:, None] * gw * (self.K / 2 * bc.T)
        F.copy_(self.dt * self.moments(ih, ib, self.v, self.u, self.w * self.v))
        fh.copy_(self.dt * self.v * ih)
        fb.copy_(self.dt * self.v * ib)

    def step(self):
        h, b, W = self.ghosts()
        hx, bx, hy, by = self.limited(h, 1), self.limited(b, 1), self.limited(h, 0), self.limited(b, 0)
        for a in (hx, bx, hy, by):  # a pressure end's ghost has no slopes
            a[:, 0] = 0
            a[:, -1] = 0
        xs = (h, b, hx, bx, hy, by)
        F, fh, fb = self.face(self.u, self.v, [a[1:-1, :-1] for a in xs], [a[1:-1, 1:] for a in xs],
                              W[:, 1:-1, :-1], W[:, 1:-1, 1:], (self.dx, self.dy))
        dW = (F[:, :, :-1] - F[:, :, 1:]) / self.dx
        dh, db = (fh[:, :-1] - fh[:, 1:]) / self.dx, (fb[:, :-1] - fb[:, 1:]) / self.dx
        ys, sw = (h, b, hy, by, hx, bx), [0, 2, 1, 3]
        F, fh, fb = self.face(self.v, self.u, [a[:-1, 1:-1] for a in ys], [a[1:, 1:-1] for a in ys],
                              W[sw][:, :-1, 1:-1], W[sw][:, 1:, 1:-1], (self.dy, self.dx))
        for side, edge, row in ((I.SIDE_S, 0, 1), (I.SIDE_N, -1, -2)):
            self.wall(side, h[row, 1:-1], b[row, 1:-1], hy[row, 1:-1], by[row, 1:-1], F[:, edge], fh[edge], fb[edge])
        dW += (F[:, :-1] - F[:, 1:])[sw] / self.dy
        dh += (fh[:-1] - fh[1:]) / self.dy
        db += (fb[:-1] - fb[1:]) / self.dy
        new = self.W + dW
        q = self.heat(self.h, self.b, self.u, self.v, *self.prim(self.W)[1:3]) if self.c.pr != 1.0 else None
        tn, t1 = (self.tau(p[0], p[3]) for p in (self.prim(self.W), self.prim(new)))
        for Wk, t in ((self.W, tn), (new, t1)):
            rho, U, V, lam = self.prim(Wk)
            gh = self.g(rho, U, V, lam)
            gb = gh * (self.K / (2 * lam))[..., None]
            if q is not None:
                s = self.shakhov(rho, U, V, lam, q)
                gb = gb + gh * self.shakhov_at(s, self.u, self.v, U, V, lam, 2)
                gh = gh + gh * self.shakhov_at(s, self.u, self.v, U, V, lam, 0)
            dh += gh.mul_((self.dt / 2 / t)[..., None])
            db += gb.mul_((self.dt / 2 / t)[..., None])
        keep, inv = (1 - self.dt / 2 / tn)[..., None], (1 / (1 + self.dt / 2 / t1))[..., None]
        self.h = (self.h * keep + dh) * inv
        self.b = (self.b * keep + db) * inv
        self.W = new
