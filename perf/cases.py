"""The work a user of this framework has it do, as measured cases.

A forward case is one logging interval of a lock-exchange run: a number of
time steps and one diagnostics pass, the loop of paper_2112_08479_gb300/run.py.
Its outputs are the diagnostics record and the populations, which live in the
workspace that the caller owns (rows of the fluid, then rows of the scalar, in
the storage type; after an even number of steps slot i of a node holds the
streamed population i).  A "macros" case is single steps with the macroscopic
fields read after each, as an interactive or coupled user does.  A "gradient"
case is one value and gradient of an objective through the discrete adjoint.

State at the start of a case: a developed gravity current made from the seed
(near-equilibrium populations of a smooth velocity field of the buoyancy
velocity's size with a shear, a wavy interface, and small non-equilibrium
parts), so that the collisions see the values of a run under way.
"""
import math

import numpy as np
import torch

from paper_2112_08479_gb300 import lbm
from paper_2112_08479_gb300.objective import friction_objective, front_objective

U_B = 0.03


def listed():
    return [
        # one step and a look at the fields, on the 128 x 8 x 16 parity box:
        # the smallest calls, where latency and launches count
        _c("macros_tiny", "macros", "bgk", "fp32", "q7", 128, 8, 16, 1, 1000.0),
        # a logging interval of the same box: launch-bound stepping
        _c("run_tiny", "run", "bgk", "fp32", "q7", 128, 8, 16, 100, 1000.0),
        # odd and ragged sizes (no even row length): one node per thread
        _c("run_ragged_bgk", "run", "bgk", "fp32", "q7", 333, 47, 59, 50, 5000.0),
        # the same for the 16-bit storage of the cumulant model
        _c("run_ragged_cumulant_bf16", "run", "cumulant", "bf16s", "q7", 509, 37, 61, 20, 5000.0),
        # the 1024 x 64 x 128 cumulant run at Re 5000
        _c("run_cumulant", "run", "cumulant", "fp32", "q7", 1024, 64, 128, 100, 5000.0),
        # the 67 M-node box: the headline run, FP32 BGK with Smagorinsky
        _c("run_large_bgk", "run", "bgk", "fp32", "q7", 2048, 128, 256, 100, 30000.0),
        # the same box with FP16 storage
        _c("run_large_bgk_fp16", "run", "bgk", "fp16s", "q7", 2048, 128, 256, 20, 30000.0),
        # the storage study: the cumulant model with FP16 storage
        _c("run_large_cumulant_fp16", "run", "cumulant", "fp16s", "q7", 2048, 128, 256, 20, 30000.0),
        # the paper's periodic array of currents (2500 x 150 x 100) with its
        # D3Q6 scalar
        _c("run_periodic_q6", "run", "bgk", "fp32", "q6", 2500, 150, 100, 50, 895.0, periodic=True),
        # the paper's walled box (1500 x 100 x 100) with its D3Q27 scalar
        _c("run_fcm", "run", "cumulant", "fp32", "q27", 1500, 100, 100, 50, 5000.0),
        # gradients on the 256 x 32 x 64 differentiation box: friction with
        # the BGK fluid, front position with the cumulant fluid
        _c("gradient_friction_bgk", "gradient", "bgk", "fp32", "q7", 256, 32, 64, 100, 2000.0,
           K=50, objective="friction"),
        _c("gradient_front_cumulant", "gradient", "cumulant", "fp32", "q7", 256, 32, 64, 60,
           2000.0, K=20, objective="front"),
    ]


def _c(name, kind, model, storage, scalar, nx, ny, nz, steps, Re, periodic=False, K=0,
       objective=""):
    return dict(name=name, kind=kind, model=model, storage=storage, scalar=scalar, nx=nx, ny=ny,
                nz=nz, steps=steps, Re=Re, periodic=periodic, K=K, objective=objective)


def draw(rng):
    """Another case of the same ranges: boxes from 32 x 4 x 8 to 67 M nodes,
    any model, scalar lattice and storage, walled or periodic ends (the larger
    models up to the sizes that cost what the 67 M-node BGK run costs)."""
    kind = rng.choice(["run"] * 7 + ["macros"] + ["gradient"] * 2)
    model, scalar = rng.choice([("bgk", "q7"), ("bgk", "q7"), ("bgk", "q6"), ("cumulant", "q7"),
                                ("cumulant", "q7"), ("cumulant", "q27")])
    storage = rng.choice(["fp32", "fp32", "fp16s", "bf16s"])
    periodic = rng.random() < 0.3
    top = 2.0 ** 26
    if kind == "gradient":
        scalar, storage, top = "q7", "fp32", 2.0 ** 19.5
    elif scalar == "q27":
        top = 2.0 ** 24
    elif model == "cumulant":
        top = 2.0 ** 25.3
    n = math.exp(rng.uniform(math.log(1024.0), math.log(top)))
    # aspect ratios of the lock-exchange boxes: long in x, thinner in y than z
    ny = max(3, round((n / 128.0) ** (1.0 / 3.0) * 2.0 * rng.uniform(0.6, 1.5)))
    nz = max(4, round(ny * rng.uniform(0.7, 2.2)))
    nx = max(2 * nz, round(n / (ny * nz)))
    while nx * ny * nz > top:
        nx -= max(1, nx // 50)
    if rng.random() < 0.6:   # most users take round sizes
        nx = max(32, nx // 32 * 32)
        ny, nz = max(4, ny // 4 * 4), max(4, nz // 4 * 4)
    # lattice viscosities of the repository's boxes: 2.6e-4 (Re 30000 at 256
    # nodes of depth) to 3.4e-3 (Re 895 at 100)
    nu = math.exp(rng.uniform(math.log(2.5e-4), math.log(3.5e-3)))
    Re = float(round(U_B * nz / nu))
    steps = rng.choice([2, 10, 20, 50, 100])
    K, objective = 0, ""
    if kind == "macros":
        steps = 1
    if kind == "gradient":
        steps = rng.choice([20, 40, 60])
        K, objective = rng.choice([10, 20]), rng.choice(["friction", "front"])
    return {k: v for k, v in _c("", kind, model, storage, scalar, nx, ny, nz, steps, Re, periodic,
                                K, objective).items() if k != "name"}


# --- inputs -------------------------------------------------------------------

def _params(case):
    nz = case["nz"]
    return lbm.lock_exchange(case["nx"], case["ny"], nz, H=nz, x0=min(nz, case["nx"] // 2),
                             u_b=U_B, Re=case["Re"], model=case["model"],
                             storage=case["storage"], scalar=case["scalar"],
                             geometry="periodic" if case["periodic"] else "walls")


# velocity sets in the documented orders (include/lbm.h)
_C27 = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1),
        (1, 1, 0), (-1, -1, 0), (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1),
        (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1), (1, 1, 1), (-1, -1, -1),
        (1, 1, -1), (-1, -1, 1), (1, -1, 1), (-1, 1, -1), (-1, 1, 1), (1, -1, -1)]


def _opp(i):
    return 0 if i == 0 else (i + 1 if i % 2 else i - 1)


def _lattice(case):
    """[(c, w)] of the fluid and of the scalar; c_s^2 of the scalar."""
    if case["model"] == "bgk":
        w = [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12
        fluid = list(zip(_C27[:19], w))
    else:
        w = [8 / 27] + [2 / 27] * 6 + [1 / 54] * 12 + [1 / 216] * 8
        fluid = list(zip(_C27, w))
    if case["scalar"] == "q7":
        return fluid, list(zip(_C27[:7], [1 / 4] + [1 / 8] * 6)), 1 / 4
    if case["scalar"] == "q6":
        return fluid, list(zip(_C27[1:7], [1 / 6] * 6)), 1 / 3
    w = [8 / 27] + [2 / 27] * 6 + [1 / 54] * 12 + [1 / 216] * 8
    return fluid, list(zip(_C27, w)), 1 / 3


def _axes(case, dev):
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    x = ((torch.arange(nx, device=dev) + 0.5) / nx).view(1, 1, nx)
    y = ((torch.arange(ny, device=dev) + 0.5) / ny).view(1, ny, 1)
    z = ((torch.arange(nz, device=dev) + 0.5) / nz).view(nz, 1, 1)
    return x, y, z


def _chi0(case, seed, dev):
    """A lock (or wavy front) with noise: 1 behind the interface, 0 ahead."""
    r = np.random.default_rng(seed)
    g = torch.Generator(device=dev)
    g.manual_seed(int(seed))
    x, y, z = _axes(case, dev)
    a, p, q = r.uniform(0.02, 0.06), r.uniform(0, 2 * np.pi), r.uniform(0, 2 * np.pi)
    # gradients start at the lock gate, an interface of about one node
    sharp = 2.0 * case["nx"] if case["kind"] == "gradient" else 25.0
    front = r.uniform(0.35, 0.55) + a * torch.sin(2 * np.pi * y + p) + 0.1 * torch.cos(np.pi * z) \
        + 0.02 * torch.sin(6 * np.pi * z + q)
    chi = 0.5 - 0.5 * torch.tanh((x - front) * sharp)
    shape = (case["nz"], case["ny"], case["nx"])
    chi = chi + 1e-3 * (2 * torch.rand(shape, generator=g, device=dev) - 1)
    return chi.clamp_(0.0, 1.0), g


def _state0(case, seed, dev):
    """The canonical state [Q + NS, nz, ny, nx] (f - w, Phi - w), FP32."""
    fluid, scal, cs2 = _lattice(case)
    chi, g = _chi0(case, seed, dev)
    r = np.random.default_rng(seed + 1)
    x, y, z = _axes(case, dev)
    ph = r.uniform(0, 2 * np.pi, 6)
    ux = U_B * (0.3 + 0.4 * torch.cos(np.pi * z) * torch.sin(np.pi * x)
                + 0.2 * torch.sin(4 * np.pi * x + ph[0]) * torch.cos(2 * np.pi * y + ph[1]))
    uy = 0.2 * U_B * torch.sin(2 * np.pi * y + ph[2]) * torch.cos(2 * np.pi * z) + 0 * x
    uz = 0.3 * U_B * torch.sin(np.pi * z) * torch.cos(4 * np.pi * x + ph[3]) \
        * (1 + 0.5 * torch.sin(2 * np.pi * y + ph[4]))
    d = 1e-3 * (0.4 + 0.5 * torch.cos(2 * np.pi * x + ph[5]) * torch.cos(np.pi * z)) + 0 * y
    us = ux * ux + uy * uy + uz * uz
    s = torch.empty((len(fluid) + len(scal),) + tuple(chi.shape), device=dev)

    def along(c):
        return c[0] * ux + c[1] * uy + c[2] * uz

    for i, (c, w) in enumerate(fluid):
        cu = along(c)
        s[i] = w * (d + (1 + d) * (3 * cu + 4.5 * cu * cu - 1.5 * us))
        s[i] += w * 1e-3 * (torch.rand(chi.shape, generator=g, device=dev) - 0.5)
    for k, (c, w) in enumerate(scal):
        s[len(fluid) + k] = w * (chi - 1 + chi * along(c) / cs2)
        s[len(fluid) + k] += w * 1e-3 * chi * (torch.rand(chi.shape, generator=g, device=dev) - 0.5)
    return s


def prepare(case, seed):
    p = _params(case)
    if case["kind"] == "gradient":
        chi, _ = _chi0(case, seed, "cuda")
        return dict(case=case, params=p, chi=chi.reshape(-1),
                    cs=torch.tensor(0.17, dtype=torch.float32, device="cuda"))
    lat = lbm.Lattice(p, device="cuda")
    lat.set_state(_state0(case, seed, "cuda"))
    return dict(case=case, params=p, lat=lat)


# --- one pass -------------------------------------------------------------------

def _rows(lat):
    """The populations in the workspace: fluid rows, scalar rows and, with
    16-bit storage, the scalar's FP32 rest row."""
    p, N = lat.params, lat.N
    t = {lbm.LBM_FP32: torch.float32, lbm.LBM_FP16S: torch.float16,
         lbm.LBM_BF16S: torch.bfloat16}[p.storage]
    es = 4 if t == torch.float32 else 2
    rest = es == 2 and p.scalar != lbm.LBM_SCALAR_Q6
    w = lat.workspace

    def rows(off, n, dt, size):
        return w[off:off + n * N * size].view(dt).view(n, N)

    off = -(-p.Q * N * es // 256) * 256
    out = {"fluid": rows(0, p.Q, t, es)}
    phi = rows(off, p.NS, t, es)
    out["scalar"] = phi[1:] if rest else phi
    if rest:
        out["rest"] = rows(off + -(-p.NS * N * es // 256) * 256, 1, torch.float32, 4)
    return out


def run(state):
    case = state["case"]
    if case["kind"] == "gradient":
        chi = state["chi"].detach().requires_grad_(True)
        cs = state["cs"].detach().requires_grad_(True)
        obj = friction_objective if case["objective"] == "friction" else front_objective
        J = obj(chi, cs, state["params"], case["steps"], K=case["K"])
        J.backward()
        return {"J": J.item(), "chi0": chi.grad, "cs": cs.grad}
    lat = state["lat"]
    lat.step(case["steps"])
    if case["kind"] == "macros":
        rho, u, chi = lat.macros()
        return {"rho": rho, "u": u, "chi": chi}
    d = lat.diag()
    out = _rows(lat)
    out["diag"] = np.array([d["front"], d["Fw"], d["mass_delta"], d["scalar_mass"]], np.float32)
    return out


# --- what one pass cannot do without ---------------------------------------------

def work(case):
    """Bytes: the state read and written once over the pass (a run keeps it
    in place), the fields or gradients written.  Flops: the collisions'
    arithmetic of every step (counted once per node update)."""
    N = case["nx"] * case["ny"] * case["nz"]
    fluid, scal, _ = _lattice(case)
    rows = len(fluid) + len(scal)
    per = {"bgk": 330, "cumulant": 420}[case["model"]] + (260 if case["scalar"] == "q27" else 40)
    if case["kind"] == "gradient":
        # forward, recompute and adjoint of every step; chi0 in, gradient out
        return {"bytes": 8.0 * N, "flops": 4.0 * per * N * case["steps"]}
    es = 4 if case["storage"] == "fp32" else 2
    bytes_ = 2.0 * rows * es * N
    if es == 2 and case["scalar"] != "q6":
        bytes_ += 4.0 * N
    if case["kind"] == "macros":
        bytes_ += 20.0 * N
    return {"bytes": bytes_, "flops": float(per) * N * case["steps"]}


# --- the same pass in 64 bits -------------------------------------------------------

class _Exact:
    """The model of include/lbm.h in float64 on torch tensors
    [rows, nz, ny, nx]: f - w and Phi - w."""

    def __init__(self, case, p, cs=None):
        self.case, self.p = case, p
        self.fluid, self.scal, self.cs2 = _lattice(case)
        self.Q, self.NS = len(self.fluid), len(self.scal)
        self.cs = p.cs_smag if cs is None else cs
        self.px = case["periodic"]
        self.F = [p.gprime * e for e in p.eg]

    def moments(self, f, phi):
        j = [0.0, 0.0, 0.0]
        m = {}
        for i, (c, _) in enumerate(self.fluid):
            for a in range(3):
                if c[a]:
                    j[a] = j[a] + c[a] * f[i]
                for b in range(a, 3):
                    if c[a] * c[b]:
                        m[a, b] = m.get((a, b), 0.0) + c[a] * c[b] * f[i]
        return f.sum(0), j, m, phi.sum(0)

    def collide(self, f, phi):
        p = self.p
        d, j, m, chit = self.moments(f, phi)
        rho, chi = 1 + d, 1 + chit
        F = [g * chi for g in self.F]
        u = [(j[a] + 0.5 * F[a]) / rho for a in range(3)]
        if self.case["model"] == "bgk":
            fo, tau = self._bgk(f, d, rho, u, F, m)
            taup = 0.5 + (p.D + (tau - (3 * p.nu + 0.5)) / 3 / p.sc_t) / self.cs2
        else:
            fo = self._cumulant(d, rho, j, F, m)
            taup = 0.5 + p.D / self.cs2
        if self.case["scalar"] == "q27":
            po = self._fcm(phi, chi, u)
        else:
            po = []
            for k, (c, w) in enumerate(self.scal):
                eq = w * (chit + chi * (c[0] * u[0] + c[1] * u[1] + c[2] * u[2]) / self.cs2)
                po.append(phi[k] - (phi[k] - eq) / taup)
            po = torch.stack(po)
        return fo, po

    def _bgk(self, f, d, rho, u, F, m):
        pi = {}
        for a in range(3):
            for b in range(a, 3):
                pi[a, b] = m[a, b] - (d / 3 if a == b else 0.0) - rho * u[a] * u[b]
        q2 = sum((1 if a == b else 2) * v * v for (a, b), v in pi.items())
        pos = q2 > 0
        q = torch.where(pos, torch.sqrt(torch.where(pos, q2, torch.ones_like(q2))),
                        torch.zeros_like(q2))
        t0 = 3 * self.p.nu + 0.5
        tau = 0.5 * (t0 + torch.sqrt(t0 * t0 + 18 * math.sqrt(2.0) * self.cs ** 2 * q / rho))
        us = u[0] * u[0] + u[1] * u[1] + u[2] * u[2]
        uF = u[0] * F[0] + u[1] * F[1] + u[2] * F[2]
        out = []
        for i, (c, w) in enumerate(self.fluid):
            cu = c[0] * u[0] + c[1] * u[1] + c[2] * u[2]
            cF = c[0] * F[0] + c[1] * F[1] + c[2] * F[2]
            eq = w * (d + rho * (3 * cu + 4.5 * cu * cu - 1.5 * us))
            S = (1 - 0.5 / tau) * w * (3 * cF - 3 * uF + 9 * cu * cF)
            out.append(f[i] - (f[i] - eq) / tau + S)
        return torch.stack(out), tau

    @staticmethod
    def _inverse(k, v):
        """Populations at c = -1, 0, 1 of the central moments k about v."""
        lead = (v * v * k[0] + 2 * v * k[1] + k[2])
        odd = v * k[0] + k[1]
        return [0.5 * (lead - odd), k[0] - lead, 0.5 * (lead + odd)]

    def _cumulant(self, d, rho, j, F, m):
        p = self.p
        v = [j[a] / rho for a in range(3)]
        c2 = {ab: (m[ab] - (d / 3 if ab[0] == ab[1] else 0.0)) / rho - v[ab[0]] * v[ab[1]]
              for ab in m}
        r1, r2 = 1 - 1 / (3 * p.nu + 0.5), 1 - p.omega_bulk
        tr = c2[0, 0] + c2[1, 1] + c2[2, 2]
        S = {ab: r1 * c2[ab] for ab in ((0, 1), (0, 2), (1, 2))}
        for a in range(3):
            S[a, a] = 1 / 3 + r1 * (c2[a, a] - tr / 3) + r2 * tr / 3
        xx, yy, zz, xy, xz, yz = (S[k] for k in ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2)))
        one, zero = torch.ones_like(d), torch.zeros_like(d)
        K = {(0, 0, 0): one, (2, 0, 0): xx, (0, 2, 0): yy, (0, 0, 2): zz, (1, 1, 0): xy,
             (1, 0, 1): xz, (0, 1, 1): yz, (2, 2, 0): xx * yy + 2 * xy * xy,
             (2, 0, 2): xx * zz + 2 * xz * xz, (0, 2, 2): yy * zz + 2 * yz * yz,
             (2, 1, 1): xx * yz + 2 * xy * xz, (1, 2, 1): yy * xz + 2 * xy * yz,
             (1, 1, 2): zz * xy + 2 * xz * yz,
             (2, 2, 2): xx * yy * zz + 2 * (xx * yz * yz + yy * xz * xz + zz * xy * xy)
             + 8 * xy * xz * yz}
        un = [(j[a] + F[a]) / rho for a in range(3)]
        T = {}
        for a in range(3):
            for b in range(3):
                line = self._inverse([K.get((a, b, c), zero) for c in range(3)], un[2])
                for c in range(3):
                    T[a, b, c] = line[c]
        for a in range(3):
            for c in range(3):
                line = self._inverse([T[a, b, c] for b in range(3)], un[1])
                for b in range(3):
                    T[a, b, c] = line[b]
        for b in range(3):
            for c in range(3):
                line = self._inverse([T[a, b, c] for a in range(3)], un[0])
                for a in range(3):
                    T[a, b, c] = line[a]
        return torch.stack([rho * T[c[0] + 1, c[1] + 1, c[2] + 1] - w for c, w in self.fluid])

    def _fcm(self, phi, chi, u):
        r1 = 1 - 1 / (3 * self.p.D + 0.5)
        one, zero = torch.ones_like(chi), torch.zeros_like(chi)
        v = []
        for a in range(3):
            jp = sum(c[a] * phi[k] for k, (c, _) in enumerate(self.scal) if c[a])
            v.append(r1 * (jp - chi * u[a]))
        E = [self._inverse([one, zero, one / 3], u[a]) for a in range(3)]
        G = [self._inverse([zero, one, zero], u[a]) for a in range(3)]
        out = []
        for c, w in self.scal:
            e = [E[a][c[a] + 1] for a in range(3)]
            g = [G[a][c[a] + 1] for a in range(3)]
            out.append(chi * e[0] * e[1] * e[2] + v[0] * g[0] * e[1] * e[2]
                       + v[1] * e[0] * g[1] * e[2] + v[2] * e[0] * e[1] * g[2] - w)
        return torch.stack(out)

    def stream(self, post, dirs, d0):
        """Pull along each direction, half-way bounce-back at the walls."""
        out = []
        for k, (c, _) in enumerate(dirs):
            t = torch.roll(post[k], shifts=(c[2], c[1], c[0]), dims=(0, 1, 2))
            back = post[_opp(k + d0) - d0] if c != (0, 0, 0) else None
            if c[0] and not self.px:
                e = 0 if c[0] > 0 else t.shape[2] - 1
                t[:, :, e] = back[:, :, e]
            if c[2]:
                e = 0 if c[2] > 0 else t.shape[0] - 1
                t[e] = back[e]
            out.append(t)
        return torch.stack(out)

    def step(self, f, phi):
        f, phi = self.collide(f, phi)
        return (self.stream(f, self.fluid, 0),
                self.stream(phi, self.scal, 1 if self.case["scalar"] == "q6" else 0))

    def step_large(self, f, phi, chunk):
        """The same in slices of z that bound the memory; f, phi are replaced."""
        nz = f.shape[1]
        for a in range(0, nz, chunk):
            f[:, a:a + chunk], phi[:, a:a + chunk] = self.collide(f[:, a:a + chunk],
                                                                  phi[:, a:a + chunk])
        for s, dirs, d0 in ((f, self.fluid, 0),
                            (phi, self.scal, 1 if self.case["scalar"] == "q6" else 0)):
            # opposite directions need each other's rows at the walls
            k = 1 - d0 if d0 == 0 else 0
            while k < len(dirs):
                s[k:k + 2] = self.stream(s[k:k + 2], dirs[k:k + 2], 1)
                k += 2
        return f, phi

    def macros(self, f, phi):
        d, j, _, chit = self.moments(f, phi)
        u = [(j[a] + 0.5 * self.F[a] * (1 + chit)) / (1 + d) for a in range(3)]
        return d, u, chit

    def friction(self, f, phi):
        u0 = self.macros(f[:, 0], phi[:, 0])[1][0]
        u1 = self.macros(f[:, 1], phi[:, 1])[1][0]
        return self.p.nu * (9 * u0 - u1).sum() / 3

    def front(self, phi):
        p = self.p
        m = (1 + phi.sum(0)).mean(1).amax(0)
        lim = max(1, (p.nx + p.x0) // 2) if self.px else p.nx
        hit = torch.nonzero(m[:lim] >= p.front_threshold)
        if not len(hit):
            return torch.full((), (-0.5 - p.x0) / p.H, dtype=torch.float64, device=phi.device)
        x = int(hit[-1])
        xn = x + (m[x] - p.front_threshold) / (m[x] - m[x + 1]) if x < lim - 1 else m[x] * 0 + x
        return (xn + 0.5 - p.x0) / p.H


def exact(case, seed):
    N = case["nx"] * case["ny"] * case["nz"]
    if N * case["steps"] > 6e8 * (4 if case["kind"] == "run" else 1):
        return None   # over 20 s
    p, dev = _params(case), "cuda"
    if case["kind"] == "gradient":
        return _exact_gradient(case, p, seed)
    ex = _Exact(case, p)
    s = _state0(case, seed, dev).double()
    f, phi = s[:ex.Q], s[ex.Q:]
    chunk = max(1, min(case["nz"], 2 ** 21 // (case["nx"] * case["ny"])))
    for _ in range(case["steps"]):
        f, phi = ex.step_large(f, phi, chunk)
    if case["kind"] == "macros":
        d, u, chit = ex.macros(f, phi)
        return {"rho": 1 + d, "u": torch.stack(u), "chi": 1 + chit}
    diag = np.array([float(ex.front(phi)), float(ex.friction(f, phi)),
                     float(sum(r.sum() for r in f)), N + float(sum(r.sum() for r in phi))])
    if case["storage"] == "fp32":
        return {"fluid": f.view(ex.Q, -1), "scalar": phi.view(ex.NS, -1), "diag": diag}
    f *= p.scale_f
    phi *= p.scale_phi
    out = {"fluid": f.view(ex.Q, -1), "scalar": phi.view(ex.NS, -1), "diag": diag}
    if case["scalar"] != "q6":
        out["rest"], out["scalar"] = out["scalar"][:1], out["scalar"][1:]
    return out


def _exact_gradient(case, p, seed):
    dev = "cuda"
    cs = torch.tensor(0.17, dtype=torch.float32).double().to(dev).requires_grad_(True)
    ex = _Exact(case, p, cs)
    chi = _chi0(case, seed, dev)[0].double()
    w = torch.tensor([w for _, w in ex.scal], dtype=torch.float64, device=dev).view(-1, 1, 1, 1)
    f = torch.zeros((ex.Q,) + tuple(chi.shape), dtype=torch.float64, device=dev)
    states = [(f, w * (chi - 1))]
    friction = case["objective"] == "friction"
    J = 0.0
    with torch.no_grad():
        for _ in range(case["steps"]):
            states.append(ex.step(*states[-1]))
            if friction:
                J += float(ex.friction(*states[-1]))
        if not friction:
            J = float(ex.front(states[-1][1]))
    lf, lp = (torch.zeros_like(t) for t in states[-1])
    gcs = 0.0
    for n in range(case["steps"], -1, -1):
        f, phi = (t.detach().requires_grad_(True) for t in states.pop())
        if n == case["steps"]:
            obj = ex.friction(f, phi) if friction else ex.front(phi)
        else:
            fo, po = ex.step(f, phi)
            obj = (fo * lf).sum() + (po * lp).sum()
            if friction and n >= 1:
                obj = obj + ex.friction(f, phi)
        g = torch.autograd.grad(obj, (f, phi, cs), allow_unused=True)
        lf, lp = (torch.zeros_like(t) if v is None else v for v, t in zip(g, (f, phi)))
        if g[2] is not None:
            gcs += float(g[2])
    return {"J": J, "chi0": (w * lp).sum(0).reshape(-1),
            "cs": torch.tensor(gcs, dtype=torch.float64)}
