"""The library's performance cases: the work its users have it do, from a 64 x 64 sheet to a 256^3
quench, through the public entry points of ``paper_1402_2920_gb300``.

``listed()`` names the cases, ``draw(rng)`` makes more of the same ranges, ``prepare`` builds the
simulation and its seeded inputs, ``run`` is one pass, ``work`` the bytes and operations a pass
cannot do without, and ``exact`` the same pass in plain torch FP64 (the method's steps S1 to S12
written out with rolls, no kernel of the library).

Kinds of pass
  run      a simulation in progress: advance ``steps`` time steps and read rho and u on the device
           (with ``monitor`` also the conservation sums, as a long run does between outputs)
  quench   a whole short simulation: initial condition, ``steps`` steps, rho and u
  restart  FP64 populations in, ``steps`` steps, FP64 populations out (coupling and restarts)
  serve    a batch of host requests of mixed lattices and sizes through ``lbm_serve``

The library hands every field out as FP64.  A simulation whose storage and arithmetic are 32 or 16
bits wide has no more than FP32 in it, and such a program keeps what it reads as FP32, so those
outputs are FP32 here; the FP64 storage's stay FP64.
"""
import math

import numpy as np
import torch

import paper_1402_2920_gb300 as P
from paper_1402_2920_gb300 import workloads as W

D2, D3 = P.LBM_D2Q21, P.LBM_D3Q59
STORAGE = {"f32": P.LBM_STORE_F32, "f32_dev": P.LBM_STORE_F32_DEV, "f16_dev": P.LBM_STORE_F16_DEV,
           "bf16_dev": P.LBM_STORE_BF16_DEV, "f64": P.LBM_STORE_F64, "f32_loc": P.LBM_STORE_F32_LOC,
           "f16_loc": P.LBM_STORE_F16_LOC, "bf16_loc": P.LBM_STORE_BF16_LOC}
POP_BYTES = {"f32": 4, "f32_dev": 4, "f32_loc": 4, "f16_dev": 2, "bf16_dev": 2, "f16_loc": 2, "bf16_loc": 2, "f64": 8}

#: largest site-steps for which exact() stays within its time
EXACT_SITE_STEPS = 40e6


def _case(name, kind, dims, start, storage="f32_dev", gamma=0.0, solver="fast", warm=0, steps=4, monitor=False):
    nx, ny, nz = tuple(dims) + (1,) * (3 - len(dims))
    return {"name": name, "kind": kind, "nx": nx, "ny": ny, "nz": nz, "start": start, "storage": storage,
            "gamma": gamma, "solver": solver, "warm": warm, "steps": steps, "monitor": monitor}


def listed():
    return [
        # the smallest simulation of the repository's workloads: a 64^2 slab, latency and launches only
        _case("slab2d_64", "run", (64, 64), "slab", warm=24, steps=10),
        # the ordinary two-dimensional run: a 512^2 disc
        _case("droplet2d_512", "run", (512, 512), "droplet", warm=8, steps=10),
        # odd sides and the library's own default parameters (plain sweeps, n_i stored as float),
        # with a relaxation that reads the populations back in the collision
        _case("ragged2d_333x217", "run", (333, 217), "droplet", storage="f32", gamma=0.2, solver="plain", warm=4, steps=6),
        # the smallest three-dimensional request of the serving stream
        _case("droplet3d_32", "run", (32, 32, 32), "droplet", warm=8, steps=8),
        # the ordinary three-dimensional run, with its conservation sums watched
        _case("droplet3d_128_monitored", "run", (128, 128, 128), "droplet", warm=4, steps=8, monitor=True),
        # odd sides in three dimensions: rows that are no multiple of 16 bytes
        _case("ragged3d_117x91x83", "run", (117, 91, 83), "droplet", warm=4, steps=4),
        # the benchmark's quench from noise, end to end: initial condition, the transient with its many
        # u-solve sweeps, fields out
        _case("quench3d_256", "quench", (256, 256, 256), "spinodal", steps=10),
        # a large simulation well past its transient: about one sweep per step
        _case("spinodal3d_288x192x224_late", "run", (288, 192, 224), "spinodal", warm=60, steps=8),
        # half-precision populations relative to the sender's equilibrium
        _case("half3d_128", "run", (128, 128, 128), "droplet", storage="f16_loc", warm=0, steps=2),
        # the FP64 path, used as the reference of the others, with the paper's plain iteration
        _case("double3d_48", "run", (48, 48, 48), "droplet", storage="f64", solver="plain", warm=1, steps=2),
        # a state handed in and out as FP64 populations
        _case("restart3d_96", "restart", (96, 96, 96), "droplet", steps=2),
        # the serving stream in small: six requests of both lattices at once
        _case("serve_mixed", "serve", (512, 512, 96), "droplet", steps=100),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["run2", "run2", "run3", "run3", "run3", "quench", "restart", "serve"])
    storage = rng.choice(["f32_dev"] * 5 + ["f32", "f16_dev", "bf16_dev", "f32_loc", "f16_loc", "bf16_loc", "f64"])
    gamma = rng.choice([0.0, 0.0, 0.0, round(rng.uniform(-0.25, 0.25), 3)])
    solver = rng.choice(["fast", "fast", "fast", "plain"])
    start = rng.choice(["droplet", "droplet", "spinodal"])
    steps = rng.randint(2, 10)
    if POP_BYTES[storage] == 2:
        steps = 2
    if kind == "run2":
        dims = (_log_int(rng, 32, 512), _log_int(rng, 32, 512))
        if rng.random() < 0.3:
            start = "slab"
        return _unnamed("run", dims, start, storage, gamma, solver, 2 if POP_BYTES[storage] > 2 else 0, steps,
                        rng.random() < 0.3)
    if kind == "serve":
        return _unnamed("serve", (rng.randrange(64, 513, 32), rng.randrange(64, 513, 32), rng.randrange(32, 97, 16)),
                        "droplet", "f32_dev", 0.0, "fast", 0, _log_int(rng, 40, 150), False)
    cap = {"f64": 5e5}.get(storage, 2e6 if kind == "restart" else 12e6)
    while True:
        dims = tuple(_log_int(rng, 12, 288) for _ in range(3))
        if rng.random() < 0.4:  # sides that are multiples of 16, as the workloads' are
            dims = tuple(max(16, 16 * round(n / 16)) for n in dims)
        if dims[0] * dims[1] * dims[2] <= cap:
            break
    if kind == "quench":
        return _unnamed("quench", dims, "spinodal", storage, gamma, solver, 0, steps, False)
    if kind == "restart":
        return _unnamed("restart", dims, start, storage, gamma, solver, 0, min(steps, 4), False)
    return _unnamed("run", dims, start, storage, gamma, solver, 2 if POP_BYTES[storage] > 2 else 0, steps,
                    rng.random() < 0.3)


def _unnamed(kind, dims, start, storage, gamma, solver, warm, steps, monitor):
    c = _case("", kind, dims, start, storage, gamma, solver, warm, steps, monitor)
    del c["name"]
    return c


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _lattice(case):
    return D2 if case["nz"] == 1 else D3


def _fluid(lattice, width=4.0):
    """The workloads' van der Waals fluid in lattice units, and kappa for an interface of that width."""
    prm = W.vdw_lattice_params(W.TR_2D if lattice == D2 else W.TR_3D, lattice)
    return prm, W.kappa_for_width(prm, width)


def _width(dims):
    return 4.0 if min(dims) >= 64 else 2.0


def _fields(dims, start, seed, flow, device="cuda"):
    """rho [z][y][x] and u [d][z][y][x] of one start, FP64, from the seed alone.

    slab and droplet: the coexisting phases of the fluid with a tanh interface, placed and sized by
    the seed, in a divergence-free shear flow with a drift; spinodal: the critical density with 1 %
    white noise (in the quench at rest, otherwise in the same flow)."""
    d = len(dims)
    lattice = D2 if d == 2 else D3
    prm, _ = _fluid(lattice)
    g = torch.Generator(device=device)
    g.manual_seed(int(seed))
    r = np.random.default_rng(int(seed))
    shape = tuple(reversed(dims))
    axes = []  # coordinate of axis a, broadcastable to the field
    for a, n in enumerate(dims):
        view = [1] * d
        view[d - 1 - a] = n
        axes.append(torch.arange(n, dtype=torch.float64, device=device).reshape(view))
    mid, half = 0.5 * (prm.rho_l + prm.rho_g), 0.5 * (prm.rho_l - prm.rho_g)
    centre = [n * (0.5 + 0.1 * r.uniform(-1, 1)) for n in dims]
    if start == "slab":
        rho = mid + half * torch.tanh((0.25 * dims[0] - (axes[0] - centre[0]).abs()) / 2.0)
        rho = rho.expand(shape).contiguous()
    elif start == "droplet":
        radius = min(dims) * r.uniform(0.15, 0.35)
        r2 = sum((x - c) ** 2 for x, c in zip(axes, centre))
        rho = mid + half * torch.tanh((radius - torch.sqrt(r2)) / _width(dims))
    else:
        rho = 1.0 + 0.01 * (2.0 * torch.rand(shape, dtype=torch.float64, device=device, generator=g) - 1.0)
    u = None
    if flow:
        u = torch.empty((d,) + shape, dtype=torch.float64, device=device)
        for a in range(d):
            b = (a + 1) % d  # the flow along a varies along the next axis: no divergence
            u[a] = 0.01 * r.uniform(0.5, 1.0) + 0.02 * torch.sin(2.0 * math.pi * axes[b] / dims[b] + r.uniform(0, 6.28))
    return rho, u


def _dims(case):
    return (case["nx"], case["ny"]) if case["nz"] == 1 else (case["nx"], case["ny"], case["nz"])


def _params(case, lattice, kappa, prm):
    kw = {}
    if case["solver"] == "fast":  # the benchmark's and the serving loop's settings of the implicit solve
        kw = {"usolve_omega": 0.0, "usolve_chebyshev": 1, "usolve_warm_start": 2}
    return P.make_params(gamma=case["gamma"], kappa=kappa, rho0=1.0, storage=STORAGE[case["storage"]],
                         rho_check_min=0.98 * prm.rho_g, rho_check_max=1.02 * prm.rho_l, **kw)


def _serve_requests(case, seed):
    """Six requests of the serving stream's kind: (dims, steps) of 2D and 3D droplets in a flow."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    sides = [(nx, nx), (nz, nz, nz), (64, 64), (32, 32, 32), (ny, 64), (nz, 32, 48)]
    steps = [case["steps"], max(1, case["steps"] // 2), case["steps"], case["steps"], case["steps"] // 2 + 7,
             case["steps"] // 2 + 3]
    return [(dims, n, seed * 16 + k) for k, (dims, n) in enumerate(zip(sides, steps))]


def prepare(case, seed):
    if case["kind"] == "serve":
        reqs = []
        for dims, steps, s in _serve_requests(case, seed):
            lattice = D2 if len(dims) == 2 else D3
            prm, kappa = _fluid(lattice, _width(dims))
            rho, u = _fields(dims, "droplet", s, True)
            rho, u = rho.cpu().numpy().reshape(-1), u.cpu().numpy().reshape(-1)
            reqs.append({"lattice": lattice, "dims": dims, "eos": P.make_eos(P.LBM_EOS_VDW, a=prm.a, b=prm.b, T=prm.T),
                         "params": _params(case, lattice, kappa, prm), "steps": steps, "arrival_s": 0.0,
                         "rho_init": rho, "u_init": u, "rho_out": np.empty_like(rho), "u_out": np.empty_like(u)})
        return {"case": case, "requests": reqs}
    dims, lattice = _dims(case), _lattice(case)
    prm, kappa = _fluid(lattice, _width(dims))
    sim = P.Sim(lattice, dims, P.make_eos(P.LBM_EOS_VDW, a=prm.a, b=prm.b, T=prm.T), _params(case, lattice, kappa, prm),
                torch.cuda.current_stream().cuda_stream)
    rho, u = _fields(dims, case["start"], seed, case["kind"] != "quench")
    st = {"case": case, "sim": sim}
    if case["kind"] == "restart":
        pops = _equilibrium(_Method(dims, case["gamma"], prm, kappa, rho.device), rho, u).reshape(sim.Q, -1)
        st.update(pops_in=pops, pops_out=torch.empty_like(pops))
        return st
    st.update(rho=torch.empty_like(rho), u=torch.empty((len(dims),) + tuple(rho.shape), dtype=torch.float64, device="cuda"))
    if case["kind"] == "quench":
        st["start"] = rho
        return st
    sim.init(rho, u)
    if case["warm"]:
        sim.step(case["warm"])
    sim.sync()
    return st


def _out(case, x):
    return x if case["storage"] == "f64" else x.float()


def run(state):
    case = state["case"]
    if case["kind"] == "serve":
        P.lbm_serve(state["requests"])
        return [{"rho": r["rho_out"].astype(np.float32), "u": r["u_out"].astype(np.float32)} for r in state["requests"]]
    sim = state["sim"]
    if case["kind"] == "restart":
        P.lbm_set_populations(sim.handle, state["pops_in"], sim.Q * sim.N)
        sim.step(case["steps"])
        P.lbm_populations(sim.handle, state["pops_out"], sim.Q * sim.N)
        return _out(case, state["pops_out"])
    if case["kind"] == "quench":
        sim.init(state["start"])
    sim.step(case["steps"])
    out = {}
    if case["monitor"]:
        st = sim.stats()
        out = {"mass": st.mass, "mom": [st.mom[k] for k in range(sim.d)]}
    P.lbm_fields(sim.handle, state["rho"], state["u"], sim.N, sim.d)
    out.update(rho=_out(case, state["rho"]), u=_out(case, state["u"]))
    return out


def work(case):
    """Every population read once and written once per step, the inputs and outputs once each.  The
    operations: about 30 per population for the collision and its share of the tensors it needs."""
    if case["kind"] == "serve":
        b = f = 0.0
        for dims, steps, _ in _serve_requests(case, 0):
            n, q, d = float(np.prod(dims)), (21 if len(dims) == 2 else 59), len(dims)
            b += n * (2.0 * q * 4 * steps + 2 * 8 * (1 + d))
            f += n * 30.0 * q * steps
        return {"bytes": b, "flops": f}
    dims = _dims(case)
    n, q, d = float(np.prod(dims)), (21 if len(dims) == 2 else 59), len(dims)
    b = n * 2.0 * q * POP_BYTES[case["storage"]] * case["steps"]
    if case["kind"] == "restart":
        b += 2 * 8 * q * n
    else:
        b += 8 * (1 + d) * n
        if case["kind"] == "quench":
            b += 8 * n
    return {"bytes": b, "flops": n * 30.0 * q * case["steps"]}


# ---------------------------------------------------------------------------
# The method in plain torch FP64
# ---------------------------------------------------------------------------
_WEIGHTS = {  # by |c|^2, the coefficients of c_s^2 to the powers 0..3 (Tables I and II)
    2: {0: (1, -21 / 8, 105 / 32, -45 / 32), 1: (0, 32 / 45, -4 / 3, 2 / 3), 2: (0, 0, 1 / 3, -1 / 4),
        4: (0, -1 / 18, 3 / 16, -1 / 12), 8: (0, 0, -1 / 192, 1 / 64), 16: (0, 1 / 1440, -1 / 384, 1 / 384)},
    3: {0: (1, -259 / 80, 273 / 64, -121 / 64), 1: (0, 16 / 45, -2 / 3, 1 / 3), 2: (0, 8 / 45, -1 / 3, 1 / 6),
        3: (0, -4 / 45, 1 / 3, -5 / 24), 4: (0, -1 / 20, 17 / 96, -3 / 32), 8: (0, -1 / 360, 1 / 192, 1 / 192),
        12: (0, 1 / 720, -1 / 192, 1 / 192), 16: (0, 1 / 1440, -1 / 384, 1 / 384)}}


class _Method:
    def __init__(self, dims, gamma, prm, kappa, device):
        self.d = len(dims)
        self.dims, self.gamma, self.kappa = dims, gamma, kappa
        self.a, self.b, self.T, self.rho0 = prm.a, prm.b, prm.T, 1.0
        # the library's velocity order (its population layout)
        self.c = [tuple(int(x) for x in v) for v in P.lbm_velocities(D2 if self.d == 2 else D3)[:, :self.d]]
        self.cs0 = float(self.p(torch.tensor(self.rho0, dtype=torch.float64))) / self.rho0

    def p(self, r):
        return r * self.T / (1 - self.b * r) - self.a * r * r

    def weight(self, c, s):
        k = _WEIGHTS[self.d][sum(x * x for x in c)]
        return k[0] + s * (k[1] + s * (k[2] + s * k[3]))

    def shift(self, g, off):
        """g(r + off)"""
        ax = [a for a in range(self.d) if off[a]]
        return torch.roll(g, [-off[a] for a in ax], [self.d - 1 - a for a in ax]) if ax else g

    def at(self, g, *pairs):
        off = [0] * self.d
        for a, n in pairs:
            off[a] += n
        return self.shift(g, off)

    def d1(self, g, a):  # Sec. IV.B
        return (2 / 3) * (self.at(g, (a, 1)) - self.at(g, (a, -1))) - (1 / 12) * (self.at(g, (a, 2)) - self.at(g, (a, -2)))

    def force(self, rho):  # Secs. IV.E and VI
        out = []
        for a in range(self.d):
            t = (-2.0 if self.d == 2 else -3.0) * (self.at(rho, (a, 1)) - self.at(rho, (a, -1)))
            t = t + 0.5 * (self.at(rho, (a, 2)) - self.at(rho, (a, -2)))
            for b in range(self.d):
                if b != a:
                    for s in (1, -1):
                        t = t + 0.5 * (self.at(rho, (a, 1), (b, s)) - self.at(rho, (a, -1), (b, s)))
            out.append(self.kappa * rho * t)
        return out

    def jacobi(self, rho, p, pm, j0, jt):
        """S3 to S5: the next j~ from the current one."""
        d = self.d
        u = [(j0[a] + jt[a]) / rho for a in range(d)]
        du = [[self.d1(u[b], a) for b in range(d)] for a in range(d)]
        div = pm * sum(du[a][a] for a in range(d))
        new = [0.0] * d
        for a in range(d):
            for b in range(a, d):
                q = p * (du[a][b] + du[b][a])
                if a == b:
                    q = q + div
                new[a] = new[a] + self.d1(q, b)
                if b != a:
                    new[b] = new[b] + self.d1(q, a)
        return [-x / 12 for x in new]

    def solve(self, rho, p, dp, j0, jt):
        """S3 to S8: the fixed point, by Chebyshev iteration on the spectrum [0, g] (Sec. IX)."""
        pm = p - rho * dp
        cs2 = p / rho
        g = min(0.95, 1.05 * self.d * 1.8831 / 12 * float(torch.maximum(3 * cs2 - dp, cs2).max()))
        sigma, delta = (1 - 0.5 * g) / (0.5 * g), 0.5 * g
        rn, step = 1 / sigma, None
        for _ in range(200):
            new = self.jacobi(rho, p, pm, j0, jt)
            res = [x - y for x, y in zip(new, jt)]
            worst = max(float(x.abs().max()) for x in res)
            if worst <= 2e-14:
                return new
            if step is None:
                step = [x / (1 - 0.5 * g) for x in res]
            else:
                nx = 1 / (2 * sigma - rn)
                step = [nx * rn * s + 2 * nx / delta * x for s, x in zip(step, res)]
                rn = nx
            jt = [x + s for x, s in zip(jt, step)]
        raise RuntimeError("the implicit solve did not converge")

    def moments(self, n):
        rho = n.sum(0)
        j = [sum(c[a] * n[i] for i, c in enumerate(self.c) if c[a]) for a in range(self.d)]
        return rho, j

    def to_u(self, n, jt):
        rho, j = self.moments(n)
        f = self.force(rho)
        j0 = [x + 0.5 * y for x, y in zip(j, f)]
        p = self.p(rho)
        dp = self.T / (1 - self.b * rho) ** 2 - 2 * self.a * rho
        jt = self.solve(rho, p, dp, j0, jt)
        return rho, p, dp, f, jt, [(x + y) / rho for x, y in zip(j0, jt)]

    def step(self, n, jt):
        d, g, c0 = self.d, self.gamma, self.cs0
        rho, p, dp, f, jt, u = self.to_u(n, jt)
        pm = p - rho * dp
        rpp = rho * (2 * self.b * self.T / (1 - self.b * rho) ** 3 - 2 * self.a)
        R = range(d)
        du = [[self.d1(u[b], a) for b in R] for a in R]
        divu = sum(du[a][a] for a in R)
        divj = sum(self.d1(rho * u[a], a) for a in R)
        A = pm * divu
        C = [self.d1(p, b) / rho + sum(u[e] * du[e][b] for e in R) for b in R]
        dA = [self.d1(A, a) for a in R]
        dC = [[self.d1(C[b], a) for b in R] for a in R]
        trdC = sum(dC[a][a] for a in R)
        divB = [sum(self.d1(p * (du[a][e] + du[e][a]), e) for e in R) for a in R]
        k1 = -0.25 * (g + 1) ** 2 / (g - 1)
        k2 = (g * g + 4 * g + 1) / (g - 1) / 6
        k3 = (g * g + 4 * g + 1) / (g + 1) / 3
        Sig = {}
        for a in R:
            for b in range(a, d):
                t = -dp * divj * (du[a][b] + du[b][a]) - p * (dC[a][b] + dC[b][a])
                if a == b:
                    t = t - pm * trdC + rpp * divu * divj
                Sig[a, b] = k1 * (u[a] * (dA[b] + divB[b]) + u[b] * (dA[a] + divB[a])) + k2 * t
        del dA, dC, divB, A, C
        dpr = [self.d1(p / rho, c) for c in R]

        def X(a, b, c):
            t = self.d1(p * u[a] * u[b], c)
            return t + p * dpr[c] + pm * u[c] * divu if a == b else t

        Xi = {}
        for a in R:
            for b in range(a, d):
                for c in range(b, d):
                    t = k3 * (X(a, b, c) + X(a, c, b) + X(b, c, a))
                    for lone, pair in ((c, (a, b)), (b, (a, c)), (a, (b, c))):
                        if pair[0] == pair[1]:
                            t = t + (1 - g) * c0 * jt[lone]
                    Xi[a, b, c] = t
        trS = sum(Sig[a, a] for a in R)
        trX = [sum(Xi[tuple(sorted((a, a, b)))] for a in R) for b in R]
        cs2 = p / rho
        uu = sum(x * x for x in u)
        out = torch.empty_like(n)
        for i, c in enumerate(self.c):
            nz = [a for a in R if c[a]]
            cu = sum((c[a] * u[a] for a in nz), torch.zeros_like(rho))
            star = g * n[i] + (1 - g) * self.weight(c, cs2) * rho * (1 + cu / cs2 + cu * cu / (2 * cs2 * cs2) - uu / (2 * cs2))
            h2 = -c0 * trS
            lin = torch.zeros_like(rho)
            for a in nz:
                lin = lin + c[a] * (0.5 * (1 + g) / c0 * f[a] + (g - 1) / c0 * jt[a] - 3 * c0 / (6 * c0 ** 3) * trX[a])
                for b in nz:
                    h2 = h2 + c[a] * c[b] * Sig[min(a, b), max(a, b)]
                    for e in nz:
                        lin = lin + c[a] * c[b] * c[e] / (6 * c0 ** 3) * Xi[tuple(sorted((a, b, e)))]
            star = star + self.weight(c, c0) * (lin + h2 / (2 * c0 * c0))
            out[i] = self.shift(star, [-x for x in c])  # n_i(r + c_i) = n*_i(r)
        return out, jt


def _equilibrium(m, rho, u):
    s = m.p(rho) / rho
    uu = sum(x * x for x in u)
    n = torch.empty((len(m.c),) + tuple(rho.shape), dtype=torch.float64, device=rho.device)
    for i, c in enumerate(m.c):
        cu = sum((c[a] * u[a] for a in range(m.d) if c[a]), torch.zeros_like(rho))
        n[i] = m.weight(c, s) * rho * (1 + cu / s + cu * cu / (2 * s * s) - uu / (2 * s))
    return n


def _simulate(dims, gamma, start, flow, seed, steps, device="cuda"):
    """The method and its populations after `steps` steps."""
    prm, kappa = _fluid(D2 if len(dims) == 2 else D3, _width(dims))
    rho, u = _fields(dims, start, seed, flow, device)
    m = _Method(dims, gamma, prm, kappa, rho.device)
    if u is None:
        u = torch.zeros((len(dims),) + tuple(rho.shape), dtype=torch.float64, device=rho.device)
    n = _equilibrium(m, rho, u)
    jt = [torch.zeros_like(rho) for _ in dims]
    for _ in range(steps):
        n, jt = m.step(n, jt)
    return m, n, jt


def exact(case, seed):
    if case["kind"] == "serve":
        out, spent = [], 0.0
        for dims, steps, s in _serve_requests(case, seed):
            spent += 2.0 * steps * (20.0 if len(dims) == 3 else 8.0) + 59.0 * steps * float(np.prod(dims)) / 3e6
            if spent > 9000.0:  # milliseconds: the rest would take too long
                out.append(None)
                continue
            m, n, jt = _simulate(dims, 0.0, "droplet", True, s, steps)
            rho, _, _, _, _, u = m.to_u(n, jt)
            out.append({"rho": rho.reshape(-1), "u": torch.stack(u).reshape(-1)})
        return out
    dims = _dims(case)
    steps = case["warm"] + case["steps"]
    if float(np.prod(dims)) * steps > EXACT_SITE_STEPS or steps > 100:
        return None
    m, n, jt = _simulate(dims, case["gamma"], case["start"], case["kind"] != "quench", seed, steps)
    if case["kind"] == "restart":
        return n.reshape(len(m.c), -1)
    out = {}
    rho, _, _, _, _, u = m.to_u(n, jt)
    if case["monitor"]:
        mass, mom = m.moments(n)
        out = {"mass": float(mass.sum()), "mom": [float(x.sum()) for x in mom]}
    out.update(rho=rho, u=torch.stack(u))
    return out
