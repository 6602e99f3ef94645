"""What the framework is timed on: whole calls of a user's program through the
public entry points, over the range of lattices, precisions and options that
the paper's experiments, the tests and the benchmark of this repository run.

A case is one simulation program in small: upload the initial order-parameter
field, advance it a number of steps (reading observables on the way where such
a program does), and read the fields back.  The float64 runs return the
library's float64 arrays; the float32 runs hand the fields to a torch program
on the GPU in float32, the type they were computed in.
"""
import math

import numpy as np
import torch
import torch.utils.checkpoint

from paper_1907_13415_gb300 import nlc
from paper_1907_13415_gb300.autograd import droplet_loss

S_COEX = 1.0 / 3.0
BASE = dict(A0=0.1, K=0.02, Gamma=0.3, xi=0.7, tau=1.0, rho0=1.0)
#: the paper's own set (Sec. 2)
PAPER = dict(A0=0.1, K=0.04, Gamma=0.34, xi=0.7, tau=1.5, rho0=1.0)
PRECISION = {"fp64": nlc.NLC_FP64, "fp32": nlc.NLC_FP32, "mixed": nlc.NLC_FP32_QF64}
LOG = ("mass", "mom_x", "mom_y", "mom_z", "s_area", "radius", "x_iface", "max_u",
       "free_energy", "u_l2")


def _run(lattice, shape, precision, steps, *, geometry="ball", size=0.0, params="base",
         gamma=2.7, noise=1e-4, every=0, profile=False, graph=0, tune=False,
         collision="bgk", stencil="standard", populations=False, **name):
    """populations: read the populations back (the state to go on from, or
    to take moments of) instead of rho and u"""
    nz, ny, nx = shape
    return dict(name, kind="run", lattice=lattice, nx=nx, ny=ny, nz=nz, precision=precision,
                steps=steps, geometry=geometry, size=float(size), params=params, gamma=gamma,
                noise=noise, every=every, profile=bool(profile and every), graph=graph, tune=tune,
                collision=collision, stencil=stencil, populations=populations)


def listed():
    return [
        # the flat-interface experiment: a tiny float64 lattice (the default
        # precision), observables with the S(x) profile on the way; all
        # latency
        _run("d2q9", (1, 8, 128), "fp64", 400, geometry="slab", noise=1e-6, every=100,
             profile=True, graph=50, name="flat_128x8_fp64"),
        # the circular-droplet experiment in its two precisions, stepped in
        # replayed graphs
        _run("d2q9", (1, 256, 256), "fp32", 200, size=32, gamma=2.705, every=100, graph=50,
             name="disc_256_fp32"),
        _run("d2q9", (1, 256, 256), "fp64", 100, size=32, gamma=2.705, every=50, graph=50,
             name="disc_256_fp64"),
        # the paper's almost static circle with the isotropic stencils: its
        # own parameters, a lattice that no tile divides
        _run("d2q9", (1, 100, 100), "fp64", 200, size=25, params="paper", gamma=2.707681,
             noise=1e-5, every=100, graph=50, stencil="isotropic", name="circle_100_iso_fp64"),
        # a large planar lattice of odd extents, plain launches, the whole
        # state read back
        _run("d2q9", (1, 1501, 2035), "fp32", 150, size=400, gamma=2.705, tune=True,
             populations=True, name="plane_2035x1501_fp32"),
        # the temperature sweep: 64 uneven lattices advanced as one batch,
        # every member's observables and Q read at the end
        dict(name="sweep_64_fp32", kind="sweep", members=64, layout=2, steps=500, graph=50,
             precision="fp32"),
        # the spherical droplet, the largest workload of the benchmark
        _run("d3q19", (256, 256, 256), "fp32", 100, size=48, gamma=2.705, tune=True,
             name="sphere_256_fp32"),
        # a monitored run: observables with the profile every few steps, odd
        # extents
        _run("d3q19", (117, 131, 149), "fp32", 60, size=30, gamma=2.705, every=5, profile=True,
             name="sphere_monitored_fp32"),
        # the multiple-relaxation-time collision with the paper's parameters,
        # populations read back for the moments
        _run("d3q19", (128, 128, 128), "fp32", 100, size=32, params="paper", gamma=2.705,
             collision="mrt", populations=True, name="sphere_128_mrt_fp32"),
        # float64 in three dimensions
        _run("d3q19", (64, 64, 64), "fp64", 20, size=16, params="paper", gamma=2.705,
             name="sphere_64_fp64"),
        # float populations with float64 Q, odd extents
        _run("d3q19", (51, 67, 90), "mixed", 20, size=14, gamma=2.705,
             name="sphere_90x67x51_mixed"),
        # gradients of a droplet loss through the torch bridge
        dict(name="adjoint_128_fp32", kind="adjoint", nx=128, ny=128, steps=400, ckpt=100,
             size=24.0, target=20.0, params="base", gamma=2.7, precision="fp32"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["flat", "disc", "disc", "plane", "sweep", "sphere", "sphere", "sphere",
                       "adjoint"])
    params = rng.choice(["base", "paper"])
    gamma = rng.uniform(2.69, 2.72)
    if kind == "sweep":
        return dict(kind="sweep", members=rng.randint(8, 64), layout=rng.randrange(1 << 20),
                    steps=50 * rng.randint(2, 8), graph=50, precision="fp32")
    if kind == "adjoint":
        nx, ny = rng.randint(48, 160), rng.randint(48, 160)
        size = rng.uniform(0.15, 0.25) * min(nx, ny)
        return dict(kind="adjoint", nx=nx, ny=ny, steps=rng.randint(60, 300),
                    ckpt=rng.choice([25, 50, 100]), size=size, target=0.8 * size, params=params,
                    gamma=gamma, precision="fp32")
    if kind == "flat":
        precision = rng.choice(["fp64", "fp64", "fp32"])
        return _run("d2q9", (1, _log_int(rng, 4, 64), _log_int(rng, 64, 1024)),
                    precision, 50 * rng.randint(1, 4),
                    geometry="slab", params=params, gamma=gamma, noise=1e-5,
                    every=rng.choice([0, 50]), profile=rng.random() < 0.5,
                    graph=rng.choice([0, 50]), populations=precision == "fp32")
    if kind == "disc":
        precision = rng.choice(["fp64", "fp32"])
        nx, ny = (_log_int(rng, 48, 320 if precision == "fp64" else 900) for _ in range(2))
        collision = rng.choice(["bgk", "bgk", "mrt"])
        return _run("d2q9", (1, ny, nx), precision, 25 * rng.randint(2, 6),
                    size=rng.uniform(0.12, 0.3) * min(nx, ny), params=params, gamma=gamma,
                    every=rng.choice([0, 50]), graph=rng.choice([0, 50]),
                    collision=collision, stencil=rng.choice(["standard", "isotropic"]),
                    populations=precision == "fp32" and (collision == "mrt" or nx * ny > 90000))
    if kind == "plane":
        nx, ny = rng.randint(900, 2200), rng.randint(900, 1500)
        return _run("d2q9", (1, ny, nx), "fp32", rng.randint(40, 120),
                    size=rng.uniform(0.12, 0.3) * min(nx, ny), params=params, gamma=gamma,
                    tune=rng.random() < 0.5, populations=True)
    precision = rng.choice(["fp32", "fp32", "fp32", "fp64", "mixed"])
    hi = 200 if precision == "fp32" else 72
    shape = tuple(_log_int(rng, 20, hi) for _ in range(3))
    collision = rng.choice(["bgk", "bgk", "mrt"]) if precision == "fp32" else "bgk"
    return _run("d3q19", shape, precision,
                rng.randint(20, 60) if precision == "fp32" else rng.randint(5, 20),
                size=rng.uniform(0.15, 0.3) * min(shape), params=params, gamma=gamma,
                every=rng.choice([0, 10]) if precision == "fp32" else 0,
                profile=rng.random() < 0.5, tune=rng.random() < 0.3,
                collision=collision, stencil=rng.choice(["standard"] * 4 + ["isotropic"]),
                populations=collision == "mrt")


# -- inputs -------------------------------------------------------------------

def _params(case):
    return dict(BASE if case["params"] == "base" else PAPER, gamma=case["gamma"])


def _mrt_rates(lattice, tau):
    """Rates of the second-order (stress) moments 1/tau, 1.2 elsewhere."""
    r = np.full(9 if lattice == "d2q9" else 19, 1.2)
    r[[7, 8] if lattice == "d2q9" else [9, 11, 13, 14, 15]] = 1.0 / tau
    return r


def _initial_q(shape, geometry, size, noise, seed, three_d, dtype):
    """Q = S (n n - I/3) of a nematic slab or ball at a place and with a
    director of its own, in an isotropic background, plus uniform noise."""
    nz, ny, nx = shape
    gen = torch.Generator(device="cuda").manual_seed(seed)
    draw_ = torch.rand(6, generator=gen, device="cuda", dtype=torch.float64).tolist()
    if geometry == "slab":
        x = torch.arange(nx, device="cuda", dtype=torch.float64)
        split = nx // 2 + int(4 * draw_[0]) - 2
        S = torch.where(x < split, S_COEX, 0.0).expand(nz, ny, nx)
        n = (0.0, 1.0, 0.0)
    else:
        r2 = 0
        for k, m in enumerate((nz, ny, nx)):
            if m == 1:
                continue
            v = torch.arange(m, device="cuda", dtype=torch.float64)
            v = v - ((m - 1) / 2.0 + (draw_[k] - 0.5) * 0.1 * m)
            r2 = r2 + (v * v).reshape([-1 if j == k else 1 for j in range(3)])
        S = torch.where(r2 < (size * (0.9 + 0.2 * draw_[3])) ** 2, S_COEX, 0.0).expand(nz, ny, nx)
        t = 2 * math.pi * draw_[4]
        c = 2 * draw_[5] - 1 if three_d else 0.0
        s = math.sqrt(1 - c * c)
        n = (s * math.cos(t), s * math.sin(t), c)
    Q = torch.empty((5, nz, ny, nx), device="cuda", dtype=dtype)
    for k, (a, b) in enumerate(((0, 0), (0, 1), (0, 2), (1, 1), (1, 2))):
        xi = torch.rand((nz, ny, nx), generator=gen, device="cuda", dtype=torch.float32)
        Q[k] = S * (n[a] * n[b] - (1.0 / 3.0 if a == b else 0.0)) + noise * (2 * xi.double() - 1)
    return Q


def _sweep_members(case):
    """(shape, gamma) of each member: extents as a seeded draw, gamma evenly
    spaced over [2.60, 2.80]."""
    rng = np.random.Generator(np.random.PCG64(case["layout"]))
    n = case["members"]
    lx = rng.choice([256, 512, 1024, 2048], size=n)
    ly = rng.choice([8, 16, 64], size=n)
    return [((1, int(ly[i]), int(lx[i])), float(g))
            for i, g in enumerate(np.linspace(2.60, 2.80, n))]


def _shape(case):
    return (case.get("nz", 1), case["ny"], case["nx"])


def _q0(case, seed):
    dtype = torch.float32 if case["precision"] == "fp32" else torch.float64
    if case["kind"] == "sweep":
        return [_initial_q(sh, "slab", 0.0, 1e-6, 64 * seed + i, False, dtype)
                for i, (sh, _) in enumerate(_sweep_members(case))]
    if case["kind"] == "adjoint":
        return _initial_q(_shape(case), "ball", case["size"], 1e-6, seed, False, dtype)
    return _initial_q(_shape(case), case["geometry"], case["size"], case["noise"], seed,
                      case["lattice"] == "d3q19", dtype)


def _pinned(shape):
    """A page-locked float64 array for read-back (torch tensor, numpy view)."""
    t = torch.empty(shape, dtype=torch.float64, pin_memory=True)
    return t, t.numpy()


def prepare(case, seed):
    torch.cuda.set_device(0)
    stream = torch.cuda.current_stream().cuda_stream
    s = dict(case=case)
    Q0 = _q0(case, seed)
    if case["kind"] == "sweep":
        members = _sweep_members(case)
        s["sim"] = sim = nlc.Batch(nlc.NLC_D2Q9, [m[0] for m in members],
                                   [dict(BASE, gamma=m[1]) for m in members],
                                   precision=nlc.NLC_FP32, stream=stream,
                                   graph_steps=case["graph"])
        # one page-locked buffer each way, a view of it per member
        q0 = torch.cat([q.reshape(-1) for q in Q0])
        s["Q0_t"] = torch.empty(q0.shape, dtype=torch.float32, pin_memory=True)
        s["Q0_t"].copy_(q0)
        s["Q_t"], qv = _pinned(q0.shape)
        s["rho_t"], rv = _pinned((q0.numel() // 5,))
        s["Q0"], s["Q"], s["rho"], at = [], [], [], 0
        for m in members:
            n = int(np.prod(m[0]))
            s["Q0"].append(s["Q0_t"].numpy()[5 * at:5 * (at + n)].reshape((5,) + m[0]))
            s["Q"].append(qv[5 * at:5 * (at + n)])
            s["rho"].append(rv[at:at + n])
            at += n
        for i in range(len(members)):
            sim.set_fields_f32(i, s["Q0"][i])
        sim.autotune()
        return s
    p = _params(case)
    if case["kind"] == "adjoint":
        s["sim"] = nlc.Simulation(nlc.NLC_D2Q9, _shape(case), p, precision=nlc.NLC_FP32,
                                  stream=stream)
        s["Q0"] = Q0.requires_grad_()
        s["theta"] = torch.tensor([p["gamma"], p["K"], p["Gamma"]], dtype=torch.float32,
                                  device="cuda", requires_grad=True)
        s["params"] = p
        return s
    s["sim"] = sim = nlc.Simulation(nlc.NLC_D2Q9 if case["lattice"] == "d2q9" else nlc.NLC_D3Q19,
                                    _shape(case), p, precision=PRECISION[case["precision"]],
                                    stream=stream)
    if case["graph"]:
        sim.set_graph(case["graph"])
    if case["collision"] == "mrt":
        sim.set_mrt(_mrt_rates(case["lattice"], p["tau"]))
    if case["stencil"] == "isotropic":
        sim.set_stencil(nlc.NLC_STENCIL_ISOTROPIC)
    if case["precision"] == "fp32":
        s["Q0"] = Q0
    else:
        s["Q0_t"] = torch.empty(Q0.shape, dtype=torch.float64, pin_memory=True)
        s["Q0_t"].copy_(Q0)
        s["Q0"] = s["Q0_t"].numpy()
    sh = _shape(case)
    s["Q_t"], s["Q"] = _pinned((5,) + sh)
    if case["populations"]:
        s["f_t"], s["f"] = _pinned((9 if case["lattice"] == "d2q9" else 19,) + sh)
    else:
        s["rho_t"], s["rho"] = _pinned(sh)
        s["u_t"], s["u"] = _pinned((3,) + sh)
    if case["tune"]:
        _upload(s)
        sim.autotune()
    torch.cuda.synchronize()
    return s


# -- one pass -----------------------------------------------------------------

def _upload(s):
    if s["case"]["precision"] == "fp32":
        s["sim"].set_fields_f32(s["Q0"].data_ptr())
    else:
        s["sim"].set_fields(s["Q0"])


def _to_gpu32(t):
    return t.to("cuda", non_blocking=True).to(torch.float32)


def run(state):
    s = state
    case, sim = s["case"], s["sim"]
    if case["kind"] == "sweep":
        for i, q in enumerate(s["Q0"]):
            sim.set_fields_f32(i, q)
        sim.step(case["steps"])
        log = []
        for i in range(len(sim)):
            o = sim.observables(i)
            log.append([o[k] for k in LOG])
            nlc.nlc_get_fields(sim.ctx, i, s["Q"][i], s["rho"][i])
        return {"Q": _to_gpu32(s["Q_t"]), "rho": _to_gpu32(s["rho_t"]),
                "log": np.array(log, dtype=np.float32)}
    if case["kind"] == "adjoint":
        loss = droplet_loss(s["Q0"], s["theta"], sim, s["params"], case["steps"], case["ckpt"],
                            case["target"], 1.0, 1.0)
        dQ0, dtheta = torch.autograd.grad(loss, (s["Q0"], s["theta"]))
        return {"loss": loss.detach(), "dQ0": dQ0, "dtheta": dtheta}
    _upload(s)
    log, profiles, done = [], [], 0
    while done < case["steps"]:
        k = min(case["every"] or case["steps"], case["steps"] - done)
        sim.step(k)
        done += k
        if case["every"]:
            o = sim.observables(profile=case["profile"])
            log.append([o[key] for key in LOG])
            if case["profile"]:
                profiles.append(o["s_profile"])
    if case["populations"]:
        nlc.nlc_get_fields(sim.ctx, 0, s["Q"])
        nlc.nlc_get_populations(sim.ctx, 0, s["f"])
        flow = ("f",)
    else:
        nlc.nlc_get_fields(sim.ctx, 0, s["Q"], s["rho"], s["u"])
        flow = ("rho", "u")
    # mixed: Q is float64, the flow comes from populations in float32
    kind = np.float64 if case["precision"] == "fp64" else np.float32
    out = {"Q": _to_gpu32(s["Q_t"]) if case["precision"] == "fp32" else s["Q"]}
    for k in flow:
        out[k] = s[k] if case["precision"] == "fp64" else _to_gpu32(s[k + "_t"])
    if log:
        out["log"] = np.array(log, dtype=kind)
    if profiles:
        out["profiles"] = np.array(profiles, dtype=kind)
    return out


# -- what a pass cannot do without --------------------------------------------

def _words(precision):
    return {"fp64": (8, 8), "fp32": (4, 4), "mixed": (4, 8)}[precision]


def work(case):
    """Bytes: the populations and Q read and written once by every step, the
    initial field read and the results written once.  Operations: each
    quantity of a step once per cell (an FMA counts two)."""
    if case["kind"] == "sweep":
        cells = sum(int(np.prod(m[0])) for m in _sweep_members(case))
        lattice, out = "d2q9", 6
    else:
        cells = int(np.prod(_shape(case)))
        lattice, out = case.get("lattice", "d2q9"), 9
    q = 9 if lattice == "d2q9" else 19
    if case.get("populations"):
        out = 5 + q
    gw, qw = _words(case["precision"])
    flops = 820 if lattice == "d2q9" else 1400
    if case.get("collision") == "mrt":
        flops += 150 if lattice == "d2q9" else 500
    if case.get("stencil") == "isotropic":
        flops += 300 if lattice == "d2q9" else 900
    step_bytes = 2 * (q * gw + 5 * qw) * cells
    if case["kind"] == "adjoint":
        # forward, and a reverse sweep that costs about twice as much
        return {"bytes": 3.0 * step_bytes * case["steps"], "flops": 3.0 * flops * cells * case["steps"]}
    ends = 5 * qw * cells + out * (8 if case["precision"] == "fp64" else 4) * cells
    return {"bytes": float(step_bytes * case["steps"] + ends),
            "flops": float(flops * cells * case["steps"])}


# -- the same in 64 bits, in plain torch --------------------------------------

class _Ref:
    """The hybrid step in float64 (Sec. 1.1, 1.2): full 3 x 3 tensors, whole
    arrays, periodic shifts."""

    def __init__(self, lattice, collision="bgk", stencil="standard"):
        self.dim = 2 if lattice == "d2q9" else 3
        # the order of the library's populations: rest, the plane with
        # opposite pairs adjacent, then the layers above and below
        plane = [(1, 0), (-1, 0), (0, 1), (0, -1)]
        self.c = [(0, 0, 0)] + [(x, y, 0) for x, y in plane + [(1, 1), (-1, -1), (1, -1), (-1, 1)]]
        if self.dim == 3:
            for z in (1, -1):
                self.c += [(0, 0, z)] + [(x, y, z) for x, y in plane]
        by_speed = (4 / 9, 1 / 9, 1 / 36) if self.dim == 2 else (1 / 3, 1 / 18, 1 / 36)
        self.w = [by_speed[sum(k * k for k in c)] for c in self.c]
        self.iso = stencil == "isotropic"
        self.mrt = collision == "mrt"
        self.lattice = lattice

    @staticmethod
    def at(v, c):
        """v(x + c) for arrays [..., z, y, x]"""
        return torch.roll(v, (-c[2], -c[1], -c[0]), (-3, -2, -1))

    def grad(self, v):
        if self.iso:
            g = [0, 0, 0]
            for c, w in zip(self.c, self.w):
                if any(c):
                    vi = self.at(v, c)
                    for a in range(self.dim):
                        if c[a]:
                            g[a] = g[a] + (3 * w * c[a]) * vi
        else:
            g = [(self.at(v, e) - self.at(v, tuple(-k for k in e))) / 2
                 for e in ((1, 0, 0), (0, 1, 0), (0, 0, 1))[:self.dim]]
        return g[:self.dim]

    def lap(self, v):
        s = 0
        if self.iso:
            for c, w in zip(self.c, self.w):
                if any(c):
                    s = s + (6 * w) * (self.at(v, c) - v)
            return s
        for e in ((1, 0, 0), (0, 1, 0), (0, 0, 1))[:self.dim]:
            s = s + (self.at(v, e) - v) + (self.at(v, tuple(-k for k in e)) - v)
        return s

    @staticmethod
    def full(q):
        return [[q[0], q[1], q[2]], [q[1], q[3], q[4]], [q[2], q[4], -q[0] - q[3]]]

    @staticmethod
    def mul(A, B):
        return [[sum(A[a][g] * B[g][b] for g in range(3)) for b in range(3)] for a in range(3)]

    def field(self, q, lap, p):
        """H of Eq. 3"""
        Q, L = self.full(q), self.full(lap)
        QQ = self.mul(Q, Q)
        tr2 = QQ[0][0] + QQ[1][1] + QQ[2][2]
        ag = p["A0"] * p["gamma"]
        return [[(-p["A0"] * (1 - p["gamma"] / 3) - ag * tr2) * Q[a][b] + ag * QQ[a][b]
                 - (ag / 3 * tr2 if a == b else 0) + p["K"] * L[a][b] for b in range(3)]
                for a in range(3)]

    def force(self, q, p):
        """div of the stress of Eq. 5 without P0"""
        H, Q = self.field(q, self.lap(q), p), self.full(q)
        dQ = [self.full(g) for g in self.grad(q)]
        X = self.mul(Q, H)
        qh = X[0][0] + X[1][1] + X[2][2]
        xi, F = p["xi"], [0, 0, 0]
        for b in range(self.dim):
            for a in range(self.dim):
                qt = Q[a][b] + (1 / 3 if a == b else 0)
                el = sum(dQ[a][i][j] * dQ[b][i][j] for i in range(3) for j in range(3))
                P = (2 * xi * qt * qh - xi * (X[b][a] + X[a][b] + 2 / 3 * H[a][b])
                     - p["K"] * el + X[a][b] - X[b][a])
                F[a] = F[a] + self.grad(P)[b]
        return F

    def moments(self, g, F, p):
        rho = p["rho0"] + g.sum(0)
        u = []
        for a in range(self.dim):
            u.append((sum(c[a] * g[i] for i, c in enumerate(self.c) if c[a]) + F[a] / 2) / rho)
        return rho, u

    def collide(self, g, rho, u, F, p):
        dot = lambda c, v: sum(c[a] * v[a] for a in range(self.dim) if c[a])  # noqa: E731
        uu, uF = sum(v * v for v in u), sum(v * f for v, f in zip(u, F))
        drho, out, src = rho - p["rho0"], [], []
        for i, c in enumerate(self.c):
            cu, cF = (dot(c, u), dot(c, F)) if any(c) else (0.0, 0.0)
            geq = self.w[i] * (drho + rho * (3 * cu + 4.5 * cu * cu - 1.5 * uu))
            src.append(self.w[i] * (3 * (cF - uF) + 9 * cu * cF))
            if self.mrt:
                out.append(g[i] - geq + src[i] / 2)
            else:
                out.append(g[i] - (g[i] - geq) / p["tau"] + (1 - 1 / (2 * p["tau"])) * src[i])
        if self.mrt:
            y = torch.stack(out)
            A = torch.tensor(self.relaxation(p["tau"]), device=g.device)
            out = [g[i] + src[i] - sum(A[i, j] * y[j] for j in range(len(self.c)))
                   for i in range(len(self.c))]
        return torch.stack(out)

    def relaxation(self, tau):
        """M^-1 S M of the moment basis: Gram-Schmidt with unit weights from
        the polynomials in the order that the library's header lists."""
        x, y, z = (np.array([c[a] for c in self.c], dtype=np.float64) for a in range(3))
        c2 = x * x + y * y + z * z
        if self.lattice == "d2q9":
            poly = [1 + 0 * x, c2, c2 * c2, x, c2 * x, y, c2 * y, x * x - y * y, x * y]
        else:
            poly = [1 + 0 * x, c2, c2 * c2, x, c2 * x, y, c2 * y, z, c2 * z, 3 * x * x - c2,
                    (3 * x * x - c2) * c2, y * y - z * z, (y * y - z * z) * c2, x * y, y * z,
                    x * z, x * (y * y - z * z), y * (z * z - x * x), z * (x * x - y * y)]
        M = []
        for v in poly:
            for m in M:
                v = v - (v @ m) / (m @ m) * m
            M.append(v)
        rates = _mrt_rates(self.lattice, tau)
        return sum(r / (m @ m) * np.outer(m, m) for r, m in zip(rates, M))

    def rhs(self, q, u, G, p):
        """Eq. 1 without its trace; G[a][b] = d_b u_a"""
        Q, H = self.full(q), self.field(q, self.lap(q), p)
        dq, n = self.grad(q), self.dim
        z = torch.zeros_like(q[0])
        g = [[G[a][b] if a < n and b < n else z for b in range(3)] for a in range(3)]
        D = [[(g[a][b] + g[b][a]) / 2 for b in range(3)] for a in range(3)]
        W = [[(g[a][b] - g[b][a]) / 2 for b in range(3)] for a in range(3)]
        Qt = [[Q[a][b] + (1 / 3 if a == b else 0) for b in range(3)] for a in range(3)]
        xi = p["xi"]
        A = self.mul([[xi * D[a][b] + W[a][b] for b in range(3)] for a in range(3)], Qt)
        B = self.mul(Qt, [[xi * D[a][b] - W[a][b] for b in range(3)] for a in range(3)])
        qg = sum(Q[a][b] * g[b][a] for a in range(n) for b in range(n))
        S = [[A[a][b] + B[a][b] - 2 * xi * Qt[a][b] * qg for b in range(3)] for a in range(3)]
        R = [[S[a][b] + p["Gamma"] * H[a][b] for b in range(3)] for a in range(3)]
        tr = (R[0][0] + R[1][1] + R[2][2]) / 3
        adv = sum(u[a] * dq[a] for a in range(n))
        r = [R[0][0] - tr, R[0][1], R[0][2], R[1][1] - tr, R[1][2]]
        return torch.stack([r[k] - adv[k] for k in range(5)])

    def stream(self, g):
        return torch.stack([torch.roll(g[i], (c[2], c[1], c[0]), (-3, -2, -1))
                            for i, c in enumerate(self.c)])

    def populations(self, g, p):
        w = torch.tensor(self.w, device=g.device, dtype=g.dtype).reshape(-1, 1, 1, 1)
        return self.stream(g) + w * p["rho0"]

    def step(self, g, q, p):
        """g: post-collision deviations f_i - w_i rho0 at their own cells"""
        g = self.stream(g)
        F = self.force(q, p)
        rho, u = self.moments(g, F, p)
        g = self.collide(g, rho, u, F, p)
        G = [self.grad(v) for v in u]
        r1 = self.rhs(q, u, G, p)
        return g, q + (r1 + self.rhs(q + r1, u, G, p)) / 2

    def state(self, g, q, p):
        rho, u = self.moments(self.stream(g), self.force(q, p), p)
        return rho, torch.stack(u + [torch.zeros_like(rho)] * (3 - self.dim))

    @staticmethod
    def order(q):
        return torch.sqrt(1.5 * (q[0] ** 2 + q[3] ** 2 + (q[0] + q[3]) ** 2
                                 + 2 * (q[1] ** 2 + q[2] ** 2 + q[4] ** 2)))

    def observe(self, q, rho, u, p):
        """The columns of LOG and the y, z-mean of S"""
        S, Q = self.order(q), self.full(q)
        tr2 = S * S / 1.5
        tr3 = sum(a * b for a, b in zip(sum(self.mul(Q, Q), []), sum(Q, [])))
        ag = p["A0"] * p["gamma"]
        en = p["A0"] / 2 * (1 - p["gamma"] / 3) * tr2 - ag / 3 * tr3 + ag / 4 * tr2 * tr2
        for e in ((1, 0, 0), (0, 1, 0), (0, 0, 1))[:self.dim]:
            en = en + p["K"] / 2 * self.order(self.at(q, e) - q) ** 2 / 1.5
        area = float(S.sum()) / S_COEX
        prof = S.mean((0, 1)).cpu().numpy()
        nxt = np.roll(prof, -1)
        hit = np.nonzero((prof >= S_COEX / 2) & (nxt < S_COEX / 2))[0]
        x = -1.0 if not len(hit) else hit[0] + (prof[hit[0]] - S_COEX / 2) / (prof[hit[0]] - nxt[hit[0]])
        planar = q.shape[1] == 1
        radius = math.sqrt(area / math.pi) if planar else (3 * area / (4 * math.pi)) ** (1 / 3)
        m = [float((rho * v).sum()) for v in u]
        uu = (u * u).sum(0)
        return [float(rho.sum()), *m, area, radius, float(x), math.sqrt(float(uu.max())),
                float(en.sum()), math.sqrt(float(uu.sum()))], prof


def _exact_adjoint(case, seed):
    p0 = _params(case)
    q0 = _q0(case, seed).double().requires_grad_()
    theta = torch.tensor([p0["gamma"], p0["K"], p0["Gamma"]], dtype=torch.float32,
                         device="cuda").double().requires_grad_()
    ref = _Ref("d2q9")

    def segment(g, q, th, n):
        p = dict(p0, gamma=th[0], K=th[1], Gamma=th[2])
        for _ in range(n):
            g, q = ref.step(g, q, p)
        return g, q

    g, q, left = torch.zeros((9,) + tuple(q0.shape[1:]), device="cuda", dtype=torch.float64), q0, case["steps"]
    while left:
        n = min(20, left)
        g, q = torch.utils.checkpoint.checkpoint(segment, g, q, theta, n, use_reentrant=False)
        left -= n
    _, u = ref.state(g, q, dict(p0, gamma=theta[0], K=theta[1], Gamma=theta[2]))
    R = torch.sqrt(ref.order(q).sum() / S_COEX / math.pi)
    loss = (R - case["target"]) ** 2 + torch.sqrt((u * u).sum())
    dQ0, dtheta = torch.autograd.grad(loss, (q0, theta))
    return {"loss": loss.detach(), "dQ0": dQ0, "dtheta": dtheta}


def exact(case, seed):
    if case["kind"] == "adjoint":
        return _exact_adjoint(case, seed)
    if case["kind"] == "sweep":
        # members of one shape are stepped together
        members, q0 = _sweep_members(case), _q0(case, seed)
        ref = _Ref("d2q9")
        Q, rho, log = ([None] * len(members) for _ in range(3))
        for sh in sorted({m[0] for m in members}):
            ids = [i for i, m in enumerate(members) if m[0] == sh]
            q = torch.stack([q0[i].double() for i in ids], 1)      # [5, k, 1, ny, nx]
            p = dict(BASE, gamma=torch.tensor([members[i][1] for i in ids], device="cuda",
                                              dtype=torch.float64).reshape(-1, 1, 1, 1))
            g = torch.zeros((9,) + tuple(q.shape[1:]), device="cuda", dtype=torch.float64)
            for _ in range(case["steps"]):
                g, q = ref.step(g, q, p)
            for k, i in enumerate(ids):
                pi = dict(BASE, gamma=members[i][1])
                r, u = ref.state(g[:, k], q[:, k], pi)
                log[i] = ref.observe(q[:, k], r, u, pi)[0]
                Q[i], rho[i] = q[:, k].reshape(-1), r.reshape(-1)
        return {"Q": torch.cat(Q), "rho": torch.cat(rho), "log": np.array(log)}
    p, q = _params(case), _q0(case, seed).double()
    ref = _Ref(case["lattice"], case["collision"], case["stencil"])
    g = torch.zeros((len(ref.c),) + tuple(q.shape[1:]), device="cuda", dtype=torch.float64)
    log, profiles = [], []
    for k in range(1, case["steps"] + 1):
        g, q = ref.step(g, q, p)
        if case["every"] and (k % case["every"] == 0 or k == case["steps"]):
            row, prof = ref.observe(q, *ref.state(g, q, p), p)
            log.append(row)
            profiles.append(prof)
    if case["populations"]:
        out = {"Q": q, "f": ref.populations(g, p)}
    else:
        rho, u = ref.state(g, q, p)
        out = {"Q": q, "rho": rho, "u": u}
    if log:
        out["log"] = np.array(log)
    if profiles and case["profile"]:
        out["profiles"] = np.array(profiles)
    return out
