"""The work that users of this framework have it do, as cases that can be timed.

A pass advances a lattice (or an ensemble of lattices) by a number of time
steps through the public interface and reads the new populations back into
host memory that the caller keeps, the state a program analyses or writes out
as a checkpoint.  Lattices, diameters, packings and flows are those of the
repository's workloads, tests and benchmark.  `exact` restates the method in
64 bits with plain torch, without the package's code.
"""
import ctypes
import math

import numpy as np
import torch

KT = 1.0 / 3.0


# ------------------------------------------------------------------ the cases
def _case(**k):
    base = dict(kind="step", nx=64, ny=8, nz=8, sigma="1,1.5", packing=0.2, amp=0.05, noise=0.002, wall=-1, wall_u=0.0,
                tails=False, meanfield="fp32", sweeps=1, drag=False, explicit=False, flow=0.0, solute=False,
                surrogate=False, upload=False, members=1, steps=10)
    base.update(k)
    return base


def listed():
    return [
        # a small box stepped often between two looks at it: the parameter scans and the decay-rate
        # measurements of the tests (64 x 8 x 8); launches and latency count
        _case(name="scan_64x8x8", nx=64, ny=8, nz=8, steps=100),
        # one odd-sized box between sheared walls, a few steps at a time (rows that are no multiple of 16 bytes)
        _case(name="channel_97x61x45", nx=97, ny=61, nz=45, packing=0.15, wall=1, wall_u=0.02, steps=20),
        # short runs from new initial fields with velocities: each pass uploads them and starts over
        _case(name="restart_96", nx=96, ny=96, nz=96, flow=0.02, upload=True, steps=5),
        # the usual production box
        _case(name="binary_128", nx=128, ny=128, nz=128, steps=20),
        # the benchmark's headline box, the largest
        _case(name="binary_256", nx=256, ny=256, nz=256, steps=40),
        # an ensemble of small systems, half of them sheared, through one batch
        _case(name="batch_256x16", kind="batch", members=256, nx=16, ny=16, nz=16, packing=0.2, steps=20),
        # larger spheres with attractive tails: contact shells of reach 3, mean field over 7 sites
        _case(name="tails_128", nx=128, ny=128, nz=128, sigma="2,3", packing=0.3, amp=0.0, noise=0.01, tails=True, steps=8),
        # the same with the mean field on the tensor cores
        _case(name="tails_bf16_128", nx=128, ny=128, nz=128, sigma="2,3", packing=0.3, amp=0.0, noise=0.01, tails=True,
              meanfield="bf16", steps=8),
        # the Taylor-dispersion channel: two solvents and a dilute solute between moving walls
        _case(name="taylor_512x64x64", nx=512, ny=64, nz=64, sigma="2,2.5,3", packing=0.211, amp=0.0, noise=0.0, wall=1,
              wall_u=0.05, solute=True, steps=8),
        # the mixture of the paper's Taylor experiment (diameters 8 and 4) in a flow held by a body force
        _case(name="paper_80x40x40", nx=80, ny=40, nz=40, sigma="8,4", packing=0.211, amp=0.01, noise=0.0, flow=0.05, steps=8),
        # three Jacobi sweeps of the half step, spheres without tails (shells of reach 3)
        _case(name="sweeps3_96x80x72", nx=96, ny=80, nz=72, sigma="2,3", packing=0.25, amp=0.02, sweeps=3, steps=8),
        # the learned hard-core force in place of the exact one (one recheck in 50 steps)
        _case(name="surrogate_128", nx=128, ny=128, nz=128, amp=0.02, noise=0.0, surrogate=True, steps=10),
    ]


def _loguniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["small", "binary", "binary", "channel", "batch", "tails", "channel3", "paper", "sweeps", "upload", "surrogate",
                       "equal", "drag"])
    side = lambda lo, hi: int(round(_loguniform(rng, lo, hi)))  # noqa: E731
    pk = lambda lo, hi: round(rng.uniform(lo, hi), 3)  # noqa: E731
    if kind == "small":
        return _case(nx=side(4, 96), ny=side(4, 20), nz=side(4, 20), packing=pk(0.05, 0.2), steps=side(1, 100))
    if kind == "binary":
        n = side(24, 224)
        return _case(nx=max(8, n + rng.randint(-7, 7)), ny=max(8, n + rng.randint(-7, 7)), nz=n, packing=pk(0.05, 0.2), steps=rng.randint(4, 24))
    if kind == "channel":
        n = side(16, 140)
        return _case(nx=n + rng.randint(0, 9), ny=n + rng.randint(0, 9), nz=n, packing=pk(0.05, 0.18), wall=rng.randint(0, 2),
                     wall_u=round(rng.uniform(0.0, 0.03), 3), steps=rng.randint(4, 24))
    if kind == "batch":
        n = side(8, 40)
        return _case(kind="batch", members=max(2, min(256, int(2.0e6 / n ** 3))) if rng.random() < 0.5 else rng.randint(2, 24), nx=n,
                     ny=max(6, n + rng.randint(-2, 2)), nz=max(6, n + rng.randint(-2, 2)), packing=pk(0.05, 0.18), steps=rng.randint(2, 20))
    if kind == "tails":
        bf = rng.random() < 0.5
        n = side(20, 128)
        return _case(nx=n + rng.randint(-3, 3), ny=n + rng.randint(-3, 3), nz=max(16, n // 8 * 8) if bf else n, sigma="2,3",
                     packing=pk(0.1, 0.3), amp=0.0, noise=0.01, tails=True, meanfield="bf16" if bf else "fp32", steps=rng.randint(2, 8))
    if kind == "channel3":
        return _case(nx=side(48, 512), ny=side(16, 64), nz=side(12, 64), sigma="2,2.5,3", packing=0.211, amp=0.0, noise=0.0, wall=1,
                     wall_u=0.05, solute=True, steps=rng.randint(2, 8))
    if kind == "paper":
        return _case(nx=rng.choice([40, 56, 80, 96]), ny=rng.choice([24, 33, 40]), nz=rng.choice([24, 40]), sigma="8,4",
                     packing=rng.choice([0.211, 0.332]), amp=0.01, noise=0.0, flow=0.04, steps=rng.randint(2, 8))
    if kind == "sweeps":
        s = rng.choice(["1,1.5", "1.5,2", "2,3"])
        n = side(16, 100)
        return _case(nx=n + rng.randint(0, 12), ny=n, nz=n + rng.randint(0, 6), sigma=s, packing=pk(0.05, 0.2), amp=0.02,
                     sweeps=rng.randint(2, 3), steps=rng.randint(2, 8))
    if kind == "upload":
        n = side(12, 128)
        return _case(nx=n + rng.randint(0, 5), ny=n + rng.randint(0, 5), nz=n, packing=pk(0.05, 0.2), flow=0.02, upload=True,
                     steps=rng.randint(1, 8))
    if kind == "surrogate":
        return _case(nx=rng.choice([32, 64, 96, 128]), ny=side(12, 96), nz=side(12, 96), amp=0.02, noise=0.0, surrogate=True,
                     steps=rng.randint(4, 12))
    if kind == "equal":
        s = rng.choice(["1", "2", "3", "4,4", "1,1.5,2"])
        n = side(16, 96)
        return _case(nx=n, ny=n + rng.randint(0, 7), nz=n + rng.randint(0, 7), sigma=s, packing=pk(0.05, 0.15), amp=0.02,
                     steps=rng.randint(2, 10))
    n = side(16, 96)
    return _case(nx=n, ny=n + rng.randint(0, 7), nz=n, packing=pk(0.05, 0.2), drag=True, steps=rng.randint(2, 12))


# ------------------------------------------------------------------ inputs
def _sigma(case):
    return [float(v) for v in case["sigma"].split(",")]


def _n0(case, packing):
    """Equal mole fractions at the packing (pi/6) sum n sigma^3 (a solute is dilute: the solvents carry the packing)."""
    s = _sigma(case)
    m = len(s) - 1 if case["solute"] else len(s)
    n0 = packing / (math.pi / 6.0 * sum(v ** 3 for v in s[:m]))
    return [n0] * m + [0.0] * (len(s) - m)


def _inputs(case, seed, member=0):
    """Fields as FP64 device tensors: n [S, N] and u [S, 3, N] or None, x fastest."""
    g = torch.Generator(device="cuda").manual_seed((int(seed) * 1009 + 7919 * member + 1) & 0x7FFFFFFF)
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    N, S = nx * ny * nz, len(_sigma(case))
    f64 = dict(dtype=torch.float64, device="cuda")
    r = torch.rand(3, generator=g, **f64).tolist()
    packing = case["packing"]
    if case["kind"] == "batch":                       # an ensemble covers a range of packings
        packing = 0.05 + (packing - 0.05) * r[2]
    n0 = _n0(case, packing)
    x = torch.arange(nx, **f64)
    wave = case["amp"] * (0.8 + 0.4 * r[0]) * torch.sin(2.0 * math.pi * (x / nx + r[1]))
    n = torch.empty(S, nz, ny, nx, **f64)
    for a in range(S):
        n[a] = n0[a] * (1.0 + (wave if a == 0 else -wave if a == 1 else 0.0 * wave))
        if case["noise"]:
            n[a] += n0[a] * case["noise"] * (2.0 * torch.rand(nz, ny, nx, generator=g, **f64) - 1.0)
    if case["solute"]:                                # a Gaussian pulse along x, peak 1e-3 of the solvents
        c = nx * (0.45 + 0.1 * r[0])
        n[S - 1] = 1e-3 * sum(n0[:-1]) * torch.exp(-0.5 * ((x - c) / 8.0) ** 2)
    u = None
    if case["flow"]:
        u = torch.zeros(S, 3, nz, ny, nx, **f64)
        y = torch.arange(ny, **f64)
        u[:, 0] = (case["flow"] * (0.9 + 0.2 * r[2]) * torch.cos(2.0 * math.pi * y / ny))[:, None]
        u = u.reshape(S, 3, N)
    return n.reshape(S, N), u


def _body_force(case, u):
    """The force that holds the cosine flow, F = nu k_y^2 u (no upload of it where fields are uploaded each pass)."""
    if u is None or case["upload"]:
        return None
    return 0.5 * (2.0 * math.pi / case["ny"]) ** 2 * u


def _lattice(case, member=0):
    from paper_1105_3634_gb300 import workloads as W
    s = _sigma(case)
    S = len(s)
    wall, wu = case["wall"], case["wall_u"]
    if case["kind"] == "batch" and member % 2:        # every other member of an ensemble is a sheared channel
        wall, wu = 1, 0.02
    kw = {}
    if wall >= 0:
        t = [0.0, 0.0, 0.0]
        t[0 if wall != 0 else 1] = wu
        kw.update(wall_axis=wall, wall_u_lo=tuple(-v for v in t), wall_u_hi=tuple(t))
    if case["tails"]:
        kw.update(eps=[[0.5 * KT] * S for _ in range(S)], lambda_c=[[2.5] * S for _ in range(S)], meanfield=case["meanfield"])
    return W.Lattice(shape=(case["nx"], case["ny"], case["nz"]), sigma=s, drag_only=case["drag"],
                     force_scheme="explicit" if case["explicit"] else "semi_implicit", predictor_sweeps=case["sweeps"], **kw)


def _response(case):
    """Linear response of the hard-core force of the uniform mixture on the 3^3 neighbourhood, [27 taps][3 S out][S in]."""
    s = np.array(_sigma(case))
    S, n0 = len(s), np.array(_n0(case, case["packing"]))

    def g(n, a, b):
        x2, x3 = math.pi / 6 * (n * s ** 2).sum(), math.pi / 6 * (n * s ** 3).sum()
        h, o = s[a] * s[b] / (s[a] + s[b]), 1.0 - x3
        return 1 / o + 3 * h * x2 / o ** 2 + 2 * h * h * x2 * x2 / o ** 3

    M = np.zeros((27, 3 * S, S))
    for a in range(S):
        for b in range(S):
            sab = 0.5 * (s[a] + s[b])
            sh = _shell(sab)
            pre = -KT * sab * sab * 4.0 * math.pi / len(sh)
            for d in sh:
                tap = (d[2] + 1) * 9 + (d[1] + 1) * 3 + d[0] + 1
                for q in range(3):
                    e = pre * d[q] / math.sqrt(sum(v * v for v in d))
                    M[tap, 3 * a + q, b] += e * g(n0, a, b)
                    for c in range(S):
                        dn = np.zeros(S)
                        dn[c] = 1e-6 * n0[c]
                        M[tap, 3 * a + q, c] += e * 0.5 * n0[b] * (g(n0 + dn, a, b) - g(n0 - dn, a, b)) / (2 * dn[c])
    return M


def _network(case, n):
    """Parameters and scales of a network that carries the linear response (the start of the training recipe)."""
    from paper_1105_3634_gb300 import surrogate as SG
    M = _response(case)
    S, shape = n.shape[0], (case["nz"], case["ny"], case["nx"])
    dn = n - n.mean(1, keepdim=True)
    F = torch.zeros(3 * S, n.shape[1], dtype=n.dtype, device=n.device)
    Mt = torch.from_numpy(M).to(n)
    for tap in range(27):
        d = (tap // 9 - 1, tap // 3 % 3 - 1, tap % 3 - 1)
        F += Mt[tap] @ torch.roll(dn.reshape(S, *shape), [-v for v in d], (1, 2, 3)).reshape(S, -1)
    ins = [0.3 / float(dn[a].square().mean().sqrt()) for a in range(S)]
    outs = [1.0 / float(F[3 * a:3 * a + 3].square().mean().sqrt()) for a in range(S)]
    k = np.repeat(outs, 3)[None, :, None] / np.array(ins)[None, None, :]
    t_max = max(float(F[3 * a:3 * a + 3].abs().max()) * outs[a] for a in range(S))
    return SG.stencil_params(M * k, 2.0 * t_max), ins, outs


def prepare(case, seed):
    from paper_1105_3634_gb300 import mlb
    S, N, M = len(_sigma(case)), case["nx"] * case["ny"] * case["nz"], case["members"]
    st = {"case": case, "lib": mlb.lib, "batch": None, "sims": []}
    # host memory for the populations that a pass reads back
    st["f"] = torch.empty((M, S, 19, N), dtype=torch.float32, pin_memory=True).numpy()
    st["n_ref"] = np.zeros((M, S))
    for m in range(M):
        n, u = _inputs(case, seed, m)
        sim = mlb.Simulation(_lattice(case, m), stream=torch.cuda.Stream() if case["kind"] == "batch" else None)
        st["sims"].append(sim)
        if case["upload"]:                            # the caller's own (pinned) field arrays
            st["n"] = n.cpu().pin_memory().numpy()
            st["u"] = None if u is None else u.cpu().pin_memory().numpy()
        sim.set_fields(n.cpu().numpy(), None if u is None else u.cpu().numpy())
        fe = _body_force(case, u)
        if fe is not None:
            sim.set_external_force(fe.cpu().numpy())
        if case["surrogate"]:
            p, ins, outs = _network(case, n)
            net = mlb.Net((case["nx"], case["ny"], case["nz"]))
            net.set_params(p)
            net.set_scales(ins, outs)
            sim.attach_surrogate(net, recheck_every=50, bound=0.05)
    if case["kind"] == "batch":
        st["batch"] = mlb.Batch(st["sims"], stream=torch.cuda.Stream())
    return st


def run(state):
    c = state["case"]
    if state["batch"] is not None:
        state["batch"].step(c["steps"])
        state["batch"].synchronize()
    else:
        sim = state["sims"][0]
        if c["upload"]:
            sim.set_fields(state["n"], state["u"])
        sim.step(c["steps"])
    for m, sim in enumerate(state["sims"]):
        sim._check(state["lib"].mlb_get_populations(sim.ctx, state["f"][m].ctypes.data_as(ctypes.POINTER(ctypes.c_float)),
                                                    state["n_ref"][m].ctypes.data_as(ctypes.POINTER(ctypes.c_double)), None))
    return {"f": state["f"], "n_ref": state["n_ref"]}


def work(case):
    """Populations in and out once a step (19 FP32 each way), once more for the copy to the host; uploaded fields once.
    Operations: 36 + 18 per ordered pair and shell point, 6 per point of the tails, about 19 x 15 of the collision."""
    s = _sigma(case)
    S, N = len(s), case["nx"] * case["ny"] * case["nz"] * case["members"]
    shell = sum(len(_shell(0.5 * (a + b))) for a in s for b in s)
    per_site = (54 + 30 * (case["sweeps"] - 1)) * shell + 285 * S
    if case["tails"]:
        per_site += 6 * sum(len(_tail(0.5 * (a + b))) for a in s for b in s)
    if case["surrogate"]:
        per_site += 2 * (27 * 2 * 32 + 27 * 32 * 32 + 6 * 32)
    b = 152.0 * S * N * case["steps"] + 76.0 * S * N
    if case["upload"]:
        b += 32.0 * S * N
    return {"bytes": b, "flops": float(per_site) * N * case["steps"]}


# ------------------------------------------------------------------ the method in 64 bits
_C = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0), (1, -1, 0), (-1, 1, 0),
      (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1)]
_W = [1.0 / 3.0] + [1.0 / 18.0] * 6 + [1.0 / 36.0] * 12


def _offsets(R, keep):
    return [(x, y, z) for z in range(-R, R + 1) for y in range(-R, R + 1) for x in range(-R, R + 1) if keep(x * x + y * y + z * z)]


def _shell(sab):
    return _offsets(int(sab) + 2, lambda q: q > 0 and (sab - 0.5) ** 2 <= q < (sab + 0.5) ** 2)


def _tail(sab):
    return _offsets(int(2.5 * sab) + 1, lambda q: sab * sab <= q <= (2.5 * sab) ** 2)


class _Exact:
    """M members of one lattice as FP64 tensors [M, ..., nz, ny, nx]."""

    def __init__(self, case, member, n, u, fext, net):
        lat = _lattice(case, member)
        self.sigma, self.S, self.shape = _sigma(case), n.shape[1], (case["nz"], case["ny"], case["nx"])
        self.case, self.wall, self.net, self.fext = case, lat.wall_axis, net, fext
        self.u_lo, self.u_hi = lat.wall_u_lo, lat.wall_u_hi
        self.pre = {}
        self.f = self.equilibrium(n, u if u is not None else torch.zeros(n.shape[0], self.S, 3, *self.shape).to(n), None)
        self.t = 0

    def at(self, x, R):
        """x padded by R sites: periodic images, zero beyond a wall.  Returns offset -> view."""
        for k in range(3):                            # lattice axis k is tensor dimension -1 - k
            dim, L = x.dim() - 1 - k, self.shape[2 - k]
            if k == self.wall:
                shape = list(x.shape)
                shape[dim] = R
                z = torch.zeros(shape, dtype=x.dtype, device=x.device)
                x = torch.cat([z, x, z], dim)
            else:
                x = x.index_select(dim, torch.arange(-R, L + R, device=x.device) % L)
        nz, ny, nx = self.shape
        return lambda d: x[..., R + d[2]:R + d[2] + nz, R + d[1]:R + d[1] + ny, R + d[0]:R + d[0] + nx]

    def equilibrium(self, n, u, acc):
        """psi_perp [M, S, 19, ...] at (n, u); with acc also the forcing term (a second tensor)."""
        rho = n.sum(1, keepdim=True)
        ub = (n[:, :, None] * u).sum(1) / rho
        psi = torch.empty(n.shape[0], self.S, 19, *self.shape, dtype=n.dtype, device=n.device)
        src = torch.empty_like(psi) if acc is not None else None
        dot = lambda c, v: sum(c[k] * v[:, k] for k in range(3) if c[k])  # noqa: E731
        for a in range(self.S):
            ua, na = u[:, a], n[:, a]
            tr = (2 * ua * ub - ub * ub).sum(1)
            trs = 2 * (ub * acc[:, a]).sum(1) if acc is not None else None
            for i, c in enumerate(_C):
                cu, cb = (dot(c, ua), dot(c, ub)) if i else (0.0, 0.0)
                psi[:, a, i] = _W[i] * na * (1 + 3 * cu + 4.5 * (2 * cu * cb - cb * cb) - 1.5 * tr)
                if acc is not None:
                    ca = dot(c, acc[:, a]) if i else 0.0
                    src[:, a, i] = _W[i] * na * (3 * ca + 9 * cb * ca - 1.5 * trs)
        return psi if acc is None else (psi, src)

    def contact(self, n):
        x2 = x3 = 0.0
        for c, s in enumerate(self.sigma):
            r2 = (0.5 * s) ** 2
            ball = _offsets(int(0.5 * s) + 1, lambda q: q <= r2)
            v = self.at(n[:, c], int(0.5 * s) + 1)
            nbar = sum(v(d) for d in ball) / len(ball)
            x2, x3 = x2 + math.pi / 6 * s * s * nbar, x3 + math.pi / 6 * s ** 3 * nbar
        o, g = 1.0 - x3, {}
        for a in range(self.S):
            for b in range(a, self.S):
                h = self.sigma[a] * self.sigma[b] / (self.sigma[a] + self.sigma[b])
                g[a, b] = g[b, a] = 1 / o + 3 * h * x2 / o ** 2 + 2 * h * h * x2 * x2 / o ** 3
        return g

    def shells(self, n, g, vel, rest):
        """Velocity-exchange gain [M, S, 3, ...]; rest: also the hard core and the friction matrix (six fields)."""
        R = max(int(s + 0.5) for s in self.sigma)
        gain = torch.zeros_like(vel)
        hc, gam = (torch.zeros_like(vel), torch.zeros(*vel.shape[:2], 6, *self.shape, dtype=n.dtype, device=n.device)) if rest else (None, None)
        nv, uv = [self.at(n[:, b], R) for b in range(self.S)], [self.at(vel[:, b], R) for b in range(self.S)]
        for a in range(self.S):
            for b in range(self.S):
                sab = 0.5 * (self.sigma[a] + self.sigma[b])
                sh, gv = _shell(sab), self.at(g[a, b], R)
                pre = sab * sab * 4.0 * math.pi / len(sh)
                K = 2.0 * math.sqrt(KT / math.pi)       # 2 sqrt(2 mu kT / pi), mu = 1/2
                for d in sh:
                    il = 1.0 / math.sqrt(d[0] * d[0] + d[1] * d[1] + d[2] * d[2])
                    s = [v * il for v in d]
                    w = (g[a, b] + gv(d)) * nv[b](d) * (0.5 * pre)
                    v = vel[:, b] if self.case["drag"] else uv[b](d)
                    sv = sum(s[k] * v[:, k] for k in range(3) if d[k]) * w
                    for k in range(3):
                        if d[k]:
                            gain[:, a, k].add_(sv, alpha=K * s[k])
                            if rest:
                                hc[:, a, k].add_(w, alpha=-KT * s[k])
                    if rest:
                        for q, (x, y) in enumerate(((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))):
                            if d[x] and d[y]:
                                gam[:, a, q].add_(w, alpha=K * s[x] * s[y])
        return (gain, hc, gam) if rest else gain

    def tails(self, n):
        """G^a = sum_b sum_d K_ab(d) n^b(r + d) by FFT (zero padding along a wall axis)."""
        R = int(2.5 * max(self.sigma)) + 1
        size = [L + (R if 2 - k == self.wall else 0) for k, L in enumerate(self.shape)]
        out = torch.zeros(n.shape[0], self.S, 3, *self.shape, dtype=n.dtype, device=n.device)
        fn = torch.fft.rfftn(n, s=size, dim=(-3, -2, -1))
        for a in range(self.S):
            for b in range(self.S):
                sab = 0.5 * (self.sigma[a] + self.sigma[b])
                if (a, b) not in self.pre:
                    k = torch.zeros(3, *size, dtype=n.dtype)
                    for d in _tail(sab):
                        c = 6.0 * 0.5 * KT * sab ** 6 / (d[0] * d[0] + d[1] * d[1] + d[2] * d[2]) ** 4
                        at = (d[2] % size[0], d[1] % size[1], d[0] % size[2])
                        for q in range(3):
                            k[(q,) + at] += c * d[q]
                    self.pre[a, b] = torch.fft.rfftn(k.to(n.device), dim=(-3, -2, -1)).conj()
                g = torch.fft.irfftn(self.pre[a, b] * fn[:, b, None], s=size, dim=(-3, -2, -1))
                out[:, a] += g[..., :self.shape[0], :self.shape[1], :self.shape[2]]
        return out

    def network(self, n):
        p, ins, outs, nref = self.net
        p = torch.from_numpy(np.asarray(p, np.float64)).to(n)
        W1, b1, W2, b2, W3, b3 = torch.split(p, [27 * 64, 32, 27 * 1024, 32, 192, 6])
        x = torch.stack([(n[0, a] - nref[a]) * ins[a] for a in range(2)])
        for W, b, ci in ((W1, b1, 2), (W2, b2, 32)):
            W, y = W.reshape(27, 32, ci), b[:, None].repeat(1, x[0].numel())
            for tap in range(27):
                d = (tap // 9 - 1, tap // 3 % 3 - 1, tap % 3 - 1)
                y += W[tap] @ torch.roll(x, [-v for v in d], (1, 2, 3)).reshape(ci, -1)
            x = torch.tanh(y).reshape(32, *self.shape)
        F = (W3.reshape(6, 32) @ x.reshape(32, -1) + b3[:, None]).reshape(1, 2, 3, *self.shape)
        return F / torch.tensor(outs).to(n).reshape(1, 2, 1, 1, 1, 1)

    @staticmethod
    def solve(G, b):
        """x of (I + G/2) x = b, G = (xx, yy, zz, xy, xz, yz)."""
        xx, yy, zz = (1 + 0.5 * G[:, :, k] for k in range(3))
        xy, xz, yz = (0.5 * G[:, :, k] for k in (3, 4, 5))
        c = [yy * zz - yz * yz, xz * yz - xy * zz, xy * yz - xz * yy, xx * zz - xz * xz, xy * xz - xx * yz, xx * yy - xy * xy]
        det = xx * c[0] + xy * c[1] + xz * c[2]
        rows = ((0, 1, 2), (1, 3, 4), (2, 4, 5))
        return torch.stack([sum(c[r[k]] * b[:, :, k] for k in range(3)) / det for r in rows], 2)

    @staticmethod
    def apply(G, v):
        rows = ((0, 3, 4), (3, 1, 5), (4, 5, 2))
        return torch.stack([sum(G[:, :, r[k]] * v[:, :, k] for k in range(3)) for r in rows], 2)

    def step(self):
        f = self.f
        n = f.sum(2)
        u = torch.stack([sum(c[k] * f[:, :, i] for i, c in enumerate(_C) if c[k]) for k in range(3)], 2)
        u /= n.clamp(min=1e-300)[:, :, None]
        g = self.contact(n)
        gain, rest, gam = self.shells(n, g, u, True)
        if self.net is not None and self.t % 50:
            rest = self.network(n)
        if self.case["tails"]:
            rest = rest + self.tails(n)
        if self.fext is not None:
            rest = rest + self.fext
        us = u
        if not self.case["explicit"]:
            for k in range(self.case["sweeps"]):
                if k:
                    gain = self.shells(n, g, us, False)
                us = self.solve(gam, u + 0.5 * (rest + gain))
            gain = self.shells(n, g, us, False)
        acc = rest + gain - self.apply(gam, us)
        del gain, rest, gam, us
        psi, src = self.equilibrium(n, u if self.case["explicit"] else u + 0.5 * acc, acc)
        post = f + 1.0 * (psi - f) + (1.0 if self.case["explicit"] else 0.5) * src           # tau = 1
        del psi, src
        out = torch.empty_like(post)
        for i, c in enumerate(_C):
            out[:, :, i] = torch.roll(post[:, :, i], (c[2], c[1], c[0]), (2, 3, 4))
        if self.wall >= 0:                            # halfway bounce-back on the moving walls
            ax = self.wall
            for i, c in enumerate(_C):
                if not c[ax]:
                    continue
                j = _C.index(tuple(-v for v in c))    # j leaves through the wall that i comes from
                edge, uw = (0, self.u_lo) if c[ax] > 0 else (self.shape[2 - ax] - 1, self.u_hi)
                cw = sum(_C[j][k] * uw[k] for k in range(3))
                dim = 4 - ax                          # of [M, S, nz, ny, nx]
                out[:, :, i].select(dim, edge).copy_((post[:, :, j] - 6.0 * _W[j] * cw * n).select(dim, edge))
        self.f = out
        self.t += 1


def exact(case, seed):
    M, shape = case["members"], (case["nz"], case["ny"], case["nx"])
    S, N = len(_sigma(case)), case["nx"] * case["ny"] * case["nz"]
    groups = [list(range(M))] if case["kind"] != "batch" else [list(range(k, M, 2)) for k in range(2) if k < M]
    f = torch.empty(M, S, 19, N, dtype=torch.float64, device="cuda")
    n_ref = torch.zeros(M, S, dtype=torch.float64, device="cuda")
    for members in groups:
        ins = [_inputs(case, seed, m) for m in members]
        n = torch.stack([v[0] for v in ins]).reshape(-1, S, *shape)
        u = None if ins[0][1] is None else torch.stack([v[1] for v in ins]).reshape(-1, S, 3, *shape)
        fe = _body_force(case, u)
        ref = n.reshape(len(members), S, N).mean(2).float().double()
        net = None
        if case["surrogate"]:
            net = _network(case, ins[0][0]) + (ref[0].tolist(),)
        del ins
        e = _Exact(case, members[0], n, u, fe, net)
        for _ in range(case["steps"]):
            e.step()
        w = torch.tensor(_W, dtype=torch.float64, device="cuda")
        f[members] = e.f.reshape(len(members), S, 19, N) - w[:, None] * ref[:, :, None, None]
        n_ref[members] = ref
        del e, n, u
    return {"f": f, "n_ref": n_ref}
