"""What this library's speed is measured on: whole calls through its public binding.

A case is one thing a program does with the library: advance a lattice and read
the fields back, log a growth run, relax an order parameter, exchange state
with the host, step a sweep of replicas, call or train the surrogate.  Every
case gives its inputs (prepare), one pass of the program's loop (run), the
bytes and operations such a pass cannot do without (work) and what it returns
in 64-bit arithmetic (exact: plain torch, none of the library's code).

Initial states are blue phase II, a cholesteric helix or isotropic noise, with a
weak vortical flow where there is flow, all from the seed.
"""

from __future__ import annotations

import math
import os

import numpy as np
import torch

from paper_0901_3293_gb300 import lcbp

WEIGHTS = os.path.join("paper_0901_3293_gb300", "weights", "slab_k50.lcbpsur")
A0 = 0.01

# LdG / kinetic parameters of the repository's parity workload
BASE = {"gamma": 3.1, "K": 0.01, "pitch": 16, "tau_f": 2.0, "xi": 0.7, "Gamma": 0.3}


def listed():
    lat = {"do": "lattice", "dtype": "f32", "mode": "flow", "init": "bpii", "log": False, **BASE}
    return [
        # the parity workload: a small periodic BPII cube, FP32 state, 100 steps between reads
        {**lat, "name": "cube_32_f32", "nx": 32, "ny": 32, "nz": 32, "steps": 100},
        # the same with FP64 state, as reference runs use it
        {**lat, "name": "cube_32_f64", "nx": 32, "ny": 32, "nz": 32, "steps": 50, "dtype": "f64"},
        # domain growth in the thin slab: free energy and mass logged every 100 steps
        {**lat, "name": "slab_64x64x256_log", "nx": 64, "ny": 64, "nz": 256, "steps": 100, "init": "slab",
         "kappa": 1.0, "tau": -0.5, "log": True},
        # the large single lattice of the benchmark, with its energy and conservation checks
        {**lat, "name": "cube_256_f32", "nx": 256, "ny": 256, "nz": 256, "steps": 20, "pitch": 32, "log": True},
        # a cell between two anchoring walls
        {**lat, "name": "walls_128x96x64", "nx": 128, "ny": 96, "nz": 64, "steps": 40, "mode": "walls"},
        # sizes that are a multiple of nothing: a cell of some physical size in lattice units
        {**lat, "name": "odd_101x75x67", "nx": 101, "ny": 75, "nz": 67, "steps": 40},
        # equilibration without flow, the usual preparation of a blue-phase state
        {**lat, "name": "relax_96_noflow", "nx": 96, "ny": 96, "nz": 96, "steps": 100, "mode": "noflow", "log": True},
        # the sequential coupling of the two updates
        {**lat, "name": "seidel_80x64x48", "nx": 80, "ny": 64, "nz": 48, "steps": 40, "mode": "gauss_seidel"},
        # another program owns the state: upload f and Q from pinned memory, one step, Q and u back
        {**lat, "name": "exchange_128_host", "do": "exchange", "nx": 128, "ny": 128, "nz": 128, "steps": 1},
        # the chirality / temperature sweep: 48 replicas of 32^3 and 48^3 in one batch
        {"do": "sweep", "name": "sweep_48_replicas", "replicas": 48, "n_a": 32, "n_b": 48, "steps": 200,
         "dtype": "f32"},
        # one segment of the judged surrogate run on the slab: calls, re-equilibration, free energy
        {"do": "surrogate", "name": "surrogate_slab", "nx": 64, "ny": 64, "nz": 256, "calls": 8, "kappa": 1.0,
         "tau": -0.5},
        # one training step on a crop with a loss mask
        {"do": "train", "name": "train_64_crop", "nx": 64, "ny": 64, "nz": 64, "kappa": 1.25, "tau": -0.5},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """Another case of the same kinds: sizes over the listed range, odd widths among them."""
    do = rng.choice(["lattice"] * 6 + ["exchange", "sweep", "surrogate", "train"])
    if do == "sweep":
        a, b = rng.choice([16, 20, 24, 32]), rng.choice([36, 40, 48, 64])
        r = rng.randint(8, 48)
        return {"do": do, "replicas": r, "n_a": a, "n_b": b, "steps": max(20, int(4e8 / (r * (a ** 3 + b ** 3) / 2)) // 2),
                "dtype": "f32"}
    if do == "surrogate":
        return {"do": do, "nx": rng.randint(24, 96), "ny": rng.randint(16, 72), "nz": rng.randint(16, 144),
                "calls": rng.randint(1, 8), "kappa": rng.uniform(0.5, 2.0), "tau": rng.uniform(-0.5, 0.5)}
    if do == "train":
        return {"do": do, "nx": rng.randint(32, 72), "ny": rng.randint(32, 64), "nz": rng.randint(32, 64),
                "kappa": rng.uniform(0.5, 2.0), "tau": rng.uniform(-0.5, 0.5)}
    mode = "flow" if do == "exchange" else rng.choice(["flow"] * 5 + ["walls", "noflow", "noflow", "gauss_seidel", "l2"])
    dtype = "f64" if do == "lattice" and rng.random() < 0.2 else "f32"
    top = 64 if dtype == "f64" else 128 if mode in ("gauss_seidel", "l2") or do == "exchange" else 224
    n = [_log(rng, 12, top) for _ in range(3)]
    if rng.random() < 0.6:
        n[0] = max(16, n[0] // 4 * 4)  # most programs choose even widths
    steps = 1 if do == "exchange" else min(100, max(5, int(1e8 / (n[0] * n[1] * n[2]))))
    case = {"do": do, "dtype": dtype, "mode": mode, "init": rng.choice(["bpii", "helix", "noise"]),
            "log": do == "lattice" and rng.random() < 0.4, **BASE, "nx": n[0], "ny": n[1], "nz": n[2], "steps": steps,
            "pitch": rng.choice([16, 24, 32])}
    if rng.random() < 0.5:
        case.update(kappa=rng.uniform(0.3, 2.0), tau=rng.uniform(-1.0, 0.5))
    return case


# ---- inputs ---------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _ldg(case):
    """gamma, K and q0 of a case (from kappa and tau where it gives them)."""
    q0 = 2.0 * math.pi / case.get("pitch", 16)
    if "kappa" in case:
        gamma = 27.0 / (9.0 + case["tau"])
        return gamma, case["kappa"] ** 2 * A0 * gamma / (108.0 * q0 * q0), q0
    return case["gamma"], case["K"], q0


def _state_dtype(case):
    return torch.float64 if case.get("dtype") == "f64" else torch.float32


def _axes(nx, ny, nz):
    o = {"device": "cuda", "dtype": torch.float64}
    return (torch.arange(nx, **o).view(1, 1, -1), torch.arange(ny, **o).view(1, -1, 1),
            torch.arange(nz, **o).view(-1, 1, 1))


def _q5(kind, nx, ny, nz, q0, gamma, seed, dtype):
    """[5, z, y, x] initial order parameter of a kind, with seeded noise."""
    x, y, z = _axes(nx, ny, nz)
    one = torch.ones((nz, ny, nx), device="cuda", dtype=torch.float64)
    k = 2.0 * q0
    bp = torch.stack([0.3 * (torch.cos(k * z) - torch.cos(k * y)) * one, 0.3 * torch.sin(k * z) * one,
                      0.3 * torch.sin(k * y) * one, 0.3 * (torch.cos(k * x) - torch.cos(k * z)) * one,
                      0.3 * torch.sin(k * x) * one])
    s = 0.25 + 0.75 * math.sqrt(max(0.0, 1.0 - 8.0 / (3.0 * gamma)))
    c, sn = torch.cos(q0 * x), torch.sin(q0 * x)  # helix along x
    hx = torch.stack([-s / 3 * one, 0 * one, 0 * one, s * (c * c - 1 / 3) * one, s * c * sn * one])
    g = _gen(seed)
    noise = torch.rand((5, nz, ny, nx), generator=g, device="cuda", dtype=torch.float64) * 2 - 1
    if kind == "noise":
        q = 1e-2 * noise
    elif kind == "helix":
        q = hx + 1e-3 * noise
    elif kind == "slab":
        q = torch.where(z < max(1, nz // 8), bp, hx) + 1e-4 * noise
    else:
        q = bp + 1e-4 * noise
    return q.to(dtype).contiguous()


def _u3(nx, ny, nz, seed, dtype):
    """[3, z, y, x] weak vortices of the box's size, amplitude 0.02, random phases."""
    x, y, z = _axes(nx, ny, nz)
    one = torch.ones((nz, ny, nx), device="cuda", dtype=torch.float64)
    p = 2 * math.pi * torch.rand(3, generator=_gen(seed + 7919), device="cuda", dtype=torch.float64)
    w = 2 * math.pi
    u = torch.stack([torch.sin(w * y / ny + p[0]) * one, torch.sin(w * z / nz + p[1]) * one,
                     torch.sin(w * x / nx + p[2]) * one])
    return (0.02 * u).to(dtype).contiguous()


Q_WALL = (0.2, 0.0, 0.0, -0.1, 0.0)  # planar anchoring S (x x - I / 3), S = 0.3


def _flow(case):
    return case["mode"] != "noflow"


def _lattice(case, seed):
    gamma, K, q0 = _ldg(case)
    dims = case["nx"], case["ny"], case["nz"]
    lat = lcbp.Lattice(*dims, dtype=case["dtype"]).set_ldg(A0, gamma, K, q0)
    lat.set_flow(case["tau_f"], case["xi"], case["Gamma"], flow_on=_flow(case),
                 coupling=lcbp.GAUSS_SEIDEL if case["mode"] == "gauss_seidel" else lcbp.JACOBI)
    if case["mode"] == "walls":
        lat.set_walls(True, Q_WALL)
    if case["mode"] == "l2":
        lat.set_l2(0.0)
    dt = _state_dtype(case)
    lat.set_q(_q5(case["init"], *dims, q0, gamma, seed, dt))
    if _flow(case):
        lat.init_f_equilibrium(1.0, _u3(*dims, seed, dt))
    return lat


def _sweep(case, seed):
    """Per-replica draws: dims, kappa, tau, initial kind, noise seed."""
    r = np.random.default_rng(seed)
    out = []
    for i in range(case["replicas"]):
        n = case["n_a"] if i % 2 == 0 else case["n_b"]
        out.append({"n": n, "kappa": float(r.uniform(0.3, 2.0)), "tau": float(r.uniform(-1.0, 0.5)), "pitch": 16,
                    "kind": ("bpii", "helix", "noise")[i % 3], "seed": seed * 1000 + i})
    return out


def _train_fields(case, seed):
    """q, u, rate, dq and mask of a crop, smooth fields of the sizes trajectories have."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    x, y, z = _axes(nx, ny, nz)
    g = _gen(seed)

    def modes(c, amp):
        out = torch.zeros((c, nz, ny, nx), device="cuda", dtype=torch.float64)
        for _ in range(3):
            k = torch.randint(0, 5, (3, c, 1, 1, 1), generator=g, device="cuda").double() * (2 * math.pi)
            p = torch.rand((c, 1, 1, 1), generator=g, device="cuda", dtype=torch.float64) * (2 * math.pi)
            out += torch.cos(k[0] * x / nx + k[1] * y / ny + k[2] * z / nz + p) * (amp / 3)
        return out

    q, u, r = modes(5, 0.3), modes(3, 1e-3), modes(5, 1e-4)
    dq = 50 * r + modes(5, 6e-6) + 1e-6 * (torch.rand(q.shape, generator=g, device="cuda", dtype=torch.float64) - 0.5)
    mask = ((z >= 10) & (z < nz - 10)).double() * torch.ones((nz, ny, nx), device="cuda", dtype=torch.float64)
    return [v.float().contiguous() for v in (q, u, r, dq, mask)]


def prepare(case, seed):
    do = case["do"]
    dev = {"device": "cuda"}
    if do == "lattice":
        lat, dt = _lattice(case, seed), _state_dtype(case)
        shape = (case["nz"], case["ny"], case["nx"])
        return {"case": case, "lat": lat, "q": torch.empty((5,) + shape, dtype=dt, **dev),
                "u": torch.empty((3,) + shape, dtype=dt, **dev) if _flow(case) else None}
    if do == "exchange":
        lat = _lattice(case, seed)
        lat.step(2)  # some state of a run, as the other program holds it
        shape = (case["nz"], case["ny"], case["nx"])
        q, f = _exchange_state(case, seed)
        pin = lambda t: torch.empty(t.shape, dtype=t.dtype, pin_memory=True).copy_(t)  # noqa: E731
        return {"case": case, "lat": lat, "q_in": pin(q), "f_in": pin(f),
                "q": torch.empty((5,) + shape, dtype=torch.float32, pin_memory=True),
                "u": torch.empty((3,) + shape, dtype=torch.float32, pin_memory=True)}
    if do == "sweep":
        rs = _sweep(case, seed)
        par, qs = [], []
        for r in rs:
            gamma, K, q0 = _ldg(r)
            par.append({"A0": A0, "gamma": gamma, "K": K, "q0": q0, "tau_f": BASE["tau_f"], "xi": BASE["xi"],
                        "Gamma": BASE["Gamma"]})
            qs.append(_q5(r["kind"], r["n"], r["n"], r["n"], q0, gamma, r["seed"], torch.float32))
        b = lcbp.Batch([(r["n"],) * 3 for r in rs], par, dtype=case["dtype"])
        for i, q in enumerate(qs):
            b.set_q(i, q)
        b.init_f_equilibrium(1.0)
        return {"case": case, "batch": b}
    if do == "surrogate":
        lc = _surrogate_lattice(case)
        lat = _lattice(lc, seed)
        snap = torch.empty(lat.snapshot_bytes(), dtype=torch.uint8, **dev)
        lat.snapshot(snap)
        sur = lcbp.Surrogate(case["nx"], case["ny"], case["nz"]).load(WEIGHTS)
        return {"case": case, "lat": lat, "sur": sur, "snap": snap,
                "q": torch.empty((5, case["nz"], case["ny"], case["nx"]), dtype=torch.float32, **dev)}
    sur = lcbp.Surrogate(case["nx"], case["ny"], case["nz"], training=True).load(WEIGHTS)
    q, u, r, dq, mask = _train_fields(case, seed)
    return {"case": case, "sur": sur, "q": q, "u": u, "r": r, "dq": dq, "mask": mask}


def run(state):
    case = state["case"]
    do = case["do"]
    if do == "lattice":
        lat = state["lat"]
        lat.step(case["steps"])
        out = {}
        if case["log"]:
            out["F"] = lat.free_energy()
            if _flow(case):
                out["mass"] = lat.totals()[0]
        out["q"] = lat.read_q(out=state["q"])
        if state["u"] is not None:
            out["u"] = lat.read_u(out=state["u"])
        return out
    if do == "exchange":
        lat = state["lat"]
        lat.set_f(state["f_in"]).set_q(state["q_in"])
        lat.step(case["steps"])
        return {"q": lat.read_q(out=state["q"]), "u": lat.read_u(out=state["u"])}
    if do == "sweep":
        b = state["batch"]
        b.step(case["steps"])
        return {"F": np.array([b.free_energy(i) for i in range(b.R)], dtype=np.float32),  # (an FP32 state's energy)
                "q": [b.read_q(i, dtype=np.float32) for i in range(b.R)]}
    if do == "surrogate":
        lat = state["lat"]
        lat.restore(state["snap"])
        state["sur"].step(lat, case["kappa"], case["tau"], case["calls"])
        lat.reequilibrate_f()
        return {"F": lat.free_energy(), "q": lat.read_q(out=state["q"])}
    sur = state["sur"]
    loss = sur.train_step(state["q"], state["u"], state["r"], case["kappa"], case["tau"], state["dq"], state["mask"],
                          lr=1e-4)
    return {"loss": loss, "grads": sur.get_grads(), "params": sur.get_params()}


# ---- the floor --------------------------------------------------------------------
STEP_FLOPS = 950    # add / multiply / fused operations a site's coupled step takes
NOFLOW_FLOPS = 330  # the same without flow
CONV_MACS = 238464  # multiply-adds per site of one network call (true channel counts)


def work(case):
    if case["do"] == "sweep":
        r = case["replicas"]
        sites = (r + 1) // 2 * case["n_a"] ** 3 + r // 2 * case["n_b"] ** 3
        return {"bytes": sites * (160.0 * case["steps"] + 40), "flops": float(sites) * STEP_FLOPS * case["steps"]}
    sites = case["nx"] * case["ny"] * case["nz"]
    if case["do"] == "surrogate":
        # Q read and written and u read in every call; f and Q restored and rebuilt once
        return {"bytes": sites * (52.0 * case["calls"] + 200), "flops": 2.0 * CONV_MACS * sites * case["calls"]}
    if case["do"] == "train":
        return {"bytes": sites * 76.0, "flops": 6.0 * CONV_MACS * sites}
    es = 8 if case["dtype"] == "f64" else 4
    flow = _flow(case)
    per = 2 * es * (5 + (15 if flow else 0))
    extra = es * (10 + (6 if flow else 0))  # the fields read back
    if case["do"] == "exchange":
        extra += 2 * es * 20
    if case["log"]:
        extra += es * (5 + (15 if flow else 0))
    return {"bytes": float(sites) * (per * case["steps"] + extra),
            "flops": float(sites) * (STEP_FLOPS if flow else NOFLOW_FLOPS) * case["steps"]}


# ---- the same in 64 bits, plain torch -----------------------------------------------
# Tensors carry a replica axis: fields are [B, z, y, x] with component axes in front.
E = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1)] + \
    [(a, b, c) for a in (1, -1) for b in (1, -1) for c in (1, -1)]
OPP = [E.index((-a, -b, -c)) for a, b, c in E]
REST = [8 / 15] + [1 / 30] * 14


def _nb(a, g, s, ghost=None):
    """a(r + s e_g), periodic; with `ghost` = (below, above), those planes stand beyond z."""
    if g == 2 and ghost is not None:
        if s > 0:
            return torch.cat([a[..., 1:, :, :], ghost[1]], dim=-3)
        return torch.cat([ghost[0], a[..., :-1, :, :]], dim=-3)
    return torch.roll(a, -s, -1 - g)


def _d0(a, g, ghost=None):
    return 0.5 * (_nb(a, g, 1, ghost) - _nb(a, g, -1, ghost))


def _mm(a, b):
    return sum(a[:, c, None] * b[None, c] for c in range(3))


def _dd(a, b):
    return (a * b).sum(dim=(0, 1))


def _tr(a):
    return a[0, 0] + a[1, 1] + a[2, 2]


def _eye_times(s):
    z = torch.zeros_like(s)
    return torch.stack([torch.stack([s if a == b else z for b in range(3)]) for a in range(3)])


def _q9(q5):
    """[5, ...] -> [3, 3, ...]"""
    xx, xy, xz, yy, yz = q5
    return torch.stack([torch.stack([xx, xy, xz]), torch.stack([xy, yy, yz]), torch.stack([xz, yz, -xx - yy])])


def _five(q):
    return torch.stack([q[0, 0], q[0, 1], q[0, 2], q[1, 1], q[1, 2]])


class _Model:
    def __init__(self, gamma, K, q0, tau_f, xi, Gamma, mode="flow"):
        self.gamma, self.K, self.q0, self.tau_f, self.xi, self.Gamma, self.mode = gamma, K, q0, tau_f, xi, Gamma, mode

    def _ghost(self, q):
        if self.mode != "walls":
            return None
        w = torch.tensor(Q_WALL, device=q.device, dtype=q.dtype).view(5, 1, 1, 1, 1)
        w = _q9(w).expand(q.shape[:3] + (1,) + q.shape[-2:])
        return w, w

    def grads(self, q):
        gh = self._ghost(q)
        return [_d0(q, g, gh) for g in range(3)]

    def field(self, q, dq):
        """H: minus the derivative of the lattice energy, made traceless."""
        gh = self._ghost(q)
        lap = sum(_nb(q, g, s, gh) for g in range(3) for s in (1, -1)) - 6.0 * q
        # C_ab = eps_agd D0_g Q_db
        C = torch.stack([dq[1][2] - dq[2][1], dq[2][0] - dq[0][2], dq[0][1] - dq[1][0]])
        tr2 = _dd(q, q)
        G = A0 * (1.0 - self.gamma / 3.0) * q - A0 * self.gamma * _mm(q, q) + A0 * self.gamma * tr2 * q - \
            self.K * lap + 2.0 * self.K * self.q0 * (C + C.transpose(0, 1)) + 4.0 * self.K * self.q0 ** 2 * q
        if self.mode == "l2":  # L2 = 0
            dv = torch.stack([dq[0][a, 0] + dq[1][a, 1] + dq[2][a, 2] for a in range(3)])
            M = torch.stack([_d0(dv, b) for b in range(3)], dim=1)
            G = G + 0.5 * self.K * (M + M.transpose(0, 1))
        return -G + _eye_times(_tr(G) / 3.0)

    def rate(self, q, h, dq, u):
        if u is None:
            return self.Gamma * h
        gh = (-u[..., :1, :, :], -u[..., -1:, :, :]) if self.mode == "walls" else None
        W = torch.stack([_d0(u, b, gh) for b in range(3)], dim=1)  # W_ab = D0_b u_a
        D, O = 0.5 * (W + W.transpose(0, 1)), 0.5 * (W - W.transpose(0, 1))
        P = q + _eye_times(torch.full_like(q[0, 0], 1 / 3))
        S = _mm(self.xi * D + O, P) + _mm(P, self.xi * D - O) - 2.0 * self.xi * P * _dd(q, D)
        S = S - _eye_times(_tr(S) / 3.0)
        return self.Gamma * h + S - (u[0] * dq[0] + u[1] * dq[1] + u[2] * dq[2])

    def stress(self, q, h):
        P = q + _eye_times(torch.full_like(q[0, 0], 1 / 3))
        s = 2.0 * self.xi * P * _dd(q, h) - self.xi * (_mm(h, P) + _mm(P, h))
        return s, _mm(q, h) - _mm(h, q)

    def force(self, h, dq, tau):
        gh = None
        if self.mode == "walls":
            z = torch.zeros_like(tau[:, 2, ..., :1, :, :])
            gh = (z, z)
        b = sum(_d0(tau[:, c], c, gh if c == 2 else None) for c in range(3))
        return b - torch.stack([_dd(h, dq[a]) for a in range(3)])

    def collide(self, f, s, b):
        """-(f - f_eq) / tau_f + p per direction (deviations from the rest weights)."""
        drho, u = _moments(f)
        rho = 1.0 + drho
        usq = (u * u).sum(0)
        out = []
        for i, e in enumerate(E):
            eu, eb = sum(c * v for c, v in zip(e, u)), sum(c * v for c, v in zip(e, b))
            if i == 0:
                feq, p = drho * (8 / 15) - rho * usq * (2 / 3), 0.0
            else:
                ese = sum(e[a] * e[c] * s[a, c] for a in range(3) for c in range(3) if e[a] * e[c])
                w = 1.0 if i <= 6 else 1 / 8
                feq = drho / 30 + rho * (w * eu / 3 + w * eu * eu / 2 - usq * (1 / 12 if i <= 6 else 1 / 24)) - \
                    0.5 * w * ese
                p = w * eb / 3
            out.append(-(f[i] - feq) / self.tau_f + p)
        return out

    def stream(self, g):
        out = []
        for i, e in enumerate(E):
            v = torch.roll(g[i], (e[0], e[1], e[2]), (-1, -2, -3))
            if self.mode == "walls" and e[2]:
                at = 0 if e[2] > 0 else -1
                v = v.clone()
                v[..., at, :, :] = g[OPP[i]][..., at, :, :]
            out.append(v)
        return out

    def lb(self, f, s, b):
        C = self.collide(f, s, b)
        half = self.stream([x + 0.5 * c for x, c in zip(f, C)])
        pred = self.stream([x + c for x, c in zip(f, C)])
        return [x + 0.5 * c for x, c in zip(half, self.collide(pred, s, b))]

    def step(self, q, f):
        dq = self.grads(q)
        h = self.field(q, dq)
        u = None
        if f is not None:
            u = _moments(f)[1]
            s, tau = self.stress(q, h)
            f = self.lb(f, s, self.force(h, dq, tau))
            if self.mode == "gauss_seidel":
                u = _moments(f)[1]
        qs = q + self.rate(q, h, dq, u)
        ds = self.grads(qs)
        return 0.5 * (q + qs + self.rate(qs, self.field(qs, ds), ds, u)), f

    def energy(self, q):
        """Total lattice energy per replica (bond form, so that walls count once)."""
        tr2 = _dd(q, q)
        e = 0.5 * A0 * (1 - self.gamma / 3) * tr2 - A0 * self.gamma / 3 * _dd(_mm(q, q), q) + \
            0.25 * A0 * self.gamma * tr2 * tr2 + 2 * self.K * self.q0 ** 2 * tr2

        def bond(a, b, g):
            d, p = b - a, (g + 1) % 3
            r = (g + 2) % 3  # eps_agd with a = r, d = p is +1: (A:eps_g B) = A_r. B_p. - A_p. B_r.
            chi = ((a[r] * b[p] - a[p] * b[r]) - (b[r] * a[p] - b[p] * a[r])).sum(0)
            return 0.5 * self.K * _dd(d, d) + self.K * self.q0 * chi

        gh = self._ghost(q)
        for g in range(3):
            e = e + bond(q, _nb(q, g, 1, gh), g)
        tot = e.sum(dim=(-1, -2, -3))
        if gh is not None:
            tot = tot + bond(gh[0], q[..., :1, :, :], 2).sum(dim=(-1, -2, -3))
        if self.mode == "l2":
            dq = self.grads(q)
            dv = torch.stack([dq[0][a, 0] + dq[1][a, 1] + dq[2][a, 2] for a in range(3)])
            tot = tot - 0.5 * self.K * (dv * dv).sum(0).sum(dim=(-1, -2, -3))
        return tot

    def equilibrium(self, q, u):
        """f of unit density, velocity u and the stress of q (deviations)."""
        dq = self.grads(q)
        s, _ = self.stress(q, self.field(q, dq))
        f = []
        usq = (u * u).sum(0)
        for i, e in enumerate(E):
            if i == 0:
                f.append(-usq * (2 / 3))
                continue
            eu = sum(c * v for c, v in zip(e, u))
            ese = sum(e[a] * e[c] * s[a, c] for a in range(3) for c in range(3) if e[a] * e[c])
            w = 1.0 if i <= 6 else 1 / 8
            f.append(w * eu / 3 + w * eu * eu / 2 - usq * (1 / 12 if i <= 6 else 1 / 24) - 0.5 * w * ese)
        return f


def _moments(f):
    drho = sum(f)
    j = torch.stack([sum(e[a] * x for e, x in zip(E, f) if e[a]) for a in range(3)])
    return drho, j / (1.0 + drho)


def _model(case):
    gamma, K, q0 = _ldg(case)
    return _Model(gamma, K, q0, case["tau_f"], case["xi"], case["Gamma"], case["mode"])


def _exchange_state(case, seed):
    """Q and full populations an outside program holds (FP32): near equilibrium, with noise."""
    gamma, _, q0 = _ldg(case)
    dims = case["nx"], case["ny"], case["nz"]
    q = _q5(case["init"], *dims, q0, gamma, seed, torch.float32)
    u = _u3(*dims, seed, torch.float64)
    m = _model(case)
    f = m.equilibrium(_q9(q.double()[:, None]), u[:, None])
    f = torch.stack([x[0] + w for x, w in zip(f, REST)])
    f += 1e-4 * (torch.rand(f.shape, generator=_gen(seed + 104729), device="cuda", dtype=torch.float64) - 0.5)
    return q, f.float().contiguous()


def _surrogate_lattice(case):
    return {"dtype": "f32", "mode": "flow", "init": "slab", **BASE, **case}


def _weights():
    """[(W [27, cin, cout], b)] and (steps, s_u, s_r, s_dq) of the shipped network."""
    raw = open(WEIGHTS, "rb").read()
    steps = int(np.frombuffer(raw, "<i4", 1, 8 + 4 * 6)[0])
    su, sr, sdq = np.frombuffer(raw, "<f8", 3, 8 + 4 * 8)
    v = torch.from_numpy(np.frombuffer(raw, "<f4", -1, 8 + 32 + 24 + 8).astype(np.float64)).cuda()
    layers, o = [], 0
    for cin, cout in [(15, 32)] + [(32, 32)] * 8 + [(32, 5)]:
        n = 27 * cin * cout
        layers.append((v[o:o + n].view(27, cin, cout), v[o + n:o + n + cout]))
        o += n + cout
    return layers, steps, float(np.float32(su)), float(np.float32(sr)), float(np.float32(sdq))


def _conv(x, W, b):
    y = b.view(-1, 1, 1, 1).expand(-1, *x.shape[1:]).clone()
    for t in range(27):
        s = torch.roll(x, (1 - t // 9, 1 - t // 3 % 3, 1 - t % 3), (1, 2, 3))
        y = y + (W[t].t() @ s.reshape(s.shape[0], -1)).view(-1, *x.shape[1:])
    return y


def _network(layers, q, u, r, kappa, tau, su, sr):
    one = torch.ones_like(q[:1])
    h = torch.relu(_conv(torch.cat([q, u / su, (kappa - 1) * one, tau * one, r / sr]), *layers[0]))
    for k in range(4):
        h = h + _conv(torch.relu(_conv(h, *layers[1 + 2 * k])), *layers[2 + 2 * k])
    return _conv(h, *layers[9])


def exact(case, seed):
    do = case["do"]
    if do == "train":
        return _exact_train(case, seed)
    with torch.no_grad():
        if do == "sweep":
            return _exact_sweep(case, seed)
        if do == "surrogate":
            return _exact_surrogate(case, seed)
        m = _model(case)
        gamma, _, q0 = _ldg(case)
        dims = case["nx"], case["ny"], case["nz"]
        f = None
        if do == "exchange":
            q5, f15 = _exchange_state(case, seed)
            f = [x.double()[None] - w for x, w in zip(f15, REST)]
        else:
            q5 = _q5(case["init"], *dims, q0, gamma, seed, _state_dtype(case))
        q = _q9(q5.double()[:, None])
        if f is None and _flow(case):
            f = m.equilibrium(q, _u3(*dims, seed, _state_dtype(case)).double()[:, None])
        for _ in range(case["steps"]):
            q, f = m.step(q, f)
        out = {}
        if do == "lattice" and case["log"]:
            out["F"] = float(m.energy(q)[0])
            if f is not None:
                out["mass"] = float((1.0 + _moments(f)[0]).sum())
        out["q"] = _five(q)[:, 0]
        if f is not None:
            out["u"] = _moments(f)[1][:, 0]
        return out


def _exact_sweep(case, seed):
    rs = _sweep(case, seed)
    F, qs = [0.0] * len(rs), [None] * len(rs)
    for n in {r["n"] for r in rs}:
        idx = [i for i, r in enumerate(rs) if r["n"] == n]
        par = [_ldg(rs[i]) for i in idx]
        col = [torch.tensor([p[c] for p in par], device="cuda", dtype=torch.float64).view(-1, 1, 1, 1) for c in range(3)]
        m = _Model(*col, BASE["tau_f"], BASE["xi"], BASE["Gamma"])
        q = _q9(torch.stack([_q5(rs[i]["kind"], n, n, n, p[2], p[0], rs[i]["seed"], torch.float32).double()
                             for i, p in zip(idx, par)], dim=1))
        f = m.equilibrium(q, torch.zeros((3,) + q.shape[2:], device="cuda", dtype=torch.float64))
        for _ in range(case["steps"]):
            q, f = m.step(q, f)
        e = m.energy(q)
        q5 = _five(q)
        for k, i in enumerate(idx):
            F[i], qs[i] = float(e[k]), q5[:, k].contiguous()
    return {"F": np.array(F), "q": qs}


def _exact_surrogate(case, seed):
    lc = _surrogate_lattice(case)
    m = _model(lc)
    gamma, _, q0 = _ldg(lc)
    dims = case["nx"], case["ny"], case["nz"]
    q = _q9(_q5("slab", *dims, q0, gamma, seed, torch.float32).double()[:, None])
    u = _moments(m.equilibrium(q, _u3(*dims, seed, torch.float32).double()[:, None]))[1]
    layers, k, su, sr, sdq = _weights()
    for _ in range(case["calls"]):
        dq = m.grads(q)
        r = _five(m.rate(q, m.field(q, dq), dq, u))
        y = _network(layers, _five(q)[:, 0], u[:, 0], r[:, 0], case["kappa"], case["tau"], su, sr)
        q = _q9(_five(q) + k * r + sdq * y[:, None])
    return {"F": float(m.energy(q)[0]), "q": _five(q)[:, 0]}


def _exact_train(case, seed):
    layers, k, su, sr, sdq = _weights()
    leaves = [(W.clone().requires_grad_(), b.clone().requires_grad_()) for W, b in layers]
    q, u, r, dq, mask = [v.double() for v in _train_fields(case, seed)]
    d = _network(leaves, q, u, r, case["kappa"], case["tau"], su, sr) - (dq - k * r) / sdq
    loss = (mask * d * d).sum() / (5 * mask.sum())
    loss.backward()
    with torch.no_grad():
        g = torch.cat([t.grad.reshape(-1) for pair in leaves for t in pair])
        w = torch.cat([t.reshape(-1) for pair in layers for t in pair])
        # the first Adam step: m / (1 - b1) = g and v / (1 - b2) = g^2
        p = w - 1e-4 * g / (g.abs() + 1e-8)
    return {"loss": float(loss), "grads": g, "params": p}
