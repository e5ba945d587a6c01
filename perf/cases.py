"""Timed workloads of the two-phase lattice Boltzmann library, called through its public C ABI.

Every case but the last advances lattices by a number of time steps in caller-owned
device memory and returns the whole state at the new time, as the caller's memory
holds it (interior columns of the buffer of that time): the colour densities (with
16-bit storage also the split form's node scalars) and the 16 deviation planes.

A case is a dict:
  kind    "single" (lbm_step on one lattice), "sweep" (one batch of `members`
          equal lattices), "uneven" (one batch of unequal lattices), "channels"
          (one batch of open channels of mixed storage), "diagnose" (read-backs)
  flow    start state and walls: "bubble" and "square" periodic, "wave" heavy over
          light between walls, "slug" gas bubbles in a channel driven by gravity,
          "drops" bubbles in a moving liquid between walls, "wet" a drop on a wall
          with a contact angle, "open" velocity inlet and pressure outlet
  nx, ny, steps, storage ("f32", "f16", "bf16"), mrt (MRT with the Hermite
  equilibrium), gamma (density ratio), visc (dynamic viscosity ratio)
"""
import math

import numpy as np
import torch

from paper_1903_01168_gb300 import lbm as L

STORAGE = {"f32": L.LBM_F32, "f16": L.LBM_F16DEV, "bf16": L.LBM_BF16DEV}
DTYPE = {"f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}
GHOST = 8          # ghost columns on each side of a stored row


def listed():
    one = dict(kind="single", storage="f32", mrt=False, gamma=1.0, visc=1.0)
    return [
        # one small static bubble (the Laplace test): thousands of short steps, latency counts
        dict(one, name="bubble_64", flow="bubble", nx=64, ny=64, steps=200),
        # the resolution study's finest box, run for up to 1.7 million steps
        dict(one, name="square_200", flow="square", nx=200, ny=200, steps=200, gamma=2.5, visc=2.5),
        # Rayleigh-Taylor between walls with gravity, the paper's 140 x 280 box
        dict(one, name="wave_140x280", flow="wave", nx=140, ny=280, steps=100, gamma=1.8),
        # gravity-driven slug train in the long periodic channel, FP32 and 16-bit storage
        dict(one, name="slug_2048x128", flow="slug", nx=2048, ny=128, steps=100, gamma=10.0),
        dict(one, name="slug_2048x128_f16", flow="slug", nx=2048, ny=128, steps=50, gamma=10.0, storage="f16"),
        # MRT with the Hermite equilibrium and its source term, ragged sizes
        dict(one, name="drops_1000x301_mrt", flow="drops", nx=1000, ny=301, steps=50, gamma=10.0, mrt=True),
        # the long open channel of the slug-generation runs
        dict(one, name="open_8192x256", flow="open", nx=8192, ny=256, steps=32, gamma=5.0),
        # the 40-run Laplace sweep as one batch (the benchmark's workload), FP32 and 16-bit
        dict(one, name="sweep_40x256", kind="sweep", flow="bubble", members=40, nx=256, ny=256, steps=50),
        dict(one, name="sweep_40x256_bf16", kind="sweep", flow="bubble", members=40, nx=256, ny=256, steps=32,
             storage="bf16"),
        # uneven ensemble of bubbles and slugs, 64..512 x 64..1024, 16-bit storage
        dict(one, name="uneven_32_f16", kind="uneven", flow="bubble", members=32, nx=512, ny=1024, sizes=1234,
             steps=32, storage="f16"),
        # what a serving loop has active: open channels of all three storage types in one batch
        dict(one, name="channels_8_mixed", kind="channels", flow="open", members=8, nx=8192, ny=256, sizes=1234,
             steps=16, gamma=5.0),
        # read-back between chunks of steps: diagnostics and slug geometry of the long channel
        dict(one, name="diagnose_2048x128", kind="diagnose", flow="slug", nx=2048, ny=128, steps=0, gamma=10.0),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["single"] * 6 + ["sweep", "uneven", "channels", "diagnose"])
    case = dict(kind=kind, storage="f32", mrt=False, gamma=rng.choice([1.0, 2.5, 10.0]), visc=rng.choice([1.0, 10.0]))
    if kind == "single":
        case["flow"] = rng.choice(["bubble", "square", "wave", "slug", "drops", "wet", "open"])
        case["storage"] = rng.choice(["f32", "f32", "f16", "bf16"])
        case["mrt"] = case["flow"] in ("drops", "wave", "wet") and rng.random() < 0.5
        nx = log_int(48, 8192)
        ny = log_int(32, max(40, min(1024, 2100000 // nx)))
        # (16-bit rounding noise grows with the steps: fewer of them there)
        case.update(nx=nx, ny=ny, steps=rng.choice({"bf16": [8, 12], "f16": [16, 32]}.get(
            case["storage"], [16, 32, 50, 100] if nx * ny < 300000 else [16, 32])))
        if case["flow"] == "open":
            case["gamma"] = 5.0
    elif kind == "sweep":
        n = log_int(64, 320)
        case.update(flow="bubble", members=rng.randint(4, 2600000 // (n * n) if n > 230 else 40), nx=n,
                    ny=n + rng.randint(0, 9), steps=rng.choice([16, 32]), storage=rng.choice(["f32", "f16", "bf16"]))
    elif kind == "uneven":
        case.update(flow="bubble", members=rng.randint(4, 32), nx=512, ny=rng.randint(256, 1024), sizes=rng.randint(0, 9999), steps=32,
                    storage=rng.choice(["f32", "f16"]))
    elif kind == "channels":
        case.update(flow="open", members=rng.randint(3, 8), nx=rng.randint(1024, 8192), ny=256, sizes=rng.randint(0, 9999),
                    steps=16, gamma=5.0)
    else:
        case.update(flow="slug", nx=log_int(200, 8192), ny=log_int(32, 256), steps=0, gamma=10.0)
    return case


# ------------------------------------------------------------------ workloads

def members(case, seed):
    """The lattices of a case: dicts with nx, ny, storage, flow, params (lbm_params fields) and the
    numbers its start state is made from."""
    rng, sizes = np.random.default_rng(seed), np.random.default_rng(case.get("sizes", 0))
    out = []
    for k in range(case.get("members", 1)):
        flow, nx, ny, storage, gamma = case["flow"], case["nx"], case["ny"], case["storage"], case["gamma"]
        p = dict(beta=0.7, sigma=0.005, tau_r=0.8, tau_b=0.8)
        m = dict(jitter=rng.uniform(-1.0, 1.0, 24))
        if case["kind"] == "sweep":        # radii x density ratio x viscosity ratio x surface tension
            gamma, visc = (1.0, 10.0)[k // 2 % 2], (1.0, 10.0)[k // 4 % 2]
            p["sigma"] = (0.001, 0.01)[k % 2]
            m["radius"] = (20, 30, 40, 50, 60)[k // 8 % 5] / 256 * min(nx, ny)
            p.update(viscosities(gamma, visc))
        elif case["kind"] == "uneven":     # lattices in multiples of 32, bubbles and slugs
            nx = 32 * int(sizes.integers(2, case["nx"] // 32 + 1))
            ny = 32 * int(sizes.integers(2, case["ny"] // 32 + 1))
            gamma, flow = float(sizes.choice([1.0, 10.0])), str(sizes.choice(["bubble", "slug"]))
        elif case["kind"] == "channels":
            nx = 32 * int(sizes.integers(16, case["nx"] // 32 + 1))
            ny = 32 * int(sizes.integers(2, case["ny"] // 32 + 1))
            storage = ("f32", "f16", "bf16")[k % 3]
        elif flow == "square":
            p.update(viscosities(gamma, case["visc"]), sigma=0.01, beta=0.99 * min(1.0, (60.0 / nx) ** 0.625))
        elif flow == "bubble":
            p.update(viscosities(gamma, case["visc"]))
        if flow == "wave":                 # Re = 420 as in the paper, gravity downwards
            tau = max(0.56, 3 * math.sqrt((ny / 2) ** 3 * 1e-4) / 420 + 0.5)
            p.update(sigma=0.0, gy=-1e-4 * 280 / max(280, ny), tau_r=tau, tau_b=tau, bc_y=L.LBM_BC_WALL)
        elif flow == "slug":               # start speed 0.02 on the centreline
            p.update(gx=8 * 0.1 * 0.02 / ny ** 2, bc_y=L.LBM_BC_WALL)
        elif flow == "drops":
            p.update(tau_r=0.6, tau_b=1.1, sigma=0.01, gx=2e-6, gy=-1e-6, bc_y=L.LBM_BC_WALL)
        elif flow == "wet":                # free slip and a contact angle, as in the open-channel walls
            p.update(sigma=0.01, tau_b=1.0, bc_y=L.LBM_BC_WALL, wall_slip=1,
                     contact_angle=math.radians(90.0 + 40.0 * m["jitter"][0]))
        elif flow == "open":
            p.update(tau_r=0.8, tau_b=0.8, sigma=1e-3, bc_x=L.LBM_BC_INOUT, bc_y=L.LBM_BC_WALL, u_in_r=0.0125,
                     u_in_b=0.025, p_out=0.48, inlet_period_r=40, inlet_period_b=20)
        if case["mrt"]:
            p.update(collision=L.LBM_MRT, equilibrium=L.LBM_EQ_HERMITE)
        p.update(gamma=gamma, storage=STORAGE[storage])
        out.append(dict(m, nx=nx, ny=ny, storage=storage, flow=flow, params=p, smooth=case["kind"] == "diagnose"))
    return out


def viscosities(gamma, visc):
    """Relaxation times with the smaller kinematic viscosity 0.1 and the ratio gamma / visc."""
    r = gamma / visc
    nu_r, nu_b = (0.1, 0.1 * r) if r >= 1 else (0.1 / r, 0.1)
    return dict(tau_r=3 * nu_r + 0.5, tau_b=3 * nu_b + 0.5)


def start_fields(m, device):
    """rho_r, rho_b, ux, uy of a lattice's start state, FP64 (ny, nx) tensors on `device`."""
    nx, ny, j, p = m["nx"], m["ny"], m["jitter"], m["params"]
    gamma = p["gamma"]
    x = torch.arange(nx, dtype=torch.float64, device=device)[None, :]
    y = torch.arange(ny, dtype=torch.float64, device=device)[:, None]
    small = min(nx, ny)

    def disc(cx, cy, r):
        dx, dy = (x - cx).abs(), (y - cy).abs()
        if p.get("bc_x", 0) == L.LBM_BC_PERIODIC:
            dx = torch.minimum(dx, nx - dx)
        if p.get("bc_y", 0) == L.LBM_BC_PERIODIC:
            dy = torch.minimum(dy, ny - dy)
        return r - torch.sqrt(dx * dx + dy * dy)

    ux, uy = torch.zeros(ny, nx, dtype=torch.float64, device=device), torch.zeros(ny, nx, dtype=torch.float64, device=device)
    wall = torch.sin(math.pi * (y + 0.5) / ny)
    flow = m["flow"]
    if flow == "bubble":
        gas = disc(nx / 2 + j[0], ny / 2 + j[1], m.get("radius", small / 4) + j[2])
    elif flow == "square":
        half = 0.165 * nx + 0.02 * nx * j[0]
        gas = half - torch.maximum((x - (nx - 1) / 2 - j[1]).abs(), (y - (ny - 1) / 2 - j[2]).abs() * nx / ny)
    elif flow == "wave":
        gas = ny / 2 - 0.1 * (1 + 0.2 * j[0]) * small * torch.sin(2 * math.pi * (x + 0.5 + 4 * j[1]) / nx) - (y + 0.5)
    elif flow == "wet":
        h = ny * (0.4 + 0.05 * j[1])
        gas = torch.minimum(h - y, nx * 0.25 - (x - nx / 2 - 2 * j[2]).abs() + 0 * y)
        ux = ux + 0.01 * wall * torch.cos(2 * math.pi * x / nx + j[3])
    else:
        n = 2 if flow == "slug" else 5
        gas = torch.full((ny, nx), -1e9, dtype=torch.float64, device=device)
        for b in range(n):
            if flow == "slug":             # elongated bubbles (stadium shape)
                half, r = nx / n * 0.25 * (1 + 0.1 * j[b]), 0.3 * ny * (1 + 0.05 * j[4 + b])
                dx = (x - nx * (b + 0.5) / n - j[8 + b]).abs()
                gap = torch.clamp(torch.minimum(dx, nx - dx) - max(half - r, 0.0), min=0.0)
                gas = torch.maximum(gas, r - torch.sqrt(gap * gap + (y - (ny - 1) / 2) ** 2))
            else:
                gas = torch.maximum(gas, disc(nx * (b + 0.5 + 0.2 * j[b]) / n, ny * (0.5 + 0.15 * j[5 + b]), 0.16 * small))
        if flow == "slug":
            nu = (p["tau_r"] - 0.5) / 3
            ux = ux + p["gx"] / (2 * nu) * (y + 0.5) * (ny - y - 0.5)
        elif flow == "drops":
            ux = ux + 0.02 * wall * torch.sin(2 * math.pi * x / nx + j[10])
            uy = uy + 0.02 * wall * torch.cos(4 * math.pi * x / nx + j[11])
        else:
            ux = ux + 0.0125 * wall
    share, scale = (gas > 0).double(), 1.0
    if m["smooth"]:                        # a diffuse interface, some flow in y and a pressure field
        share = torch.sigmoid(2 * gas / 1.5)
        uy = uy + 0.01 * wall * (1 + 0.5 * torch.cos(2 * math.pi * x / nx + j[12]))
        scale = 1 + 0.05 * torch.exp(-((x - nx / 2) / (0.3 * nx)) ** 2 - ((y - ny / 2) / ny) ** 2)
    return [a.expand(ny, nx).contiguous() for a in (gamma * (1 - share) * scale, share * scale, ux, uy)]


STREAM = []        # the program's one work stream


class State:
    """Simulations on caller-owned memory, all on the program's stream, and their batch."""

    def __init__(self, case, seed):
        self.case, self.ms, self.sims, self.batch = case, members(case, seed), [], 0
        if not STREAM:
            STREAM.append(torch.cuda.Stream())
        with torch.cuda.stream(STREAM[0]):
            ps = [L.make_params(**m["params"]) for m in self.ms]
            sizes = [-(-L.lbm_bytes_required(m["nx"], m["ny"], p) // 256) * 256 for m, p in zip(self.ms, ps)]
            self.memory = torch.zeros(sum(sizes), dtype=torch.uint8, device="cuda")
            self.parts = list(torch.split(self.memory, sizes))
            for m, p, part in zip(self.ms, ps, self.parts):
                h = L.lbm_create_ex(m["nx"], m["ny"], p, part.data_ptr(), part.numel(), STREAM[0].cuda_stream)
                self.sims.append(h)
                L.lbm_init_fields(h, *[f.cpu().numpy() for f in start_fields(m, "cuda")])
        if case["kind"] in ("sweep", "uneven"):
            self.batch = L.lbm_batch_create(self.sims)
        elif case["kind"] == "channels":   # the serving loop's plan
            self.batch = L.lbm_batch_create(self.sims, row_overhead=4.0, plan=L.LBM_PLAN_BALANCED)
        if case["kind"] == "sweep":
            self.views = [state_views(self.memory.view(len(sizes), sizes[0]), self.ms[0])]
        else:
            self.views = [state_views(part[None], m) for m, part in zip(self.ms, self.parts)]

    def __del__(self):
        if self.batch:
            L.lbm_batch_destroy(self.batch)
        for h in self.sims:
            L.lbm_destroy(h)


def state_views(memory, m):
    """Both time buffers of the stored state, (member, buffer, row, plane, column) views of the interior:
    FP32 node planes, then deviation planes."""
    nx, ny = m["nx"], m["ny"]
    scalars = 2 if m["storage"] == "f32" else 5
    pitch = [(nx + 2 * GHOST + 3) // 4 * 4, 0]
    pitch[1] = pitch[0] if m["storage"] == "f32" else (nx + 2 * GHOST + 7) // 8 * 8
    head = 2 * ny * scalars * pitch[0] * 4
    dev = torch.empty(0, dtype=DTYPE[m["storage"]]).element_size()
    at = -(-head // 256) * 256
    rho = memory[:, :head].view(torch.float32).unflatten(1, (2, ny, scalars, pitch[0]))
    pop = memory[:, at:at + 2 * ny * 16 * pitch[1] * dev].view(DTYPE[m["storage"]]).unflatten(1, (2, ny, 16, pitch[1]))
    return rho[..., GHOST:GHOST + nx], pop[..., GHOST:GHOST + nx]


def prepare(case, seed):
    return State(case, seed)


def run(s):
    if s.case["kind"] == "diagnose":
        d = L.lbm_diagnostics(s.sims[0])
        g, gas = L.lbm_slug_geometry(s.sims[0], s.case["nx"])
        return {"diagnostics": d, "slug": g, "gas": gas}
    if s.batch:
        L.lbm_batch_step(s.batch, s.case["steps"])
    else:
        L.lbm_step(s.sims[0], s.case["steps"])
    b = L.lbm_time(s.sims[0]) & 1
    return [(rho[:, b], pop[:, b]) for rho, pop in s.views]


def work(case):
    """Per pass: the state read once and written once (144 bytes a node in FP32; 104 with 16-bit storage),
    about 350 operations per node and step; the read-backs read it once."""
    ms = members(case, 0)
    size = sum(m["nx"] * m["ny"] * (72 if m["storage"] == "f32" else 52) for m in ms)
    nodes = sum(m["nx"] * m["ny"] for m in ms)
    if case["kind"] == "diagnose":
        return {"bytes": size, "flops": 150 * nodes}
    return {"bytes": 2 * size, "flops": 350 * nodes * case["steps"]}


# ------------------------------------------------- the same in 64 bits, in plain torch

CX, CY = (0, 1, 0, -1, 0, 1, -1, -1, 1), (0, 0, 1, 0, -1, 1, 1, -1, -1)
OPP, MIRROR = (0, 3, 4, 1, 2, 7, 8, 5, 6), (0, 1, 4, 3, 2, 8, 7, 6, 5)


def exact(case, seed):
    device = "cuda" if torch.cuda.is_available() else "cpu"
    if case["kind"] == "diagnose":
        return exact_diagnose(members(case, seed)[0], case, device)
    got = [Lattice64(m, device).steps(case["steps"]) for m in members(case, seed)]
    if case["kind"] == "sweep":
        return [(torch.stack([g[0] for g in got]), torch.stack([g[1] for g in got]))]
    return [(g[0][None], g[1][None]) for g in got]


class Lattice64:
    """D2Q9 colour-gradient steps in FP64 (arXiv 1903.01168, Sec. 2)."""

    def __init__(self, m, device):
        self.m, self.nx, self.ny, self.dev = m, m["nx"], m["ny"], device
        p = dict(alpha_b=0.2, delta=0.1, gx=0.0, gy=0.0, u_in_r=0.0, u_in_b=0.0, p_out=0.0, bc_x=0, bc_y=0,
                 wall_slip=0, contact_angle=0.0, collision=0, equilibrium=0)
        p.update(m["params"])
        self.p = p
        alpha = (1 - (1 - p["alpha_b"]) / p["gamma"], p["alpha_b"])
        self.cs2 = [3 * (1 - a) / 5 for a in alpha]
        self.q = [1.8 * a - 0.8 for a in alpha]
        c2 = [x * x + y * y for x, y in zip(CX, CY)]

        def t(v):
            return torch.tensor(v, dtype=torch.float64, device=device)[:, None, None]

        self.phi = [t([a if c == 0 else (1 - a) / (5 if c == 1 else 20) for c in c2]) for a in alpha]
        self.w = t([4 / 9 if c == 0 else 1 / 9 if c == 1 else 1 / 36 for c in c2])
        self.B = t([-4 / 27 if c == 0 else 2 / 27 if c == 1 else 5 / 108 for c in c2])
        self.cx, self.cy, self.c2 = t([float(v) for v in CX]), t([float(v) for v in CY]), t([float(v) for v in c2])
        self.abs_c = torch.sqrt(self.c2)
        self.hermite = p["equilibrium"] == L.LBM_EQ_HERMITE
        self.walls, self.open = p["bc_y"] == L.LBM_BC_WALL, p["bc_x"] == L.LBM_BC_INOUT
        self.t = 0
        rr, rb, ux, uy = start_fields(m, device)
        cu, usq = self.cx * ux + self.cy * uy, ux * ux + uy * uy
        self.N = []
        for k, rho in enumerate((rr, rb)):
            lin = 3 * cu
            if self.hermite:
                lin = 3 * cu * (1 + 0.5 * (3 * self.cs2[k] - 1) * (3 * self.c2 - 4))
            self.N.append(rho * self.phi[k] + rho * self.w * (lin + 4.5 * cu * cu - 1.5 * usq))
        self.zou_he()

    def zou_he(self):
        if not self.open:
            return
        p, (Nr, Nb) = self.p, self.N
        period = p["inlet_period_r"] + p["inlet_period_b"]
        f = 1.0 if self.t % period < p["inlet_period_r"] else 0.0
        n = (Nr + Nb)[:, :, 0]
        h = [3 * c - 1 for c in self.cs2]
        V = f * p["u_in_r"] + (1 - f) * p["u_in_b"]
        rho = (n[0] + n[2] + n[4] + 2 * (n[3] + n[6] + n[7])) / (1 - V)
        H = -rho * (f * h[0] + (1 - f) * h[1]) * V / 3 if self.hermite else 0.0
        new = {1: n[3] + 2 / 3 * rho * V + H, 5: n[7] + 0.5 * (n[4] - n[2]) + rho * V / 6 - 0.5 * H,
               8: n[6] + 0.5 * (n[2] - n[4]) + rho * V / 6 - 0.5 * H}
        for i, v in new.items():
            Nr[i, :, 0], Nb[i, :, 0] = f * v, (1 - f) * v
        kr, kb = [sum(N[i, :, -1] for i in (0, 1, 2, 4, 5, 8)) for N in (Nr, Nb)]
        a = kr / p["gamma"]
        fr = 0.5 * (1 + (a - kb) / (a + kb))
        n = (Nr + Nb)[:, :, -1]
        rho = (1 - fr) * p["p_out"] / self.cs2[1] + fr * p["p_out"] / self.cs2[0]
        V = (n[0] + n[2] + n[4] + 2 * (n[1] + n[5] + n[8]) - rho) / rho
        H = rho * (fr * h[0] + (1 - fr) * h[1]) * V / 3 if self.hermite else 0.0
        new = {3: n[1] - 2 / 3 * rho * V + H, 6: n[8] - 0.5 * (n[2] - n[4]) - rho * V / 6 - 0.5 * H,
               7: n[5] + 0.5 * (n[2] - n[4]) - rho * V / 6 - 0.5 * H}
        for i, v in new.items():
            Nr[i, :, -1], Nb[i, :, -1] = fr * v, (1 - fr) * v

    def pad(self, f, is_psi):
        """f with one node around the domain: periodic, zero gradient in an open x, walls."""
        f = torch.cat([f[:, :1], f, f[:, -1:]], 1) if self.open else torch.cat([f[:, -1:], f, f[:, :1]], 1)
        if not self.walls:
            return torch.cat([f[-1:], f, f[:1]], 0)
        ends = []
        for row in (f[:1], f[-1:]):
            if not is_psi:
                ends.append(torch.zeros_like(row))
                continue
            inner = row[:, 1:-1]
            one = torch.ones_like(inner)

            def spread(v):
                v = torch.nn.functional.pad(v, (2, 2)) if self.open else torch.cat([v[:, -2:], v, v[:, :2]], 1)
                return v[:, 1:-1] / 9 + (v[:, :-2] + v[:, 2:]) / 36

            ends.append(spread(inner) / spread(one))
        return torch.cat([ends[0], f, ends[1]], 0)

    @staticmethod
    def gradient(f):
        gx = (f[1:-1, 2:] - f[1:-1, :-2]) / 3 + (f[2:, 2:] - f[:-2, :-2] + f[:-2, 2:] - f[2:, :-2]) / 12
        gy = (f[2:, 1:-1] - f[:-2, 1:-1]) / 3 + (f[2:, 2:] - f[:-2, :-2] - f[:-2, 2:] + f[2:, :-2]) / 12
        return gx, gy

    def collide(self, last):
        p, (Nr, Nb) = self.p, self.N
        rr, rb = Nr.sum(0), Nb.sum(0)
        rho, N = rr + rb, Nr + Nb
        ux = (self.cx * N).sum(0) / rho + 0.5 * p["gx"]
        uy = (self.cy * N).sum(0) / rho + 0.5 * p["gy"]
        a = rr / p["gamma"]
        psi = (a - rb) / (a + rb)
        wr, wb, d = 1 / p["tau_r"], 1 / p["tau_b"], p["delta"]
        chi = 2 * wr * wb / (wr + wb)
        eta, lam = 2 * (wr - chi) / d, 2 * (chi - wb) / d
        w = torch.where(psi > 0, chi + eta * psi - eta / (2 * d) * psi * psi, chi + lam * psi + lam / (2 * d) * psi * psi)
        w = torch.where(psi > d, torch.full_like(w, wr), torch.where(psi < -d, torch.full_like(w, wb), w))
        Fx, Fy = self.gradient(self.pad(psi, True))
        if p["contact_angle"] > 0 and self.walls:
            Fx, Fy = Fx.clone(), Fy.clone()
            for y, s in ((0, 1.0), (self.ny - 1, -1.0)):
                self.turn(Fx[y], Fy[y], s)
        cu, usq = self.cx * ux + self.cy * uy, ux * ux + uy * uy
        e = N - rr * self.phi[0] - rb * self.phi[1]
        lin = 3 * rho * cu
        if self.hermite:
            h = rr * (3 * self.cs2[0] - 1) + rb * (3 * self.cs2[1] - 1)
            lin = lin + 3 * cu * 0.5 * h * (3 * self.c2 - 4)
        weq = self.w * (lin + rho * (4.5 * cu * cu - 1.5 * usq))
        cG, uG = rho * (self.cx * p["gx"] + self.cy * p["gy"]), rho * (ux * p["gx"] + uy * p["gy"])
        src = self.w * (3 * cG + 9 * cu * cG - 3 * uG)
        if p["collision"] == L.LBM_MRT:
            M = torch.tensor([[1] * 9, [-4, -1, -1, -1, -1, 2, 2, 2, 2], [4, -2, -2, -2, -2, 1, 1, 1, 1],
                              [0, 1, 0, -1, 0, 1, -1, -1, 1], [0, -2, 0, 2, 0, 1, -1, -1, 1],
                              [0, 0, 1, 0, -1, 1, 1, -1, -1], [0, 0, -2, 0, 2, 1, 1, -1, -1],
                              [0, 1, -1, 1, -1, 0, 0, 0, 0], [0, 0, 0, 0, 0, 1, -1, 1, -1]],
                             dtype=torch.float64, device=self.dev)
            s = torch.stack([0.8 * w] * 7 + [w] * 2)
            mm = s * torch.einsum("ab,byx->ayx", M, e - weq) - (1 - 0.5 * s) * torch.einsum("ab,byx->ayx", M, src)
            if self.hermite:
                q = self.q[0] * rr + self.q[1] * rb
                dQx, dQy = self.gradient(self.pad(q * ux, False))[0], self.gradient(self.pad(q * uy, False))[1]
                mm[1] -= 3 * (1 - 0.4 * w) * (dQx + dQy)
                mm[7] -= (1 - 0.5 * w) * (dQx - dQy)
            e = e - torch.einsum("ab,byx->ayx", torch.linalg.inv(M), mm)
        else:
            e = e - w * (e - weq) + (1 - 0.5 * w) * src
        Fn = torch.sqrt(Fx * Fx + Fy * Fy)
        inv = torch.where(Fn > 0, 1 / torch.where(Fn > 0, Fn, torch.ones_like(Fn)), torch.zeros_like(Fn))
        Fc = self.cx * Fx + self.cy * Fy
        E = e + 2.25 * p["sigma"] * w * (self.w * Fc * Fc * inv - self.B * Fn)
        rest = rr * self.phi[0] + rb * self.phi[1]
        mix = rr * rb / rho
        kk = p["beta"] * mix / rho * inv
        shift = mix * (self.phi[1] - self.phi[0]) + kk * Fc / torch.where(self.abs_c > 0, self.abs_c, torch.ones_like(self.abs_c)) * rest
        if not last:
            # the rest direction's flux is zero (Fc = 0), its shift is the mixing part
            self.N = [rr * self.phi[0] + shift + rr / rho * E, rb * self.phi[1] - shift + rb / rho * E]
            return None
        if self.m["storage"] == "f32":
            node, dev = [rr, rb], [shift + rr / rho * E, rb / rho * E - shift]
        else:
            node, dev = [rr, rb, mix, kk * Fx, kk * Fy], [rr / rho * E, rb / rho * E]
        return torch.stack(node, 1), torch.cat([d[1:] for d in dev]).permute(1, 0, 2).contiguous()

    def turn(self, Fx, Fy, s):
        th = self.p["contact_angle"]
        n = torch.sqrt(Fx * Fx + Fy * Fy)
        ux, uy = Fx / n, Fy / n
        tx, ty = math.sin(th), s * math.cos(th)
        d1, d2 = (ux + s * tx) ** 2 + (uy - ty) ** 2, (ux - s * tx) ** 2 + (uy - ty) ** 2
        on = n > 0
        nx_ = torch.where(d1 < d2, -s * tx * n, torch.where(d1 > d2, s * tx * n, torch.zeros_like(n)))
        ny_ = torch.where(d1 == d2, s * n, ty * n)
        Fx.copy_(torch.where(on, nx_, Fx))
        Fy.copy_(torch.where(on, ny_, Fy))

    def stream(self):
        new = []
        for P in self.N:
            Q = torch.stack([torch.roll(P[i], (CY[i], CX[i]), (0, 1)) for i in range(9)])
            if self.walls:
                for i in range(1, 9):
                    if CY[i]:
                        y = 0 if CY[i] > 0 else -1
                        back = P[OPP[i], y]
                        if self.p["wall_slip"]:
                            along = torch.roll(P[MIRROR[i], y], CX[i], 0)
                            if self.open and CX[i]:
                                x = 0 if CX[i] > 0 else -1
                                along[x] = back[x]
                            back = along
                        Q[i, y] = back
            new.append(Q)
        self.N = new
        self.t += 1
        self.zou_he()

    def steps(self, n):
        for k in range(n - 1):
            self.collide(False)
            self.stream()
        return self.collide(True)


def exact_diagnose(m, case, device):
    """The read-backs of a start state, from its fields."""
    nx, ny, p = m["nx"], m["ny"], m["params"]
    rr, rb, ux, uy = start_fields(m, device)
    ux = ux + 0.5 * p["gx"]
    rho, a = rr + rb, rr / p["gamma"]
    psi = (a - rb) / (a + rb)
    wb = 0.5 * (1 - psi)
    x = torch.arange(nx, dtype=torch.float64, device=device)[None, :].expand(ny, nx)
    y = torch.arange(ny, dtype=torch.float64, device=device)[:, None].expand(ny, nx)
    area = wb.sum()
    cx, cy, r = (wb * x).sum() / area, (wb * y).sum() / area, torch.sqrt(area / math.pi)
    dx = (x - cx).abs()
    far = torch.sqrt(torch.minimum(dx, nx - dx) ** 2 + (y - cy) ** 2)
    pr = rr * 0.48 / p["gamma"] + rb * 0.48
    inside, outside = far < r / 2, far > r + 8
    p_in = pr[inside].mean() if bool(inside.any()) else torch.zeros(())
    p_out = pr[outside].mean() if bool(outside.any()) else torch.zeros(())
    d = dict(mass_r=rr.sum(), mass_b=rb.sum(), mom_x=(rho * ux).sum(), mom_y=(rho * uy).sum(), area_b=area,
             max_u=torch.sqrt(ux * ux + uy * uy).max(), cx_b=cx, cy_b=cy, ux_b=(wb * ux).sum() / area,
             ux_r=((1 - wb) * ux).sum() / (1 - wb).sum(), r_eff=r, p_in=p_in, p_out=p_out, dp=p_in - p_out)
    return {"diagnostics": {k: float(v) for k, v in d.items()}, "slug": None, "gas": wb.sum(0)}
