"""What a user of this package has it do, as measurable cases.

A pass of a "march" case advances a simulation by `steps` timesteps and reads its densities and
velocity back (`Lbm3.step`, `Lbm3.fields`), as a program does that marches a droplet for tens of
thousands of steps and looks at it now and then; the next pass goes on from there.  A pass of an
"adjoint" case is one evaluation of the centroid objective and its gradient
(`adjoint.centroid` and the backward pass), as in an optimisation over wall angles and inflow.

The set-ups are those of arXiv:2102.04709 Section III (Janus droplet on a flat wall and on a
cylinder, capillary intrusion through a modified periodic seam, compound droplet among pillars
behind a Zou-He inlet), with droplet positions, contact angles and pillars drawn from the seed.
`exact` advances the same inputs with the method written out in 64 bits in plain torch.
"""
import math

import numpy as np
import torch

from paper_2102_04709_gb300 import adjoint, lbm3

STORAGE = {"fp32": lbm3.LBM3_FP32, "fp16": lbm3.LBM3_FP16, "bf16": lbm3.LBM3_BF16}
PERIODIC, SEAM, ZOUHE = 0, 1, 2  # x boundary

MOST_NODES = 4096 * 2048  # of a drawn grid: the largest listed one


def listed():
    return [
        # a small droplet on a wall coupled to another program, which wants it every few steps:
        # the smallest calls, where launches and latency count
        {"name": "coupled_flat_128x64", "kind": "flat", "nx": 128, "ny": 64, "R": 20.0,
         "storage": "fp32", "steps": 8},
        # contact-angle table at the paper's size: one of the runs of 10^5 steps each
        {"name": "flat_320x180", "kind": "flat", "nx": 320, "ny": 180, "R": 80.0,
         "storage": "fp32", "steps": 200},
        # capillary intrusion at the paper's size (an odd width, viscosity contrast)
        {"name": "capillary_450x31", "kind": "capillary", "nx": 450, "ny": 31, "wall": 1,
         "s0": 90, "Lg": 90, "nu0": 0.35, "nu1": 0.0035, "storage": "fp32", "steps": 200},
        # the same in a long, wide channel with thick walls
        {"name": "capillary_2048x128", "kind": "capillary", "nx": 2048, "ny": 128, "wall": 24,
         "s0": 256, "Lg": 256, "nu0": 0.1, "nu1": 0.1, "storage": "fp32", "steps": 200},
        # Janus droplet on a cylinder in a periodic box, the standard size
        {"name": "cylinder_512x512", "kind": "cylinder", "nx": 512, "ny": 512, "Rs": 60.0,
         "Rj": 50.0, "storage": "fp32", "steps": 200},
        # compound droplet through five pillars, the paper's size
        {"name": "pillars_800x375", "kind": "pillars", "nx": 800, "ny": 375, "count": 5,
         "r_lo": 36.0, "r_hi": 40.0, "core": 30.0, "shell": 50.0, "nu": 0.163, "u_in": 0.00245,
         "storage": "fp32", "steps": 200},
        # a ragged channel of pillars: no dimension is a multiple of a vector or a tile
        {"name": "pillars_1030x517", "kind": "pillars", "nx": 1030, "ny": 517, "count": 24,
         "r_lo": 10.0, "r_hi": 30.0, "core": 40.0, "shell": 70.0, "nu": 0.1, "u_in": 0.004,
         "storage": "fp32", "steps": 200},
        # reduced storage, brain floats, on a grid of medium size
        {"name": "pillars_2048x1024_bf16", "kind": "pillars", "nx": 2048, "ny": 1024, "count": 60,
         "r_lo": 20.0, "r_hi": 40.0, "core": 60.0, "shell": 100.0, "nu": 0.04, "u_in": 0.01,
         "storage": "bf16", "steps": 200},
        # the largest standard grid: sixty pillars, full and reduced storage
        {"name": "pillars_4096x2048", "kind": "pillars", "nx": 4096, "ny": 2048, "count": 60,
         "r_lo": 40.0, "r_hi": 80.0, "core": 120.0, "shell": 200.0, "nu": 0.04, "u_in": 0.01,
         "storage": "fp32", "steps": 256},
        {"name": "pillars_4096x2048_fp16", "kind": "pillars", "nx": 4096, "ny": 2048, "count": 60,
         "r_lo": 40.0, "r_hi": 80.0, "core": 120.0, "shell": 200.0, "nu": 0.04, "u_in": 0.01,
         "storage": "fp16", "steps": 256},
        # gradient of the droplet's position with respect to every wall node's angles, every
        # state kept
        {"name": "adjoint_512x256", "kind": "adjoint", "nx": 512, "ny": 256, "count": 6,
         "r_lo": 20.0, "r_hi": 40.0, "core": 30.0, "shell": 50.0, "nu": 0.04, "u_in": 0.01,
         "storage": "fp32", "steps": 200, "every": 200},
        # the same on a small ragged grid, states recomputed from checkpoints
        {"name": "adjoint_250x125", "kind": "adjoint", "nx": 250, "ny": 125, "count": 3,
         "r_lo": 10.0, "r_hi": 18.0, "core": 15.0, "shell": 25.0, "nu": 0.04, "u_in": 0.01,
         "storage": "fp32", "steps": 100, "every": 25},
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def fp():
        return rng.choice(["fp32", "fp32", "fp16", "bf16"])

    kind = rng.choice(["flat", "capillary", "cylinder", "pillars", "pillars", "adjoint"])
    steps = size(8, 256)
    if kind == "flat":
        ny = size(48, 512)
        nx = max(96, int(ny * rng.uniform(1.5, 2.5)))
        return {"kind": kind, "nx": nx, "ny": ny, "R": round(0.3 * ny, 1), "storage": fp(), "steps": steps}
    if kind == "capillary":
        nx = size(160, 2048)
        ny = size(31, 192)
        return {"kind": kind, "nx": nx, "ny": ny, "wall": rng.randint(1, max(1, ny // 5)), "s0": nx // 5,
                "Lg": nx // 5, "nu0": 0.1, "nu1": round(rng.uniform(0.01, 0.1), 3), "storage": fp(), "steps": steps}
    if kind == "cylinder":
        n = size(96, 1024)
        ny = max(96, int(n * rng.uniform(0.8, 1.2)))
        m = min(n, ny)
        return {"kind": kind, "nx": n, "ny": ny, "Rs": round(0.12 * m, 1), "Rj": round(0.1 * m, 1),
                "storage": fp(), "steps": steps}
    ny = size(96, 320) if kind == "adjoint" else size(96, 1600)
    nx = int(ny * rng.uniform(1.8, 2.4))
    nx = min(nx, MOST_NODES // ny)
    case = {"kind": kind, "nx": nx, "ny": ny, "count": rng.randint(2, 24), "r_lo": round(0.04 * ny, 1),
            "r_hi": round(0.08 * ny, 1), "core": round(0.08 * ny, 1), "shell": round(0.14 * ny, 1),
            "nu": round(rng.uniform(0.04, 0.16), 3), "u_in": round(rng.uniform(0.002, 0.008), 4),
            "storage": "fp32" if kind == "adjoint" else fp(), "steps": steps}
    if kind == "adjoint":
        case["steps"] = min(steps, 150)
        case["every"] = rng.choice([case["steps"], max(1, case["steps"] // 4), 16])
    return case


# ---- inputs ---------------------------------------------------------------------------------
def scene(case, seed):
    """Geometry, wall angles, initial densities and parameters of a case, from the seed."""
    g = np.random.default_rng(seed)
    nx, ny = case["nx"], case["ny"]
    x = np.arange(nx, dtype=np.float64)[None, :]
    y = np.arange(ny, dtype=np.float64)[:, None]
    solid = np.zeros((ny, nx), np.uint8)
    label = np.zeros((ny, nx), np.uint8)  # fluid by node
    s = {"nx": nx, "ny": ny, "per_y": 1, "bc_x": PERIODIC, "sigma": (0.01, 0.01, 0.01), "u_in": 0.0,
         "nu": (1.0 / 6.0,) * 3}
    t = float(g.uniform(-5.0, 5.0))  # contact angles jittered by up to 5 degrees
    if case["kind"] == "flat":
        s["per_y"] = 0
        solid[0] = solid[-1] = 1
        cx, R = nx / 2.0 + g.uniform(-2.0, 2.0), case["R"]
        inside = (x - cx) ** 2 + (y - 0.5) ** 2 < R * R
        label[:] = 1
        label[inside & (x < cx)] = 0
        label[inside & (x >= cx)] = 2
        # equal tensions: the three cosines sum to 0 (Eq.18)
        rg, br = 90.0 + t, 60.0 + float(g.uniform(-5.0, 5.0))
        gb = math.degrees(math.acos(-math.cos(math.radians(rg)) - math.cos(math.radians(br))))
        triple = (rg, br, gb)
    elif case["kind"] == "capillary":
        s["per_y"], s["bc_x"] = 0, SEAM
        w = case["wall"]
        solid[:w] = solid[ny - w:] = 1
        s0 = case["s0"] + int(g.integers(-4, 5))
        label[:] = 2
        label[:, :s0] = 0
        label[:, s0:s0 + case["Lg"]] = 1
        s["nu"] = (case["nu0"], case["nu1"], case["nu0"])
        triple = (90.0, 135.0 - t, 45.0 + t)
    elif case["kind"] == "cylinder":
        cx, cy = nx / 2.0 + g.uniform(-2.0, 2.0), ny / 2.0 + g.uniform(-2.0, 2.0)
        Rs, Rj = case["Rs"], case["Rj"]
        solid[(x - cx) ** 2 + (y - cy) ** 2 <= Rs * Rs] = 1
        inside = (x - cx) ** 2 + (y - cy - Rs) ** 2 < Rj * Rj
        label[:] = 1
        label[inside & (x < cx)] = 0
        label[inside & (x >= cx)] = 2
        s["sigma"] = (0.01, 0.005, 0.01)
        triple = (60.0 + t, 90.0, 120.0 - t)
    else:
        if case["kind"] == "adjoint":  # an optimisation keeps its geometry: the angles differ
            g = np.random.default_rng(nx * ny + case["count"])
        core, shell = case["core"], case["shell"]
        dx, dy = 1.2 * shell + 8.0, ny / 2.0 + g.uniform(-4.0, 4.0)
        s["bc_x"], s["u_in"], s["nu"] = ZOUHE, case["u_in"], (case["nu"],) * 3
        discs = []
        if case["kind"] == "adjoint":  # the first pillar stands in the shell's front: it is wetted
            r = g.uniform(case["r_lo"], case["r_hi"])
            discs.append((dx + shell + r - 0.15 * shell, dy + g.uniform(-0.3, 0.3) * shell, r))
        lo, hi = dx + shell + case["r_hi"] + 4.0, nx - 8.0 - case["r_hi"]
        for _ in range(200 * case["count"]):
            if len(discs) >= case["count"] or hi <= lo:
                break
            r, cx, cy = g.uniform(case["r_lo"], case["r_hi"]), g.uniform(lo, hi), g.uniform(0.0, ny)
            gaps = [math.hypot(cx - a, min(abs(cy - b), ny - abs(cy - b))) - r - q for a, b, q in discs]
            if all(d >= 6.0 for d in gaps):
                discs.append((cx, cy, r))
        for cx, cy, r in discs:
            rows = np.arange(math.floor(cy - r), math.ceil(cy + r) + 1)
            cols = np.arange(math.floor(cx - r), math.ceil(cx + r) + 1)
            hit = (cols[None, :] - cx) ** 2 + (rows[:, None] - cy) ** 2 <= r * r
            rr, cc = np.nonzero(hit)
            solid[rows[rr] % ny, cols[cc]] = 1
        d2 = (x - dx) ** 2 + (y - dy) ** 2
        label[:] = 2
        label[d2 < shell * shell] = 1
        label[d2 < core * core] = 0
        triple = (90.0, 90.0 - t, 90.0 + t)
    rho = np.zeros((3, ny, nx))
    for k in range(3):
        rho[k][(label == k) & (solid == 0)] = 1.0
    angles = np.empty((ny, nx, 3))
    angles[...] = np.float32(triple)
    if case["kind"] == "adjoint":
        # every wall node has its own angle, and the densities are not exactly those of pure
        # fluids (there the gradient has a kink)
        g = np.random.default_rng(seed)
        th = g.uniform(60.0, 120.0, (ny, nx)).astype(np.float32)
        angles[..., 0], angles[..., 1], angles[..., 2] = 90.0, 180.0 - th, th
        rho *= 1.0 + 1e-6 * g.standard_normal(rho.shape)
    s.update(solid=solid, rho=rho, angles=angles)
    return s


def prepare(case, seed):
    s = scene(case, seed)
    sim = lbm3.Lbm3(s["nx"], s["ny"], s["per_y"], s["bc_x"], s["solid"], s["angles"], s["sigma"], s["nu"],
                    u_in=s["u_in"], precision=STORAGE[case["storage"]])
    if case["kind"] == "adjoint":
        wall = s["angles"].reshape(-1, 3)[sim.wall_nodes()]
        return {"sim": sim, "steps": case["steps"], "every": case["every"], "rho": s["rho"],
                "angles": torch.tensor(wall, dtype=torch.float32, device="cuda"),
                "u_in": torch.tensor(s["u_in"], dtype=torch.float32, device="cuda")}
    sim.set_fields(s["rho"])
    return {"sim": sim, "steps": case["steps"]}


def run(state):
    sim = state["sim"]
    if "every" in state:
        angles = state["angles"].detach().requires_grad_()
        u_in = state["u_in"].detach().requires_grad_()
        J = adjoint.centroid(sim, angles, u_in, state["rho"], state["steps"], state["every"])
        g_angles, g_u = torch.autograd.grad(J, (angles, u_in))
        return {"J": J.float(), "dJ_dangles": g_angles, "dJ_du": g_u}
    sim.step(state["steps"])
    rho, u = sim.fields()
    # the populations are single precision (or less): so are the snapshots that are kept
    return {"rho": torch.from_numpy(rho).float(), "u": torch.from_numpy(u).float()}


def work(case):
    """A timestep reads and writes the nine populations of every fluid that a node holds: of one
    fluid far from the droplets, of all three in and around them; in the reduced storage a density
    in 32 bits and eight 16-bit numbers per fluid.  An adjoint step reads and writes the 27 adjoint
    populations besides and reads the stored state.  Per node and step about 300 operations
    forwards, three times that backwards."""
    n = case["nx"] * case["ny"]
    if case["kind"] == "flat":
        fluid, mixed = n - 2 * case["nx"], 0.5 * math.pi * (case["R"] + 12) ** 2
    elif case["kind"] == "capillary":
        fluid = case["nx"] * (case["ny"] - 2 * case["wall"])
        mixed = 3 * 24 * (case["ny"] - 2 * case["wall"])
    elif case["kind"] == "cylinder":
        fluid, mixed = n - math.pi * case["Rs"] ** 2, math.pi * (case["Rj"] + 12) ** 2
    else:
        r2 = (case["r_lo"] ** 2 + case["r_lo"] * case["r_hi"] + case["r_hi"] ** 2) / 3
        fluid, mixed = n - case["count"] * math.pi * r2, math.pi * (case["shell"] + 12) ** 2
    mixed = min(mixed, fluid)
    one = 2 * 36 if case["storage"] == "fp32" else 2 * 20  # bytes of one fluid at a node, in and out
    step = one * (fluid + 2 * mixed)
    if case["kind"] == "adjoint":
        step += fluid * 4 * (27 + 2 * 27) + n * 16
        return {"bytes": step * case["steps"] + 24 * n, "flops": 1200 * fluid * case["steps"]}
    return {"bytes": step * case["steps"] + 5 * 8 * n, "flops": 300 * fluid * case["steps"]}


# ---- the method in 64 bits --------------------------------------------------------------------
EX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
EY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
WQ = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4
OPP = (0, 3, 4, 1, 2, 7, 8, 5, 6)
PAIRS = ((0, 1), (0, 2), (1, 2))


class Method:
    """Eq.(1)-(22) of the paper on [k, a, y, x] tensors of doubles; every operation can be
    differentiated."""

    def __init__(self, s, dev):
        def as_t(v, dtype=torch.float64):
            return torch.as_tensor(np.ascontiguousarray(v), device=dev).to(dtype)

        self.s, self.dev, self.nx, self.ny = s, dev, s["nx"], s["ny"]
        self.solid = as_t(s["solid"], torch.bool)
        self.fluid = ~self.solid
        # node classes (C_SB: solid with a fluid neighbour), with what lies beyond the grid: solid
        # behind a wall side, the boundary column behind an open one
        self.Sp = self.pad(self.solid, 2, outside=True)
        touch = torch.zeros_like(self.solid)
        for a in range(1, 9):
            touch |= ~self.at(self.Sp, 2, EX[a], EY[a])
        self.wall = self.solid & touch
        self.valued = self.pad(self.fluid | self.wall, 2, outside=False)
        self.P = torch.nonzero(self.wall.reshape(-1)).reshape(-1)
        self.px, self.py = self.P % self.nx, self.P // self.nx
        # outward normals, Eq.(19)-(20); D2Q9 weights where those cancel
        w8 = {1: 4 / 21, 2: 4 / 45, 4: 1 / 60, 5: 2 / 315, 8: 1 / 5040}
        nrm = torch.zeros(2, self.ny, self.nx, dtype=torch.float64, device=dev)
        alt = torch.zeros_like(nrm)
        for cy in range(-2, 3):
            for cx in range(-2, 3):
                c2 = cx * cx + cy * cy
                sol = self.at(self.Sp, 2, cx, cy).double()
                d9 = {1: 1 / 9, 2: 1 / 36}.get(c2, 0.0)
                for j, c in enumerate((cx, cy)):
                    nrm[j] += w8.get(c2, 0.0) * c * sol
                    alt[j] += d9 * c * sol
        small = nrm.norm(dim=0) < 1e-12
        nrm = torch.where(small, alt, nrm)
        none = nrm.norm(dim=0) < 1e-12
        nrm[0][none], nrm[1][none] = 0.0, -1.0
        nrm = -nrm / nrm.norm(dim=0)
        self.n = nrm.reshape(2, -1)[:, self.P]
        e2 = [EX[a] ** 2 + EY[a] ** 2 for a in range(9)]
        rows = [[1] * 9, [-4 + 3 * q for q in e2], [4 - 10.5 * q + 4.5 * q * q for q in e2], EX,
                [EX[a] * (3 * e2[a] - 5) for a in range(9)], EY, [EY[a] * (3 * e2[a] - 5) for a in range(9)],
                [EX[a] ** 2 - EY[a] ** 2 for a in range(9)], [EX[a] * EY[a] for a in range(9)]]
        self.M = torch.tensor(rows, dtype=torch.float64, device=dev)
        self.Mi = torch.linalg.inv(self.M.cpu()).to(dev)
        self.nu = s["nu"]
        self.sig = dict(zip(PAIRS, s["sigma"]))
        s01, s02, s12 = s["sigma"]

        def gfun(X):
            X = max(-1.0, min(1.0, X))
            r = math.sqrt(1.0 - X * X)
            return 1.0 - r if X < 0 else r - 1.0

        self.g = {(0, 1): gfun((s02 ** 2 + s12 ** 2 - s01 ** 2) / (2 * s02 * s12)),
                  (0, 2): gfun((s01 ** 2 + s12 ** 2 - s02 ** 2) / (2 * s01 * s12)),
                  (1, 2): gfun((s01 ** 2 + s02 ** 2 - s12 ** 2) / (2 * s01 * s02))}
        self.w = torch.tensor(WQ, dtype=torch.float64, device=dev)
        self.ex = torch.tensor(EX, dtype=torch.float64, device=dev)
        self.ey = torch.tensor(EY, dtype=torch.float64, device=dev)

    def pad(self, v, p, outside=None, swap=False):
        """v with p rows and columns more on every side, as the boundaries continue it; `outside`:
        its value behind a wall side; swap: fluids 0 and 2 (first dimension) change places across
        the modified periodic seam."""
        nx, ny = self.nx, self.ny
        iy = torch.arange(-p, ny + p, device=self.dev)
        ix = torch.arange(-p, nx + p, device=self.dev)
        iy = iy % ny if self.s["per_y"] else iy.clamp(0, ny - 1)
        ix = ix.clamp(0, nx - 1) if self.s["bc_x"] == ZOUHE else ix % nx
        r = v.index_select(-2, iy).index_select(-1, ix)
        if swap and self.s["bc_x"] == SEAM:
            other = torch.tensor([2, 1, 0], device=self.dev)
            r = torch.cat([r[..., :p].index_select(0, other), r[..., p:-p], r[..., -p:].index_select(0, other)], -1)
        if outside is not None and not self.s["per_y"]:
            r[..., :p, :] = outside
            r[..., -p:, :] = outside
        return r

    def at(self, v, p, cx, cy, more=0):
        """The padded v seen from (x + cx, y + cy), on the grid and `more` nodes around it."""
        b = p - more
        return v[..., b + cy:v.shape[-2] - b + cy, b + cx:v.shape[-1] - b + cx]

    # -- wetting
    def look(self, C, k, X, Y):
        """C_k at unwrapped fluid positions."""
        swap = (torch.div(X, self.nx, rounding_mode="floor") % 2 == 1) if self.s["bc_x"] == SEAM else torch.zeros_like(X, dtype=torch.bool)
        return C.reshape(-1)[torch.where(swap, 2 - k, k) * (self.nx * self.ny) + (Y % self.ny) * self.nx + X % self.nx]

    def is_fluid(self, X, Y):
        ok = torch.ones_like(X, dtype=torch.bool)
        if not self.s["per_y"]:
            ok &= (Y >= 0) & (Y < self.ny)
        if self.s["bc_x"] == ZOUHE:
            ok &= (X >= 0) & (X < self.nx)
        return ok & self.fluid.reshape(-1)[(Y % self.ny) * self.nx + X % self.nx]

    def mean(self, C):
        """w-weighted mean of the fluid neighbours of every C_SB node, [3, wall]."""
        num, den = 0.0, 0.0
        for a in range(1, 9):
            X, Y = self.px + EX[a], self.py + EY[a]
            w = WQ[a] * self.is_fluid(X, Y).double()
            num = num + torch.stack([w * self.look(C, torch.full_like(X, k), X, Y) for k in range(3)])
            den = den + w
        return torch.where(den > 0, num / den.clamp(min=1e-300), 0.0)

    def march(self, px, py, dx, dy):
        """First crossing of each line with fluid nodes on both sides: (kind, X, Y): 0 none, 1 node,
        2 vertical grid line X above node Y, 3 horizontal grid line Y right of node X."""
        inf = torch.full_like(dx, math.inf)
        sx = torch.where(dx > 0, 1, -1)
        sy = torch.where(dy > 0, 1, -1)
        X, Y = px + sx, py + sy
        useX, useY = dx.abs() > 1e-14, dy.abs() > 1e-14
        tX = torch.where(useX, (X - px) / dx, inf)
        tY = torch.where(useY, (Y - py) / dy, inf)
        kind = torch.zeros_like(px)
        hx, hy = px.clone(), py.clone()
        done = torch.zeros_like(px, dtype=torch.bool)
        for _ in range(64):
            t = torch.minimum(tX, tY)
            done = done | ~(t <= 16.0)
            if bool(done.all()):
                break
            onX, onY = (tX - t) <= 1e-6, (tY - t) <= 1e-6
            s = torch.where(onX, py + t * dy, px + t * dx)
            s = torch.where(done, torch.zeros_like(s), s)
            sr, s0 = torch.floor(s + 0.5).long(), torch.floor(s).long()
            both = onX & onY
            hit = ((s - sr).abs() < 1e-6) & ~both
            nX = torch.where(both, X, torch.where(onX, X, sr))
            nY = torch.where(both, Y, torch.where(onX, sr, Y))
            aX, aY = torch.where(onX, X, s0), torch.where(onX, s0, Y)
            bX, bY = torch.where(onX, X, s0 + 1), torch.where(onX, s0 + 1, Y)
            node = (both | hit) & self.is_fluid(nX, nY)
            edge = ~(both | hit) & self.is_fluid(aX, aY) & self.is_fluid(bX, bY)
            new = (node | edge) & ~done
            kind = torch.where(new, torch.where(node, 1, torch.where(onX, 2, 3)), kind)
            hx = torch.where(new, torch.where(node, nX, aX), hx)
            hy = torch.where(new, torch.where(node, nY, aY), hy)
            done = done | new
            X, Y = torch.where(onX, X + sx, X), torch.where(onY, Y + sy, Y)
            tX = torch.where(useX, (X - px) / dx, inf)
            tY = torch.where(useY, (Y - py) / dy, inf)
        return kind, hx, hy

    def wet(self, C, Cw, ang):
        """Eq.(21)-(22): the wall values of this step from those of the last one."""
        t_rg, t_br, t_gb = ang[:, 0], ang[:, 1], ang[:, 2]

        def local(wm, tm, wl, tl):
            d = wm + wl
            return torch.where(d < 1e-12, 0.5 * (tm + tl), tl + wm / d.clamp(min=1e-12) * (tm - tl))

        th = torch.stack([local(Cw[2], 180.0 - t_br, Cw[1], t_rg), local(Cw[2], t_gb, Cw[0], 180.0 - t_rg)])
        dev = (90.0 - th).abs()
        phi = torch.where(dev < 1e-6, torch.zeros_like(dev), dev * (math.pi / 180.0))
        cs, sn = torch.cos(phi), torch.sin(phi)
        nx, ny = self.n[0], self.n[1]
        fallback = self.mean(C)
        got = []
        for side in (1.0, -1.0):
            dx, dy = cs * nx - side * sn * ny, cs * ny + side * sn * nx
            px, py = self.px.expand_as(dx), self.py.expand_as(dx)
            k = torch.arange(2, device=self.dev)[:, None].expand_as(px)
            with torch.no_grad():
                kind, X, Y = self.march(px.contiguous(), py.contiguous(), dx.detach(), dy.detach())
            s2 = py + (X - px) / torch.where(kind == 2, dx, 1.0) * dy
            s3 = px + (Y - py) / torch.where(kind == 3, dy, 1.0) * dx
            fr = torch.where(kind == 2, s2 - Y, torch.where(kind == 3, s3 - X, torch.zeros_like(s2)))
            ca = self.look(C, k, X, Y)
            cb = self.look(C, k, X + (kind == 3).long(), Y + (kind == 2).long())
            got.append(torch.where(kind == 0, fallback[:2], torch.where(kind == 1, ca, ca + fr * (cb - ca))))
        second = torch.where(th <= 90.0, got[1] > got[0], got[1] < got[0])
        c = torch.where(second, got[1], got[0])
        tot = c[0] + c[1]
        c = torch.where(tot > 1.0, c / torch.where(tot > 1.0, tot, 1.0), c)
        return torch.stack([c[0], c[1], (1.0 - c[0] - c[1]).clamp(min=0.0)])

    # -- one timestep
    def fractions(self, f):
        r = f.sum(1)
        return r, r / torch.where(self.solid, 1.0, r.sum(0))

    def gradients(self, C):
        """Eq.(12) on the grid and one node around it; a C_SB node's missing neighbour is
        extrapolated through it."""
        Cp = self.pad(C, 2, swap=True)
        c0 = self.at(Cp, 2, 0, 0, 1)
        gx, gy = torch.zeros_like(c0), torch.zeros_like(c0)
        for a in range(1, 9):
            here, there = self.at(self.valued, 2, EX[a], EY[a], 1), self.at(self.valued, 2, -EX[a], -EY[a], 1)
            v = torch.where(here, self.at(Cp, 2, EX[a], EY[a], 1),
                            torch.where(there, 2.0 * c0 - self.at(Cp, 2, -EX[a], -EY[a], 1), c0))
            gx = gx + 3.0 * WQ[a] * EX[a] * v
            gy = gy + 3.0 * WQ[a] * EY[a] * v
        return c0, gx, gy

    def zou_he(self, f, U):
        f = f.clone()
        q = f[..., 0].sum(0)
        rho = (q[0] + q[2] + q[4] + 2.0 * (q[3] + q[6] + q[7])) / (1.0 - U)
        h = 0.5 * (q[2] - q[4])
        inl = {1: q[3] + 2.0 / 3.0 * rho * U, 5: q[7] - h + rho * U / 6.0, 8: q[6] + h + rho * U / 6.0}
        for a, v in inl.items():
            f[:, a, :, 0] = torch.stack([torch.zeros_like(v), torch.zeros_like(v), v])
        q = f[..., -1].sum(0)
        ux = -1.0 + q[0] + q[2] + q[4] + 2.0 * (q[1] + q[5] + q[8])
        h = 0.5 * (q[2] - q[4])
        out = {3: q[1] - 2.0 / 3.0 * ux, 7: q[5] + h - ux / 6.0, 6: q[8] - h - ux / 6.0}
        part = f[:, [0, 1, 2, 4, 5, 8], :, -1].sum(1)
        for a, v in out.items():
            f[:, a, :, -1] = v * part / part.sum(0)
        return f

    def start(self, rho, U):
        f = self.w[None, :, None, None] * rho[:, None]
        if self.s["bc_x"] == ZOUHE:
            f = self.zou_he(f, U)
        return f, self.mean(self.fractions(f)[1])

    def step(self, f, Cw, ang, U):
        r, C = self.fractions(f)
        if len(self.P):
            Cw = self.wet(C, Cw, ang)
            C = C.reshape(3, -1).index_copy(1, self.P, Cw).reshape(C.shape)
        c0, gx, gy = self.gradients(C)
        rp = self.pad(torch.where(self.solid, C, r), 1, swap=True)  # rho := 1 at solid nodes
        T = [0.0, 0.0, 0.0]
        normal = {}
        for k, l in PAIRS:
            Gx, Gy = c0[l] * gx[k] - c0[k] * gx[l], c0[l] * gy[k] - c0[k] * gy[l]
            G2 = Gx * Gx + Gy * Gy
            some = G2 > 1e-24
            Gn = torch.sqrt(torch.where(some, G2, 1.0))
            s = torch.where(some, self.sig[k, l] * (1e6 * rp[k] * rp[l]).clamp(max=1.0) / Gn, 0.0)
            T = [T[0] + s * Gy * Gy, T[1] - s * Gx * Gy, T[2] + s * Gx * Gx]
            normal[k, l] = tuple(self.at(torch.where(some, G / Gn, 0.0), 1, 0, 0) for G in (Gx, Gy))
        Fx, Fy = 0.0, 0.0
        for a in range(1, 9):
            xx, xy, yy = (self.at(t, 1, EX[a], EY[a]) for t in T)
            Fx = Fx + 3.0 * WQ[a] * (xx * EX[a] + xy * EY[a])
            Fy = Fy + 3.0 * WQ[a] * (xy * EX[a] + yy * EY[a])
        zero = torch.zeros_like(Fx)
        Fx, Fy = torch.where(self.fluid, Fx, zero), torch.where(self.fluid, Fy, zero)
        # Eq.(1)-(9), (11)
        t = f.sum(0)
        rho = torch.where(self.solid, 1.0, r.sum(0))
        ex, ey, w = self.ex[:, None, None], self.ey[:, None, None], self.w[:, None, None]
        ux = ((t * ex).sum(0) + 0.5 * Fx) / rho
        uy = ((t * ey).sum(0) + 0.5 * Fy) / rho
        eu = ex * ux + ey * uy
        feq = rho * w * (1.0 + 3.0 * eu + 4.5 * eu * eu - 1.5 * (ux * ux + uy * uy))
        Ft = w * ((3.0 * (ex - ux) + 9.0 * eu * ex) * Fx + (3.0 * (ey - uy) + 9.0 * eu * ey) * Fy)
        inv = sum(r[k] / self.nu[k] for k in range(3))
        s1 = 1.0 / (0.5 + 3.0 / torch.where(self.solid, 1.0, inv))
        s4 = 8.0 * (2.0 - s1) / (8.0 - s1)
        S = torch.stack([zero, s1, s1, zero, s4, zero, s4, s1, s1])
        m = -S * torch.tensordot(self.M, t - feq, 1) + (1.0 - 0.5 * S) * torch.tensordot(self.M, Ft, 1)
        t = t + torch.tensordot(self.Mi, m, 1)
        # Eq.(13)-(15)
        trip = (35.0 * r[0] * r[1] * r[2] / rho ** 3).clamp(max=1.0)
        V = [[0.0, 0.0], [0.0, 0.0], [0.0, 0.0]]
        for k, l in PAIRS:
            b = 0.7 * (1.0 + trip * self.g[k, l]) * r[k] * r[l] / rho
            for j in range(2):
                V[k][j] = V[k][j] + b * normal[k, l][j]
                V[l][j] = V[l][j] - b * normal[k, l][j]
        out = torch.stack([r[k] / rho * t + w * (V[k][0] * ex + V[k][1] * ey) for k in range(3)])
        out = torch.where(self.fluid, out, 0.0)
        # Eq.(16) with halfway bounce-back
        op = self.pad(out, 1, swap=True)
        new = torch.stack([torch.where(self.at(self.Sp, 2, -EX[a], -EY[a]), out[:, OPP[a]],
                                       self.at(op[:, a], 1, -EX[a], -EY[a])) for a in range(9)], 1)
        new = torch.where(self.fluid, new, 0.0)
        if self.s["bc_x"] == ZOUHE:
            new = self.zou_he(new, U)
        return new, Cw, torch.where(self.fluid, torch.stack([ux, uy]), 0.0)


def exact(case, seed):
    s = scene(case, seed)
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    m = Method(s, dev)
    rho = torch.as_tensor(s["rho"], device=dev)
    ang = torch.as_tensor(s["angles"].reshape(-1, 3), device=dev)[m.P]
    U = torch.tensor(float(np.float32(s["u_in"])), dtype=torch.float64, device=dev)
    if case["kind"] == "adjoint":
        from torch.utils.checkpoint import checkpoint
        ang.requires_grad_()
        U.requires_grad_()
        f, Cw = m.start(rho, U)
        for _ in range(case["steps"]):
            f, Cw, _u = checkpoint(m.step, f, Cw, ang, U, use_reentrant=False)
        r0 = f[0].sum(0)
        J = (torch.arange(m.nx, device=dev) * r0).sum() / r0.sum()
        g = torch.autograd.grad(J, (ang, U))
        return {"J": J.detach(), "dJ_dangles": g[0], "dJ_du": g[1]}
    with torch.no_grad():
        f, Cw = m.start(rho, U)
        u = None
        for _ in range(case["steps"]):
            f, Cw, u = m.step(f, Cw, ang, U)
        return {"rho": m.fractions(f)[0], "u": u}
