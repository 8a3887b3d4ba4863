"""The workloads whose speed this framework is judged by.

Each case is one call sequence of a user's program on a handle that it keeps: advance the
lattices by a number of steps and read the result (the whole state in its storage format,
and for single lattices the observables the study reports), or one gradient by the discrete
adjoint.  Sizes and parameters are those of ``paper_1707_00198_gb300.inputs``: the paper's
static droplets, cylinder droplets, capillary filling, viscous fingering and wettability
study, the 64-channel batch and the adjoint channel, with the schedules a user of them runs
(the default one; ``autotune`` for the batches).
"""
import math

import numpy as np
import torch

from paper_1707_00198_gb300 import inputs as I

DTYPES = {"fp64": torch.float64, "fp32": torch.float32, "fp16": torch.float16, "bf16": torch.bfloat16}


def listed():
    return [
        # the static droplet on a flat wall, whose steady state the paper checks every 500 steps:
        # the smallest lattice, in the validation precision
        dict(name="droplet_fp64", kind="droplet", nx=100, ny=50, radius=20.0, closed=False, theta=60.0,
             precision="fp64", steps=500),
        # a program that looks at its observables every few steps (a coupling loop, a monitor)
        # on the paper's closed 160 x 100 box: the shortest call
        dict(name="droplet_monitor_fp32", kind="droplet", nx=160, ny=100, radius=45.0, closed=True, theta=120.0,
             precision="fp32", steps=10),
        # a droplet on a cylinder, curved walls with analytic normals
        dict(name="cylinder_fp64", kind="cylinder", nx=200, ny=200, rs=40.0, rd=40.0, theta=60.0, analytic=True,
             precision="fp64", steps=200),
        # capillary filling between two solid blocks, in both precisions it is reported in
        dict(name="capillary_fp64", kind="capillary", length=800, d=40, reservoir=200, wall=20, theta=30.0,
             precision="fp64", steps=100),
        dict(name="capillary_fp32", kind="capillary", length=800, d=40, reservoir=200, wall=20, theta=30.0,
             precision="fp32", steps=200),
        # one point of the viscous-fingering study: FP32 against 16-bit storage
        dict(name="fingering_fp32", kind="channel", width=100, length=2000, M=5.0, Ca=0.05, theta=60.0, profile=0,
             precision="fp32", steps=400),
        dict(name="fingering_fp16", kind="channel", width=100, length=2000, M=5.0, Ca=0.05, theta=60.0, profile=0,
             precision="fp16", steps=400),
        # an odd-sized channel with a Poiseuille inlet
        dict(name="odd_channel_bf16", kind="channel", width=77, length=1013, M=20.0, Ca=0.1, theta=120.0, profile=1,
             precision="bf16", steps=300),
        # the wettability study: eight contact angles as one batch
        dict(name="wettability_fp32", kind="study", width=58, length=630, n=8, precision="fp32", steps=200),
        # the batched parameter sweep: 64 channels of uneven width, state larger than the L2 cache
        dict(name="channels64_fp32", kind="channels", n=64, widths=0, wmin=40, wmax=200, aspect=10,
             precision="fp32", steps=192),
        dict(name="channels64_fp16", kind="channels", n=64, widths=0, wmin=40, wmax=200, aspect=10,
             precision="fp16", steps=192),
        # the adjoint through fingering: gradient of the finger length
        dict(name="adjoint_fp32", kind="adjoint", width=40, length=400, M=10.0, Ca=0.05, theta=60.0,
             precision="fp32", reverse="fp32", steps=800, checkpoint=100),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["droplet", "droplet", "cylinder", "capillary", "channel", "channel", "channel", "study",
                       "channels", "adjoint"])
    theta = rng.choice([30.0, 45.0, 60.0, 90.0, 120.0, 150.0])
    grid = dict(M=rng.choice(I.M_GRID[:3]), Ca=rng.choice(I.CA_GRID), theta=rng.choice(I.THETA_GRID))
    if kind == "droplet":
        ny = _log(rng, 32, 200)
        return dict(kind=kind, nx=2 * ny + rng.randrange(40), ny=ny, radius=round(ny * rng.uniform(0.3, 0.45), 1),
                    closed=rng.random() < 0.5, theta=theta, precision=rng.choice(["fp64", "fp32"]),
                    steps=_log(rng, 8, 400))
    if kind == "cylinder":
        n = _log(rng, 80, 260)
        return dict(kind=kind, nx=n, ny=n + rng.randrange(20), rs=round(0.2 * n, 1), rd=round(0.18 * n, 1),
                    theta=rng.choice([60.0, 90.0, 120.0]), analytic=rng.random() < 0.5,
                    precision=rng.choice(["fp64", "fp32"]), steps=_log(rng, 20, 200))
    if kind == "capillary":
        return dict(kind=kind, length=_log(rng, 200, 800), d=rng.randrange(20, 44), reservoir=rng.randrange(80, 200),
                    wall=rng.randrange(6, 21), theta=rng.choice([30.0, 60.0]),
                    precision=rng.choice(["fp64", "fp32", "fp32", "fp16"]), steps=_log(rng, 20, 150))
    if kind == "channel":
        w = _log(rng, 30, 200)
        return dict(kind=kind, width=w, length=w * rng.randrange(8, 16) + rng.randrange(32), profile=rng.randrange(2),
                    precision=rng.choice(["fp64", "fp32", "fp32", "fp16", "bf16"]), steps=_log(rng, 20, 150), **grid)
    if kind == "study":
        return dict(kind=kind, width=rng.randrange(40, 80), length=rng.randrange(400, 800), n=rng.randrange(2, 9),
                    precision=rng.choice(["fp32", "fp16"]), steps=_log(rng, 20, 100))
    if kind == "channels":
        return dict(kind=kind, n=_log(rng, 4, 24), widths=rng.randrange(1, 1000), wmin=40, wmax=200, aspect=10,
                    precision=rng.choice(["fp32", "fp16", "bf16"]), steps=_log(rng, 20, 100))
    w = rng.randrange(20, 41)
    precision = rng.choice(["fp32", "fp32", "fp64"])
    return dict(kind="adjoint", width=w, length=10 * w + rng.randrange(20), M=10.0, Ca=0.05, theta=60.0,
                precision=precision, reverse=precision, steps=_log(rng, 40, 200), checkpoint=rng.choice([20, 25, 50]))


def _lattices(case, seed):
    """(geometries, parameters) of a case; the seed gives the noise and the interfaces."""
    th = math.radians(case.get("theta", 90.0))
    kind = case["kind"]
    if kind == "droplet":
        return ([I.flat_wall_droplet(case["nx"], case["ny"], R=case["radius"], noise=1e-3, seed=seed,
                                     closed_x=case["closed"])], [I.Params(theta=th)])
    if kind == "cylinder":
        nx, ny, rs = case["nx"], case["ny"], case["rs"]
        return ([I.cylinder_droplet(nx, ny, Rs=rs, cx=nx / 2, cy=1.5 * rs, Rd=case["rd"], theta=th, noise=1e-3,
                                    seed=seed, analytic_normal=case["analytic"])], [I.Params(theta=th)])
    if kind == "capillary":
        return ([I.capillary_filling(L=case["length"], d=case["d"], reservoir=case["reservoir"], wall=case["wall"],
                                     red_into=case["length"] // 8, noise=1e-3, seed=seed)], [I.Params(theta=th)])
    if kind in ("channel", "adjoint"):
        p = I.fingering_params(case["M"], case["Ca"], case["theta"])
        p.inlet_profile = case.get("profile", 0)
        return [I.displacement_channel(W=case["width"], L=case["length"], x_I=0.05 * case["length"] + 20,
                                       seed=seed)], [p]
    if kind == "study":
        angles = [20.0 + 140.0 * i / max(1, case["n"] - 1) for i in range(case["n"])]
        gs = [I.displacement_channel(W=case["width"], L=case["length"], x_I=30.0, seed=seed * 100 + i)
              for i in range(case["n"])]
        return gs, [I.Params(nu_R=0.3, nu_B=0.3, sigma=0.06, theta=math.radians(a), u_in=0.1, inlet_profile=1)
                    for a in angles]
    return I.channel_sweep(case["n"], seed=case["widths"], wmin=case["wmin"], wmax=case["wmax"],
                           aspect=case["aspect"], param_seed=seed)


def prepare(case, seed):
    from paper_1707_00198_gb300.lbcg import Lattice
    gs, ps = _lattices(case, seed)
    L = Lattice(gs, ps, case["precision"])
    state = dict(case=case, lattice=L)
    if case["kind"] == "adjoint":
        # every gradient of an optimisation starts from the same state
        state["start"] = torch.empty(L.state_bytes, dtype=torch.uint8, pin_memory=torch.cuda.is_available())
        _download(L, state["start"])
        return state
    if case["kind"] == "channels":
        L.autotune()
    dtype = DTYPES[case["precision"]]
    state["out"] = torch.empty(L.state_bytes // dtype.itemsize, dtype=dtype, pin_memory=torch.cuda.is_available())
    return state


def _download(L, buf):
    from paper_1707_00198_gb300 import lbcg
    lbcg.lbcg_download_state(L.h, buf.data_ptr(), buf.numel() * buf.element_size())


REPORT = ("mass_R", "mass_B", "umax", "x_tip", "x_cl")


def run(state):
    case, L = state["case"], state["lattice"]
    if case["kind"] == "adjoint":
        from paper_1707_00198_gb300 import lbcg
        lbcg.lbcg_upload_state(L.h, state["start"].data_ptr(), state["start"].numel())
        g = L.adjoint(case["steps"], case["checkpoint"], reverse_fp32=case["reverse"] == "fp32")
        dt = np.float32 if case["precision"] == "fp32" else np.float64
        return {k: np.asarray(g[k], dtype=dt) for k in ("J", "dsigma", "dnu_R", "dnu_B", "dtheta", "dtheta_node")}
    L.step(case["steps"])
    out = {"state": state["out"]}
    if case["precision"] in ("fp64", "fp32") and len(L.geoms) == 1:
        o = L.observables()
        out["report"] = torch.tensor([o[k] for k in REPORT], dtype=DTYPES[case["precision"]])
    _download(L, state["out"])
    return out


def _fluid(case):
    kind = case["kind"]
    if kind == "droplet":
        return (case["nx"] - (2 if case["closed"] else 0)) * (case["ny"] - 2)
    if kind == "cylinder":
        return int((case["nx"] - 2) * (case["ny"] - 2) - math.pi * case["rs"] ** 2)
    if kind == "capillary":
        d = case["d"]
        return case["length"] * d + 2 * case["reservoir"] * (d + 2 * case["wall"])
    if kind == "study":
        return case["n"] * case["width"] * case["length"]
    if kind == "channels":
        # the widths as inputs.channel_sweep draws them: after each, one (M, Ca, theta)
        rng, total = np.random.default_rng(case["widths"]), 0
        for _ in range(case["n"]):
            w = int(rng.integers(case["wmin"], case["wmax"] + 1))
            for values in (I.M_GRID, I.CA_GRID, I.THETA_GRID):
                rng.choice(values)
            total += w * w * case["aspect"]
        return total
    return case["width"] * case["length"]


def work(case):
    """Every step reads and writes the 18 populations of each fluid node once, and spends about
    280 operations on it (an adjoint step: twice that on top of the forward step)."""
    n, size = _fluid(case) * case["steps"], DTYPES[case["precision"]].itemsize
    if case["kind"] == "adjoint":
        return {"bytes": 3 * 36 * size * n, "flops": 3 * 280 * n}
    return {"bytes": 36 * size * n, "flops": 280 * n}


# ------------------------------------------------------------------ the same in 64 bits
EX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
EY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
OPP = (0, 3, 4, 1, 2, 7, 8, 5, 6)
WT = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4
MOMENTS = ((1, 1, 1, 1, 1, 1, 1, 1, 1), (-4, -1, -1, -1, -1, 2, 2, 2, 2), (4, -2, -2, -2, -2, 1, 1, 1, 1),
           (0, 1, 0, -1, 0, 1, -1, -1, 1), (0, -2, 0, 2, 0, 1, -1, -1, 1), (0, 0, 1, 0, -1, 1, 1, -1, -1),
           (0, 0, -2, 0, 2, 1, 1, -1, -1), (0, 1, -1, 1, -1, 0, 0, 0, 0), (0, 0, 0, 0, 0, 1, -1, 1, -1))


class Plain:
    """One lattice's step (arXiv 1707.00198, Sec. II) in plain float64 tensor operations."""

    def __init__(self, g, p, device):
        self.g, self.p, self.dev = g, p, device
        self.nx, self.ny = g.nx, g.ny
        self.px, self.py, self.inout = g.bc_x == "periodic", g.bc_y == "periodic", g.bc_x == "inout"
        t = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device=device)  # noqa: E731
        solid = np.asarray(g.solid) != 0
        self.iy = torch.as_tensor(self._index(self.ny, self.py), device=device)
        self.ix = torch.as_tensor(self._index(self.nx, self.px), device=device)
        iy, ix = self._index(self.ny, self.py), self._index(self.nx, self.px)
        nb = [solid[np.ix_(iy, ix)][1 + EY[a]: 1 + EY[a] + self.ny, 1 + EX[a]: 1 + EX[a] + self.nx] for a in range(9)]
        y, x = np.mgrid[0:self.ny, 0:self.nx]
        inside = [(self.px | ((x + EX[a] >= 0) & (x + EX[a] < self.nx))) &
                  (self.py | ((y + EY[a] >= 0) & (y + EY[a] < self.ny))) for a in range(9)]
        wall = ~solid & np.any(nb[1:], axis=0)
        outer = solid & ~np.all(nb[1:], axis=0)
        b = lambda a: torch.as_tensor(np.ascontiguousarray(a), device=device)  # noqa: E731
        self.fluid, self.wall, self.outer = b(~solid), b(wall), b(outer)
        self.nb_fluid = [t(~nb[a]) for a in range(9)]
        # direction a arrives from x - e_a, a fluid node of the lattice, or bounces back at x + e_a
        self.arrives = [b(~solid & ~nb[OPP[a]] & inside[OPP[a]]) for a in range(9)]
        self.bounces = [b(~solid & nb[a] & inside[a]) for a in range(9)]
        den = sum(WT[a] * (~nb[a]).astype(float) for a in range(1, 9))
        self.virt_den = t(np.where(outer, den, 1.0))
        n = np.asarray(g.normal) * wall if g.normal is not None else self._e8(solid, wall)
        self.ns = t(n)
        th = g.theta_node if g.theta_node is not None else np.full((self.ny, self.nx), p.theta)
        self.theta = t(th)
        self.sigma, self.nuR, self.nuB = t(p.sigma), t(p.nu_R), t(p.nu_B)
        m = np.array(MOMENTS, float)
        self.M, self.Minv = t(m), t(np.linalg.inv(m))
        r = t(g.rhoN0)
        w = t(np.array(WT))[:, None, None]
        self.first = torch.stack([w * p.rho0 * (1 + r) / 2, w * p.rho0 * (1 - r) / 2]) * self.fluid
        if p.inlet_profile:
            rows = np.nonzero(~solid[:, 0])[0]
            s = (np.arange(self.ny) - (rows[0] - 0.5)) / (rows[-1] - rows[0] + 1.0)
            self.u_in = t(4 * p.u_in * s * (1 - s))
        else:
            self.u_in = t(np.full(self.ny, p.u_in))

    @staticmethod
    def _index(n, periodic):
        i = np.arange(-1, n + 1)
        return i % n if periodic else np.clip(i, 0, n - 1)

    def _e8(self, solid, wall):
        """Eq. 32-33 with the weights as integers over 5040."""
        k = {1: 960, 2: 448, 4: 84, 5: 32, 8: 1}
        s = solid.astype(np.int64)
        mode = {"periodic": "wrap", "inout": "edge"}
        pad = ((0, 0), (2, 2))
        s = np.pad(s, pad, mode=mode[self.g.bc_x]) if self.g.bc_x in mode else np.pad(s, pad, constant_values=1)
        pad = ((2, 2), (0, 0))
        s = np.pad(s, pad, mode="wrap") if self.py else np.pad(s, pad, constant_values=1)
        vx, vy = np.zeros(solid.shape), np.zeros(solid.shape)
        for cy in range(-2, 3):
            for cx in range(-2, 3):
                w = k.get(cx * cx + cy * cy, 0)
                v = w * s[2 + cy: 2 + cy + self.ny, 2 + cx: 2 + cx + self.nx]
                vx += v * cx
                vy += v * cy
        mag = np.sqrt(vx * vx + vy * vy)
        ok = wall & (mag > 0)
        mag = np.where(ok, mag, 1.0)
        return np.stack([np.where(ok, vx / mag, 0.0), np.where(ok, vy / mag, 0.0)])

    def around(self, f):
        """f at x + e_a for a = 0..8 (periodic axes wrap, others repeat the edge)."""
        f = f.index_select(-2, self.iy).index_select(-1, self.ix)
        return [f[..., 1 + EY[a]: 1 + EY[a] + self.ny, 1 + EX[a]: 1 + EX[a] + self.nx] for a in range(9)]

    def filled(self, f):
        nb, num = self.around(f), torch.zeros_like(f)
        for a in range(1, 9):
            num = num + WT[a] * nb[a] * self.nb_fluid[a]
        return torch.where(self.fluid, f, torch.where(self.outer, num / self.virt_den, 0.0))

    def gradient(self, f):
        nb = self.around(self.filled(f))
        gx = gy = torch.zeros_like(f)
        for a in range(1, 9):
            if EX[a]:
                gx = gx + WT[a] * nb[a] * EX[a]
            if EY[a]:
                gy = gy + WT[a] * nb[a] * EY[a]
        return gx / (1 / 3), gy / (1 / 3)

    def open_columns(self, F):
        if not self.inout:
            return F
        F = F.clone()
        f = F[:, :, :, 0].sum(0)
        u = self.u_in
        rho = (f[0] + f[2] + f[4] + 2 * (f[3] + f[6] + f[7])) / (1 - u)
        red = torch.stack([f[0], f[3] + 2 / 3 * rho * u, f[2], f[3], f[4], f[7] - 0.5 * (f[2] - f[4]) + rho * u / 6,
                           f[6], f[7], f[6] + 0.5 * (f[2] - f[4]) + rho * u / 6])
        inlet = torch.where(self.fluid[:, 0], torch.stack([red, torch.zeros_like(red)]), F[:, :, :, 0])
        o = F[:, :, :, -1]
        f, r = o.sum(0), self.p.rho_out
        ux = -1 + (f[0] + f[2] + f[4] + 2 * (f[1] + f[5] + f[8])) / r
        new = {3: f[1] - 2 / 3 * r * ux, 7: f[5] + 0.5 * (f[2] - f[4]) - r * ux / 6,
               6: f[8] - 0.5 * (f[2] - f[4]) - r * ux / 6}
        known = [0, 1, 2, 4, 5, 8]
        kT = f[known].sum(0)
        part = o[0][known].sum(0) / torch.where(kT != 0, kT, torch.ones_like(kT))
        outlet = torch.stack([torch.stack([part * new[a] if a in new else o[0, a] for a in range(9)]),
                              torch.stack([(1 - part) * new[a] if a in new else o[1, a] for a in range(9)])])
        outlet = torch.where(self.fluid[:, -1], outlet, o)
        return torch.cat([inlet[..., None], F[:, :, :, 1:-1], outlet[..., None]], dim=-1)

    def macro(self, F):
        """Densities, rho^N, corrected gradient, n, force and velocity of a post-streaming state."""
        p = self.p
        rR, rB = F[0].sum(0), F[1].sum(0)
        rho = torch.where(self.fluid, rR + rB, 1.0)
        rn = torch.where(self.fluid, (rR - rB) / rho, 0.0)
        gx, gy = self.gradient(rn)
        mag, ok = self._norm(gx, gy)
        safe = torch.where(ok, mag, 1.0)
        c, s = torch.cos(self.theta), torch.sin(self.theta)
        sx, sy = self.ns[0], self.ns[1]
        f1, f2 = (sx * c - sy * s, sx * s + sy * c), (sx * c + sy * s, -sx * s + sy * c)
        with torch.no_grad():
            d1 = torch.sqrt((f1[0] - gx / safe) ** 2 + (f1[1] - gy / safe) ** 2)
            d2 = torch.sqrt((f2[0] - gx / safe) ** 2 + (f2[1] - gy / safe) ** 2)
            pick, sel = d1 <= d2, self.wall & ok
        gx = torch.where(self.fluid, torch.where(sel, mag * torch.where(pick, f1[0], f2[0]), gx), 0.0)
        gy = torch.where(self.fluid, torch.where(sel, mag * torch.where(pick, f1[1], f2[1]), gy), 0.0)
        mag, ok = self._norm(gx, gy)
        safe = torch.where(ok, mag, 1.0)
        nx, ny = torch.where(ok, gx / safe, 0.0), torch.where(ok, gy / safe, 0.0)
        (xx, xy), (yx, yy) = self.gradient(nx), self.gradient(ny)
        kappa = torch.where(self.fluid, -nx * nx * yy - ny * ny * xx + nx * ny * (xy + yx), 0.0)
        Fx, Fy = 0.5 * self.sigma * kappa * gx, 0.5 * self.sigma * kappa * gy
        f = F.sum(0)
        ux = torch.where(self.fluid, (f[1] - f[3] + f[5] - f[6] - f[7] + f[8] + 0.5 * Fx) / rho, 0.0)
        uy = torch.where(self.fluid, (f[2] - f[4] + f[5] + f[6] - f[7] - f[8] + 0.5 * Fy) / rho, 0.0)
        return rR, rB, rho, rn, nx, ny, Fx, Fy, ux, uy, f

    def _norm(self, gx, gy):
        m2 = gx * gx + gy * gy
        ok = torch.sqrt(m2.detach()) > self.p.grad_eps
        return torch.where(ok, torch.sqrt(torch.where(ok, m2, 1.0)), 0.0), ok

    def step(self, F):
        p = self.p
        rR, rB, rho, rn, nx, ny, Fx, Fy, ux, uy, f = self.macro(self.open_columns(F))
        u2, feq, src = ux * ux + uy * uy, [], []
        for a in range(9):
            eu = EX[a] * ux + EY[a] * uy
            feq.append(WT[a] * rho * (1 + 3 * eu + 4.5 * eu * eu - 1.5 * u2))
            src.append(WT[a] * ((3 * (EX[a] - ux) + 9 * eu * EX[a]) * Fx + (3 * (EY[a] - uy) + 9 * eu * EY[a]) * Fy))
        inv_nu = (1 + rn) / (2 * self.nuR) + (1 - rn) / (2 * self.nuB)
        sv, one = 1 / (3 / inv_nu + 0.5), torch.ones_like(rn)
        S = torch.stack([one, p.s_e * one, p.s_eps * one, one, p.s_q * one, one, p.s_q * one, sv, sv])
        flat = lambda m, v: (m @ v.reshape(9, -1)).reshape(v.shape)  # noqa: E731
        d = -S * flat(self.M, f - torch.stack(feq)) + (1 - 0.5 * S) * flat(self.M, torch.stack(src))
        f = f + flat(self.Minv, d)
        pert = [p.beta * rR * rB / rho * WT[a] * (EX[a] * nx + EY[a] * ny) for a in range(9)]
        pert = torch.stack(pert)
        P = torch.stack([rR / rho * f + pert, rB / rho * f - pert])
        out = []
        for a in range(9):
            moved = self.around(P[:, a])[OPP[a]]
            back = torch.where(self.bounces[OPP[a]], P[:, OPP[a]], self.first[:, a])
            out.append(torch.where(self.arrives[a], moved, back))
        return torch.stack(out, dim=1)

    def stored(self, F, precision):
        """The state in its storage format: [y][x / 32][direction][x % 32][pair]."""
        if precision in ("fp16", "bf16"):
            k = 1024.0 if precision == "fp16" else 1.0
            w = torch.tensor(WT, dtype=torch.float64, device=self.dev)[:, None, None]
            F = torch.stack([k * (F[0] + F[1] - w * self.p.rho0 * self.fluid), k * (F[0] - F[1])])
        pad = -self.nx % 32
        F = torch.nn.functional.pad(F, (0, pad)).reshape(2, 9, self.ny, -1, 32)
        return F.permute(2, 3, 1, 4, 0).reshape(-1)

    def crossing(self, prof):
        """The first rho^N >= 0 -> < 0 change along a profile (None without one)."""
        at = torch.nonzero((prof[:-1] >= 0) & (prof[1:] < 0))
        if not len(at):
            return None
        i = int(at[0])
        return i + prof[i] / (prof[i] - prof[i + 1])

    def tip_and_line(self, rn):
        ny = self.ny
        rows = (ny // 2 - 1, ny // 2) if ny % 2 == 0 else (ny // 2, ny // 2)
        tip = self.crossing(0.5 * (rn[rows[0]] + rn[rows[1]]))
        ends = [c for c in (self.crossing(rn[1]), self.crossing(rn[ny - 2])) if c is not None]
        return tip, sum(ends) / len(ends) if ends else None


def exact(case, seed):
    if case["steps"] * (_fluid(case) / 2e8 + case.get("n", 1) * 0.004) > 15:
        return None
    device = "cuda" if torch.cuda.is_available() else "cpu"
    lattices = [Plain(g, p, device) for g, p in zip(*_lattices(case, seed))]
    if case["kind"] == "adjoint":
        P = lattices[0]
        for v in (P.theta, P.sigma, P.nuR, P.nuB):
            v.requires_grad_(True)
        F = P.first
        for _ in range(case["steps"]):
            F = P.step(F)
        tip, line = P.tip_and_line(P.macro(P.open_columns(F))[3])
        (tip - line).backward()
        return {"J": float((tip - line).detach()), "dsigma": float(P.sigma.grad), "dnu_R": float(P.nuR.grad),
                "dnu_B": float(P.nuB.grad), "dtheta": float(P.theta.grad.sum()), "dtheta_node": P.theta.grad}
    states, report = [], None
    with torch.no_grad():
        for P in lattices:
            F = P.first
            for _ in range(case["steps"]):
                F = P.step(F)
            states.append(P.stored(F, case["precision"]))
        if case["precision"] in ("fp64", "fp32") and len(lattices) == 1:
            rR, rB, _, rn, _, _, _, _, ux, uy, _ = P.macro(P.open_columns(F))
            tip, line = P.tip_and_line(rn)
            u = torch.where(P.fluid, torch.sqrt(ux * ux + uy * uy), 0.0).max()
            report = torch.tensor([float((rR * P.fluid).sum()), float((rB * P.fluid).sum()), float(u),
                                   -1.0 if tip is None else float(tip), -1.0 if line is None else float(line)],
                                  dtype=torch.float64)
    out = {"state": torch.cat(states)}
    if report is not None:
        out["report"] = report
    return out
