"""What the framework is timed on: one pass of each piece of work that its users have it do, through its public entry
points, over the range of sizes, storage precisions, link rules and directions (forward and adjoint) they use.

A pass advances a prepared lattice and hands back what a program reads afterwards: the density and velocity fields (device
tensors), the forces on the bodies, or the gradients.  Lattices, geometry and output buffers are kept between passes, as a
simulation loop keeps them; the flow goes on from pass to pass.  Fields, forces and gradients of an FP32 lattice are kept in
FP32 (its storage precision), those of an FP64 lattice in FP64.

``exact`` restates the method on the dense lattice in plain FP64 torch (gradients by torch.autograd).
"""
import functools
import math

import numpy as np
import torch

from paper_1903_01111_gb300 import batch as B
from paper_1903_01111_gb300 import geometry as G
from paper_1903_01111_gb300 import lbm

FP64, FP32 = "fp64", "fp32"
RULES = ("halfway", "bouzidi", "vibb", "yu")


def listed():
    return [
        # Sec. 4.1's plane Poiseuille cell between off-node walls: the smallest lattice, run for thousands of steps in the
        # accuracy studies; a step is launches and latency
        dict(name="poiseuille_32x24_fp64", kind="poiseuille", nx=32, ny=24, q=0.3, rule="vibb", prec=FP64, steps=200),
        # Sec. 4.3's spinning cylinder (Magnus lift) with the paper's MRT operator, in the reference precision, lift read
        # every 100 steps
        dict(name="magnus_400x400_mrt_fp64", kind="channel", nx=400, ny=400, cx=100.37, cy=199.61, r=10.0, spin=1.0,
             u_max=0.05, tau=0.65, collision="mrt", monitor=False, prec=FP64, steps=100),
        # flow past a cylinder in a 2000 x 400 channel (Re = 100) with the drag of every step on the host: the state fits L2
        dict(name="cylinder_2000x400_fp32", kind="channel", nx=2000, ny=400, cx=400.37, cy=200.61, r=20.3, spin=0.0,
             u_max=0.1, tau=0.5812, collision="bgk", monitor=True, prec=FP32, steps=64),
        # body-force flow through the 384^3 random sphere pack, 31 M cut links: the headline workload
        dict(name="pack_384_fp32", kind="pack", n=384, rule="vibb", prec=FP32, steps=10),
        # the same flow in FP64, the precision the FP32 runs are checked against
        dict(name="pack_200_fp64", kind="pack", n=200, rule="vibb", prec=FP64, steps=5),
        # solid-free boxes: the bulk pass alone, 2-D and 3-D, both precisions, with even and odd sizes
        dict(name="box_8192x4096_fp32", kind="box", stencil=2, nx=8192, ny=4096, nz=1, prec=FP32, steps=10),
        dict(name="box_301x257x259_fp32", kind="box", stencil=3, nx=301, ny=257, nz=259, prec=FP32, steps=10),
        dict(name="box_4097x2049_fp64", kind="box", stencil=2, nx=4097, ny=2049, nz=1, prec=FP64, steps=6),
        dict(name="box_192x192x192_fp64", kind="box", stencil=3, nx=192, ny=192, nz=192, prec=FP64, steps=5),
        # 256 channels of different sizes, cylinders and Reynolds numbers stepped as one lattice, all drags read
        dict(name="batch_256_fp32", kind="batch", domains=256, prec=FP32, steps=20),
        # drag gradient (every link's q, and tau) of a 1024 x 256 channel: forward, recompute and adjoint sweep
        dict(name="adjoint_1024x256_fp32", kind="adjoint", nx=1024, ny=256, prec=FP32, steps=200, every=50),
        # gradient of the summed drag of 64 channels at once
        dict(name="adjoint_batch_64_fp32", kind="adjoint_batch", domains=64, prec=FP32, steps=64, every=16),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["poiseuille", "channel", "channel", "pack", "box", "box", "batch", "adjoint", "adjoint_batch"])
    prec = rng.choice([FP64, FP32])
    if kind == "poiseuille":
        return dict(kind=kind, nx=_log(rng, 8, 128), ny=_log(rng, 6, 100), q=round(rng.uniform(0.1, 0.9), 3),
                    rule=rng.choice(RULES), prec=prec, steps=rng.randint(50, 300))
    if kind == "channel":
        nx, ny = _log(rng, 120, 2000), _log(rng, 40, 400)
        r = rng.uniform(3.0, min(nx, ny) / 8.0)
        # tau: a cell Reynolds number the collision is stable at (the spinning study's, and above)
        return dict(kind=kind, nx=nx, ny=ny, cx=round(nx * rng.uniform(0.2, 0.3), 2), cy=round(ny * rng.uniform(0.45, 0.55), 2),
                    r=round(r, 2), spin=round(rng.choice([0.0, rng.uniform(0.2, 1.5)]), 2), u_max=0.05,
                    tau=round(rng.uniform(0.62, 0.9), 3), collision=rng.choice(["bgk", "mrt"]), monitor=rng.random() < 0.5,
                    prec=prec, steps=rng.randint(20, 100))
    if kind == "pack":
        return dict(kind=kind, n=_log(rng, 40, 240), rule=rng.choice(RULES), prec=prec, steps=rng.randint(2, 10))
    if kind == "box":
        if rng.random() < 0.5:
            nx, ny = _log(rng, 64, 8192), _log(rng, 64, 8192)
            ny = min(ny, (1 << 25) // nx)
            return dict(kind=kind, stencil=2, nx=nx, ny=ny, nz=1, prec=prec, steps=rng.randint(2, 10))
        n = [_log(rng, 16, 320) for _ in range(3)]
        n[2] = min(n[2], 24_000_000 // (n[0] * n[1]))
        return dict(kind=kind, stencil=3, nx=n[0], ny=n[1], nz=n[2], prec=prec, steps=rng.randint(2, 10))
    if kind == "batch":
        return dict(kind=kind, domains=_log(rng, 2, 128), prec=prec, steps=rng.randint(5, 40))
    if kind == "adjoint":
        every = rng.randint(5, 40)
        return dict(kind=kind, nx=_log(rng, 100, 1024), ny=_log(rng, 40, 256), prec=prec, steps=rng.randint(every, 120),
                    every=every)
    every = rng.randint(4, 16)
    return dict(kind=kind, domains=_log(rng, 2, 24), prec=prec, steps=rng.randint(every, 48), every=every)


# ------------------------------------------------------------------ inputs --

@functools.lru_cache(maxsize=2)
def _geometry_of(key):
    """The case's geometry (mask, cut links, domains): fixed by its sizes, whatever the seed of the flow."""
    c = dict(key)
    k = c["kind"]
    if k == "poiseuille":
        return G.channel(0, c["nx"], c["ny"], q_lo=c["q"], q_hi=c["q"])
    if k == "channel":
        return G.cylinder_channel(nx=c["nx"], ny_fluid=c["ny"], center=(c["cx"], c["cy"]), radius=c["r"],
                                  u_max=c["u_max"], omega=c["spin"] * c["u_max"] / c["r"])
    if k == "pack":
        n = c["n"]
        return G.sphere_pack(n) if n >= 64 else G.sphere_pack(n, rmin=3.0, rmax=6.0)
    if k == "box":
        return G.build(G.D2Q9 if c["stencil"] == 2 else G.D3Q19, (c["nx"], c["ny"], c["nz"]), (1, 1, 1), [])
    if k in ("batch", "adjoint_batch"):
        return B.stack(B.draw_channels(c["domains"], seed=0))
    if k == "adjoint":
        nx, ny = c["nx"], c["ny"]
        return G.cylinder_channel(nx=nx, ny_fluid=ny, center=(0.2503 * nx, 0.5024 * ny), radius=ny / 15.52, u_max=0.1)
    raise ValueError(k)


def _geometry(case):
    g = _geometry_of(tuple(sorted((k, v) for k, v in case.items() if k not in ("name", "prec", "steps", "every", "monitor"))))
    return (g.geometry, g) if isinstance(g, B.Batch) else (g, None)


def _setup(case, seed):
    """(geometry, lattice configuration without the precision, domains, rho, u): what a program hands to the lattice.  The
    flow starts from a developed or uniform profile with a few random long waves, and is driven as the case's study drives
    it."""
    geo, batch = _geometry(case)
    gen = np.random.default_rng([seed, 17])
    k = case["kind"]
    D = 2 if geo.stencil == G.D2Q9 else 3
    cfg = dict(tau=0.8, g=(0.0, 0.0, 0.0), bc=lbm.LBM_BC_VIBB)
    rows = None
    amp = 5e-3
    if k == "poiseuille":
        cfg.update(tau=0.8, g=(float(gen.uniform(0.5e-6, 2e-6)), 0.0, 0.0), bc=RULES.index(case["rule"]))
        amp = 2e-4
    elif k == "channel":
        cfg.update(tau=case["tau"], inlet_umax=case["u_max"], inlet_y0=0.5, inlet_y1=case["ny"] + 0.5,
                   collision=lbm.LBM_MRT if case["collision"] == "mrt" else lbm.LBM_BGK)
    elif k == "pack":
        cfg.update(tau=0.7, g=(float(gen.uniform(0.5e-6, 2e-6)), 0.0, 0.0), bc=RULES.index(case["rule"]),
                   vibb_density=lbm.LBM_VIBB_RHO_LOCAL)
        amp = 5e-4
    elif k == "box":
        cfg.update(tau=float(gen.uniform(0.6, 0.9)), g=(float(gen.uniform(0.5e-7, 1e-7)), 0.0, 0.0))
        amp = 2e-2
    elif k == "adjoint":
        # Re = 40 on the mean inflow and the diameter at the study's 256 rows
        cfg.update(tau=0.665, inlet_umax=0.1, inlet_y0=0.5, inlet_y1=case["ny"] + 0.5)
    else:
        cfg.update(tau=1.0, inlet_y0=0.0, inlet_y1=1.0)
        rows = batch.domains
    nx, ny, nz = geo.shape
    dev = torch.device("cuda")
    x = torch.arange(nx, device=dev, dtype=torch.float64)[None, None, :]
    y = torch.arange(ny, device=dev, dtype=torch.float64)[None, :, None]
    z = torch.arange(nz, device=dev, dtype=torch.float64)[:, None, None]

    def waves(a):
        out = torch.zeros((nz, ny, nx), device=dev, dtype=torch.float64)
        for _ in range(3):
            m = gen.integers(1, 4, 3)
            ph = gen.uniform(0, 2 * np.pi, 3)
            px = torch.sin(2 * np.pi * int(m[0]) * x / nx + float(ph[0]))
            py = torch.cos(2 * np.pi * int(m[1]) * y / max(ny, 16) + float(ph[1]))
            pz = torch.cos(2 * np.pi * int(m[2]) * z / nz + float(ph[2])) if nz > 1 else torch.ones_like(z)
            out += a * float(gen.uniform(0.3, 0.6)) * px * py * pz
        return out

    u = torch.zeros((nz, ny, nx, 3), device=dev, dtype=torch.float64)
    if k in ("channel", "adjoint"):
        H = case["ny"]
        u[..., 0] = 4 * cfg["inlet_umax"] * (y - 0.5) * (H + 0.5 - y) / H ** 2
    for a in range(D):
        u[..., a] += waves(amp)
    u = u.reshape(-1, 3)
    if rows is not None:
        u += torch.from_numpy(batch.initial_velocity()).to(dev)
    rho = 1.0 + waves(amp * 0.2).reshape(-1)
    fluid = torch.from_numpy(geo.solid).to(dev) == 0
    u = torch.where(fluid[:, None], u, torch.zeros_like(u))
    rho = torch.where(fluid, rho, torch.ones_like(rho))
    return geo, cfg, rows, rho.cpu().numpy(), u.cpu().numpy()


# --------------------------------------------------------------- the passes --

def prepare(case, seed):
    geo, cfg, rows, rho, u = _setup(case, seed)
    stream = torch.cuda.Stream()
    cfg.update(precision=lbm.LBM_FP64 if case["prec"] == FP64 else lbm.LBM_FP32_SHIFTED, stream=stream.cuda_stream)
    lat = lbm.Lattice(geo, domains=rows, **cfg)
    lat.init_equilibrium(rho, u)
    D = 2 if geo.stencil == G.D2Q9 else 3
    st = dict(case=case, lat=lat, stream=stream)
    if not case["kind"].startswith("adjoint"):
        st["rho"] = torch.empty(geo.N, dtype=torch.float64, device="cuda")
        st["u"] = torch.empty((D, geo.N), dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    return st


def run(st):
    case, lat = st["case"], st["lat"]
    single = case["prec"] == FP32
    host = np.float32 if single else np.float64
    out = {}
    if case["kind"].startswith("adjoint"):
        # drag of the cylinder, or of every cylinder of the batch
        if case["kind"] == "adjoint":
            body, w = 0, (1.0, 0.0, 0.0)
        else:
            body, w = -1, np.tile([1.0, 0.0, 0.0], (lat.info().n_bodies, 1))
        J, dq, dtau, _ = lbm.lbm_adjoint_step(lat.h, body, w, case["steps"], case["every"])
        return {"J": np.asarray([J], host), "dJ_dq": dq.astype(host), "dJ_dtau": np.atleast_1d(np.asarray(dtau, host))}
    if case.get("monitor"):
        out["forces"] = lat.step_forces(case["steps"], 0).astype(host)
    else:
        lat.step(case["steps"])
        if case["kind"] == "channel":
            out["forces"] = lat.force(0).astype(host)
        elif case["kind"] == "batch":
            out["forces"] = lat.forces().astype(host)
    with torch.cuda.stream(st["stream"]):
        lat.moments(st["rho"], st["u"])
        out["rho"] = st["rho"].float() if single else st["rho"]
        out["u"] = st["u"].float() if single else st["u"]
    return out


def work(case):
    """Per step and fluid node every population read and written once, and per cut link its wall fraction, node and
    direction; the fields written once at the end.  Flops as the update and the rules need them: 263 (D3Q19) and 125 (D2Q9)
    per node, 118 per VIBB link.  A gradient: the steps forward, again for the recompute, and per step back the populations
    and both adjoint states."""
    geo, _ = _geometry(case)
    Q, D, fl = (9, 2, 125) if geo.stencil == G.D2Q9 else (19, 3, 263)
    s = 8 if case["prec"] == FP64 else 4
    nf, nl, n = geo.fluid_count(), len(geo.links), case["steps"]
    by, flops = nf * 2 * Q * s + nl * (8 + s), nf * fl + nl * 118
    if case["kind"].startswith("adjoint"):
        return {"bytes": n * (2 * by + nf * 3 * Q * s + nl * (8 + s)), "flops": n * flops * 5}
    return {"bytes": n * by + 8 * (1 + D) * geo.N, "flops": n * flops}


# ------------------------------------------------- the same in 64-bit torch --

_M9 = [[1] * 9, [-4, -1, -1, -1, -1, 2, 2, 2, 2], [4, -2, -2, -2, -2, 1, 1, 1, 1], [0, 1, 0, -1, 0, 1, -1, -1, 1],
       [0, -2, 0, 2, 0, 1, -1, -1, 1], [0, 0, 1, 0, -1, 1, 1, -1, -1], [0, 0, -2, 0, 2, 1, 1, -1, -1],
       [0, 1, -1, 1, -1, 0, 0, 0, 0], [0, 0, 0, 0, 0, 1, -1, 1, -1]]


class _Dense:
    """Post-collision populations f [Q, N] on the whole lattice; solid nodes are held at rest."""

    def __init__(self, geo, cfg, rows):
        self.shape, N = geo.shape, geo.N
        nx, ny, nz = geo.shape
        dev = self.dev = torch.device("cuda")
        e2 = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
        e3 = [(0, 0, 0)]
        for a, b in ((0, None), (1, None), (2, None), (0, 1), (0, 2), (1, 2)):
            for sa, sb in (((1, 0), (-1, 0)) if b is None else ((1, 1), (-1, -1), (1, -1), (-1, 1))):
                v = [0, 0, 0]
                v[a] = sa
                if b is not None:
                    v[b] = sb
                e3.append(tuple(v))
        self.two = geo.stencil == G.D2Q9
        if self.two:
            E = [(a, b, 0) for a, b in e2]
            W = [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4
        else:
            E = e3[:7] + [(1, 1, 0), (-1, -1, 0), (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1),
                          (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1)]
            W = [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12
        self.E, self.Q, self.N = E, len(E), N
        t = lambda v, k=torch.float64: torch.as_tensor(np.asarray(v), device=dev).to(k)  # noqa: E731
        self.e, self.w = t(E), t(W)[:, None]
        self.opp = t([E.index(tuple(-v for v in x)) for x in E], torch.int64)
        self.g = t(cfg["g"])[:, None]
        self.mrt = cfg.get("collision", lbm.LBM_BGK) == lbm.LBM_MRT
        self.local = cfg.get("vibb_density", lbm.LBM_VIBB_RHO_PRINTED) == lbm.LBM_VIBB_RHO_LOCAL
        solid = t(geo.solid, torch.bool)
        # domains: per-row width, inlet profile and relaxation time
        row = np.arange(ny)
        width, uin, dom = np.full(ny, nx), np.zeros(ny), np.zeros(ny, np.int64)
        taus = [cfg["tau"]]
        prof = lambda r, m, a, b: 4.0 * m * (r - a) * (b - r) / (b - a) ** 2  # noqa: E731
        if rows is not None:
            taus = [r["tau"] for r in rows]
            for d, r in enumerate(rows):
                own = slice(r["lo"], r["lo"] + r["n"])
                width[own], dom[own] = r["nx"], d
                uin[own] = prof(np.arange(r["n"]), r["inlet_umax"], r["inlet_y0"], r["inlet_y1"])
        elif geo.open_x[0]:
            uin = prof(row, cfg["inlet_umax"], cfg["inlet_y0"], cfg["inlet_y1"])
        self.tau = t(taus)
        self.dom = t(np.tile(np.repeat(dom, nx), nz), torch.int64) if len(taus) > 1 else None
        self.open = bool(geo.open_x[0])
        live = ~solid
        if self.open:
            m = geo.solid.reshape(ny, nx) == 0
            yi, yo = np.flatnonzero(m[:, 0]), np.flatnonzero(m[row, width - 1])
            self.k_in, self.u_in = t(yi * nx, torch.int64), t(uin[yi])
            self.k_out = t(yo * nx + width[yo] - 1, torch.int64)
            live = live.clone()
            live[self.k_in] = False
            live[self.k_out] = False
        self.live = live
        L = geo.links
        self.nl = len(L)
        self.ln, self.ld = t(L["node"], torch.int64), t(L["dir"], torch.int64)
        self.q, self.body = t(L["q"]), t(L["body"], torch.int64)
        self.uw = t(L["uw"]).T
        self.rule = torch.where(t(L["bc"], torch.int64) >= 0, t(L["bc"], torch.int64), torch.full_like(self.ln, cfg["bc"]))
        c = [self.ln % nx, (self.ln // nx) % ny, self.ln // (nx * ny)]
        ei = self.e.to(torch.int64)[self.ld]
        per, inside, p = geo.periodic, torch.ones_like(self.ln, dtype=torch.bool), []
        for a, n in enumerate((nx, ny, nz)):
            v = c[a] - ei[:, a]
            if not per[a]:
                inside &= (v >= 0) & (v < n)
            p.append(v % n)
        ff = p[0] + nx * (p[1] + ny * p[2])
        self.lff = torch.where(inside & live[ff], ff, self.ln)

    def collide(self, f, tau):
        om = 1.0 / (tau[0] if self.dom is None else tau[self.dom])
        rho = f.sum(0)
        u = (self.e.T @ f + 0.5 * self.g) / rho
        eu, eg = self.e @ u, self.e @ self.g
        ug = (u * self.g).sum(0)
        n = f - self.w * rho * (1.0 + 3.0 * eu + 4.5 * eu * eu - 1.5 * (u * u).sum(0))
        src = self.w * (3.0 * (eg - ug) + 9.0 * eu * eg)
        if self.mrt:
            M = torch.tensor(_M9, dtype=torch.float64, device=self.dev)
            s = torch.tensor([0.3, 1.5, 1.5, 0.3, 1.2, 0.3, 1.2, 0.0, 0.0], dtype=torch.float64, device=self.dev)[:, None]
            s = torch.cat([s[:7], om.reshape(1, 1).expand(2, 1)])
            out = f - (M.T / (M * M).sum(1)) @ (s * (M @ n) - (1.0 - 0.5 * s) * (M @ src))
        else:
            out = f - om * n + (1.0 - 0.5 * om) * src
        return torch.where(self.live[None], out, self.w.expand_as(out))

    def start(self, rho, u, tau):
        rho, u = torch.from_numpy(rho).to(self.dev), torch.from_numpy(u).to(self.dev).T
        eu = self.e @ u
        return self.collide(self.w * rho * (1.0 + 3.0 * eu + 4.5 * eu * eu - 1.5 * (u * u).sum(0)), tau)

    def moments(self, f):
        rho = f.sum(0)
        return rho, (self.e.T @ f - 0.5 * self.g) / rho

    def _eq(self, ex, w, rho, u):
        eu = (ex * u).sum(0)
        return w * rho * (1.0 + 3.0 * eu + 4.5 * eu * eu - 1.5 * (u * u).sum(0))

    def link_values(self, f, q):
        n, ff, d = self.ln, self.lff, self.ld
        flat = f.reshape(-1)
        a, b, c = flat[d * self.N + n], flat[d * self.N + ff], flat[self.opp[d] * self.N + n]
        ex, w, uw = self.e[d].T, self.w[d, 0], self.uw
        wall = -6.0 * w * (ex * uw).sum(0)
        out = torch.zeros_like(a)
        near = q <= 0.5
        for rule in sorted(set(self.rule.unique().tolist())):
            if rule == 0:
                v = a + wall
            elif rule == 1:
                v = torch.where(near, 2 * q * a + (1 - 2 * q) * b + wall, (a + wall) / (2 * q) + (2 * q - 1) / (2 * q) * c)
            elif rule == 3:
                v = (q * a + (1 - q) * b + wall + q * c) / (1 + q)
            else:
                # moments of f+ at both nodes (the collision keeps mass and adds g to the momentum)
                rf, rff = f[:, n].sum(0), f[:, ff].sum(0)
                uf = (self.e.T @ f[:, n] - 0.5 * self.g) / rf
                uff = (self.e.T @ f[:, ff] - 0.5 * self.g) / rff
                rd = 2 * q * rf + (1 - 2 * q) * rff
                if self.local:
                    rd = torch.where(near, rd, rf)
                neq = rd * (2 * q * (a - self._eq(ex, w, rf, uf)) / rf + (1 - 2 * q) * (b - self._eq(ex, w, rff, uff)) / rff)
                us = torch.where(near, 2 * q * uf + (1 - 2 * q) * uff, ((1 - q) * uf + (2 * q - 1) * uw) / q)
                uss = ((1 - q) * uff + 2 * q * uw) / (1 + q)
                v = self._eq(ex, w, rd, us / 3 + 2 * uss / 3) + neq + wall
            out = torch.where(self.rule == rule, v, out)
        return out, a

    def step(self, f, q, tau, want=None):
        """f+(t+1), and sum_b want[b] . F_b (or the force on body `want`) of the step."""
        nx, ny, nz = self.shape
        F = None
        if self.nl:
            val, a = self.link_values(f, q)
            if want is not None:
                t = (a + val) * self.e[self.ld].T
                if isinstance(want, int):
                    nb = max(int(self.body.max()) + 1, 1) if want < 0 else 1
                    sel = torch.where(self.body >= 0, self.body, nb) if want < 0 else torch.where(self.body == want, 0, 1)
                    F = torch.zeros((nb + 1, 3), dtype=torch.float64, device=self.dev).index_add(0, sel, t.T)[:nb]
                else:
                    on = self.body >= 0
                    F = (t * torch.where(on, want[self.body.clamp(min=0)].T, torch.zeros_like(t))).sum()
        if self.open:
            k1 = self.k_in + 1
            rho, u = self.moments(f[:, k1])
            eu = self.e @ u
            eq1 = self.w * rho * (1.0 + 3.0 * eu + 4.5 * eu * eu - 1.5 * (u * u).sum(0))
            ein = self.e[:, :1] * self.u_in
            eqi = self.w * rho * (1.0 + 3.0 * ein + 4.5 * ein * ein - 1.5 * self.u_in ** 2)
            f = f.index_copy(1, self.k_in, eqi + f[:, k1] - eq1).index_copy(1, self.k_out, f[:, self.k_out - 1])
        p = torch.stack([f[i].reshape(nz, ny, nx).roll((x[2], x[1], x[0]), (0, 1, 2)).reshape(-1) for i, x in enumerate(self.E)])
        if self.nl:
            p = p.reshape(-1).index_copy(0, self.opp[self.ld] * self.N + self.ln, val).reshape(self.Q, self.N)
        return self.collide(p, tau), F


def exact(case, seed):
    geo, cfg, rows, rho, u = _setup(case, seed)
    ref = _Dense(geo, cfg, rows)
    if case["kind"].startswith("adjoint"):
        from torch.utils.checkpoint import checkpoint

        q, tau = ref.q.clone().requires_grad_(True), ref.tau.clone().requires_grad_(True)
        nb = max(int(ref.body.max()) + 1, 1)
        want = torch.tensor([[1.0, 0.0, 0.0]], dtype=torch.float64, device=ref.dev).expand(nb, 3)
        f = ref.start(rho, u, tau)
        for s in range(case["steps"] - 1):
            f = checkpoint(lambda f, q, tau: ref.step(f, q, tau)[0], f, q, tau, use_reentrant=False)
        _, J = ref.step(f, q, tau, want)
        dq, dtau = torch.autograd.grad(J, (q, tau))
        return {"J": J.detach().reshape(1), "dJ_dq": dq, "dJ_dtau": dtau}
    out = {}
    with torch.no_grad():
        f = ref.start(rho, u, ref.tau)
        want = 0 if case["kind"] == "channel" else -1 if case["kind"] == "batch" else None
        seen = []
        for s in range(case["steps"]):
            f, F = ref.step(f, ref.q, ref.tau, want if case.get("monitor") or s == case["steps"] - 1 else None)
            if F is not None:
                seen.append(F)
        if case.get("monitor"):
            out["forces"] = torch.cat(seen)
        elif want is not None:
            out["forces"] = seen[-1][0] if case["kind"] == "channel" else seen[-1]
        r, v = ref.moments(f)
        D = 2 if ref.two else 3
        out["rho"] = torch.where(ref.live, r, torch.zeros_like(r))
        out["u"] = torch.where(ref.live[None], v[:D], torch.zeros_like(v[:D]))
    return out
