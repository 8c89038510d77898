"""Performance cases of the library's public entry points.

A case is one pass a user's program makes: a whole scene (medium -> flux
matrix -> solve -> detector radiance), a scene with its gradient, a batch of
queued scenes, or a solve on a caller's own matrix.  Every case names its
sizes and options as plain values; the fields are made from the seed.

``exact`` restates the method in FP64 on torch tensors (translation-invariant
rays, one array per direction and chain member) and shares nothing with the
library but the input recipes in ``scenes``.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2503_16037_gb300 import scenes
from paper_2503_16037_gb300 import tursca as T

EDGES_R = {1: 27.5, 2: 124.4}  # stored entries of K per node, about


# ---------------------------------------------------------------------------
# The cases

def listed():
    scene = dict(kind="scene", field="plume", R=2, S=2, fp64=False, mode="full", rtol=1e-10, sza=60.0, saa=0.0,
                 vza=30.0, vaa=180.0, albedo=0.1, ppv=1)
    return [
        # the smallest configuration (26 neighbours, FP64): a call is all latency and launches
        dict(scene, name="plain 8x8x8 fp64", field="plain", nx=8, ny=8, nz=8, R=1, S=1, fp64=True, rtol=1e-12,
             sza=30.0, vza=0.0, vaa=0.0, albedo=0.2),
        # the smallest scene of the serving mix, one call at a time: a retrieval's inner loop over small scenes
        dict(scene, name="plume 16x16x16", nx=16, ny=16, nz=16),
        # odd sizes, three species, a brighter ground, oblique sun and view off the grid's axes
        dict(scene, name="random 45x37x29", field="random", nx=45, ny=37, nz=29, S=3, sza=50.0, saa=20.0, vza=25.0,
             vaa=200.0, albedo=0.3),
        # the benchmark's scene: an industrial plume on the full 124-neighbour stencil
        dict(scene, name="plume 64x64x32", nx=64, ny=64, nz=32),
        # the largest configuration: a broken cloud, nearly conservative scattering, solver at its hardest
        dict(scene, name="cloud 128x128x40", field="cloud", nx=128, ny=128, nz=40, sza=70.0, vza=20.0, vaa=0.0,
             albedo=0.04),
        # the same plume in full FP64: reference runs and validation
        dict(scene, name="plume 64x64x32 fp64", nx=64, ny=64, nz=32, fp64=True, rtol=1e-12),
        # one retrieval step: radiance and its gradient with respect to every voxel's absorption
        dict(scene, name="plume 48x48x32 gradient", nx=48, ny=48, nz=32, mode="gradient"),
        # first scattering order only: fast previews and optically thin scenes
        dict(scene, name="plume 64x64x32 single", nx=64, ny=64, nz=32, mode="single"),
        # coupling selection: the scattering graph keeps the couplings above a threshold
        dict(scene, name="plume 64x64x32 c_min 2", nx=64, ny=64, nz=32, mode="c_min", c_min=2.0),
        # edge unknowns: the arrival direction is kept into every scattering
        dict(scene, name="plume 32x32x24 aniso", nx=32, ny=32, nz=24, mode="aniso", rtol=1e-8),
        # a queue of scenes of the serving shapes, in pinned host memory, on eight workers
        dict(kind="serve", name="serve 16 mixed", requests=16, workers=8, small=False, sizes=7, rtol=1e-10),
        # a caller's own CSR matrix, solved without allocating: real-time loops with fixed memory
        dict(kind="csr", name="csr 65536 x 124", n=65536, band=4096, row=124, sweeps=20, refinements=4),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    what = rng.choice(["full", "full", "full", "fp64", "gradient", "single", "c_min", "top_k", "aniso", "serve",
                       "cloud", "csr"])
    if what == "csr":
        n = _log(rng, 2000, 100000)
        return dict(kind="csr", n=n, band=min(n - 1, _log(rng, 500, 8000)), row=rng.randint(20, 130),
                    sweeps=rng.randint(18, 30), refinements=rng.randint(4, 6))
    if what == "serve":
        return dict(kind="serve", requests=rng.randint(5, 14), workers=rng.randint(2, 8), small=rng.random() < 0.5,
                    sizes=rng.randint(0, 10 ** 6), rtol=1e-10)
    most = {"full": 250_000, "fp64": 100_000, "gradient": 120_000, "single": 400_000, "c_min": 60_000,
            "top_k": 60_000, "aniso": 20_000, "cloud": 200_000}[what]
    while True:
        nx, ny, nz = _log(rng, 8, 128), _log(rng, 8, 128), _log(rng, 6, 40)
        if what == "cloud":
            nx, ny, nz = max(nx, 24), max(ny, 24), rng.randint(28, 40)
        if most / 100 <= nx * ny * nz <= most:
            break
    field = "cloud" if what == "cloud" else rng.choice(["plume", "random"])
    c = dict(kind="scene", field=field, nx=nx, ny=ny, nz=nz, R=2 if rng.random() < 0.8 or field == "cloud" else 1,
             S=rng.randint(1, 4) if field == "random" else 2, fp64=what == "fp64" or rng.random() < 0.1,
             mode=what if what in ("gradient", "single", "c_min", "top_k", "aniso") else "full",
             rtol=1e-10, sza=round(rng.uniform(15.0, 72.0), 1), saa=round(rng.uniform(0.0, 180.0), 1),
             vza=round(rng.uniform(3.0, 50.0), 1), vaa=round(rng.uniform(0.0, 360.0), 1),
             albedo=round(rng.uniform(0.02, 0.4), 2), ppv=2 if rng.random() < 0.15 else 1)
    if field == "cloud" or what in ("c_min", "top_k"):
        c["fp64"] = False
    if what == "c_min":
        c["c_min"] = round(rng.uniform(0.5, 4.0), 2)
    if what == "top_k":
        c["keep"] = round(rng.uniform(0.1, 0.9), 2)
    if what == "aniso":
        c["fp64"], c["rtol"] = False, 1e-8
    if c["fp64"]:
        c["rtol"] = 1e-12
    return c


def work(case):
    """Inputs read once and outputs written once; products and edge weights of the path's arithmetic."""
    if case["kind"] == "csr":
        nnz = case["n"] * case["row"] * 0.75
        return {"bytes": 8.0 * nnz + 16.0 * case["n"],
                "flops": 2.0 * nnz * (case["sweeps"] + 1) * case["refinements"]}
    if case["kind"] == "serve":
        ws = [work(_serve_case(case, k)) for k in range(case["requests"])]
        return {m: sum(w[m] for w in ws) for m in ("bytes", "flops")}
    n, np_ = case["nx"] * case["ny"] * case["nz"], case["nx"] * case["ny"] * case["ppv"] ** 2
    es = 8.0 if case["fp64"] else 4.0
    out = 2.0 * np_ + (n - np_ if case["mode"] == "gradient" else 0)
    edges = EDGES_R[case["R"]] * n
    # an edge's weight takes about 20 operations; the solve about 30 products with K
    # (100 for a cloud), the gradient as many again, the edge form a dense 147 x 98 one per node and term
    flops = 30.0 * n if case["mode"] == "single" else edges * (20.0 + 2.0 * (100.0 if case["field"] == "cloud" else 30.0))
    flops *= 2.0 if case["mode"] == "gradient" else 1.0
    if case["mode"] == "aniso":
        nd, ngd = (26, 9) if case["R"] == 1 else (98, 49)
        flops += 30.0 * 2.0 * n * (nd + ngd) * nd * case["S"]
    return {"bytes": es * (n * (1 + case["S"]) + out), "flops": flops}


# ---------------------------------------------------------------------------
# Inputs

def _scene(case, seed):
    """The fields: the repository's recipes, the plume with a seeded turbulent modulation."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    if case["field"] == "plain":
        sc = scenes.make_plain(seed)
    elif case["field"] == "cloud":
        sc = scenes.make_cloud(nx, ny, nz, seed=seed)
    elif case["field"] == "random":
        sc = scenes.make_random(nx, ny, nz, seed=seed, S=case["S"], R=case["R"], M=8192)
    else:
        sc = scenes.make_plume(nx, ny, nz)
        t = np.exp(0.25 * scenes.periodic_grf((nz, ny, nx), (sc.hz, sc.hy, sc.hx), 0.3, seed))
        sc = sc.replace(mu_a=sc.mu_a * t, mu_s=sc.mu_s * t)
    sc = sc.replace(R=case["R"], precision=T.FP64 if case["fp64"] else T.FP32_REFINE, sza=case["sza"],
                    saa=case["saa"], vza=case["vza"], vaa=case["vaa"], albedo=case["albedo"],
                    npx=nx * case["ppv"], npy=ny * case["ppv"])
    if case["mode"] == "c_min":
        sc = sc.replace(c_min=case["c_min"])
    if case["mode"] == "top_k":
        nd = 98 if case["R"] == 2 else 26
        sc = sc.replace(max_couplings=int(case["keep"] * nd * nx * ny * nz))
    return sc


SERVE_SHAPES = ((16, 16, 16), (32, 32, 24), (48, 48, 32), (64, 64, 32), (96, 96, 32))


def _serve_case(case, k):
    """Request k of a queue: the serving mix's shapes and sun heights."""
    r = np.random.default_rng([case["sizes"], k])
    nx, ny, nz = SERVE_SHAPES[int(r.integers(3 if case["small"] else 5))]
    return dict(kind="scene", field="plume", nx=nx, ny=ny, nz=nz, R=2, S=2, fp64=False, mode="full",
                rtol=case["rtol"], sza=round(float(r.uniform(20.0, 75.0)), 1), saa=0.0, vza=30.0, vaa=180.0,
                albedo=0.1, ppv=1)


def _csr(case, seed, dev):
    """Ragged rows (half to all of ``row`` entries) in a band, row sums of K about 0.45 to 0.9."""
    n, row = case["n"], case["row"]
    gen = torch.Generator(device="cpu").manual_seed(seed)
    length = torch.randint(row // 2, row + 1, (n,), generator=gen)
    ptr = torch.zeros(n + 1, dtype=torch.int64)
    ptr[1:] = torch.cumsum(length, 0)
    nnz = int(ptr[-1])
    rows = torch.repeat_interleave(torch.arange(n), length)
    col = (rows + torch.randint(-case["band"], case["band"] + 1, (nnz,), generator=gen)) % n
    val = (torch.rand(nnz, generator=gen) * (1.8 * 0.45 / row)).float()
    s = (0.1 + torch.rand(n, generator=gen)).float()
    return ptr.int().to(dev), col.int().to(dev), val.to(dev), s.to(dev), rows


def prepare(case, seed):
    if case["kind"] == "csr":
        ptr, col, val, s, _ = _csr(case, seed, "cuda")
        return dict(case=case, ptr=ptr, col=col, val=val, s=s,
                    x=torch.empty(case["n"], dtype=torch.float64, device="cuda"))
    if case["kind"] == "serve":
        req = []
        for k in range(case["requests"]):
            sc = _scene(_serve_case(case, k), seed * 1000 + k)
            f = [torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float32).pin_memory() for a in (sc.mu_a, sc.mu_s)]
            req.append((sc, tuple(f), torch.empty((sc.npy, sc.npx), dtype=torch.float32).pin_memory()))
        return dict(case=case, server=T.Server(16 << 30, case["workers"]), req=req)
    sc = _scene(case, seed)
    rn = T.Runner(sc)
    if case["mode"] == "single":
        T.tursca_set_option(rn.handle, T.OPT_SINGLE_SCATTER, 1)
    if case["mode"] == "aniso":
        T.tursca_set_option(rn.handle, T.OPT_ANISO, 1)
    mu_a, mu_s = rn.fields("cuda")
    if case["mode"] == "gradient":
        mu_a.requires_grad_(True)
    return dict(case=case, rn=rn, mu_a=mu_a, mu_s=mu_s)


def run(st):
    case = st["case"]
    if case["kind"] == "csr":
        T.tursca_csr_solve_noalloc(st["ptr"], st["col"], st["val"], case["n"], st["s"], st["x"], case["sweeps"],
                                   case["refinements"], None, torch.cuda.current_stream().cuda_stream)
        return st["x"]
    if case["kind"] == "serve":
        srv = st["server"]
        tickets = [srv.submit(sc, T.FP32_REFINE, case["rtol"], fields=f, out=o) for sc, f, o in st["req"]]
        return [srv.wait(t)[0] for t in tickets]
    if case["mode"] == "gradient":
        # J = sum of L^2 over the detector
        rad = T.render(st["mu_a"], st["rn"], st["mu_s"], case["rtol"])
        (grad,) = torch.autograd.grad(rad.square().sum(), st["mu_a"])
        return {"rad": rad.detach(), "grad": grad}
    rad, refl = st["rn"].run(st["mu_a"], st["mu_s"], rtol=case["rtol"])
    return {"rad": rad, "refl": refl}


# ---------------------------------------------------------------------------
# The method in FP64

def exact(case, seed):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    if case["kind"] == "csr":
        _, col, val, s, rows = _csr(case, seed, dev)
        col, val, rows, s = col.long(), val.double(), rows.to(dev), s.double()
        x = s.clone()
        for _ in range(2000):
            xn = s.index_add(0, rows, val * x[col])
            done = bool((xn - x).abs().max() <= 1e-15 * xn.abs().max())
            x = xn
            if done:
                break
        return x
    if case["kind"] == "serve":
        return [_Method(_scene(c, seed * 1000 + k), c["mode"], dev).radiance()[0]
                for k, c in ((k, _serve_case(case, k)) for k in range(case["requests"]))]
    m = _Method(_scene(case, seed), case["mode"], dev)
    if case["mode"] == "gradient":
        rad, grad = m.gradient()
        return {"rad": rad, "grad": grad}
    rad, refl = m.radiance()
    return {"rad": rad, "refl": refl}


def _pieces(P, V, tend, lphys):
    """Cells and lengths along P + t V, t in [0, tend] (cell units), in order."""
    ts = [0.0, tend]
    for a in range(3):
        if abs(V[a]) > 1e-14:
            lo, hi = sorted((P[a], P[a] + tend * V[a]))
            for f in range(math.ceil(lo - 1e-9), math.floor(hi + 1e-9) + 1):
                t = (f - P[a]) / V[a]
                if 0.0 < t < tend:
                    ts.append(t)
    ts.sort()
    out = []
    for t0, t1 in zip(ts, ts[1:]):
        if t1 - t0 > 1e-12 * tend:
            m = 0.5 * (t0 + t1)
            out.append((*(math.floor(P[a] + m * V[a]) for a in range(3)), (t1 - t0) * lphys))
    return out


def _hg(g, mu):
    return (1.0 - g * g) / (4.0 * math.pi * (1.0 + g * g - 2.0 * g * mu) ** 1.5)


class _Method:
    """One scene in FP64: node arrays are (nz, ny, nx), ground arrays (ny, nx);
    a slot is (from layer, to layer or -1 for the ground, column offset, deposit)."""

    def __init__(self, sc, mode, dev):
        self.sc, self.mode, self.dev = sc, mode, dev
        dt = torch.float64 if sc.precision == T.FP64 else torch.float32
        f64 = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=dt).double().to(dev)  # noqa: E731
        self.mu_a, self.mu_s = f64(sc.mu_a), f64(sc.mu_s)
        self.h = (sc.hx, sc.hy, sc.hz)
        R = sc.R
        rng = range(-R, R + 1)
        self.dirs = [(x, y, z) for z in rng for y in rng for x in rng if math.gcd(math.gcd(x, y), z) == 1]
        # ground chains: members of one line from the ground point, nearest first
        lines = {}
        for z in range(1, R + 1):
            for y in rng:
                for x in rng:
                    q = (2 * x, 2 * y, 2 * z - 1)
                    k = math.gcd(math.gcd(q[0], q[1]), q[2])
                    lines.setdefault(tuple(c // k for c in q), []).append((x, y, z))
        self.gdirs = list(lines.values())
        self.uhat = self._unit([u for u in self.dirs])
        self.ghat = self._unit([(m[0][0], m[0][1], m[0][2] - 0.5) for m in self.gdirs])
        rad = math.pi / 180.0
        a, b = sc.sza * rad, sc.saa * rad
        self.s0 = np.array([-math.sin(a) * math.cos(b), -math.sin(a) * math.sin(b), -math.cos(a)])
        a, b = sc.vza * rad, sc.vaa * rad
        self.v = np.array([math.sin(a) * math.cos(b), math.sin(a) * math.sin(b), math.cos(a)])
        self.mu0 = math.cos(sc.sza * rad)
        M = sc.M
        m = np.arange(M)
        q = m / ((1.0 + math.sqrt(5.0)) / 2.0)
        z = 1.0 - (2.0 * m + 1.0) / M
        lam, r = 2.0 * math.pi * (q - np.floor(q)), np.sqrt(1.0 - z * z)
        self.pts = np.stack([r * np.cos(lam), r * np.sin(lam), z], 1)
        self.wsp = None

    def _unit(self, v):
        p = np.asarray(v, dtype=np.float64) * np.asarray(self.h)
        return p / np.linalg.norm(p, axis=1, keepdims=True)

    def _len(self, v):
        return math.sqrt(sum((c * h) ** 2 for c, h in zip(v, self.h)))

    def _tau_up(self, start, V, lphys, layers):
        """Optical depth to the TOA from ``start`` of each cell (relative, in
        the layer or at its bottom) along V: one path, cut where it leaves.
        layers: the start layers are 0 .. layers - 1."""
        nz = self.sc.nz
        tau = torch.zeros((layers, *self.mu_e.shape[1:]), dtype=torch.float64, device=self.dev)
        for dx, dy, dz, ln in _pieces(start, V, (nz - start[2]) / V[2], lphys):
            n = min(layers, nz - dz)
            if n > 0:
                tau = torch.cat([tau[:n] + ln * torch.roll(self.mu_e[dz:dz + n], (-dy, -dx), (1, 2)), tau[n:]])
        return tau

    def _tau(self, z, P, V, tend, lphys):
        """Optical depth of a short path that starts in layer z (P relative to the cell)."""
        tau = 0.0
        for dx, dy, dz, ln in _pieces(P, V, tend, lphys):
            if 0 <= z + dz < self.sc.nz:
                tau = tau + ln * torch.roll(self.mu_e[z + dz], (-dy, -dx), (0, 1))
        return tau

    def medium(self, mu_a):
        sc = self.sc
        self.mus = self.mu_s.sum(0)
        self.mu_e = mu_a + self.mus
        self.om = torch.where(self.mu_e > 0, self.mus / self.mu_e, torch.zeros_like(self.mu_e))
        self.wsp = torch.where(self.mus > 0, self.mu_s / self.mus, torch.full_like(self.mu_s, 1.0 / sc.n_species))
        self.lamb = sc.albedo * float(self.mus.max())
        V = [-s / h for s, h in zip(self.s0, self.h)]
        tau = self._tau_up((0.5, 0.5, 0.0), V, 1.0, sc.nz + 1)  # from the bottom of layer Z (the ground: Z = 0)
        ts = torch.exp(-tau)
        p = sc.f0 * self.mu0 * sc.hx * sc.hy
        self.e1 = self.om * p * ts[1:] * -torch.expm1(-self.mu_e * sc.hz / self.mu0)
        self.e1g = sc.albedo * p * ts[0]

    def chains(self):
        """Deposits: self.slots[d] = [(z, target layer or -1, (dy, dx), P)] per direction
        (atmospheric, then ground), and the coupling C per direction (< 0: no receiver)."""
        sc, nz = self.sc, self.sc.nz
        self.slots, self.C = [], []
        for u in self.dirs:
            L, kmax = self._len(u), sc.R // max(abs(c) for c in u)
            tinf = self._tau_up((0.5, 0.5, 0.5), u, L, nz) if u[2] > 0 else None
            out, cl = [], []
            for z in range(nz):
                pre, zc, k, C = 0.0, z, 0, -torch.ones_like(self.mus[z])
                col = lambda a, k: torch.roll(a, (-k * u[1], -k * u[0]), (0, 1))  # noqa: E731
                done = False
                while k < kmax and not done:
                    zn = zc + 0.5 + u[2]
                    if zn > nz:  # leaves through the TOA: the rest goes to the last node
                        t = col(tinf[zc], k)
                        out.append((z, zc, (k * u[1], k * u[0]), torch.exp(-pre) * -torch.expm1(-t)
                                    if k else -torch.expm1(-t)))
                        done = True
                    elif zn < 0:  # hits the ground
                        th = (zc + 0.5) / -u[2]
                        t = col(self._tau(zc, (0.5, 0.5, 0.5), u, th, L), k)
                        T0 = torch.exp(-pre) if k else torch.ones_like(t)
                        out.append((z, zc, (k * u[1], k * u[0]), T0 * -torch.expm1(-t)))
                        hit = [0.5 + k * u[a] + th * u[a] for a in range(2)]
                        ax = [[round(c) - 1, round(c)] if abs(c - round(c)) < 1e-9 else [math.floor(c)] for c in hit]
                        for x in ax[0]:
                            for y in ax[1]:
                                out.append((z, -1, (y, x), T0 * torch.exp(-t) / (len(ax[0]) * len(ax[1]))))
                        if k == 0:
                            C = torch.sqrt(self.mus[z] * self.lamb) / (th * L)
                        done = True
                    else:
                        t = col(self._tau(zc, (0.5, 0.5, 0.5), u, 1.0, L), k)
                        T0 = torch.exp(-pre) if k else torch.ones_like(t)
                        k, zc = k + 1, zc + u[2]
                        out.append((z, zc, (k * u[1], k * u[0]), T0 * -torch.expm1(-t)))
                        pre = pre + t
                        if k == 1:
                            C = torch.sqrt(self.mus[z] * col(self.mus[zc], 1)) / L
                if not done:  # the stencil ended inside the domain
                    T0 = torch.exp(-pre)
                    out.append((z, zc, (k * u[1], k * u[0]),
                                T0 * -torch.expm1(-col(tinf[zc], k)) if u[2] > 0 else T0))
                cl.append(C)
            self.slots.append(out)
            self.C.append(torch.stack(cl))
        for mem in self.gdirs:
            out, pre, P = [], 0.0, (0.5, 0.5, 0.0)
            for k, (x, y, z) in enumerate(mem):
                Q = (x + 0.5, y + 0.5, z - 0.5)
                V = [b - a for a, b in zip(P, Q)]
                t = self._tau(0, P, V, 1.0, self._len(V))
                T0 = torch.exp(-pre) if k else torch.ones_like(t)
                out.append((0, z - 1, (y, x), T0 * -torch.expm1(-t)))
                if k == 0:
                    self.C.append(torch.sqrt(self.lamb * torch.roll(self.mus[z - 1], (-y, -x), (0, 1))) / self._len(V))
                pre, P = pre + t, Q
            x, y, z = mem[-1]
            V = (mem[0][0], mem[0][1], mem[0][2] - 0.5)
            t = torch.roll(self._tau_up((0.5, 0.5, 0.5), V, self._len(V), sc.nz)[z - 1], (-y, -x), (0, 1))
            out.append((0, z - 1, (y, x), torch.exp(-pre) * -torch.expm1(-t)))
            self.slots.append(out)

    def weights(self):
        """W_iso, W_sun (direction, node) and the ground's W (ground direction, column)."""
        sc, dev, nd = self.sc, self.dev, len(self.dirs)
        cos_u, cos_g = self.pts @ self.uhat.T, self.pts @ self.ghat.T
        mu = self.pts @ self.s0
        hg = np.stack([_hg(g, mu) for g in sc.g])
        up = self.pts[:, 2] > 0.0
        C, Cg = torch.stack(self.C[:nd]).reshape(nd, -1), torch.stack(self.C[nd:]).reshape(len(self.gdirs), -1)
        thr = 0.0
        if self.mode == "c_min":
            thr = sc.c_min
        elif self.mode == "top_k":
            every = torch.cat([C[C >= 0], Cg.reshape(-1)])
            if sc.max_couplings < every.numel():
                thr = max(float(torch.sort(every, descending=True)[0][sc.max_couplings]), 5e-324)

        def cells(cosines, C, pts_w, everyone):
            """Shares of the lattice weights pts_w (rows) by kept direction, per source."""
            w = torch.as_tensor(np.ascontiguousarray(pts_w / everyone[:, None]), device=dev)  # (rows, points)
            n = cosines.shape[1]
            rank = torch.as_tensor(np.argsort(-cosines, axis=1, kind="stable"), device=dev)
            if thr <= 0.0:
                q = torch.zeros((len(w), n), dtype=torch.float64, device=dev).index_add_(1, rank[:, 0], w)
                return q[:, :, None]
            kept, inv = torch.unique(((C < 0) | (C > thr)).T, dim=0, return_inverse=True)
            q = torch.zeros((len(w), len(kept), n), dtype=torch.float64, device=dev)
            for b in range(0, len(kept), 64):
                kb = kept[b:b + 64]
                near = torch.full((len(kb), len(rank)), n, dtype=torch.int64, device=dev)
                for p in range(n - 1, -1, -1):  # the first kept direction in each point's ranking
                    near = torch.where(kb[:, rank[:, p]], rank[:, p], near)
                for r in range(len(w)):
                    full = torch.zeros((len(kb), n + 1), dtype=torch.float64, device=dev)
                    q[r, b:b + 64] = full.scatter_add_(1, near, w[r].expand(len(kb), -1))[:, :n]
            return q[:, inv].permute(0, 2, 1)  # (rows, direction, source)

        def route(C, q):
            has = (C >= 0).double()
            sq, sqc = (has * q).sum(0), (has * q * C.clamp(min=0)).sum(0)
            on = (sqc > 0) & (sc.coupling != 0)
            f = torch.where(on, sq / torch.where(on, sqc, torch.ones_like(sqc)), torch.zeros_like(sqc))
            return q * torch.where(on & (C >= 0), C * f, torch.ones_like(C))

        q = cells(cos_u, C, np.concatenate([np.ones((1, sc.M)), hg]), np.concatenate([[sc.M], hg.sum(1)]))
        qs = (self.wsp.reshape(sc.n_species, 1, -1) * q[1:]).sum(0)
        shape = (nd, *self.mus.shape)
        self.Wi, self.Ws = route(C, q[0]).reshape(shape), route(C, qs).reshape(shape)
        zw = np.where(up, self.pts[:, 2], 0.0)
        qg = cells(cos_g[up], Cg, zw[up][None], np.array([zw.sum()]))
        self.Wg = route(Cg, qg[0]).reshape(len(self.gdirs), *self.mus.shape[1:])
        self.CA = C.reshape(shape)

    def _src(self, d, z, W):
        return W[d][z] if d < len(self.dirs) else self.Wg[d - len(self.dirs)]

    def apply(self, x, xg, W, take=None):
        """Deposits of the sources' power (x on voxels, xg on the ground): the
        arriving power, scattered (om, albedo); take(d, layer, power) sees each arrival."""
        nz = self.sc.nz
        acc = [0.0] * (nz + 1)
        for d, out in enumerate(self.slots):
            for z, zt, (dy, dx), P in out:
                src = (W[d][z] * x[z] if W is not None else x[d][z]) if d < len(self.dirs) else \
                    (self.Wg[d - len(self.dirs)] * xg if W is not None else xg[d - len(self.dirs)])
                a = torch.roll(P * src, (dy, dx), (0, 1))
                rho = self.om[zt] if zt >= 0 else self.sc.albedo
                if take is not None:
                    take(d, zt, rho * a)
                else:
                    acc[zt] = acc[zt] + rho * a
        return None if take is not None else (torch.stack(acc[:nz]), acc[nz] + torch.zeros_like(xg))

    def matrix(self):
        """K as a sparse FP64 matrix over (voxels, ground columns)."""
        sc = self.sc
        nxy, na = sc.nx * sc.ny, sc.nx * sc.ny * sc.nz
        idx = torch.arange(nxy, device=self.dev).reshape(sc.ny, sc.nx)
        rows, cols, vals = [], [], []
        with torch.no_grad():
            for d, out in enumerate(self.slots):
                for z, zt, (dy, dx), P in out:
                    t = torch.roll(idx, (-dy, -dx), (0, 1))
                    rho = torch.roll(self.om[zt], (-dy, -dx), (0, 1)) if zt >= 0 else sc.albedo
                    rows.append((t + (zt * nxy if zt >= 0 else na)).reshape(-1).int())
                    cols.append((idx + (z * nxy if d < len(self.dirs) else na)).reshape(-1).int())
                    vals.append((rho * self._src(d, z, self.Wi) * P).reshape(-1))
            r, c, v = torch.cat(rows), torch.cat(cols), torch.cat(vals)
        return r, c, v, na + nxy

    @staticmethod
    def _csr(r, c, v, n):
        o = torch.argsort(r)
        ptr = torch.zeros(n + 1, dtype=torch.int32, device=r.device)
        ptr[1:] = torch.cumsum(torch.bincount(r, minlength=n), 0)
        return torch.sparse_csr_tensor(ptr, c[o], v[o], (n, n))

    @staticmethod
    def solve(K, s, tol=2e-14, m=60):
        """Restarted GMRES on (I - K) x = s."""
        x, bn = torch.zeros_like(s), float(s.norm())
        for _ in range(200):
            r = s - x + K @ x
            beta = float(r.norm())
            if bn == 0.0 or beta <= tol * bn:
                break
            V = torch.zeros((m + 1, len(s)), dtype=s.dtype, device=s.device)
            H = np.zeros((m + 1, m))
            V[0] = r / beta
            k = 0
            for k in range(m):
                w = V[k] - K @ V[k]
                h = V[:k + 1] @ w
                w = w - h @ V[:k + 1]
                h2 = V[:k + 1] @ w
                w = w - h2 @ V[:k + 1]
                H[:k + 1, k] = (h + h2).cpu().numpy()
                H[k + 1, k] = float(w.norm())
                if H[k + 1, k] <= 1e-15 * beta:
                    break
                V[k + 1] = w / H[k + 1, k]
                if k % 10 == 9:
                    e = np.zeros(k + 2)
                    e[0] = beta
                    y = np.linalg.lstsq(H[:k + 2, :k + 1], e, rcond=None)[0]
                    if np.linalg.norm(H[:k + 2, :k + 1] @ y - e) <= 0.3 * tol * bn:
                        break
            e = np.zeros(k + 2)
            e[0] = beta
            y = np.linalg.lstsq(H[:k + 2, :k + 1], e, rcond=None)[0]
            x = x + torch.as_tensor(y, device=s.device) @ V[:k + 1]
        return x

    def _theta(self, mu):
        """The species mixture's HG at the cosine mu, per voxel."""
        return sum(self.wsp[k] * _hg(float(g), float(mu)) for k, g in enumerate(self.sc.g))

    def detector(self, emis, xg):
        """Lines of sight from the TOA down to each pixel's ground point."""
        sc = self.sc
        npx, npy, nz = sc.npx, sc.npy, sc.nz
        rad = torch.zeros((npy, npx), dtype=torch.float64, device=self.dev)
        gx, gy = (np.arange(npx) + 0.5) * sc.nx / npx, (np.arange(npy) + 0.5) * sc.ny / npy
        ln = nz * sc.hz / self.v[2]
        vol = sc.hx * sc.hy * sc.hz
        px, py = np.round(gx % 1.0, 9), np.round(gy % 1.0, 9)
        for fx in np.unique(px):
            for fy in np.unique(py):
                a, b = np.nonzero(px == fx)[0], np.nonzero(py == fy)[0]
                X = torch.as_tensor(np.floor(gx[a]).astype(np.int64), device=self.dev)
                Y = torch.as_tensor(np.floor(gy[b]).astype(np.int64), device=self.dev)[:, None]
                tau, L = 0.0, 0.0
                V = [c / h for c, h in zip(self.v, self.h)]
                for dx, dy, dz, ds in reversed(_pieces((fx, fy, 0.0), V, ln, 1.0)):
                    me, em = (f[dz][(Y + dy) % sc.ny, (X + dx) % sc.nx] for f in (self.mu_e, emis))
                    f = torch.where(me > 0, -torch.expm1(-me * ds) / torch.where(me > 0, me, torch.ones_like(me)),
                                    torch.full_like(me, ds))
                    L = L + (torch.exp(-tau) if torch.is_tensor(tau) else 1.0) * f * em / vol
                    tau = tau + me * ds
                L = L + torch.exp(-tau) * (self.e1g + xg)[Y % sc.ny, X % sc.nx] / (math.pi * sc.hx * sc.hy)
                rad = rad.index_put((torch.as_tensor(b, device=self.dev)[:, None],
                                     torch.as_tensor(a, device=self.dev)[None]), L)
        return rad

    def emission(self, x, xg):
        """E toward the instrument: the first scattering and every arrival by its direction."""
        mu = np.concatenate([self.uhat, self.ghat]) @ self.v
        th = [self._theta(m) for m in mu]
        acc = [self.e1[z] * self._theta(float(self.s0 @ self.v))[z] for z in range(self.sc.nz)]

        def take(d, zt, a):
            if zt >= 0:
                acc[zt] = acc[zt] + th[d][zt] * a

        self.apply(x, xg, self.Wi, take)
        self.apply(self.e1, self.e1g, self.Ws, take)
        return torch.stack(acc)

    def _edge_form(self):
        """X(node, arrival direction) by the series, then E and the ground's total."""
        sc, nd = self.sc, len(self.dirs)
        w = np.concatenate([self.uhat, self.ghat])
        cell = np.argmax(self.pts @ self.uhat.T, axis=1)
        Q = []
        for g in sc.g:
            h = _hg(float(g), w @ self.pts.T)
            q = np.zeros((len(w), nd))
            for u in range(nd):
                q[:, u] = h[:, cell == u].sum(1)
            Q.append(torch.as_tensor(q / h.sum(1, keepdims=True), device=self.dev))
        n = self.mus.numel()
        wsp, C = self.wsp.reshape(sc.n_species, n), self.CA.reshape(nd, n)
        has = (C >= 0).double()
        sq = sum(wsp[k] * (Q[k] @ has) for k in range(len(Q)))
        sqc = sum(wsp[k] * (Q[k] @ (has * C.clamp(min=0))) for k in range(len(Q)))
        on = (sqc > 0) & (sc.coupling != 0)
        zf = torch.where(on, sq / torch.where(on, sqc, torch.ones_like(sqc)), torch.zeros_like(sqc))  # (w, node)
        shape, gshape = (len(w), *self.mus.shape), (len(w), *self.mus.shape[1:])

        def arrivals(x, xg, W):
            X, Xg = torch.zeros(shape, dtype=torch.float64, device=self.dev), \
                torch.zeros(gshape, dtype=torch.float64, device=self.dev)

            def take(d, zt, a):
                if zt >= 0:
                    X[d, zt] += a
                else:
                    Xg[d] += a

            self.apply(x, xg, W, take)
            return X, Xg

        Xs, Xsg = arrivals(self.e1, self.e1g, self.Ws)
        X, Xg = Xs, Xsg
        for _ in range(3000):
            Xf = X.reshape(len(w), n)
            Lc = sum(wsp[k] * (Q[k].T @ (Xf * zf)) for k in range(len(Q))) * C.clamp(min=0)
            L1 = sum(wsp[k] * (Q[k].T @ Xf) for k in range(len(Q)))  # no receiver: routed with weight 1
            Lo = sum(wsp[k] * (Q[k].T @ torch.where(on, torch.zeros_like(Xf), Xf)) for k in range(len(Q)))
            L = torch.where(C >= 0, Lc + Lo, L1).reshape(nd, *self.mus.shape)
            A, Ag = arrivals(L, self.Wg * Xg.sum(0), None)
            Xn, Xng = Xs + A, Xsg + Ag
            done = float((Xn - X).norm() + (Xng - Xg).norm()) <= 1e-13 * float(Xn.norm())
            X, Xg = Xn, Xng
            if done:
                break
        th = torch.stack([self._theta(m) for m in w @ self.v])
        E = self.e1 * self._theta(float(self.s0 @ self.v)) + (th * X).sum(0)
        return E, Xg.sum(0)

    def radiance(self):
        sc = self.sc
        self.medium(self.mu_a)
        if self.mode == "single":
            rad = self.detector(self.e1 * self._theta(float(self.s0 @ self.v)), torch.zeros_like(self.e1g))
        else:
            self.chains()
            self.weights()
            if self.mode == "aniso":
                rad = self.detector(*self._edge_form())
            else:
                s = torch.cat([a.reshape(-1) for a in self.apply(self.e1, self.e1g, self.Ws)])
                x = self.solve(self._csr(*self.matrix()), s)
                x, xg = x[:self.mus.numel()].reshape(self.mus.shape), x[self.mus.numel():].reshape(self.e1g.shape)
                rad = self.detector(self.emission(x, xg), xg)
        return rad, math.pi * rad / (self.mu0 * sc.f0)

    def gradient(self):
        """rad and d(sum rad^2)/d mu_a: the adjoint system, then one backward pass at fixed x."""
        mu_a = self.mu_a.clone().requires_grad_(True)
        self.medium(mu_a)
        self.chains()
        self.weights()
        S, Sg = self.apply(self.e1, self.e1g, self.Ws)
        s = torch.cat([S.reshape(-1), Sg.reshape(-1)])
        r, c, v, n = self.matrix()
        x = self.solve(self._csr(r, c, v, n), s.detach())
        na = self.mus.numel()
        X = x[:na].reshape(self.mus.shape).requires_grad_(True)
        Xg = x[na:].reshape(self.e1g.shape).requires_grad_(True)
        rad = self.detector(self.emission(X, Xg), Xg)
        w = 2.0 * rad.detach()
        gx = torch.autograd.grad((w * rad).sum(), [X, Xg], retain_graph=True)
        lam = self.solve(self._csr(c, r, v, n), torch.cat([g.reshape(-1) for g in gx]))
        A, Ag = self.apply(X.detach(), Xg.detach(), self.Wi)
        J = (w * rad).sum() + (lam[:na].reshape(A.shape) * (S + A)).sum() + (lam[na:].reshape(Ag.shape) * (Sg + Ag)).sum()
        (grad,) = torch.autograd.grad(J, [mu_a])
        return rad.detach(), grad
