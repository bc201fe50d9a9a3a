"""Measured cases: what users of this library have it compute, through its public entry points.

Every case is one call sequence of a solver run: advance a prepared phonon state by a few time
steps (or implicit iterations, or one gradient evaluation) and take the results a program takes,
the lattice temperature on the host and the state where the program keeps it on the device.  Sizes
are those of the workloads in ``paper_2306_14181_gb300.inputs`` and odd sizes around them.

``exact`` restates the schemes in plain 64-bit torch, without the library: limited second-order
upwind faces, the wall types, the lattice temperature, the first-order implicit increment, the
interface and, by automatic differentiation step by step, the gradients of a probe temperature.
"""
import math

import numpy as np
import torch

from paper_2306_14181_gb300 import bte, inputs

ISO, DIF, SPE, PER = 0, 1, 2, 3
_STORE = {"f32": bte.BTE_STORE_F32, "f16": bte.BTE_STORE_F16, "bf16": bte.BTE_STORE_BF16}
_DTYPE = {"f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}
_LIMITER = {"first": bte.BTE_LIM_FIRST_ORDER, "minmod": bte.BTE_LIM_MINMOD, "vanalbada": bte.BTE_LIM_VANALBADA}


# -------------------------------------------------------------------------------------------
# the cases
# -------------------------------------------------------------------------------------------
def _case(name, family, nx, ny, nz, nb, ntheta, nphi, steps, **more):
    c = dict(name=name, family=family, nx=nx, ny=ny, nz=nz, nb=nb, ntheta=ntheta, nphi=nphi, steps=steps,
             storage="f32", rounding="nearest", limiter="vanalbada")
    c.update(more)
    return c


def listed():
    return [
        # the cross-plane film between two isothermal walls: the smallest problem, a parameter
        # study runs thousands of them
        _case("film_1d", "film", 100, 1, 1, 10, 16, 0, 200),
        # the transient grating: one gray band, many directions, long runs of small steps
        _case("grating_1d", "grating", 1000, 1, 1, 1, 512, 0, 128),
        # in-plane conduction: marching to the steady state with the residual stop
        _case("inplane_steady_2d", "inplane", 64, 64, 1, 3, 2, 3, 128),
        # the device hot spot, in the two storages it is run with
        _case("hotspot_2d_f32", "hotspot", 256, 256, 1, 40, 4, 4, 10),
        _case("hotspot_2d_f16", "hotspot", 256, 256, 1, 40, 4, 4, 10, storage="f16"),
        # a device cross-section whose extents nobody rounded, with the fields a plot needs
        _case("odd_2d_f32", "hotspot", 203, 157, 1, 24, 3, 4, 10, moments=True),
        # the laser-heated block, in both storages
        _case("laser_3d_f32", "laser", 128, 128, 64, 40, 4, 3, 6),
        _case("laser_3d_f16", "laser", 128, 128, 64, 40, 4, 3, 6, storage="f16"),
        # gradients of a probe temperature with respect to the source and the relaxation times
        _case("film_adjoint_2d", "adjoint2d", 128, 128, 1, 20, 2, 4, 40, ckpt=10),
        _case("block_adjoint_3d_f16", "adjoint3d", 96, 96, 96, 32, 4, 3, 4, ckpt=2, storage="f16"),
        # the steady state of the hot spot by implicit iterations
        _case("implicit_2d", "implicit", 256, 256, 1, 40, 4, 4, 4),
        # two materials side by side
        _case("interface_2d", "pair", 256, 128, 1, 40, 4, 4, 10),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same kinds: rows of any length (multiples of four and others), 2 to 40
    bands, few and many directions, the three limiters and storages.  The sizes are cut back until
    the pass costs less than the largest listed one."""
    family = rng.choice(["film", "grating", "inplane", "hotspot", "hotspot", "hotspot", "laser", "laser", "laser",
                         "adjoint2d", "adjoint3d", "implicit", "pair"])
    nb = _logint(rng, 2, 40)
    nt, npz = rng.choice([(2, 2), (2, 3), (3, 3), (2, 4), (3, 4), (4, 4)])
    lim = rng.choice(["vanalbada", "vanalbada", "vanalbada", "minmod", "first"])
    store, rnd = rng.choice([("f32", "nearest")] * 3 + [("f16", "nearest"), ("f16", "nearest"), ("bf16", "stochastic")])

    def extent(lo, hi):
        n = _logint(rng, lo, hi)
        return n if rng.random() < 0.5 else max(lo, n // 4 * 4)

    if family == "film":
        return _case("", "film", extent(24, 400), 1, 1, rng.randint(2, 16), rng.choice([8, 16, 24]), 0,
                     _logint(rng, 50, 400), limiter=lim)
    if family == "grating":
        return _case("", "grating", extent(200, 4000), 1, 1, rng.choice([1, 1, 2, 4]), rng.choice([64, 128, 256, 512]),
                     0, _logint(rng, 20, 200))
    if family == "inplane":
        return _case("", "inplane", extent(24, 200), extent(24, 160), 1, 3, nt, npz, _logint(rng, 40, 160))
    if family in ("hotspot", "implicit", "pair", "adjoint2d"):
        nx, ny = extent(32, 400), extent(32, 400)
        if family == "hotspot":
            return _case("", family, nx, ny, 1, nb, nt, npz, rng.randint(2, 12), storage=store, rounding=rnd,
                         limiter=lim, moments=rng.random() < 0.3)
        if family == "implicit":
            return _case("", family, nx, ny, 1, nb, nt, npz, rng.randint(1, 4))
        if family == "pair":
            return _case("", family, nx, ny, 1, nb, nt, npz, rng.randint(2, 10), limiter=lim)
        if rng.random() < 0.5:
            nx = rng.choice([96, 128, 256])  # rows that many device studies use
        return _case("", family, nx, ny, 1, min(nb, 20), nt, npz, rng.randint(4, 20), ckpt=rng.randint(2, 6), limiter=lim)
    nx, ny, nz = extent(20, 140), extent(16, 128), extent(8, 64)
    if family == "laser":
        steps = rng.randint(2, 6)
        while nx * ny * nz * nb * 8 * nt * npz * steps > 4.0e9:
            nb = max(1, nb // 2)
            if nb == 1:
                nz = max(8, nz // 2)
        return _case("", family, nx, ny, nz, nb, nt, npz, steps, storage=store, rounding=rnd, limiter=lim)
    if rng.random() < 0.5:
        nx = rng.choice([64, 96, 128])
    steps = rng.randint(2, 6)
    while nx * ny * nz * nb * 8 * nt * npz * steps > 1.2e9:
        nb = max(1, nb // 2)
        if nb == 1:
            nz = max(8, nz // 2)
    return _case("", family, nx, ny, nz, nb, nt, npz, steps, ckpt=rng.randint(1, 3),
                 storage="f32" if store == "bf16" else store, limiter=lim)


def _workload(case):
    """The workload dict(s) of a case: [cfg] or [cfg of side A, cfg of side B]."""
    f, nx, ny, nz = case["family"], case["nx"], case["ny"], case["nz"]
    nb, nt, npz = case["nb"], case["ntheta"], case["nphi"]
    if f == "film":
        cfg = inputs.film_1d(nx=nx)
        cfg["C"], cfg["v"], cfg["tau"] = inputs.bands(1001, nb)
        cfg.update(nb=nb, quad=("gl1d", nt))
        cfg["dt"] = inputs.cfl_time_step(cfg["h"][:1], cfg["v"])
        return [cfg]
    if f == "grating":
        return [inputs.ttg_1d(xi=1.0, nx=nx, ntheta=nt, nb=nb)]
    if f == "inplane":
        return [inputs.inplane_film_2d(nx=nx, ny=ny, ntheta=nt, nphi=npz)]
    if f in ("hotspot", "implicit"):
        return [inputs.hotspot_2d(nx=nx, ny=ny, nb=nb, ntheta=nt, nphi=npz)]
    if f == "laser":
        return [inputs.laser_3d(nx=nx, ny=ny, nz=nz, nb=nb, ntheta=nt, nphi=npz)]
    if f == "adjoint2d":
        return [inputs.film_adjoint_2d(nx=nx, ny=ny, nb=nb, ntheta=nt, nphi=npz)]
    if f == "adjoint3d":
        return [inputs.block_adjoint_3d(nx=nx, ny=ny, nz=nz, nb=nb, ntheta=nt, nphi=npz)]
    pair = inputs.interface_2d(nx=nx, ny=ny, nb=nb, ntheta=nt, nphi=npz)
    A, B = pair["A"], pair["B"]
    A["iface"], B["iface"] = pair["wall_a"], pair["wall_b"]
    A["beta_ab"], A["beta_ba"] = pair["beta_ab"], pair["beta_ba"]
    return [A, B]


def _amplitude(case):
    """Size (K) of the temperature field the state starts from, and the scale of 16-bit codes."""
    return {"hotspot": (5.0, 10.0), "laser": (0.5, 1.0), "adjoint3d": (0.5, 1.0)}.get(case["family"], (0.5, 1.0))


# -------------------------------------------------------------------------------------------
# inputs
# -------------------------------------------------------------------------------------------
def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _quadrature(cfg):
    """Directions [nd, 3] and weights [nd] of the library's rules (Gauss-Legendre in the cosine of
    the polar angle, Gauss-Legendre in the azimuth of each octant)."""
    q = cfg["quad"]
    if q[0] == "gl1d":
        mu, w = np.polynomial.legendre.leggauss(q[1])
        s = np.zeros((q[1], 3))
        s[:, 0] = mu
        return s, 2 * math.pi * w
    x, wx = np.polynomial.legendre.leggauss(q[1])
    y, wy = np.polynomial.legendre.leggauss(q[2])
    mu, wm = 0.5 * (x + 1), 0.5 * wx
    ph, wp = 0.25 * math.pi * (y + 1), 0.25 * math.pi * wy
    s, w = [], []
    for o in range(8):
        sg = [-1.0 if o >> a & 1 else 1.0 for a in range(3)]
        for m, a in zip(mu, wm):
            for p, b in zip(ph, wp):
                st = math.sqrt(1 - m * m)
                s.append([sg[0] * st * math.cos(p), sg[1] * st * math.sin(p), sg[2] * m])
                w.append(a * b)
    return np.array(s), np.array(w)


class _Fields:
    """The start state of one context: a smooth temperature field of a few modes, direction- and
    band-dependent departures from equilibrium (as a flux makes them) and a little roughness."""

    def __init__(self, cfg, case, seed, side):
        self.cfg, self.case = cfg, case
        self.nx, self.ny, self.nz = cfg["n"]
        self.nb = len(cfg["C"])
        self.s, self.w = _quadrature(cfg)
        self.nd = len(self.w)
        self.W = float(np.sum(self.w))
        self.A, self.Ts = _amplitude(case)
        dev = _device()
        rng = np.random.default_rng([int(seed), side, 77])
        self.seed = int(seed) * 8 + side

        def modes(n):
            z = torch.arange(self.nz, device=dev, dtype=torch.float64)[:, None, None] / max(self.nz, 8)
            y = torch.arange(self.ny, device=dev, dtype=torch.float64)[None, :, None] / max(self.ny, 8)
            x = torch.arange(self.nx, device=dev, dtype=torch.float64)[None, None, :] / max(self.nx, 8)
            f = 0
            for _ in range(n):
                k, p = rng.uniform(0.5, 9.0, 3), rng.uniform(0, 2 * math.pi, 3)
                f = f + float(rng.standard_normal()) * (torch.cos(k[0] * x + p[0]) * torch.cos(k[1] * y + p[1]) * torch.cos(k[2] * z + p[2]))
            return f

        self.T = (self.A * (0.3 + 0.5 * modes(3))).to(torch.float32)
        self.G = torch.stack([self.A * 0.4 * modes(2) for _ in range(3)]).to(torch.float32)
        lam = np.asarray(cfg["v"]) * np.asarray(cfg["tau"])
        self.g = lam / (lam + 50e-9)  # bands of long mean free path are further from equilibrium
        self.sdir = torch.tensor(self.s, device=dev, dtype=torch.float32)

    def band(self, k):
        """e of band k over C_k / W, float32 [nd, nz, ny, nx]."""
        gen = torch.Generator(device=self.T.device).manual_seed(self.seed * 1000 + k)
        t = torch.randn((self.nd, self.nz, self.ny, self.nx), generator=gen, device=self.T.device).mul_(0.004 * self.A)
        t += self.T
        for a in range(3):
            t += float(self.g[k]) * self.sdir[:, a].view(-1, 1, 1, 1) * self.G[a]
        return t

    def scale(self, k):
        """s_k of the 16-bit codes as the library holds it (single precision)."""
        return float(np.float32(self.cfg["C"][k] * self.Ts / self.W))

    def stored(self):
        """(state in the storage format, code reference or None)."""
        kind = self.case["storage"]
        out = torch.empty((self.nb, self.nd, self.nz, self.ny, self.nx), dtype=_DTYPE[kind], device=self.T.device)
        for k in range(self.nb):
            t = self.band(k)
            if kind == "f32":
                out[k] = t * float(self.cfg["C"][k] / self.W)
            else:
                out[k] = ((t - self.T) / self.Ts).to(_DTYPE[kind])
            del t
        return out, None if kind == "f32" else self.T.clone()


def _probe(cfg):
    return inputs.probe_weights(cfg)


def prepare(case, seed):
    state = {"case": case, "ctx": [], "out": [], "ref": []}
    for side, cfg in enumerate(_workload(case)):
        f = _Fields(cfg, case, seed, side)
        opts = dict(storage=_STORE[case["storage"]], limiter=_LIMITER[case["limiter"]], T_scale=f.Ts, seed=1 + seed % 1000,
                    rounding=bte.BTE_ROUND_STOCHASTIC if case["rounding"] == "stochastic" else bte.BTE_ROUND_NEAREST)
        if "iface" in cfg:
            cfg["bc"][cfg["iface"]] = bte.BTE_BC_INTERFACE
        ctx = bte.bte_from_workload(cfg, **opts)
        Q = inputs.source_field(cfg)
        if Q is not None:
            bte.bte_set_source(ctx, Q, inputs.source_amplitudes(cfg, 400))
        e, R = f.stored()
        bte.bte_set_state(ctx, e, ref=R)
        bte.bte_synchronize(ctx)
        state["ctx"].append(ctx)
        state["out"].append(e)  # where the program keeps the state it takes back
        state["ref"].append(R)
        if case["family"] in ("adjoint2d", "adjoint3d"):
            state["probe"] = _probe(cfg)
    if case["family"] == "pair":
        a, b = _workload(case)
        bte.bte_interface(state["ctx"][0], a["iface"], state["ctx"][1], b["iface"], a["beta_ab"], a["beta_ba"])
    return state


# -------------------------------------------------------------------------------------------
# one pass
# -------------------------------------------------------------------------------------------
def _results(state, i):
    """The lattice temperature on the host (single precision, as it is formed) and the state."""
    ctx = state["ctx"][i]
    out = {"TL": bte.bte_lattice_temperature(ctx).astype(np.float32)}
    bte.bte_get_state(ctx, out=state["out"][i], ref=state["ref"][i])
    out["state"] = state["out"][i]
    if state["ref"][i] is not None:
        out["ref"] = state["ref"][i]
    return out


def run(state):
    case, ctx = state["case"], state["ctx"][0]
    f = case["family"]
    if f in ("adjoint2d", "adjoint3d"):
        J, gQ, gt = bte.bte_adjoint(ctx, case["steps"], state["probe"], case["ckpt"])
        return {"J": np.float32(J), "dJ_dQ": gQ.astype(np.float32), "dJ_dlogtau": gt.astype(np.float32)}
    if f == "pair":
        bte.bte_step_pair(ctx, state["ctx"][1], case["steps"])
        return [_results(state, 0), _results(state, 1)]
    if f == "implicit":
        bte.bte_sis_iterate(ctx, case["steps"])
    elif f == "inplane":
        bte.bte_run_steady(ctx, case["steps"], max(1, case["steps"] // 2), 1e-9, 1e-9)
    else:
        bte.bte_step(ctx, case["steps"])
    out = _results(state, 0)
    if case.get("moments"):
        T, _, q = bte.bte_moments(ctx)
        out["T"], out["q"] = T.astype(np.float32), q.astype(np.float32)
    return out


def _sizes(case):
    nd = case["ntheta"] if case["family"] in ("film", "grating") else 8 * case["ntheta"] * case["nphi"]
    sides = 2 if case["family"] == "pair" else 1
    return case["nx"] * case["ny"] * case["nz"], sides * case["nx"] * case["ny"] * case["nz"] * case["nb"] * nd


def work(case):
    """A step reads the state and writes the next one; a state that fits the chip (100 MB) is read
    and written once a pass.  An implicit iteration writes and reads the explicit residual too; a
    reverse step reads the adjoint and the state and writes the adjoint, after a forward run and
    its recomputation.  Taking the state back is one read and one write."""
    ncell, nelem = _sizes(case)
    es = 4 if case["storage"] == "f32" else 2
    dim = 1 + (case["ny"] > 1) + (case["nz"] > 1)
    n = case["steps"]
    f = case["family"]
    flops = nelem * n * (24.0 * dim + 8)
    if f in ("adjoint2d", "adjoint3d"):
        return {"bytes": nelem * n * (2 * 2 * es + 8.0 + es), "flops": 4 * flops}
    per = 2.0 * es * nelem
    if f == "implicit":
        per *= 2
    if per / 2 <= 100e6:
        n = 1
    return {"bytes": per * n + 2.0 * es * nelem + 4.0 * ncell + (es * nelem if case.get("moments") else 0.0),
            "flops": flops}


# -------------------------------------------------------------------------------------------
# the same in 64 bits, without the library
# -------------------------------------------------------------------------------------------
def _limit(kind, a, b):
    if kind == "first":
        return torch.zeros_like(a)
    ab = a * b
    if kind == "minmod":
        return torch.where(ab > 0, torch.where(a.abs() < b.abs(), a, b), torch.zeros_like(a))
    pos = ab > 0
    den = torch.where(pos, a * a + b * b, torch.ones_like(a))
    return torch.where(pos, ab * (a + b), torch.zeros_like(a)) / den


class _Plain:
    """One material's scheme in 64 bits, band by band; fields [nd, nz, ny, nx]."""

    def __init__(self, cfg, limiter):
        dev = _device()
        self.cfg, self.limiter = cfg, limiter
        self.dim, self.n = cfg["dim"], cfg["n"]
        s, w = _quadrature(cfg)
        self.nd, self.nb = len(w), len(cfg["C"])
        self.W, self.sumC = float(np.sum(w)), float(np.sum(cfg["C"]))
        self.s = torch.tensor(s, device=dev)
        self.w = torch.tensor(w, device=dev)
        self.bc = [DIF if (b == bte.BTE_BC_INTERFACE or i == cfg.get("iface")) else b for i, b in enumerate(cfg["bc"])]
        self.jump = cfg.get("jump") or [0.0, 0.0, 0.0]
        self.mirror = []
        for a in range(3):
            m = s.copy()
            m[:, a] *= -1
            self.mirror.append(torch.tensor([int(np.argmin(np.sum((s - r) ** 2, axis=1))) for r in m], device=dev))
        self.D = sum(float(c / t) for c, t in zip(cfg["C"], cfg["tau"]))

    def wall_values(self, e):
        """Plain diffuse values {wall: [wall cells, kept dim]} of one band's field e."""
        out = {}
        for wall in range(2 * self.dim):
            if self.bc[wall] != DIF:
                continue
            a, side = wall // 2, wall % 2
            sn = (self.s[:, a] if side else -self.s[:, a]) * self.w
            cells = e.narrow(3 - a, self.n[a] - 1 if side else 0, 1)
            lead = sn.clamp(min=0).view(-1, 1, 1, 1)
            out[wall] = (lead * cells).sum(0) / (-sn).clamp(min=0).sum()
        return out

    def _extended(self, e, k, a, diffuse):
        ax, n = 3 - a, self.n[a]
        pos = (self.s[:, a] > 0).view(-1, 1, 1, 1)
        ghosts = []
        for side in (0, 1):
            wall, bc = 2 * a + side, self.bc[2 * a + side]
            edge = e.narrow(ax, n - 1 if side else 0, 1)
            if bc == PER:
                off = self.cfg["C"][k] * self.jump[a] / self.W
                g = [e.narrow(ax, L if side else n - 1 - L, 1) + (-off if side else off) for L in (0, 1)]
            elif bc == SPE:
                m = e[self.mirror[a]]
                g = [m.narrow(ax, n - 1 - L if side else L, 1) for L in (0, 1)]
            else:
                val = diffuse[wall].expand_as(edge) if bc == DIF else torch.full_like(edge, self.cfg["C"][k] * self.cfg["Tw"][wall] / self.W)
                g0 = torch.where(pos if side == 0 else ~pos, val, edge)
                g = [g0, g0]
            ghosts.append(g)
        lo, hi = ghosts
        return torch.cat([lo[1], lo[0], e, hi[0], hi[1]], dim=ax), pos

    def step_band(self, e, k, TL, src, tau, diffuse):
        """e of band k after one explicit step; TL [nz, ny, nx], src = a(t) Q or None, tau a number
        or a tensor."""
        dt, C, v = self.cfg["dt"], float(self.cfg["C"][k]), float(self.cfg["v"][k])
        new = e + (dt / tau) * (C / self.W * TL - e)
        if src is not None:
            new = new + src * (dt * C / (self.sumC * self.W))
        for a in range(self.dim):
            ax, n = 3 - a, self.n[a]
            x, pos = self._extended(e, k, a, diffuse)
            d = x.narrow(ax, 1, n + 3) - x.narrow(ax, 0, n + 3)
            L = 0.5 * _limit(self.limiter, d.narrow(ax, 0, n + 2), d.narrow(ax, 1, n + 2))
            u = x.narrow(ax, 1, n + 2)  # cells -1 .. n
            F = torch.where(pos, (u + L).narrow(ax, 0, n + 1), (u - L).narrow(ax, 1, n + 1))
            nu = (dt * v / self.cfg["h"][a]) * self.s[:, a].view(-1, 1, 1, 1)
            new = new - nu * (F.narrow(ax, 1, n) - F.narrow(ax, 0, n))
        return new

    def numerator(self, e, k):
        return (self.w.view(-1, 1, 1, 1) * e).sum(0) / float(self.cfg["tau"][k])

    def sweep_band(self, r, k):
        """The increment of one implicit iteration of a 2-D band from r = dt R (first-order upwind,
        no increment across walls), by wavefronts x + y = const in upwind orientation."""
        dt, v = self.cfg["dt"], float(self.cfg["v"][k])
        nx, ny = self.n[0], self.n[1]
        nd = r.shape[0]
        r = r[:, 0]
        fx, fy = (self.s[:, 0] < 0).view(-1, 1, 1), (self.s[:, 1] < 0).view(-1, 1, 1)
        r = torch.where(fx, r.flip(2), r)
        r = torch.where(fy, r.flip(1), r)
        nux = (dt * v / self.cfg["h"][0] * self.s[:, 0].abs()).view(-1, 1)
        nuy = (dt * v / self.cfg["h"][1] * self.s[:, 1].abs()).view(-1, 1)
        diag = dt / float(self.cfg["tau"][k]) + nux + nuy
        y = torch.arange(ny, device=r.device)
        S = nx + ny - 1
        x = torch.arange(S, device=r.device)[:, None] - y[None, :]  # [S, ny]
        ok = (x >= 0) & (x < nx)
        at = (y[None, :] * nx + x.clamp(0, nx - 1)).reshape(-1)
        sk = torch.where(ok, r.reshape(nd, -1)[:, at].reshape(nd, S, ny), torch.zeros((), dtype=r.dtype, device=r.device))
        sk = sk.permute(1, 0, 2).contiguous()  # [S, nd, ny]
        prev = torch.zeros((nd, ny), dtype=r.dtype, device=r.device)
        up = torch.zeros_like(prev)
        okf = ok.to(r.dtype)
        for t in range(S):
            up[:, 1:] = prev[:, :-1]
            prev = (sk[t] + nux * prev + nuy * up) / diag * okf[t]
            sk[t] = prev
        back = (torch.arange(nx, device=r.device)[None, :] + y[:, None]).reshape(-1)  # wavefront of (y, x)
        ycol = y[:, None].expand(ny, nx).reshape(-1)
        d = sk[back, :, ycol].t().reshape(nd, ny, nx)
        d = torch.where(fy, d.flip(1), d)
        d = torch.where(fx, d.flip(2), d)
        return d[:, None]


def _start64(cfg, case, seed, side):
    """The start state of one side in 64 bits, decoded from what prepare() stores."""
    f = _Fields(cfg, case, seed, side)
    e, R = f.stored()
    out = []
    for k in range(f.nb):
        if R is None:
            out.append(e[k].double())
        else:
            out.append(f.scale(k) * (e[k].double() + R.double() / f.Ts))
    return out, f


def _source(cfg):
    Q = inputs.source_field(cfg)
    if Q is None:
        return None, None
    return torch.tensor(Q, device=_device()).double(), inputs.source_amplitudes(cfg, 400)


def _TL(P, E):
    return sum(P.numerator(E[k], k) for k in range(P.nb)) / P.D


def _exact_adjoint(case, seed):
    cfg = _workload(case)[0]
    P = _Plain(cfg, case["limiter"])
    E, _ = _start64(cfg, case, seed, 0)
    Q, amp = _source(cfg)
    N = case["steps"]
    probe = torch.tensor(_probe(cfg), device=_device())
    tau = [float(t) for t in cfg["tau"]]
    states, TLs = [E], [_TL(P, E)]
    for n in range(N):
        a = 1.0 if amp is None else float(amp[n])
        states.append([P.step_band(states[n][k], k, TLs[n], a * Q, tau[k], P.wall_values(states[n][k])) for k in range(P.nb)])
        TLs.append(_TL(P, states[-1]))
    J = float((probe * TLs[N]).sum())
    gQ, gt = torch.zeros_like(Q), [0.0] * P.nb
    mu, lam = probe.clone(), [None] * P.nb
    for n in range(N, -1, -1):
        # T_L^n = sum_k (sum_d w e / tau_k) / D
        for k in range(P.nb):
            gt[k] += float((mu * (TLs[n] * float(cfg["C"][k]) / tau[k] - P.numerator(states[n][k], k))).sum()) / P.D
            add = mu * P.w.view(-1, 1, 1, 1) / (tau[k] * P.D)
            lam[k] = add if lam[k] is None else lam[k] + add
        states[n] = None if n == N else states[n]
        if n == 0:
            break
        a = 1.0 if amp is None else float(amp[n - 1])
        new_mu = torch.zeros_like(mu)
        for k in range(P.nb):
            e = states[n - 1][k].clone().requires_grad_(True)
            tl = TLs[n - 1].clone().requires_grad_(True)
            q = Q.clone().requires_grad_(True)
            lt = torch.tensor(math.log(tau[k]), device=e.device, dtype=torch.float64, requires_grad=True)
            new = P.step_band(e, k, tl, a * q, torch.exp(lt), P.wall_values(e))
            ge, gtl, gq, glt = torch.autograd.grad(new, [e, tl, q, lt], lam[k])
            del new
            lam[k] = ge
            new_mu += gtl
            gQ += gq
            gt[k] += float(glt)
        states[n] = None
        mu = new_mu
    return {"J": J, "dJ_dQ": gQ, "dJ_dlogtau": np.array(gt)}


def exact(case, seed):
    ncell, nelem = _sizes(case)
    f, N = case["family"], case["steps"]
    if nelem * N * (6 if "adjoint" in f else 3 if f == "implicit" else 1) > 7e10:
        return None
    with torch.no_grad():
        if f not in ("adjoint2d", "adjoint3d"):
            return _exact_forward(case, seed)
    return _exact_adjoint(case, seed)


def _exact_forward(case, seed):
    f, N = case["family"], case["steps"]
    cfgs = _workload(case)
    Ps = [_Plain(c, case["limiter"]) for c in cfgs]
    Es = [_start64(c, case, seed, i)[0] for i, c in enumerate(cfgs)]
    Ts = _amplitude(case)[1]
    src = [_source(c) for c in cfgs]
    TLs = [_TL(P, E) for P, E in zip(Ps, Es)]
    prev = [t.clone() for t in TLs]
    for n in range(N):
        walls = [[P.wall_values(E[k]) for k in range(P.nb)] for P, E in zip(Ps, Es)]
        if f == "pair":
            a, b = cfgs
            for k in range(Ps[0].nb):
                sa, sb = walls[0][k][a["iface"]], walls[1][k][b["iface"]]
                ab, ba = float(a["beta_ab"][k]), float(a["beta_ba"][k])
                walls[0][k][a["iface"]] = ba * sb + (1 - ab) * sa
                walls[1][k][b["iface"]] = ab * sa + (1 - ba) * sb
        for i, P in enumerate(Ps):
            Q, amp = src[i]
            s = None if Q is None else Q if amp is None else float(amp[n]) * Q
            num = 0
            for k in range(P.nb):
                new = P.step_band(Es[i][k], k, TLs[i], s, float(cfgs[i]["tau"][k]), walls[i][k])
                if f == "implicit":
                    new = Es[i][k] + P.sweep_band(new - Es[i][k], k)
                Es[i][k] = new
                num = num + P.numerator(new, k)
            prev[i] = TLs[i]
            TLs[i] = num / P.D
    outs = []
    for i, P in enumerate(Ps):
        E = Es[i]
        out = {"TL": TLs[i].reshape(-1)}
        if case.get("moments"):
            out["T"] = sum((P.w.view(-1, 1, 1, 1) * e).sum(0) for e in E) / P.sumC
            out["q"] = torch.stack([sum(float(cfgs[i]["v"][k]) * ((P.w * P.s[:, a]).view(-1, 1, 1, 1) * E[k]).sum(0) for k in range(P.nb))
                                    for a in range(3)])
        if case["storage"] == "f32":
            out["state"] = torch.stack(E)
        else:
            g = _Fields(cfgs[i], case, seed, i)
            for k in range(P.nb):
                E[k] = E[k] / g.scale(k) - prev[i] / Ts
            out["state"] = torch.stack(E)
            out["ref"] = prev[i]
        del E
        Es[i] = None
        outs.append(out)
    return outs if f == "pair" else outs[0]
