"""Performance cases of the WDLB library: what its users have it do, through the
public calls of ``paper_1304_7880_gb300.wdlb``.

A case is a dict of plain values.  ``kind`` says which calls one pass makes:

* ``lattice``: ``wdlb_step(steps)`` of one lattice, then its moments on the
  device (n and u of every node), the block of steps every run repeats;
* ``steady``: ``wdlb_run_steady`` of one slit for at most ``steps`` steps with
  its FP64 residual tests, then the moments;
* ``batch``: ``wdlb_batch_step(steps)`` of many pores of uneven sizes, the
  residual test of every pore, then every pore's moments: one block of the
  serving loop.

The lattices are the library's own workloads: the plain 8x8x41 slit, the 128^3
bulk box, the 256x256x161 slit, the 64 uneven pores, the serving mix
(sigma 3, 4, 6; cross-sections 16..64; H lognormal) and the sigma 8 bulk box of
the viscosity sweep.  Densities stay below the scheme's stability limit in
slits (n* <= 0.57), so any number of passes is a valid run.  Slits start from
uniform density and a parabolic u_x of up to 0.1, as a solve does that
continues from the flow of a similar one: a slit started at rest, or stepped
until its layering has settled, has a wall-normal velocity of rounding noise
alone (1e-8, FP32), against which no result can be compared.

Outputs are n, u (and the residual tests' results) of every node, in the
precision that the lattice stores its populations in: FP64 storage as float64,
FP32 as float32, FP16 as float16.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1304_7880_gb300 import wdlb as w

KT = 1.0 / 3.0
_CHECK = 50          # steps between the residual tests of a steady solve


def _case(name=None, **kw):
    c = dict(kind="lattice", nx=8, ny=8, nz=41, walls=True, sigma=4.0, tau=1.0, gx=1e-6, nstar=0.5, noise=1e-3,
             u0=0.08, storage="f32", rule="full", closure="CS", collision="fp32", steps=50)
    c.update(kw)
    if name is not None:
        c["name"] = name
    return c


def _bulk(name=None, **kw):
    # shear wave on a noisy fluid at packing fraction 0.3 (n* = 0.573 whatever sigma)
    base = dict(walls=False, gx=0.0, nstar=1.8 / math.pi, noise=1e-4, u0=1e-4, steps=10)
    base.update(kw)
    return _case(name, **base)


def listed():
    return [
        # the plain slit of the smallest configuration in FP64: the reference run of the scheme
        _case("slit_8x8x41_f64", storage="f64"),
        # the same slit in FP32: one thin pore of a viscosity sweep, where latency and launches count
        _case("slit_8x8x41_f32"),
        # one serving request solved alone to its steady state (odd cross-section, sigma 3)
        _case("steady_27x27x46_s3", kind="steady", nx=27, ny=27, nz=46, sigma=3.0, nstar=0.45, gx=3e-6, steps=100),
        # the bulk-viscosity sweep's box at sigma 8 (762 shell vectors)
        _bulk("sweep_8x8x256_s8", nx=8, ny=8, nz=256, sigma=8.0, nstar=1.5 / math.pi, noise=0.0, u0=1e-6, steps=20),
        # a ragged FP64 box: the plain path that results are checked against
        _bulk("bulk_45x38x51_f64", nx=45, ny=38, nz=51, storage="f64", steps=4),
        # a driven slit at the accuracy option (double-word collision), ragged
        _case("slit_41x37x81_dw", nx=41, ny=37, nz=81, nstar=0.4, collision="dw", steps=20),
        # the bulk box in the default precision, on both contact shells
        _bulk("bulk_128_f32", nx=128, ny=128, nz=128),
        _bulk("bulk_128_compact", nx=128, ny=128, nz=128, rule="compact"),
        # half-precision storage (periodic boxes only) at sigma 6
        _bulk("bulk_96_f16_s6", nx=96, ny=96, nz=96, sigma=6.0, storage="f16"),
        # the single large slit
        _case("slit_256x256x161", nx=256, ny=256, nz=161, tau=0.8, nstar=0.3, steps=4),
        # 64 uneven pores of one cross-section: the headline batch
        _case("batch_64_pores", kind="batch", pores=64, nxy_min=32, nxy_max=32, h_min=3.0, h_max=30.0,
              sigmas="4", sizes=4, steps=20),
        # a full serving mix: three diameters, ragged cross-sections
        _case("serving_mix_32", kind="batch", pores=32, nxy_min=16, nxy_max=64, h_min=3.0, h_max=60.0,
              sigmas="3,4,6", sizes=5, steps=20),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    pick = rng.choice(["slit", "slit", "bulk", "bulk", "sigma8", "f64", "dw", "steady", "batch", "batch"])
    tau = rng.choice([0.8, 1.0, 1.0])
    if pick in ("slit", "dw", "steady"):
        sigma = 4.0 if pick == "dw" and rng.random() < 0.5 else rng.choice([3.0, 4.0, 4.0, 6.0])
        top = 192 if pick == "slit" else 64
        nx = _log_int(rng, 8, top)
        ny = nx if rng.random() < 0.5 else _log_int(rng, 8, top)
        nz = int(round(sigma * rng.uniform(7.0, 40.0 if pick == "slit" else 25.0))) + 1
        kw = dict(nx=nx, ny=ny, nz=nz, sigma=sigma, tau=tau, nstar=round(rng.uniform(0.1, 0.57), 3),
                  gx=10.0 ** round(rng.uniform(-7.0, -5.0), 2), steps=20)
        if pick == "steady":
            return _case(kind="steady", **dict(kw, nz=max(nz, 45), steps=100 if nx * ny * nz < 60000 else 50))
        if pick == "dw":
            return _case(collision="dw", **kw)
        return _case(rule=rng.choice(["full", "full", "compact"]) if kw["nstar"] < 0.45 else "full",
                     closure=rng.choice(["CS"] * 7 + ["PY"]), **kw)
    if pick in ("bulk", "sigma8", "f64"):
        sigma = 8.0 if pick == "sigma8" else rng.choice([3.0, 4.0, 4.0, 6.0])
        hi = {"bulk": 144, "sigma8": 48, "f64": 48}[pick]
        nx, ny, nz = (_log_int(rng, 8, hi) for _ in range(3))
        nz = _log_int(rng, 24, 256 if pick == "sigma8" else hi)
        if pick == "sigma8":
            if rng.random() < 0.5:
                nx = ny = 8
        storage = "f64" if pick == "f64" else rng.choice(["f32", "f32", "f16"]) if pick == "bulk" else "f32"
        rule = "compact" if pick != "f64" and rng.random() < 0.3 else "full"
        top = 0.5 if rule == "compact" else 0.57
        return _bulk(nx=nx, ny=ny, nz=nz, sigma=sigma, tau=tau, storage=storage, rule=rule,
                     nstar=round(rng.uniform(0.1, top), 3), closure=rng.choice(["CS"] * 7 + ["PY"]), u0=1e-2,
                     steps=4 if pick != "bulk" or nx * ny * nz > 200000 else 10)
    sig = rng.choice(["4", "3,4,6", "3,4,6"])
    lo = _log_int(rng, 8, 32)
    return _case(kind="batch", pores=_log_int(rng, 3, 32), nxy_min=lo, nxy_max=max(lo, _log_int(rng, 16, 56)),
                 h_min=3.0, h_max=rng.choice([10.0, 20.0, 30.0]), sigmas=sig, sizes=rng.randrange(1000),
                 rule="full", storage="f32", tau=tau, steps=20)


# ---- inputs ----------------------------------------------------------------------------

def _pores(case):
    """Lattice of every pore of a batch: (nx, ny, nz, sigma, nstar, gx), from the case alone."""
    r = np.random.RandomState(int(case["sizes"]))
    sigmas = [float(s) for s in case["sigmas"].split(",")]
    out = []
    for _ in range(int(case["pores"])):
        sigma = sigmas[r.randint(len(sigmas))]
        nxy = r.randint(int(case["nxy_min"]), int(case["nxy_max"]) + 1)
        if len(sigmas) == 1:
            h = r.uniform(case["h_min"], case["h_max"])
        else:
            h = min(case["h_max"], max(case["h_min"], 10.0 * math.exp(0.5 * r.randn())))
        out.append((nxy, nxy, int(round(h * sigma)) + 1, sigma, r.uniform(0.1, 0.57), 10.0 ** r.uniform(-7.0, -5.0)))
    return out


def _device():
    return torch.device("cuda") if torch.cuda.is_available() else torch.device("cpu")


def _fields(nx, ny, nz, walls, n0, noise, u0, gen, dev):
    """Density n0 (1 + noise (2U - 1)) and u_x: a shear wave of amplitude u0 with
    a random phase, or between walls a parabola."""
    n = torch.rand((nz, ny, nx), generator=gen, dtype=torch.float64, device=dev)
    n = n0 * (1.0 + noise * (2.0 * n - 1.0))
    phase = torch.rand((2,), generator=gen, dtype=torch.float64, device=dev)
    u = torch.zeros((3, nz, ny, nx), dtype=torch.float64, device=dev)
    if u0:
        z = torch.arange(nz, dtype=torch.float64, device=dev)
        s = (z - 0.5) / (nz - 2)
        prof = 4.0 * s * (1.0 - s) if walls else torch.sin(2.0 * math.pi * (z / nz + phase[0]))
        u[0] = (u0 * (0.8 + 0.4 * phase[1]) * prof)[:, None, None]
    if walls:
        n[0] = n[-1] = 0.0
        u[:, 0] = u[:, -1] = 0.0
    return n.contiguous(), u


def _gen(seed, dev):
    g = torch.Generator(device=dev)
    g.manual_seed(int(seed))
    return g


def _out_type(case):
    return {"f64": torch.float64, "f32": torch.float32, "f16": torch.float16}[case["storage"]]


def prepare(case, seed):
    dev = _device()
    gen = _gen(seed, dev)
    st = {"case": case}
    if case["kind"] == "batch":
        pores = _pores(case)
        total = sum(p[0] * p[1] * p[2] for p in pores)
        probe = w.wdlb_batch_create(1, 1 << 20, closure=case["closure"], storage=case["storage"],
                                    shell_rule=case["rule"], collision=case["collision"])
        need = sum((w.wdlb_batch_pore_bytes(probe, p[:3], p[3], True) + 255) // 256 * 256 for p in pores)
        w.wdlb_batch_destroy(probe)
        b = w.wdlb_batch_create(len(pores), need + 4096, closure=case["closure"], storage=case["storage"],
                                shell_rule=case["rule"], collision=case["collision"])
        st.update(batch=b, stream=b.stream, slots=[])
        for nx, ny, nz, sigma, nstar, gx in pores:
            n, u = _fields(nx, ny, nz, True, nstar / sigma ** 3, case["noise"], case["u0"], gen, dev)
            st["slots"].append(w.wdlb_batch_add(b, (nx, ny, nz), sigma, True, case["tau"], (gx, 0.0, 0.0),
                                                n.cpu().numpy(), u.cpu().numpy()))
        st["ctx"] = [w.wdlb_batch_context(b, s) for s in st["slots"]]
        w.wdlb_batch_residuals(b, case["steps"])        # the pores' first flux, as at admission
    else:
        nx, ny, nz = case["nx"], case["ny"], case["nz"]
        total = nx * ny * nz
        ctx = w.wdlb_create((nx, ny, nz), case["sigma"], case["walls"], case["tau"], (case["gx"], 0.0, 0.0),
                            closure=case["closure"], storage=case["storage"], shell_rule=case["rule"],
                            collision=case["collision"])
        n, u = _fields(nx, ny, nz, case["walls"], case["nstar"] / case["sigma"] ** 3, case["noise"], case["u0"], gen,
                       dev)
        ctx.stream.wait_stream(torch.cuda.current_stream())
        w.wdlb_init_fields_device(ctx, n, u)
        ctx.stream.synchronize()
        st.update(ctx=[ctx], stream=ctx.stream)
    # moments of every pore, one after the other in one buffer
    st["n"] = torch.empty(total, dtype=torch.float64, device=dev)
    st["u"] = torch.empty(3 * total, dtype=torch.float64, device=dev)
    st["views"], at = [], 0
    for c in st["ctx"]:
        st["views"].append((st["n"][at:at + c.N], st["u"][3 * at:3 * (at + c.N)]))
        at += c.N
    torch.cuda.synchronize()
    return st


# ---- one pass --------------------------------------------------------------------------

def run(st):
    case = st["case"]
    out = {}
    if case["kind"] == "batch":
        w.wdlb_batch_step(st["batch"], case["steps"])
        res, status = w.wdlb_batch_residuals(st["batch"], case["steps"])
        out["residual"] = res.astype(np.float32)
        out["status"] = status
    elif case["kind"] == "steady":
        done, res = w.wdlb_run_steady(st["ctx"][0], 1e-30, _CHECK, case["steps"])
        out["steps"] = done
        out["residual"] = np.float32(res)
    else:
        w.wdlb_step(st["ctx"][0], case["steps"])
    for c, (n, u) in zip(st["ctx"], st["views"]):
        w.wdlb_moments_device(c, n, u)
    with torch.cuda.stream(st["stream"]):
        out["n"] = st["n"].to(_out_type(case))
        out["u"] = st["u"].to(_out_type(case))
    return out


# ---- what a pass cannot do without ---------------------------------------------------------

def _shell(sigma):
    r = int(math.floor(sigma + 0.5))
    a = np.arange(-r, r + 1)
    x, y, z = (t.ravel() for t in np.meshgrid(a, a, a, indexing="ij"))
    r2 = x * x + y * y + z * z
    keep = (r2 > (sigma - 0.5) ** 2) & (r2 <= (sigma + 0.5) ** 2)
    e = np.stack([x, y, z], 1)[keep]
    return e, e / np.sqrt(r2[keep])[:, None]


# vectors of the compact rule per sigma: its cubic orbits (sorted |components|)
_ORBITS = {3.0: [(0, 0, 3), (0, 2, 2), (2, 2, 2)], 4.0: [(0, 0, 4), (0, 2, 3), (0, 3, 3)],
           6.0: [(0, 0, 6), (2, 4, 4)], 8.0: None}


def _weighted_shell(sigma, rule):
    """Vectors, unit vectors and weights: uniform with the virial moment, or the
    compact rule's orbits with the virial, viscosity and isotropy moments."""
    e, k = _shell(sigma)
    if rule == "full":
        return e, k, np.full(len(e), 4.0 * math.pi / 3.0 * sigma / np.sum(k[:, 2] * e[:, 2]))
    rhs = np.array([4.0 * math.pi * sigma / 3.0, 4.0 * math.pi * sigma ** 2 / 15.0, 0.0])
    keys = [tuple(sorted(abs(int(c)) for c in v)) for v in e]
    orbits = _ORBITS[sigma]
    if orbits is None:                     # the rule's selection: fewest vectors, then the smallest radial spread
        import itertools
        names = sorted(set(keys), key=lambda t: (sum(c * c for c in t), t))
        best = None
        for m in (2, 3):
            for group in itertools.combinations(names, m):
                got = _orbit_weights(e, k, keys, group, rhs)
                if got is None:
                    continue
                sel = [key in group for key in keys]
                rank = (sum(sel), round(float(np.sum((np.sum(e[sel] ** 2, 1) - sigma ** 2) ** 2)), 6))
                if best is None or rank < best[0]:
                    best = (rank, group)
        orbits = _ORBITS[sigma] = list(best[1])
    wts = _orbit_weights(e, k, keys, orbits, rhs)
    wv = np.array([wts[orbits.index(key)] if key in orbits else 0.0 for key in keys])
    return e[wv > 0], k[wv > 0], wv[wv > 0]


def _orbit_weights(e, k, keys, group, rhs):
    cols = []
    for o in group:
        s = np.array([key == o for key in keys])
        vc = np.sum(k[s, 0] ** 2 * e[s, 2] ** 2)
        cols.append([np.sum(k[s, 2] * e[s, 2]), vc, np.sum(k[s, 2] ** 2 * e[s, 2] ** 2) - 3.0 * vc])
    a = np.array(cols).T
    wts, _, rank, _ = np.linalg.lstsq(a, rhs, rcond=None)
    mag = np.abs(rhs) + np.sum(np.abs(a * wts), 1)
    if rank < len(group) or np.any(np.abs(a @ wts - rhs) > 1e-9 * mag) or np.any(wts <= 1e-3 * np.max(wts)):
        return None
    return wts


def _lattices(case):
    if case["kind"] == "batch":
        return [p[:4] for p in _pores(case)]
    return [(case["nx"], case["ny"], case["nz"], case["sigma"])]


def work(case):
    """Per time step and node: the 19 populations read and written once, 52
    operations per shell vector and 475 for the moments, the collision and the
    forces; per pass, n and u written once."""
    size = {"f64": 8, "f32": 4, "f16": 2}[case["storage"]]
    nbytes = flops = 0.0
    for nx, ny, nz, sigma in _lattices(case):
        nodes = float(nx * ny * nz)
        m = len(_weighted_shell(sigma, case["rule"])[0])
        nbytes += nodes * (case["steps"] * 2 * 19 * size + 4 * size)
        flops += nodes * case["steps"] * (52.0 * m + 475.0)
    return {"bytes": nbytes, "flops": flops}


# ---- the scheme in 64 bits with torch --------------------------------------------------------

_C = [(0, 0, 0)] + [tuple(s if a == d else 0 for a in range(3)) for d in range(3) for s in (1, -1)] + \
     [(s, t, 0) for s in (1, -1) for t in (1, -1)] + [(s, 0, t) for s in (1, -1) for t in (1, -1)] + \
     [(0, s, t) for s in (1, -1) for t in (1, -1)]
_W = [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12


class _Scheme:
    """One lattice of the discretised equations, stepped in FP64 (BGK with
    second-order forcing, shell sums with the contact value at the mean smeared
    density, lagged implicit field velocity, half-way bounce-back)."""

    def __init__(self, nx, ny, nz, walls, sigma, tau, gx, rule, closure, n, u):
        self.dim, self.walls, self.tau, self.closure, self.sigma = (nz, ny, nx), walls, tau, closure, sigma
        dev = n.device
        self.dev = dev
        e, k, wt = _weighted_shell(sigma, rule)
        self.shell = self._table(e)
        self.k = torch.from_numpy(k).to(dev)
        self.wt = torch.from_numpy(wt).to(dev)
        r = int(math.floor(sigma / 2))
        a = np.arange(-r, r + 1)
        x, y, z = (t.ravel() for t in np.meshgrid(a, a, a, indexing="ij"))
        keep = x * x + y * y + z * z <= (sigma / 2) ** 2
        self.ball = self._table(np.stack([x, y, z], 1)[keep])
        self.g = torch.tensor([gx, 0.0, 0.0], dtype=torch.float64, device=dev)[:, None]
        self.N = nx * ny * nz
        self.fluid = torch.ones(self.dim, dtype=torch.float64, device=dev)
        if walls:
            self.fluid[0] = self.fluid[-1] = 0.0
        self.fluid = self.fluid.reshape(-1)
        self.c = torch.tensor(_C, dtype=torch.float64, device=dev)
        self.w = torch.tensor(_W, dtype=torch.float64, device=dev)
        n, u = n.reshape(-1) * self.fluid, u.reshape(3, -1) * self.fluid
        self.f = self._feq(n, u)
        self.C = torch.zeros((3, self.N), dtype=torch.float64, device=dev)
        self.t = torch.zeros(self.N, dtype=torch.float64, device=dev)
        self.v = u.clone()
        self.beta = 2.0 * sigma ** 2 * math.sqrt(KT / math.pi)

    def _table(self, e):
        """Wrapped coordinates of every node's neighbours, per axis, and 1 where z stays inside."""
        nz, ny, nx = self.dim
        x = (np.arange(nx)[None] + e[:, :1]) % nx
        y = (np.arange(ny)[None] + e[:, 1:2]) % ny
        z = np.arange(nz)[None] + e[:, 2:3]
        inside = ((z >= 0) & (z < nz)) if self.walls else np.ones(z.shape, bool)
        to = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(self.dev)  # noqa: E731
        return to(x), to(nx * y), to(nx * ny * (z % nz)), to(inside.astype(np.float64))

    def _chunks(self, table):
        nz, ny, nx = self.dim
        x, y, z, inside = table
        step = max(1, min(x.shape[0], 24_000_000 // self.N))
        for a in range(0, x.shape[0], step):
            s = slice(a, a + step)
            idx = (z[s, :, None, None] + y[s, None, :, None]) + x[s, None, None, :]
            keep = inside[s, :, None, None].expand(-1, nz, ny, nx).reshape(-1, self.N)
            yield s, idx.reshape(-1, self.N), keep

    def _feq(self, n, u):
        cu = self.c @ u
        return self.w[:, None] * n * (1.0 + 3.0 * cu + 4.5 * cu * cu - 1.5 * (u * u).sum(0))

    def moments(self):
        n = self.f.sum(0)
        safe = torch.where(self.fluid > 0, n, torch.ones_like(n))
        j = self.c.T @ self.f
        H = self.beta * 2.0 * self.t / 6.0
        v = ((j + 0.5 * (n * self.g + self.C)) / safe + H * self.v) / (1.0 + H)
        return n * self.fluid, v * self.fluid, j

    def _contact(self, chi):
        s = 1.0 - chi
        return (0.5 + 0.5 * s) / s ** 3 if self.closure == "CS" else (1.5 - 0.5 * s) / (s * s)

    def step(self):
        n, v, j = self.moments()
        nbar = torch.zeros_like(n)
        count = 0
        for s, idx, keep in self._chunks(self.ball):
            nbar += (n[idx] * keep).sum(0)
            count += idx.shape[0]
        h = math.pi * self.sigma ** 3 / 12.0 * nbar / count
        V = torch.zeros((3, self.N), dtype=torch.float64, device=self.dev)
        Wv, M, t = torch.zeros_like(V), torch.zeros((3, 3, self.N), dtype=torch.float64, device=self.dev), \
            torch.zeros_like(n)
        for s, idx, keep in self._chunks(self.shell):
            k = self.k[s]
            q = self._contact(h + h[idx]) * n[idx] * keep * self.wt[s, None]
            du = [v[a][idx] - v[a] for a in range(3)]
            kdu = k[:, 0:1] * du[0] + k[:, 1:2] * du[1] + k[:, 2:3] * du[2]
            t += q.sum(0)
            V += k.T @ q
            Wv += k.T @ (q * kdu)
            for a in range(3):
                M[a] += k.T @ (q * du[a])
        C = n * (-KT * self.sigma ** 2 * V + self.beta * Wv)
        A = -(KT / 5.0) * n * self.sigma ** 2 * (M + M.transpose(0, 1))
        F = n * self.g + C
        safe = torch.where(self.fluid > 0, n, torch.ones_like(n))
        u = (j + 0.5 * F) / safe
        tr = (A[0, 0] + A[1, 1] + A[2, 2]) / 3.0
        om = 1.0 / self.tau
        cu, cF, uF = self.c @ u, self.c @ F, (u * F).sum(0)
        cac = torch.zeros_like(cu)
        for a in range(3):
            for b in range(3):
                cac += (self.c[:, a] * self.c[:, b])[:, None] * (A[a, b] - (tr if a == b else 0.0))
        src = self.w[:, None] * (3.0 * (cF - uF) + 9.0 * cu * cF + 2.0 * 4.5 * cac)
        post = self.f - om * (self.f - self._feq(n, u)) + (1.0 - 0.5 * om) * src
        post *= self.fluid
        nz, ny, nx = self.dim
        post = post.reshape(19, nz, ny, nx)
        solid = (1.0 - self.fluid).reshape(self.dim)
        new = torch.empty_like(post)
        for q, (cx, cy, cz) in enumerate(_C):
            new[q] = torch.roll(post[q], (cz, cy, cx), (0, 1, 2))
            if self.walls and cz:
                opp = _C.index((-cx, -cy, -cz))
                new[q] += torch.roll(solid, cz, 0) * post[opp]
        self.f = new.reshape(19, -1) * self.fluid
        self.C, self.t, self.v = C * self.fluid, t * self.fluid, v


def _exact_cost(case):
    return sum(nx * ny * nz * len(_shell(sigma)[0]) for nx, ny, nz, sigma in _lattices(case)) * case["steps"]


def exact(case, seed):
    if _exact_cost(case) > 3e10:
        return None
    dev = _device()
    gen = _gen(seed, dev)
    out = {}
    if case["kind"] == "batch":
        todo = [(p[:3], p[3], p[4], p[5], case["u0"], True) for p in _pores(case)]
    else:
        todo = [((case["nx"], case["ny"], case["nz"]), case["sigma"], case["nstar"], case["gx"], case["u0"],
                 case["walls"])]
    ns, us, res = [], [], []
    for (nx, ny, nz), sigma, nstar, gx, u0, walls in todo:
        n, u = _fields(nx, ny, nz, walls, nstar / sigma ** 3, case["noise"], u0, gen, dev)
        s = _Scheme(nx, ny, nz, walls, sigma, case["tau"], gx, case["rule"], case["closure"], n, u)
        every = min(_CHECK, case["steps"]) if case["kind"] == "steady" else case["steps"]
        flux = []
        for k in range(case["steps"] + 1):
            if k % every == 0 or k == case["steps"]:
                m = s.moments()
                flux.append((k, (m[0] * m[1][0]).sum()))
            if k < case["steps"]:
                s.step()
        n, v, _ = s.moments()
        ns.append(n)
        us.append(v.reshape(-1))
        (ka, qa), (kb, qb) = flux[-2:]
        res.append(float(abs(qb - qa) / ((kb - ka) * abs(qb))) if float(qb) else math.inf)
    if case["kind"] != "lattice":
        out["residual"] = np.array(res) if case["kind"] == "batch" else np.float64(res[0])
    if case["kind"] == "steady":
        out["steps"] = None
    if case["kind"] == "batch":
        out["status"] = None
    out["n"], out["u"] = torch.cat(ns), torch.cat(us)
    return out
