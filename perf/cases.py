"""Performance cases: what users of the framework have it compute, through its
public entry points, from the smallest grids to the largest.

A case is a dict of plain values. kind:
  "heat"      Grid.run, the time loop of the heat-diffusion solver (nt steps);
  "batch"     Batch.run, many independent diffusion problems of uneven sizes;
  "gradient"  autograd.solve and its backward pass (misfit gradient in T0 and Ci);
  "acoustic"  Grid.acoustic_step, a time loop of the staggered-grid acoustics;
  "gp"        Grid.gp_step, a time loop of the Gross-Pitaevskii solver.
Sizes are local: nx, ny, nz points per subdomain, dx, dy, dz subdomains per
dimension, px periodic in x (1) or not (0).

Work is counted per time step (T_eff, the metric this solver is quoted in):
a step reads each of its input fields once and writes each of its output
fields once.
"""
from __future__ import annotations

import math
import random

import torch

import paper_2211_15716_gb300 as igg
from paper_2211_15716_gb300 import autograd as ag

DTYPES = {"f64": torch.float64, "f32": torch.float32, "bf16": torch.bfloat16}
SIZE = {"f64": 8, "f32": 4, "bf16": 2}
DEV = "cuda"


def _case(name, kind, dtype, n, d=(1, 1, 1), px=0, nt=10, overlap=2, hidden=0, field="gaussian",
          count=0, nmin=32, nmax=192):
    return {"name": name, "kind": kind, "dtype": dtype, "nx": n[0], "ny": n[1], "nz": n[2],
            "dx": d[0], "dy": d[1], "dz": d[2], "px": px, "nt": nt, "overlap": overlap,
            "hidden": hidden, "field": field, "count": count, "nmin": nmin, "nmax": nmax}


def listed():
    return [
        # the smallest real grid: one 64^3 FP64 array, a whole run of 100
        # steps (launches and latency count, everything fits in L2)
        _case("heat_64_f64", "heat", "f64", (64, 64, 64), nt=100),
        # the headline workload: 2x2x2 subdomains of 512x256x256, FP64, halo
        # update hidden with widths (16, 2, 2); a stretch of its time loop
        _case("heat_2x2x2_512x256x256_f64", "heat", "f64", (512, 256, 256), (2, 2, 2), 1, 10,
              hidden=1),
        # the same physics with a field that changes sign (stencils across
        # zero and powers of two), a quarter of the size per dimension pair
        _case("heat_signed_2x2x2_256x128x128_f64", "heat", "f64", (256, 128, 128), (2, 2, 2), 1,
              20, hidden=1, field="signed"),
        # rows of an odd length (a grid the user did not round up), FP64
        _case("heat_odd_2x2x2_255x127x129_f64", "heat", "f64", (255, 127, 129), (2, 2, 2), 0, 10),
        # the headline grid in the reduced precisions
        _case("heat_2x2x2_512x256x256_f32", "heat", "f32", (512, 256, 256), (2, 2, 2), 1, 10,
              hidden=1),
        _case("heat_2x2x2_512x256x256_bf16", "heat", "bf16", (512, 256, 256), (2, 2, 2), 1, 10,
              hidden=1),
        # the batched solver: 256 uneven FP32 problems of 32 to 192 points
        _case("batch_256_f32", "batch", "f32", (0, 0, 0), nt=20, count=256),
        # the inverse problem: misfit gradient through 48 steps at 256^3, FP64
        _case("gradient_256_f64", "gradient", "f64", (256, 256, 256), nt=48),
        # the same on subdomains (transposed halo updates), FP32, small arrays
        _case("gradient_2x2x2_64_f32", "gradient", "f32", (64, 64, 64), (2, 2, 2), 1, 32),
        # acoustics on 2x2x2 subdomains of 256^3 cells, FP64
        _case("acoustic_2x2x2_256_f64", "acoustic", "f64", (256, 256, 256), (2, 2, 2), nt=4),
        # acoustics in FP32 on sizes nobody rounded
        _case("acoustic_2x1x2_255x193x130_f32", "acoustic", "f32", (255, 193, 130), (2, 1, 2), 1,
              10),
        # Gross-Pitaevskii on 2x2x2 subdomains of 256^3 points, FP64
        _case("gp_2x2x2_256_f64", "gp", "f64", (256, 256, 256), (2, 2, 2), nt=4),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    while True:
        kind = rng.choice(["heat", "heat", "heat", "batch", "gradient", "acoustic", "gp"])
        dtype = rng.choice(["f64", "f64", "f32", "bf16"] if kind in ("heat", "batch") else ["f64", "f32"])
        d = rng.choice([(1, 1, 1), (2, 2, 2), (2, 2, 2), (3, 1, 2), (1, 2, 1), (4, 2, 1)])
        hi = {"heat": 512, "gradient": 192, "acoustic": 320, "gp": 320, "batch": 512}[kind]
        n = [_logint(rng, 24, hi) for _ in range(3)]
        if rng.random() < 0.5:  # rows of a round length
            n[0] = max(24, n[0] // 8 * 8)
        px = rng.randint(0, 1)
        nt = _logint(rng, 4, 64)
        field = "signed" if kind == "heat" and rng.random() < 0.2 else "gaussian"
        c = _case("", kind, dtype, n, d, px, nt, rng.choice([2, 2, 2, 3]), rng.randint(0, 1), field)
        if kind == "batch":
            c.update(nx=0, ny=0, nz=0, dx=1, dy=1, dz=1, px=0, overlap=2, hidden=0,
                     count=_logint(rng, 8, 256), nmin=_logint(rng, 16, 48),
                     nmax=_logint(rng, 64, 192))
        del c["name"]
        if _points(c) <= 1 << 27 and work(c)["bytes"] <= 24e9:
            return c


# -- sizes ------------------------------------------------------------------
def _problems(c):
    """The batched workload's problems: sizes, lam, Ci, spacings, dt (a
    catalogue of problems, the same for every seed of the fields)."""
    r = random.Random(3)
    sizes = [tuple(r.randint(c["nmin"], c["nmax"]) for _ in range(3)) for _ in range(c["count"])]
    lam = [r.uniform(0.5, 2.0) for _ in sizes]
    ci = [1.0 / r.uniform(1.5, 2.5) for _ in sizes]
    dd = [[1.0 / (m - 1) for m in s] for s in sizes]
    dts = [min(x * x for x in d) / l / k / 6.1 for d, l, k in zip(dd, lam, ci)]
    return sizes, lam, ci, dd, dts


def _points(c):
    if c["kind"] == "batch":
        return sum(a * b * e for a, b, e in _problems(c)[0])
    return c["nx"] * c["ny"] * c["nz"] * c["dx"] * c["dy"] * c["dz"]


def work(c):
    N, s, nt = _points(c), SIZE[c["dtype"]], c["nt"]
    if c["kind"] in ("heat", "batch"):  # T, Ci read, T2 written; 7-point update
        return {"bytes": 3 * N * s * nt, "flops": 13 * N * nt}
    if c["kind"] == "gradient":
        # the forward steps twice (checkpoint every ~sqrt(nt) states: all but
        # one step of each segment again), and per backward step lam, Ci, T_n
        # and the FP64 gCi read, lam and gCi written
        every = ag.default_every(nt)
        fwd = 2 * nt - (nt + every - 1) // every
        return {"bytes": N * (3 * s * fwd + (4 * s + 16) * nt), "flops": N * (13 * fwd + 30 * nt)}
    if c["kind"] == "acoustic":  # P, Vx, Vy, Vz read and written once per step
        return {"bytes": 8 * N * s * nt, "flops": 18 * N * nt}
    # gp: per half step u, v, V read and one of u, v written
    return {"bytes": 8 * N * s * nt, "flops": 2 * 20 * N * nt}


# -- inputs -----------------------------------------------------------------
class _Topo:
    """The case's global grid in plain arithmetic: global sizes, and per
    subdomain the global index of each local point and the neighbours."""

    def __init__(self, c):
        self.n = (c["nx"], c["ny"], c["nz"])
        self.dims = (c["dx"], c["dy"], c["dz"])
        self.per = (c["px"], 0, 0)
        self.o = (c["overlap"],) * 3
        self.nsub = self.dims[0] * self.dims[1] * self.dims[2]
        self.ng = tuple(self.dims[k] * (self.n[k] - self.o[k]) + (0 if self.per[k] else self.o[k])
                        for k in range(3))

    def coords(self, s):
        return (s % self.dims[0], (s // self.dims[0]) % self.dims[1], s // (self.dims[0] * self.dims[1]))

    def neighbour(self, s, k, side):
        c = list(self.coords(s))
        c[k] += side
        if not 0 <= c[k] < self.dims[k]:
            if not self.per[k]:
                return -1
            c[k] %= self.dims[k]
        return c[0] + self.dims[0] * (c[1] + self.dims[1] * c[2])

    def index(self, s, k, n=None, ng=None):
        c = self.coords(s)[k]
        i = torch.arange(n or self.n[k], device=DEV) + c * (self.n[k] - self.o[k])
        return i % self.ng[k] if self.per[k] else i

    def cut(self, G, dtype):
        """The global field G [ngz][ngy][ngx] as [nsub][nz][ny][nx]."""
        out = torch.empty((self.nsub, self.n[2], self.n[1], self.n[0]), dtype=dtype, device=DEV)
        for s in range(self.nsub):
            z, y, x = self.index(s, 2), self.index(s, 1), self.index(s, 0)
            out[s] = G[z][:, y][:, :, x].to(dtype)
        return out


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) & 0x7FFFFFFF)
    return g


def _axes(ng):
    return [torch.linspace(0.0, 1.0, m, dtype=torch.float64, device=DEV) for m in ng]


def _bump(ng, seed, base, amp, width, jitter=0.05):
    """base + amp * Gaussian of the given width about a centre near the middle."""
    u = torch.rand(4, generator=_gen(seed + 11), device=DEV, dtype=torch.float64).tolist()
    w = width * (0.9 + 0.2 * u[3])
    e = [torch.exp(-(a - 0.5 - jitter * (2 * u[k] - 1)) ** 2 / (2 * w * w)) for k, a in enumerate(_axes(ng))]
    return base + amp * (e[2][:, None, None] * e[1][None, :, None] * e[0][None, None, :])


def _sines(ng, seed, base, amp, count=8, mmax=8):
    """base + amp * the sum of `count` products of sines (mode numbers from the seed)."""
    m = torch.randint(1, mmax + 1, (count, 3), generator=_gen(seed + 13), device=DEV).tolist()
    ax = _axes(ng)
    out = torch.full((ng[2], ng[1], ng[0]), base, dtype=torch.float64, device=DEV)
    for mx, my, mz in m:
        s = [torch.sin(math.pi * k * a) for k, a in zip((mx, my, mz), ax)]
        out += amp * (s[2][:, None, None] * s[1][None, :, None] * s[0][None, None, :])
    return out


def _uniform(ng, seed, lo, hi):
    G = torch.rand((ng[2], ng[1], ng[0]), generator=_gen(seed + 17), device=DEV, dtype=torch.float64)
    return G.mul_(hi - lo).add_(lo)


def _inputs(c, seed):
    """The case's fields and numbers, without any call of the library's kernels."""
    dt = DTYPES[c["dtype"]]
    kind = c["kind"]
    if kind == "batch":
        sizes, lam, ci, dd, dts = _problems(c)
        r = torch.rand((len(sizes), 5), generator=_gen(seed), dtype=torch.float64, device=DEV).tolist()
        T = [_bump(s, int(1e6 * r[b][0]) + seed, 1.7, 0.5 + r[b][1], 0.1) for b, s in enumerate(sizes)]
        return {"sizes": sizes, "lam": lam, "ci": ci, "dd": dd, "dts": dts, "T": T}
    t = _Topo(c)
    h = [1.0 / (m - 1) for m in t.ng]
    if kind == "heat":
        # Fig. 1's physics: a warm bump on 1.7 (or modes about zero), Ci = 1/c0
        G = _sines(t.ng, seed, 0.0, 0.1) if c["field"] == "signed" else _bump(t.ng, seed, 1.7, 1.0, 0.1)
        T = t.cut(G, dt)
        del G
        Ci = t.cut(_uniform(t.ng, seed, 1.5, 2.5).reciprocal_(), dt)
        return {"T": T, "Ci": Ci, "h": h, "lam": 1.0}
    if kind == "gradient":
        # a smooth heat capacity to be found from noisy observations
        T0 = t.cut(_bump(t.ng, seed, 1.7, 1.0, 0.15), dt)
        Ci = t.cut(_sines(t.ng, seed, 0.53, 0.02, 4, 3).clamp_(0.4, 0.667), dt)
        noise = torch.randn((t.ng[2], t.ng[1], t.ng[0]), generator=_gen(seed + 19), device=DEV,
                            dtype=torch.float64)
        obs = t.cut(_bump(t.ng, seed + 1, 1.7, 0.95, 0.155) + 1e-3 * noise, dt)
        return {"T0": T0, "Ci": Ci, "obs": obs, "h": h, "lam": 1.0}
    if kind == "acoustic":
        # a pressure pulse and background modes, medium at rest
        G = _bump(t.ng, seed, 0.0, 1.0, 0.08) + _sines(t.ng, seed, 0.0, 0.05, 6, 12)
        rho, K = 1.0, 2.0
        return {"P": t.cut(G, dt), "h": h, "rho": rho, "K": K, "dt": 0.3 * min(h) / math.sqrt(K / rho)}
    # gp: a moving wave packet in a harmonic trap
    ax = _axes(t.ng)
    env = _bump(t.ng, seed, 0.0, 1.0, 0.16)
    k = (torch.rand(3, generator=_gen(seed + 23), device=DEV, dtype=torch.float64) * 40 + 10).tolist()
    ph = k[2] * ax[2][:, None, None] + k[1] * ax[1][None, :, None] + k[0] * ax[0][None, None, :]
    u, v = t.cut(env * torch.cos(ph), dt), t.cut(env * torch.sin(ph), dt)
    q = [50.0 * (a - 0.5) ** 2 for a in ax]
    V = t.cut(q[2][:, None, None] + q[1][None, :, None] + q[0][None, None, :], dt)
    g = 1.0
    return {"u": u, "v": v, "V": V, "h": h, "g": g,
            "dt": 0.3 / (2 * sum(1 / x ** 2 for x in h) + 40.0 + 2 * g)}


def _heat_dt(a, ci_max):
    return min(x * x for x in a["h"]) / a["lam"] / ci_max / 6.1


def _grid(c):
    return igg.Grid((c["nx"], c["ny"], c["nz"]), dims=(c["dx"], c["dy"], c["dz"]),
                    overlap=(c["overlap"],) * 3, periods=(c["px"], 0, 0))


def prepare(c, seed):
    a = _inputs(c, seed)
    st = {"c": c, "a": a}
    dt = DTYPES[c["dtype"]]
    if c["kind"] == "batch":
        b = igg.Batch(a["sizes"], dt)
        b.set_coefs(a["lam"], a["dts"], *[[d[k] for d in a["dd"]] for k in range(3)])
        T, Ci = b.empty().zero_(), b.empty().zero_()
        for i in range(len(a["sizes"])):
            b.view(T, i).copy_(a["T"][i])
            b.view(Ci, i).fill_(float(a["ci"][i]))
        del a["T"]
        st.update(b=b, T=T, T2=T.clone(), Ci=Ci)
        return st
    st["g"] = _grid(c)
    if c["kind"] == "heat":
        st["T2"] = a["T"].clone()
        st["dt"] = _heat_dt(a, float(igg.reduce(igg.RED_MAX, a["Ci"]).item()))
    elif c["kind"] == "gradient":
        st["dt"] = _heat_dt(a, float(igg.reduce(igg.RED_MAX, a["Ci"]).item()))
        a["T0"].requires_grad_(True)
        a["Ci"].requires_grad_(True)
    elif c["kind"] == "acoustic":
        P, st["Vx"], st["Vy"], st["Vz"] = st["g"].acoustic_fields(dt)
        P.copy_(a["P"])
        st["P"] = P
        del a["P"]
    return st


def run(st):
    c, a = st["c"], st["a"]
    nt = c["nt"]
    if c["kind"] == "heat":
        w = (16, max(2, c["overlap"]), max(2, c["overlap"])) if c["hidden"] else None
        return st["g"].run(nt, a["T"], st["T2"], a["Ci"], a["lam"], st["dt"], *a["h"], widths=w)
    if c["kind"] == "batch":
        return st["b"].run(nt, st["T"], st["T2"], st["Ci"])
    if c["kind"] == "gradient":
        T = ag.solve(a["T0"], a["Ci"], st["g"], nt, a["lam"], st["dt"], *a["h"])
        mis = ag.residual(T.detach(), a["obs"])
        gT, gC = torch.autograd.grad(T, (a["T0"], a["Ci"]), grad_outputs=mis)
        return {"T": T.detach(), "gT0": gT, "gCi": gC}
    if c["kind"] == "acoustic":
        for _ in range(nt):
            st["g"].acoustic_step(st["P"], st["Vx"], st["Vy"], st["Vz"], a["rho"], a["K"], a["dt"], *a["h"])
        return {"P": st["P"], "Vx": st["Vx"], "Vy": st["Vy"], "Vz": st["Vz"]}
    for _ in range(nt):
        st["g"].gp_step(a["u"], a["v"], a["V"], a["g"], a["dt"], *a["h"])
    return {"u": a["u"], "v": a["v"]}


# -- the same in plain 64-bit torch -----------------------------------------
def _plane(F, k, i):
    """The plane i of dimension k (0 = x) of every subdomain's field."""
    return F.select(F.dim() - 1 - k, i)


def _halo(t, F, delta=(0, 0, 0)):
    """The halo update of F [nsub][..] (staggered by delta), x, y, z in order."""
    for k in range(3):
        n, o = F.shape[3 - k], t.o[k] + delta[k]
        if o < 2:
            continue
        for s in range(t.nsub):
            l, r = t.neighbour(s, k, -1), t.neighbour(s, k, 1)
            if l >= 0:
                _plane(F[s], k, 0).copy_(_plane(F[l], k, n - o))
            if r >= 0:
                _plane(F[s], k, n - 1).copy_(_plane(F[r], k, o - 1))


def _halo_t(t, F):
    """The transpose of _halo: z, y, x; each halo entry into its source."""
    for k in (2, 1, 0):
        n, o = F.shape[3 - k], t.o[k]
        for s in range(t.nsub):
            for nb, dst, src in ((t.neighbour(s, k, -1), 0, n - o), (t.neighbour(s, k, 1), n - 1, o - 1)):
                if nb >= 0:
                    _plane(F[nb], k, src).add_(_plane(F[s], k, dst))
                    _plane(F[s], k, dst).zero_()


def _sh(F, k, d):
    """Inner points of one array [nz][ny][nx], shifted by d in dimension k."""
    sl = [slice(1, -1)] * 3
    sl[2 - k] = slice(1 + d, F.shape[2 - k] - 1 + d)
    return F[tuple(sl)]


def _lap(F, w):
    c = _sh(F, 0, 0)
    out = (-2.0 * (w[0] + w[1] + w[2])) * c
    for k in range(3):
        out += w[k] * (_sh(F, k, 1) + _sh(F, k, -1))
    return out


def _heat_step(t, T, Ci, w):
    out = T.clone()
    for s in range(T.shape[0]):
        _sh(out[s], 0, 0).add_(_sh(Ci[s], 0, 0) * _lap(T[s], w))
    if t is not None:
        _halo(t, out)
    return out


def exact(c, seed):
    a = _inputs(c, seed)
    nt = c["nt"]
    dt = DTYPES[c["dtype"]]
    if c["kind"] == "batch":
        # the packed layout: rows padded to 16 bytes, problems to 256 bytes
        es, at, places = SIZE[c["dtype"]], 0, []
        for nx, ny, nz in a["sizes"]:
            pitch = -(-nx * es // 16) * 16 // es
            places.append((at, pitch))
            at += -(-pitch * ny * nz * es // 256) * 256 // es
        out = torch.zeros(at, dtype=torch.float64, device=DEV)
        for i, s in enumerate(a["sizes"]):
            T = a["T"][i].to(dt).double()[None]
            Ci = torch.full_like(T, float(a["ci"][i])).to(dt).double()
            w = [a["dts"][i] * float(a["lam"][i]) / x ** 2 for x in a["dd"][i]]
            for _ in range(nt):
                T = _heat_step(None, T, Ci, w)
            p0, pitch = places[i]
            nx, ny, nz = s
            out[p0:p0 + pitch * ny * nz].view(nz, ny, pitch)[:, :, :nx].copy_(T[0])
        return out
    t = _Topo(c)
    if c["kind"] == "heat":
        T, Ci = a.pop("T").double(), a["Ci"].double()
        w = [_heat_dt(a, float(Ci.max())) * a["lam"] / x ** 2 for x in a["h"]]
        for _ in range(nt):
            T = _heat_step(t, T, Ci, w)
        return T
    if c["kind"] == "gradient":
        T, Ci, obs = a["T0"].double(), a["Ci"].double(), a["obs"].double()
        w = [_heat_dt(a, float(Ci.max())) * a["lam"] / x ** 2 for x in a["h"]]
        states = [T]
        for _ in range(nt):
            states.append(_heat_step(t, states[-1], Ci, w))
        lam = states[-1] - obs
        gCi = torch.zeros_like(Ci)
        for n in reversed(range(nt)):
            _halo_t(t, lam)
            new = lam.clone()
            for s in range(t.nsub):
                _sh(gCi[s], 0, 0).add_(_sh(lam[s], 0, 0) * _lap(states[n][s], w))
                v = _sh(Ci[s], 0, 0) * _sh(lam[s], 0, 0)
                _sh(new[s], 0, 0).add_(v * (-2.0 * (w[0] + w[1] + w[2])))
                for k in range(3):
                    _sh(new[s], k, 1).add_(v * w[k])
                    _sh(new[s], k, -1).add_(v * w[k])
            lam = new
        return {"T": states[-1], "gT0": lam, "gCi": gCi}
    if c["kind"] == "acoustic":
        P = a["P"].double()
        n = t.n
        V = []
        for k in range(3):
            m = [n[2], n[1], n[0]]
            m[2 - k] += 1
            V.append(torch.zeros([t.nsub] + m, dtype=torch.float64, device=DEV))
        for _ in range(nt):
            for k in range(3):
                ax = 3 - k
                V[k].narrow(ax, 1, n[k] - 1).sub_(a["dt"] / a["rho"] / a["h"][k] * P.diff(dim=ax))
            for k in range(3):
                P.sub_(a["dt"] * a["K"] / a["h"][k] * V[k].diff(dim=3 - k))
            _halo(t, P)
            for k in range(3):
                _halo(t, V[k], tuple(int(j == k) for j in range(3)))
        return {"P": P, "Vx": V[0], "Vy": V[1], "Vz": V[2]}
    u, v, V = (a[x].double() for x in ("u", "v", "V"))
    w = [-0.5 * a["dt"] / x ** 2 for x in a["h"]]
    for _ in range(nt):
        for o, r, sg in ((u, v, 1.0), (v, u, -1.0)):
            for s in range(t.nsub):
                q = a["dt"] * (V[s] + a["g"] * (u[s] ** 2 + v[s] ** 2))
                _sh(o[s], 0, 0).add_(sg * (_lap(r[s], w) + _sh(q, 0, 0) * _sh(r[s], 0, 0)))
            _halo(t, o)
    return {"u": u, "v": v}
