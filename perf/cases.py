"""Performance cases of the SPH density/force library: what a user's program has it do.

A case names a call sequence (``call``), a particle distribution (``dist``) with its
size, and the parameters a program sets.  The call sequences:

* ``static``   -- the allocation-free density of a small box (one call);
* ``density``  -- hand over a state, density at the given h (a program with its own h rule);
* ``fixed``    -- the same, then the force pass: both passes at the given h;
* ``h_update`` -- hand over a state, iterate h to N_ngb (density, ghost quantities);
* ``force``    -- the force pass alone, on a box whose density pass has run;
* ``passes``   -- hand over a state, one ``sph_step(0)``: build, h iteration, force (a
  program that integrates on its own and asks for the forces at new positions);
* ``kdk``      -- one kick-drift-kick step of a running simulation (fixed time step);
* ``served``   -- requests of several boxes through the batching server, from and to
  host memory, as a client sees them.

Sizes come from the repository's workloads and tests: the 16^3 lattice, the 262,144
Plummer box, the 977,621-particle Sod tube, the 8.4M log-normal field, the 33.5M clustered box
and its octant, the served lattices.  Inputs are drawn on the GPU from the seed
with the recipes of ``paper_1309_3783_gb300.inputs``.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1309_3783_gb300 import sph

GAMMA_K = 1.825742          # support radius / h
GAMMA_GAS = 5.0 / 3.0
ALPHA = 2.0
ETA = 1.2348                # h0 / local spacing at 48 neighbours
SOUND = math.sqrt(GAMMA_GAS * (GAMMA_GAS - 1.0))    # at u = 1


# ------------------------------------------------------------------------- the cases
def listed():
    return [
        # the smallest call: a small box, no context, nothing allocated
        {"name": "static 4096", "call": "static", "dist": "lattice", "side": 16, "periodic": True},
        # the smallest box through a kept handle: launches and the host path count
        {"name": "fixed 4096", "call": "fixed", "dist": "lattice", "side": 16, "periodic": True},
        # open box, ragged size, L not a power of two, high neighbour number (compensated sums)
        {"name": "passes open 59319 ngb128", "call": "passes", "dist": "lattice", "side": 39, "periodic": False,
         "L": 2.5, "n_ngb": 128.0, "h_tol": 1e-5},
        # a running simulation of a medium box, odd size
        {"name": "kdk 103823", "call": "kdk", "dist": "lattice", "side": 47, "periodic": True, "h_tol": 1e-5},
        # the mid-size clustered box: h iterated from an estimate, then forces
        {"name": "passes plummer 262144", "call": "passes", "dist": "plummer", "n": 262144, "spheres": 16,
         "scale": 0.02, "h_tol": 1e-5},
        # the Sod tube at the paper's size: density alone, forces alone, and the running
        # simulation that keeps its decomposition over steps
        {"name": "density sod 977621", "call": "density", "dist": "sod", "side": 116},
        {"name": "force lognormal 1000003", "call": "force", "dist": "lognormal", "n": 1000003, "grid": 128},
        {"name": "kdk sod 977621 reuse", "call": "kdk", "dist": "sod", "side": 116, "reuse": 1},
        # h iteration of an octant of the large box at the default leaf size
        {"name": "h_update clustered 4194304", "call": "h_update", "dist": "clustered", "n": 4194304, "spheres": 512,
         "L": 0.5},
        # running simulations of the large boxes, at the leaf sizes the autotuner keeps for them
        {"name": "kdk lognormal 8388608", "call": "kdk", "dist": "lognormal", "n": 8388608, "grid": 256,
         "leaf_max": 3200},
        {"name": "kdk clustered 33554432", "call": "kdk", "dist": "clustered", "n": 33554432, "spheres": 4096,
         "leaf_max": 4800},
        # a burst of served requests, log-uniform sizes, host memory to host memory
        {"name": "served 12 boxes", "call": "served", "dist": "lattice", "boxes": 12, "n_min": 1000, "n_max": 262144,
         "steps": 4, "h_tol": 1e-5},
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    call = rng.choice(["static", "density", "fixed", "h_update", "force", "passes", "passes", "kdk", "kdk", "kdk",
                       "served"])
    if call == "static":
        return {"call": call, "dist": "lattice", "side": rng.randint(11, 25), "periodic": rng.random() < 0.7}
    if call == "served":
        return {"call": call, "dist": "lattice", "boxes": rng.randint(3, 12), "n_min": rng.randint(1000, 4000),
                "n_max": size(8000, 262144), "steps": rng.randint(1, 6), "h_tol": 1e-5}
    c = {"call": call, "dist": rng.choice(["lattice", "plummer", "lognormal", "clustered"])}
    if c["dist"] == "lattice":
        c["n_ngb"] = rng.choice([48.0, 48.0, 64.0, 128.0])
        c["side"] = max(16, int(round(size(4000, 3000000) ** (1.0 / 3.0))))
        c["periodic"] = rng.random() < 0.6
        c["L"] = rng.choice([1.0, 1.0, 2.5, 0.7])
        n = c["side"] ** 3
    elif c["dist"] == "plummer":
        n = c["n"] = size(20000, 2000000) | 1
        c["spheres"] = rng.randint(4, 24)
        c["scale"] = round(rng.uniform(0.01, 0.05), 4)
    elif c["dist"] == "lognormal":
        n = c["n"] = size(500000, 8000000) | 1
        c["grid"] = 128
        c["leaf_max"] = rng.choice([400, 1600, 3200])
    else:
        n = c["n"] = size(500000, 16000000) | 1
        c["spheres"] = max(8, n // 8192)
        c["L"] = rng.choice([0.5, 1.0])
        c["leaf_max"] = rng.choice([400, 1600, 4800])
    if call == "kdk":
        c["reuse"] = rng.choice([0, 0, 1])
    if call in ("kdk", "passes", "h_update"):
        c["h_tol"] = 1e-5 if n < 1000000 else 1e-4
    return c


# --------------------------------------------------------------------------- inputs
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _uniform(g, *shape, lo=0.0, hi=1.0):
    return torch.rand(*shape, generator=g, device="cuda", dtype=torch.float64) * (hi - lo) + lo


def _wrap(x, L):
    x = torch.remainder(x, L)
    return torch.where(x >= L, torch.zeros_like(x), x)


def _eta(case):
    # h0 for the asked neighbour number (ETA gives 48)
    return ETA * (case.get("n_ngb", 48.0) / 48.0) ** (1.0 / 3.0)


def _state(x, h, n, L, g, v_sigma, u=None):
    v = (torch.randn(n, 3, generator=g, device="cuda", dtype=torch.float32) * v_sigma)
    m = torch.full((n,), L ** 3 / n, dtype=torch.float32, device="cuda")
    if u is None:
        u = torch.ones(n, dtype=torch.float32, device="cuda")
    h = h.clamp(max=0.2 * L / GAMMA_K)       # a first guess that fits the box
    return {"x": x.contiguous(), "v": v, "m": m, "u": u, "h": h.to(torch.float32).contiguous()}


def _lattice(case, seed, side=None):
    g, L = _gen(seed), float(case.get("L", 1.0))
    side = int(side or case["side"])
    a = L / side
    k = torch.arange(side, device="cuda", dtype=torch.float64)
    idx = torch.stack(torch.meshgrid(k, k, k, indexing="ij"), dim=-1).reshape(-1, 3)
    x = (idx + 0.5 + _uniform(g, *idx.shape, lo=-0.2, hi=0.2)) * a
    x = _wrap(x, L) if case.get("periodic", True) else x.clamp(0.0, math.nextafter(L, 0.0))
    n = side ** 3
    # h off its converged value by a few per cent, as a program's last values are
    h = _eta(case) * a * (1.0 + 0.03 * (2.0 * _uniform(g, n) - 1.0))
    return _state(x, h, n, L, g, 0.05)


def _sod(case, seed):
    # dense half: side/2 x side x side, thin half about a quarter of the density (side / 4^(1/3))
    g, s = _gen(seed), int(case["side"])
    t = int(round(s / 4.0 ** (1.0 / 3.0)))
    parts, hs = [], []
    for x0, nx, ny in ((0.0, s // 2, s), (0.5, (t + 1) // 2, t)):
        ax, a = 0.5 / nx, 1.0 / ny
        ix = torch.arange(nx, device="cuda", dtype=torch.float64)
        iy = torch.arange(ny, device="cuda", dtype=torch.float64)
        idx = torch.stack(torch.meshgrid(ix, iy, iy, indexing="ij"), dim=-1).reshape(-1, 3) + 0.5
        idx = idx + _uniform(g, *idx.shape, lo=-0.02, hi=0.02)
        parts.append(idx * torch.tensor([ax, a, a], device="cuda", dtype=torch.float64)
                     + torch.tensor([x0, 0.0, 0.0], device="cuda", dtype=torch.float64))
        hs.append(torch.full((idx.shape[0],), ETA * a, device="cuda", dtype=torch.float64))
    nl, nr = parts[0].shape[0], parts[1].shape[0]
    n = nl + nr
    u = torch.cat([torch.full((nl,), 1.5, device="cuda"), torch.full((nr,), 0.1795 * 1.5 * nl / nr, device="cuda")])
    st = _state(_wrap(torch.cat(parts), 1.0), torch.cat(hs), n, 1.0, g, 0.0, u)
    st["m"].fill_(0.5 / nl)
    return st


def _isotropic(g, n):
    z = _uniform(g, n, lo=-1.0, hi=1.0)
    phi = _uniform(g, n, hi=2.0 * math.pi)
    s = torch.sqrt(1.0 - z * z)
    return torch.stack([s * torch.cos(phi), s * torch.sin(phi), z], dim=1)


def _spheres(case, seed):
    """Uniform background plus Plummer spheres (``plummer``: equal ones; ``clustered``: log-uniform scales)."""
    g, L, n, ns = _gen(seed), float(case.get("L", 1.0)), int(case["n"]), int(case["spheres"])
    equal = case["dist"] == "plummer"
    n_bg = int(round(n * (0.5 if equal else 0.3)))
    n_sp = n - n_bg
    sid = torch.arange(n_sp, device="cuda") * ns // n_sp              # sphere by sphere
    per = n_sp / ns
    centres = _uniform(g, ns, 3, hi=L)
    if equal:
        scale = torch.full((ns,), float(case["scale"]) * L, device="cuda", dtype=torch.float64)
    else:
        scale = torch.exp(_uniform(g, ns, lo=math.log(1e-4), hi=math.log(1e-2)))
    a = scale[sid]
    r_max = 0.5
    top = (r_max ** 2 / (r_max ** 2 + a * a)) ** 1.5                  # enclosed fraction at r_max
    X = (1.0 - _uniform(g, n_sp)) * top
    r = a / torch.sqrt((X ** (-2.0 / 3.0) - 1.0).clamp(min=1e-12))
    x = torch.cat([_uniform(g, n_bg, 3, hi=L), centres[sid] + r[:, None] * _isotropic(g, n_sp)])
    x = _wrap(x, L)
    dens = torch.full((n,), n_bg / L ** 3, device="cuda", dtype=torch.float64)
    if equal:
        for s in range(ns):
            d = x - centres[s]
            d = d - L * torch.round(d / L)
            q2 = (d * d).sum(1) / scale[s] ** 2
            dens += 3.0 * per / (4.0 * math.pi * scale[s] ** 3) * (1.0 + q2) ** -2.5
    else:
        dens[n_bg:] += 3.0 * per / (4.0 * math.pi * a ** 3) * (1.0 + (r / a) ** 2) ** -2.5
    return _state(x, _eta(case) * dens ** (-1.0 / 3.0), n, L, g, 0.1)


def _lognormal(case, seed):
    g, n, m = _gen(seed), int(case["n"]), int(case["grid"])
    k = torch.fft.fftfreq(m, device="cuda", dtype=torch.float64) * m
    kz = torch.fft.rfftfreq(m, device="cuda", dtype=torch.float64) * m
    k2 = k[:, None, None] ** 2 + k[None, :, None] ** 2 + kz[None, None, :] ** 2
    amp = torch.where(k2 > 0, k2.clamp(min=1e-30) ** -0.5, torch.zeros_like(k2))       # P(k) ~ k^-2
    f = torch.fft.irfftn(torch.fft.rfftn(torch.randn(m, m, m, generator=g, device="cuda", dtype=torch.float64)) * amp,
                         s=(m, m, m))
    f = (f - f.mean()) / f.std()
    p = torch.exp(2.0 * f).reshape(-1)
    p = p / p.sum()
    cell = torch.searchsorted(torch.cumsum(p, 0), _uniform(g, n).sort().values).clamp(max=m ** 3 - 1)
    ijk = torch.stack([cell // (m * m), cell // m % m, cell % m], dim=1).to(torch.float64)
    x = _wrap((ijk + _uniform(g, n, 3)) / m, 1.0)
    dens = n * p[cell] * m ** 3
    return _state(x, _eta(case) * dens ** (-1.0 / 3.0), n, 1.0, g, 0.1)


_DIST = {"lattice": _lattice, "sod": _sod, "plummer": _spheres, "clustered": _spheres, "lognormal": _lognormal}


def _inputs(case, seed):
    return _DIST[case["dist"]](case, seed)


def _dt(st):
    # a Courant step of the initial state, from its first-guess supports
    c = SOUND * math.sqrt(float(st["u"].max()))
    return 0.3 * GAMMA_K * float(st["h"].min()) / (2.2 * c + 1.0)


def _served_sides(case, seed):
    # the sizes belong to the case (spread evenly over the logarithm), the particles to the seed
    k = int(case["boxes"])
    lo, hi = math.log(case["n_min"]), math.log(case["n_max"])
    return [min(64, max(10, int(round(math.exp((lo + (hi - lo) * (i + 0.5) / k) / 3.0))))) for i in range(k)]


# ------------------------------------------------------------------------ the handles
_CTX = {}


def _ctx(case):
    """The program's context for these parameters (one per process and parameter set)."""
    key = (case.get("n_ngb", 48.0), case.get("h_tol", 1e-4), case.get("reuse", 0), case.get("leaf_max", 400))
    if key not in _CTX:
        p = sph.sph_params_default()
        p.n_ngb, p.h_tol, p.reuse, p.leaf_max = key
        _CTX[key] = sph.sph_ctx_create(p, 0)
    return _CTX[key]


class _Server:
    def __init__(self, ctx):
        self.h = sph.sph_server_create(ctx)

    def __del__(self):
        sph.sph_server_destroy(self.h)


_OUT = {"rho": (torch.float32, 1), "drho_dh": (torch.float32, 1), "nngb": (torch.float32, 1),
        "count": (torch.int32, 1), "h": (torch.float32, 1), "a": (torch.float32, 3), "dudt": (torch.float32, 1),
        "vsig": (torch.float32, 1), "x": (torch.float64, 3), "v": (torch.float32, 3), "u": (torch.float32, 1)}
_READ = {"density": ("rho", "drho_dh", "nngb", "count"), "fixed": ("rho", "count", "a", "dudt", "vsig"),
         "h_update": ("rho", "nngb", "h"), "force": ("a", "dudt", "vsig"), "passes": ("rho", "h", "a", "dudt", "vsig"),
         "kdk": ("x", "v", "u", "h", "a", "dudt"), "served": ("x", "v", "u", "h", "rho")}


def prepare(case, seed):
    call = case["call"]
    if call == "served":
        boxes = []
        for i, s in enumerate(_served_sides(case, seed)):
            st = _lattice(case, 1000 * int(seed) + i, side=s)
            boxes.append({k: t.cpu().numpy() for k, t in st.items()})
        dts = [0.2 * GAMMA_K * ETA / s / (2.2 * SOUND + 1.0) for s in _served_sides(case, seed)]
        return {"call": call, "boxes": boxes, "dt": dts, "steps": int(case["steps"]), "server": _Server(_ctx(case))}
    st = _inputs(case, seed)
    n, L, periodic = st["m"].numel(), float(case.get("L", 1.0)), bool(case.get("periodic", True))
    if call == "static":
        sph.load()
        return {"call": call, "in": st, "L": L, "periodic": periodic,
                "rho": torch.empty(n, device="cuda"), "count": torch.empty(n, device="cuda", dtype=torch.int32)}
    torch.cuda.synchronize()            # the context has a stream of its own
    box = sph.Box(_ctx(case), n, L, periodic)
    out = {k: torch.empty((n, _OUT[k][1]) if _OUT[k][1] > 1 else n, device="cuda", dtype=_OUT[k][0])
           for k in _READ[call]}
    s = {"call": call, "in": st, "box": box, "out": out}
    if call == "force":
        box.set(**st)
        box.density()
    if call == "kdk":
        s["dt"] = _dt(st)
        box.set(**st)
        box.step(0.0)                   # the starting forces of the simulation
    torch.cuda.synchronize()
    return s


# -------------------------------------------------------------------------- one pass
def run(s):
    call = s["call"]
    if call == "static":
        i = s["in"]
        sph.sph_density_static(i["x"], i["m"], i["h"], s["L"], s["periodic"], s["rho"], s["count"])
        return {"rho": s["rho"], "count": s["count"]}
    if call == "served":
        srv = s["server"].h
        ids = [sph.sph_server_submit(srv, b["x"], b["v"], b["m"], b["u"], b["h"], 1.0, True, s["steps"], dt)
               for b, dt in zip(s["boxes"], s["dt"])]
        while sph.sph_server_tick(srv):
            pass
        res = []
        for rid, b in zip(ids, s["boxes"]):
            res.append([sph.sph_server_get(srv, rid, f, len(b["m"])) for f in _READ["served"]])
            sph.sph_server_release(srv, rid)
        return res
    box = s["box"]
    if call in ("density", "fixed", "h_update", "passes"):
        box.set(**s["in"])
    if call in ("density", "fixed"):
        box.density()
    if call in ("fixed", "force"):
        box.force()
    if call == "h_update":
        box.h_update()
    if call == "passes":
        box.step(0.0)
    if call == "kdk":
        box.step(s["dt"])
    for f, t in s["out"].items():
        box.get(f, t)
    return s["out"]


# ------------------------------------------------------------------------- the floor
def work(case):
    """Bytes: the state in and the results out, once.  Flops: the interacting pairs only (11 per
    unordered pair and 16 per side for density, 75 per unordered pair for force; N_ngb
    neighbours each)."""
    call = case["call"]
    if call == "served":
        n, steps = sum(s ** 3 for s in _served_sides(case, 0)), int(case["steps"])
    elif case["dist"] == "lattice":
        n, steps = int(case["side"]) ** 3, 1
    elif case["dist"] == "sod":
        s = int(case["side"])
        t = int(round(s / 4.0 ** (1.0 / 3.0)))
        n, steps = s // 2 * s * s + (t + 1) // 2 * t * t, 1
    else:
        n, steps = int(case["n"]), 1
    pairs = 0.5 * case.get("n_ngb", 48.0) * n
    dens, force = (11 + 32) * pairs, 75 * pairs
    per = {"static": (40, dens), "density": (48 + 16, dens), "fixed": (48 + 28, dens + force),
           "h_update": (48 + 12, dens), "force": (48 + 16 + 20, force), "passes": (48 + 28, dens + force),
           "kdk": (64 + 60, dens + force), "served": (48 / steps + 48 / steps + 76, dens + force)}[call]
    return {"bytes": float(per[0]) * n * steps, "flops": float(per[1]) * steps}


# ------------------------------------------------------------------ values in 64 bits
def _near(x, reach, L, periodic):
    """Ordered pairs (i, j), i != j, with r < max(reach_i, reach_j): i, j, d = x_i - x_j, r (all pairs tested)."""
    n = x.shape[0]
    rows = max(1, (1 << 27) // n)
    got = []
    for a in range(0, n, rows):
        b = min(n, a + rows)
        r2 = torch.zeros(b - a, n, device=x.device, dtype=torch.float64)
        for k in range(3):
            d = x[a:b, k, None] - x[None, :, k]
            if periodic:
                d -= L * torch.round(d / L)
            r2 += d * d
        i, j = torch.nonzero(r2 < torch.maximum(reach[a:b, None], reach[None, :]) ** 2, as_tuple=True)
        keep = i + a != j
        got.append((i[keep] + a, j[keep]))
    i, j = (torch.cat(t) for t in zip(*got))
    d = x[i] - x[j]
    if periodic:
        d = torch.where(d > 0.5 * L, d - L, torch.where(d < -0.5 * L, d + L, d))
    return i, j, d, torch.sqrt((d * d).sum(1))


def _kernel(r, H):
    """W and dW/dr of the cubic spline with support H."""
    q = r / H
    k = 8.0 / math.pi / H ** 3
    w = torch.where(q < 0.5, 1 - 6 * q * q + 6 * q ** 3, torch.where(q < 1, 2 * (1 - q) ** 3, torch.zeros_like(q)))
    dw = torch.where(q < 0.5, -12 * q + 18 * q * q, torch.where(q < 1, -6 * (1 - q) ** 2, torch.zeros_like(q)))
    return k * w, k / H * dw


def _sums(p, m, H):
    """Density sums at supports H over the pair list p."""
    i, j, _, r = p
    k = r < H[i]
    i, j, r = i[k], j[k], r[k]
    w, dw = _kernel(r, H[i])
    zero = torch.zeros_like(H)
    w0 = 8.0 / math.pi / H ** 3
    return {"rho": zero.index_add(0, i, m[j] * w) + m * w0, "srm": zero.index_add(0, i, m[j] * r * dw),
            "nw": zero.index_add(0, i, w) + w0, "sr": zero.index_add(0, i, r * dw),
            "count": torch.zeros(H.numel(), device=H.device, dtype=torch.int64).index_add(
                0, i, torch.ones_like(i))}


def _iterate(x, m, h0, L, periodic, n_ngb, tol):
    """Newton on (4 pi/3) H^3 n = n_ngb per particle, kept inside its bracket and [h/2, 2h]; (h, sums, pairs)."""
    h = h0.clone()
    room, reach = 1.3, None
    lo, hi = torch.zeros_like(h), torch.full_like(h, math.inf)
    act = torch.ones_like(h, dtype=torch.bool)
    for it in range(1, 31):
        if reach is None or bool((GAMMA_K * h > reach).any()):
            reach = torch.maximum(room * GAMMA_K * h, reach if reach is not None else torch.zeros_like(h))
            pairs = _near(x, reach, L, periodic)
        H = GAMMA_K * h
        s = _sums(pairs, m, H)
        F = 4.0 * math.pi / 3.0 * H ** 3 * s["nw"] - n_ngb
        act = act & (F.abs() > tol * n_ngb)
        if it == 30 or not bool(act.any()):
            break
        dN = -GAMMA_K * (4.0 * math.pi / 3.0) * H * H * s["sr"]
        lo = torch.where(act & (F < 0), h, lo)
        hi = torch.where(act & (F >= 0), h, hi)
        hn = torch.where(dN > 0, h - F / dN, torch.where(F < 0, 2 * h, 0.5 * h))
        hn = torch.minimum(torch.maximum(hn, 0.5 * h), 2 * h)
        out = (lo > 0) & torch.isfinite(hi) & ~((hn > lo) & (hn < hi))
        h = torch.where(act, torch.where(out, 0.5 * (lo + hi), hn), h)
    return h, s, pairs


def _forces(p, m, v, u, H, s):
    i, j, d, r = p
    k = (r < torch.maximum(H[i], H[j])) & (r > 0)
    i, j, d, r = i[k], j[k], d[k], r[k]
    P = (GAMMA_GAS - 1.0) * s["rho"] * u
    c = torch.sqrt(GAMMA_GAS * P / s["rho"])
    f = torch.where(s["srm"] < 0, -3.0 * s["rho"] / s["srm"].clamp(max=-1e-300), torch.ones_like(P))
    F = f * P / s["rho"] ** 2
    wi, wj = _kernel(r, H[i])[1], _kernel(r, H[j])[1]
    w = ((v[i] - v[j]) * d).sum(1) / r
    mu = w.clamp(max=0.0)
    vs = c[i] + c[j] - 3.0 * mu
    pi = -ALPHA * vs * mu / (s["rho"][i] + s["rho"][j])
    wb = 0.5 * (wi + wj)
    a = torch.zeros(H.numel(), 3, device=H.device, dtype=torch.float64).index_add(
        0, i, -(m[j] * (F[i] * wi + F[j] * wj + pi * wb) / r)[:, None] * d)
    du = torch.zeros_like(H).index_add(0, i, m[j] * (F[i] * wi + 0.5 * pi * wb) * w)
    vsig = torch.zeros_like(H).index_reduce(0, i, vs, "amax", include_self=True)
    return {"a": a, "dudt": du, "vsig": vsig}


def exact(case, seed):
    call = case["call"]
    if call == "served":
        return None
    n = case.get("n", int(case.get("side", 0)) ** 3)
    if case["dist"] in ("sod", "clustered") or n > 300000:
        return None                     # every pair is tested: larger boxes take too long
    st = _inputs(case, seed)
    L, periodic = float(case.get("L", 1.0)), bool(case.get("periodic", True))
    n_ngb, tol = case.get("n_ngb", 48.0), case.get("h_tol", 1e-4)
    x = st["x"]
    v, m, u, h = (st[k].double() for k in ("v", "m", "u", "h"))
    if call in ("static", "density", "fixed", "force"):
        H = (st["h"] * torch.tensor(GAMMA_K, dtype=torch.float32, device="cuda")).double()   # rounded once, as documented
        p = _near(x, H, L, periodic)
        s = _sums(p, m, H)
        s["nngb"] = 4.0 * math.pi / 3.0 * H ** 3 * s["nw"]
        s["drho_dh"] = -(3.0 * s["rho"] + s["srm"]) / h
        s.update(_forces(p, m, v, u, H, s))
        if call == "static":
            return {"rho": s["rho"], "count": None}
        return {k: None if k == "count" else s[k] for k in _READ[call]}
    h, s, p = _iterate(x, m, h, L, periodic, n_ngb, tol)
    s["nngb"] = 4.0 * math.pi / 3.0 * (GAMMA_K * h) ** 3 * s["nw"]
    s["h"] = h
    if call == "h_update":
        return {k: s[k] for k in _READ[call]}
    s.update(_forces(p, m, v, u, GAMMA_K * h, s))
    if call == "passes":
        return {k: s[k] for k in _READ[call]}
    # one kick-drift-kick step from these forces; the passes see v and u predicted to its end
    dt = _dt(st)
    v = v + 0.5 * dt * s["a"]
    u = (u + 0.5 * dt * s["dudt"]).clamp(min=0.0)
    x = x + dt * v
    x = _wrap(x, L) if periodic else x.clamp(0.0, math.nextafter(L, 0.0))
    vp, up = v + 0.5 * dt * s["a"], (u + 0.5 * dt * s["dudt"]).clamp(min=0.0)
    h, s, p = _iterate(x, m, h, L, periodic, n_ngb, tol)
    s.update(_forces(p, m, vp, up, GAMMA_K * h, s))
    s.update({"x": x, "h": h, "v": v + 0.5 * dt * s["a"], "u": (u + 0.5 * dt * s["dudt"]).clamp(min=0.0)})
    return {k: s[k] for k in _READ[call]}
