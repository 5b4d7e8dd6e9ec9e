"""The work that users of this framework have it do, as measurable cases.

Each case is one pass through public entry points: whole solves from 32^3 to
1024^3 in FP32 and FP64 with each weighting, the batched and the parameter-study
forms, ranking and matching of a caller's own intensities at ragged counts, and
the source-field pipeline.  Grid sizes, boxes (about 0.8 h^-1 Mpc per cell),
histories and mean free paths are those of the tests, the benchmark and the
serving loop.  Inputs follow the recipe of paper_2109_10375_gb300.synth (a
Gaussian density with P(k) = k^-2.5 exp(-(k/k_c)^2), excursion-set sources),
made here on the GPU in one go so that they are quick to make at any size.
"""
import math
import os

import numpy as np
import torch

from paper_2109_10375_gb300 import binding as B

HISTORY = (8.0, 4.0, 3.0)  # (z_mid, dz, Az) of the benchmark
WEIGHTS = {"mass": 0, "growth": 1, "volume": 2}


def listed():
    return [
        # smoke-sized field: tests, interactive use; latency and launches count
        {"name": "solve_32", "kind": "solve", "n": 32, "l_mfp": 3.0, "weighting": "mass", "want_J": True},
        # the serving loop's most frequent grid, growth-rescaled matching (the paper's full equation)
        {"name": "solve_128_growth", "kind": "solve", "n": 128, "l_mfp": 3.0, "weighting": "growth", "want_J": False},
        # the serving loop's largest grid, a first request for a field
        {"name": "solve_512", "kind": "solve", "n": 512, "l_mfp": 10.0, "weighting": "mass", "want_J": True},
        # the benchmark's headline workload (paper-size box)
        {"name": "solve_1024", "kind": "solve", "n": 1024, "l_mfp": 5.0, "weighting": "mass", "want_J": False},
        # the FP64 intensity form at its largest grid (accuracy studies)
        {"name": "solve_f64_256", "kind": "solve_f64", "n": 256, "l_mfp": 3.0, "weighting": "mass", "want_J": True},
        # the batched workload: 32 x 128^3 + 16 x 256^3 realisations in one captured graph
        {"name": "batch_48", "kind": "batch", "n_a": 128, "count_a": 32, "n_b": 256, "count_b": 16},
        # parameter study, new mean free path: from the kept transformed source
        {"name": "new_mfp_256", "kind": "spectrum", "n": 256, "l_mfp": 5.0, "weighting": "mass", "want_J": True},
        # parameter study, new history only (70 % of the serving requests): matching alone
        {"name": "new_history_512", "kind": "history", "n": 512, "l_mfp": 3.0, "weighting": "mass"},
        # a caller's own intensities on a ragged cell count: rank, then match, with the fraction F
        {"name": "rank_match_10m", "kind": "rank_match", "cells": 10_000_019, "weighting": "mass"},
        # 2LPT displacements of a linear field
        {"name": "lpt_512", "kind": "lpt", "n": 512},
        # mesh density from displaced particles: TSC, interlaced and deconvolved
        {"name": "density_512", "kind": "density", "n": 512, "order": 3, "interlace": True},
        # ESF-L source field: 2LPT, collapsed fraction, weighted CIC interlaced mesh
        {"name": "esf_l_256", "kind": "esf_l", "n": 256},
    ]


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "solve_f64", "batch", "spectrum", "history", "rank_match",
                       "rank_match", "lpt", "density", "esf_l"])
    weighting = rng.choice(["mass", "mass", "growth", "volume"])
    l_mfp = round(rng.uniform(1.0, 20.0), 3)
    if kind == "solve":
        return {"kind": kind, "n": rng.choice([32, 64, 128, 256, 512]), "l_mfp": l_mfp, "weighting": weighting,
                "want_J": rng.random() < 0.5}
    if kind == "solve_f64":
        return {"kind": kind, "n": rng.choice([32, 64, 128, 256]), "l_mfp": l_mfp, "weighting": weighting,
                "want_J": True}
    if kind == "batch":
        return {"kind": kind, "n_a": rng.choice([32, 64, 128]), "count_a": rng.randint(1, 24), "n_b": 256,
                "count_b": rng.randint(0, 8)}
    if kind == "spectrum":
        return {"kind": kind, "n": rng.choice([64, 128, 256, 512]), "l_mfp": l_mfp, "weighting": weighting,
                "want_J": rng.random() < 0.5}
    if kind == "history":
        return {"kind": kind, "n": rng.choice([64, 128, 256, 512]), "l_mfp": l_mfp, "weighting": weighting}
    if kind == "rank_match":
        return {"kind": kind, "cells": int(10 ** rng.uniform(3.5, 7.8)) | 1, "weighting": weighting}
    if kind == "density":
        return {"kind": kind, "n": rng.choice([64, 128, 256, 512]), "order": rng.choice([1, 2, 3, 3]),
                "interlace": rng.random() < 0.7}
    return {"kind": kind, "n": rng.choice([64, 128, 256, 512])}


# ---------------------------------------------------------------------------
# Inputs (from the seed alone, on the GPU)
# ---------------------------------------------------------------------------
def _box(n):
    return 1000.0 if n == 1024 else n * 0.78125


def _wave(n, device, dtype):
    """(kx [n/2+1], ky [n]) as signed integer wave numbers."""
    kx = torch.arange(n // 2 + 1, device=device, dtype=dtype)
    ky = torch.arange(n, device=device, dtype=dtype)
    return kx, torch.where(ky < n // 2, ky, ky - n)


def _delta(n, seed, sigma, dtype):
    """Gaussian density of the recipe, mean 0 and the given rms."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    w = torch.randn((n, n, n), generator=g, device="cuda", dtype=dtype)
    wk = torch.fft.rfftn(w)
    del w
    kx, ky = _wave(n, "cuda", dtype)
    for z in range(0, n, 64):  # plane blocks, so that temporaries stay small
        k2 = ky[z:z + 64, None, None] ** 2 + ky[None, :, None] ** 2 + kx[None, None, :] ** 2
        k2[k2 == 0] = math.inf
        wk[z:z + 64] *= k2.pow(-0.625) * torch.exp(k2 * (-0.5 / (0.25 * n) ** 2))
    d = torch.fft.irfftn(wk, s=(n, n, n))
    del wk
    d -= d.mean()
    d *= sigma / d.square().mean().sqrt()
    return d


def _source_and_mass(n, seed, dtype=torch.float32):
    d = _delta(n, seed, 1.5, dtype)
    mass = 1.0 + d.clamp(min=-0.99)
    S = d.mul_(-1.0).add_(1.686).mul_(1.0 / (math.sqrt(2.0) * 0.7)).erfc_().mul_(mass)
    S /= S.mean()
    return S, mass.to(torch.float32)


def _batch_items(case, seed):
    """(n, l_mfp, history, weighting, field seed) of each realisation."""
    rng = np.random.default_rng(seed)
    sizes = [case["n_a"]] * case["count_a"] + [case["n_b"]] * case["count_b"]
    return [(n, float(rng.uniform(1, 20)),
             (float(rng.uniform(6.5, 9)), float(rng.uniform(2, 6)), float(rng.uniform(1.5, 5))), "mass",
             seed * 1000 + i) for i, n in enumerate(sizes)]


def _intensity(cells, seed):
    """A few-octave positive intensity field and masses on a plain list of cells."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    J = torch.randn(cells, generator=g, device="cuda").mul_(0.8).exp_()
    mass = torch.randn(cells, generator=g, device="cuda").mul_(0.5).exp_()
    return J, mass


def _ranked(S, mass, box, l_mfp):
    """(order, masses in rank order) that an earlier solve of this field left behind."""
    order = torch.sort(_field(S, box, l_mfp).float().reshape(-1), descending=True, stable=True).indices
    return order.to(torch.int32), mass.reshape(-1)[order]


def _zeldovich(n, seed, box):
    """First-order displacement of a linear field: smooth, a few cells at most."""
    H = torch.fft.rfftn(_delta(n, seed, 1.0, torch.float32))
    kx, ky = _wave(n, "cuda", torch.float32)
    k = [kx[None, None, :], ky[None, :, None], ky[:, None, None]]
    k2 = k[0] ** 2 + k[1] ** 2 + k[2] ** 2
    k2[0, 0, 0] = math.inf
    return tuple(torch.fft.irfftn(H * (k[a] / k2) * (1j * D1 * box / (2.0 * math.pi)), s=(n, n, n))
                 for a in range(3))


D1 = 0.25  # growth factor of the benchmark's source pipeline (linear field of rms 1)
D2 = -3.0 / 7.0 * D1 ** 2


def _history(case, point=HISTORY):
    return B.history(*point, weighting=WEIGHTS[case.get("weighting", "mass")])


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        # the size's default choices, not timed ones: the same work on every run
        os.environ.setdefault("AMBER_AUTOTUNE", "0")
        todo = _batch_items(case, seed)
        ctx = B.Context(max(t[0] for t in todo) ** 3)
        items = []
        for n, l, point, weighting, s in todo:
            S, mass = _source_and_mass(n, s)
            items.append((S, mass, _box(n), l, B.history(*point, weighting=WEIGHTS[weighting]), torch.empty_like(S)))
        return {"kind": kind, "ctx": ctx, "batch": B.Batch([ctx], items), "out": [it[5] for it in items]}
    if kind == "rank_match":
        J, mass = _intensity(case["cells"], seed)
        return {"kind": kind, "ctx": B.Context(case["cells"]), "J": J, "mass": mass, "h": _history(case),
                "order": torch.empty(case["cells"], dtype=torch.int32, device="cuda"), "z": torch.empty_like(J),
                "F": torch.empty(case["cells"], dtype=torch.float64, device="cuda")}
    n, box = case["n"], _box(case["n"])
    st = dict(case, ctx=B.Context(n ** 3), box=box)
    if kind == "density":
        st["psi"] = _zeldovich(n, seed, box)
        st["rho"] = torch.empty_like(st["psi"][0])
        return st
    if kind in ("lpt", "esf_l"):
        st["delta"] = _delta(n, seed, 1.0, torch.float32)
        return st
    S, mass = _source_and_mass(n, seed, torch.float64 if kind == "solve_f64" else torch.float32)
    st |= {"h": _history(case), "z": torch.empty_like(mass), "J": torch.empty_like(S) if case.get("want_J") else None}
    if kind == "history":
        st["order"], st["mass_rank"] = _ranked(S, mass, box, case["l_mfp"])
        return st
    st["mass"] = mass
    if kind == "spectrum":
        st["spec"] = st["ctx"].source_spectrum(S)
    else:
        st["S"] = S
    return st


def run(state):
    ctx, kind = state["ctx"], state["kind"]
    if kind == "batch":
        state["batch"].launch()
        return state["out"]
    if kind == "rank_match":
        ctx.rank(state["J"], out=state["order"])
        ctx.assign_zre(state["order"], state["mass"], state["h"], out=state["z"], F=state["F"])
        return {"order": state["order"], "z": state["z"], "F": state["F"]}
    box = state["box"]
    if kind == "density":
        return ctx.mesh_density(state["psi"], box, state["order"], state["interlace"], out=state["rho"])
    if kind in ("lpt", "esf_l"):
        psi = ctx.lpt_displacement(state["delta"], box, D1, D2)
        if kind == "lpt":
            return {"psi": psi}
        f = ctx.esf_fcoll(state["delta"], box, 2.0 * box / state["n"], 1.686 / D1, 1.0)
        return {"psi": psi, "f": f, "rho": ctx.mesh_density(psi, box, 2, True, mass=f)}
    z, J, h, l = state["z"], state["J"], state["h"], state["l_mfp"]
    if kind == "spectrum":
        ctx.solve_spectrum(state["spec"], state["mass"], box, l, h, z, J_out=J)
    elif kind == "history":
        ctx.assign_zre_ranked(state["order"], state["mass_rank"], h, z)
    else:
        ctx.solve(state["S"], state["mass"], box, l, h, out=z, J_out=J)
    return {"z": z} if J is None else {"z": z, "J": J}


# ---------------------------------------------------------------------------
# Bytes and operations that one pass cannot do without
# ---------------------------------------------------------------------------
def _fft_flops(n):
    return 2.5 * n ** 3 * 3 * math.log2(n)  # one real transform of n^3 cells


def work(case):
    kind = case["kind"]
    if kind == "batch":
        cells = case["count_a"] * case["n_a"] ** 3 + case["count_b"] * case["n_b"] ** 3
        return {"bytes": 12.0 * cells,
                "flops": 2 * (case["count_a"] * _fft_flops(case["n_a"]) + case["count_b"] * _fft_flops(case["n_b"]))}
    if kind == "rank_match":
        return {"bytes": (4 + 4 + 4 + 4 + 8) * float(case["cells"]), "flops": 10.0 * case["cells"]}
    n = case["n"]
    c = float(n) ** 3
    if kind == "lpt":
        return {"bytes": 16 * c, "flops": 11 * _fft_flops(n)}
    if kind == "density":
        return {"bytes": 16 * c, "flops": 60 * c + (3 * _fft_flops(n) if case["interlace"] else 0)}
    if kind == "esf_l":
        return {"bytes": 24 * c, "flops": 16 * _fft_flops(n) + 30 * c}
    if kind == "history":
        return {"bytes": 12 * c, "flops": 10 * c}
    word = 8 if kind == "solve_f64" else 4
    source = 8 * n * n * (n // 2 + 1) if kind == "spectrum" else word * c
    return {"bytes": source + 8 * c + (word * c if case.get("want_J") else 0),
            "flops": (1 if kind == "spectrum" else 2) * _fft_flops(n)}


# ---------------------------------------------------------------------------
# The same results in 64 bits, as plain torch and numpy give them
# ---------------------------------------------------------------------------
def _weibull(point):
    """(a, b, c) of x(z) = exp(-max((z - a)/b, 0)^c) through (early, mid, late) = (0.05, 0.5, 0.95)."""
    zm, dz, Az = point
    ze = zm + dz * Az / (1 + Az)
    zl = ze - dz
    Le, Lm, Ll = (abs(math.log(x)) for x in (0.05, 0.5, 0.95))

    def offset(c):
        pm, pl = Lm ** (1 / c), Ll ** (1 / c)
        return (zl * pm - zm * pl) / (pm - pl)

    def f(c):
        a = offset(c)
        return (Le / Lm) ** (1 / c) - (ze - a) / (zm - a)

    grid = np.exp(np.linspace(math.log(0.05), math.log(100.0), 401))
    for lo, hi in zip(grid[:-1], grid[1:]):
        if f(lo) * f(hi) > 0:
            continue
        up = f(lo) > 0
        for _ in range(200):
            mid = 0.5 * (lo + hi)
            lo, hi = (mid, hi) if (f(mid) > 0) == up else (lo, mid)
        c = 0.5 * (lo + hi)
        a = offset(c)
        b = (zm - a) / Lm ** (1 / c)
        if a > 0 and b > 0:
            return a, b, c
    raise ValueError("no Weibull history through these points")


def _growth(z, om=0.3):
    """Linear growth factor of flat LCDM (any normalisation)."""
    x, w = np.polynomial.legendre.leggauss(64)
    a = 1.0 / (1.0 + np.asarray(z, dtype=np.float64))[..., None]
    s = np.sqrt(a) * 0.5 * (x + 1.0)
    f = 2.0 * s ** 4 / (om + (1 - om) * s ** 6) ** 1.5
    I = (f * w).sum(-1) * 0.5 * np.sqrt(a[..., 0])
    return np.sqrt(om / a[..., 0] ** 3 + 1 - om) * I


def _match(order, mass, point, weighting):
    """(z per cell, F per rank) of the ranked cells."""
    a, b, c = _weibull(point)
    zt = np.linspace(min(5.0, a), 20.0, 2000)
    x = np.exp(-np.maximum((zt - a) / b, 0.0) ** c)
    M = torch.cumsum(mass[order].double(), 0)
    N, T = M.numel(), M[-1].item()
    F = M / T
    xt = torch.from_numpy(x).cuda()
    if weighting == "mass":
        j = torch.searchsorted(-xt, -F, right=True) - 1
        del M
        k = j.clamp(0, 1998)
        t = (xt[k] - F) / (xt[k] - xt[k + 1])
    else:
        g = _growth(zt) / _growth(point[0]) if weighting == "growth" else np.zeros_like(zt)
        al, be = 1.0 - g, g
        W = al * N + be * T
        rank = torch.arange(1, N + 1, device="cuda", dtype=torch.float64)
        j = torch.full((N,), -1, device="cuda", dtype=torch.int64)
        t = torch.zeros(N, device="cuda", dtype=torch.float64)
        above = None
        for q in range(1999, -1, -1):  # the highest root: a cell's first ionization
            h = x[q] * W[q] - al[q] * rank - be[q] * M
            new = (j < 0) & (h >= 0)
            j = torch.where(new, q, j)
            if above is not None:
                t = torch.where(new, h / (h - above), t)
            above = h
        k = j
    z = zt[0] + (k + t) * ((zt[-1] - zt[0]) / 1999.0)
    z = torch.where(j < 0, zt[0], torch.where(j >= 1999, zt[-1], z))
    del k, t, j
    cell = torch.empty_like(z)
    cell[order] = z
    return cell, F


def _field(S, box, l):
    """Radiation intensity: the periodic convolution with exp(-r/l)/(4 pi r^2)."""
    n = S.shape[0]
    H = torch.fft.rfftn(S.double())
    kf = 2.0 * math.pi / box
    kx, ky = _wave(n, "cuda", torch.float64)
    for z in range(0, n, 64):
        k = kf * torch.sqrt(ky[z:z + 64, None, None] ** 2 + ky[None, :, None] ** 2 + kx[None, None, :] ** 2)
        K = torch.atan(k * l) / k
        if z == 0:
            K[0, 0, 0] = l
        H[z:z + 64] *= K
    return torch.fft.irfftn(H, s=(n, n, n))


def _solve64(S, mass, box, l, point, weighting):
    J = _field(S, box, l)
    order = torch.sort(J.reshape(-1), descending=True, stable=True).indices
    return _match(order, mass.reshape(-1), point, weighting)[0].reshape(S.shape), J


def _lpt64(delta, box):
    n = delta.shape[0]
    H = torch.fft.rfftn(delta.double())
    kx, ky = _wave(n, "cuda", torch.float64)
    k = [kx[None, None, :], ky[None, :, None], ky[:, None, None]]
    odd = [torch.where(v == n // 2, 0.0, v) if i == 0 else torch.where(v == -(n // 2), 0.0, v)
           for i, v in enumerate(k)]  # odd derivatives vanish at the Nyquist wave number
    k2 = k[0] ** 2 + k[1] ** 2 + k[2] ** 2
    k2[0, 0, 0] = math.inf

    def back(X):
        return torch.fft.irfftn(X, s=delta.shape)

    def hess(a, b):
        return back(H * (k[a] * k[a] if a == b else odd[a] * odd[b]) / k2)

    d = [hess(0, 0), hess(1, 1), hess(2, 2)]
    s2 = d[0] * d[1] + d[0] * d[2] + d[1] * d[2]
    del d
    for a, b in ((0, 1), (0, 2), (1, 2)):
        s2 -= hess(a, b) ** 2
    H = -D1 * H + D2 * torch.fft.rfftn(s2)
    del s2
    kf = 2.0 * math.pi / box
    return tuple(back(H * (-1j * odd[a]) / (k2 * kf)) for a in range(3))


def _mesh64(psi, box, order, interlace, mass=None):
    n = psi[0].shape[0]
    lat = torch.arange(n, device="cuda", dtype=torch.float64)
    q = [lat[None, None, :], lat[None, :, None], lat[:, None, None]]

    def deposit(shift):
        rho = torch.zeros(n ** 3, device="cuda", dtype=torch.float64)
        base, wt = [], []
        for a in range(3):
            pos = q[a] + psi[a].double() * (n / box) + shift
            b = torch.floor(pos + 0.5)
            d = pos - b
            base.append(b.to(torch.int64))
            wt.append([(-d).clamp(min=0), 1 - d.abs(), d.clamp(min=0)] if order == 2 else
                      [0.5 * (0.5 - d) ** 2, 0.75 - d * d, 0.5 * (0.5 + d) ** 2])
            del pos, d, b
        m = 1.0 if mass is None else mass.double()
        for oz in range(3):
            for oy in range(3):
                wzy = wt[2][oz] * wt[1][oy] * m
                row = ((base[2] + oz - 1) % n * n + (base[1] + oy - 1) % n) * n
                for ox in range(3):
                    rho.index_add_(0, (row + (base[0] + ox - 1) % n).reshape(-1), (wzy * wt[0][ox]).reshape(-1))
        return rho.reshape(n, n, n)

    total = float(n) ** 3 if mass is None else mass.double().sum().item()
    if not interlace:
        return deposit(0.0) * (n ** 3 / total)
    A, Bk = torch.fft.rfftn(deposit(0.0)), torch.fft.rfftn(deposit(0.5))
    kx, ky = _wave(n, "cuda", torch.float64)
    k = [kx[None, None, :], ky[None, :, None], ky[:, None, None]]
    A = 0.5 * (A + Bk * torch.exp(1j * (math.pi / n) * (k[0] + k[1] + k[2])))
    for v in k:
        A /= torch.sinc(v / n) ** order
    A[:, :, n // 2] = 0
    A[:, n // 2] = 0
    A[n // 2] = 0
    return torch.fft.irfftn(A, s=(n, n, n)) * (n ** 3 / total)


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        out = []
        for n, l, point, weighting, s in _batch_items(case, seed):
            S, mass = _source_and_mass(n, s)
            out.append(_solve64(S, mass, _box(n), l, point, weighting)[0])
        return out
    if kind == "rank_match":
        J, mass = _intensity(case["cells"], seed)
        order = torch.sort(J, descending=True, stable=True).indices
        z, F = _match(order, mass, HISTORY, case["weighting"])
        return {"order": order.to(torch.int32), "z": z, "F": F}
    n, box = case["n"], _box(case["n"])
    if kind == "density":
        if case["order"] == 1:
            return None  # nearest point: a rounding of the position moves a whole particle
        return _mesh64(_zeldovich(n, seed, box), box, case["order"], case["interlace"])
    if kind in ("lpt", "esf_l"):
        delta = _delta(n, seed, 1.0, torch.float32)
        psi = _lpt64(delta, box)
        if kind == "lpt":
            return {"psi": psi}
        H = torch.fft.rfftn(delta.double())
        kx, ky = _wave(n, "cuda", torch.float64)
        k2 = ky[:, None, None] ** 2 + ky[None, :, None] ** 2 + kx[None, None, :] ** 2
        H[k2 > (n / (4.0 * math.pi)) ** 2] = 0
        f = torch.special.erfc((1.686 / D1 - torch.fft.irfftn(H, s=(n, n, n))) / math.sqrt(2.0))
        return {"psi": psi, "f": f, "rho": _mesh64(psi, box, 2, True, f)}
    S, mass = _source_and_mass(n, seed, torch.float64 if kind == "solve_f64" else torch.float32)
    if kind == "history":
        order, _ = _ranked(S, mass, box, case["l_mfp"])
        return {"z": _match(order.long(), mass.reshape(-1), HISTORY, case["weighting"])[0].reshape(S.shape)}
    z, J = _solve64(S, mass, box, case["l_mfp"], HISTORY, case["weighting"])
    return {"z": z, "J": J} if case.get("want_J") else {"z": z}
