"""Performance cases of the solver: what its users run, through its public entry points.

A case is a dict of plain values:
  kind       "force" (Plan.solve into the caller's arrays), "potential" (Plan.solve_potential),
             "host" (Plan.solve_host on numpy arrays), "batch" (Batch.solve of many nests)
  n, levels  cells a side of every patch, refinement levels; "forest": a named forest instead
  precision  "fp32", "bf16x" or "fp64"
  zero_rim   the density vanishes on the two outermost rings (SGF_PLAN_ZERO_RIM)
  cx, cy     point the nest is centred on (level 0 spans [-1, 1]^2)
  shapes     batch only: "n x levels x count" triples
"""
import math

import numpy as np
import torch

from paper_1603_03142_gb300 import sgf


# ------------------------------------------------------------------ geometry
class Nest:
    """One patch per level, refinement ratio 2 (the descriptor Plan takes)."""

    def __init__(self, n, levels, cx=0.0, cy=0.0):
        self.n, self.levels = n, levels
        self.x0 = self.y0 = -1.0
        self.h0 = 2.0 / n
        self.off = [(0, 0)]
        x, y = self.x0, self.y0
        for l in range(1, levels):
            hp = self.h0 / (1 << (l - 1))
            half = 0.5 * n * self.h0 / (1 << l)
            ox = min(max(int(round((cx - half - x) / hp)), 0), n // 2)
            oy = min(max(int(round((cy - half - y) / hp)), 0), n // 2)
            self.off.append((ox, oy))
            x, y = x + ox * hp, y + oy * hp

    def patches(self):
        """[(level, corner x, corner y)], corners in cells of the patch's level."""
        out, px, py = [], 0, 0
        for l in range(self.levels):
            if l > 0:
                px, py = 2 * (px + self.off[l][0]), 2 * (py + self.off[l][1])
            out.append((l, px, py))
        return out


class Forest:
    """Several patches per level (the descriptor Plan takes for forests)."""

    def __init__(self, n, level, org, x0, y0, h0):
        self.n, self.level, self.org = n, level, org
        self.x0, self.y0, self.h0 = x0, y0, h0
        self.levels = len(level)

    def patches(self):
        return [(l, o[0], o[1]) for l, o in zip(self.level, self.org)]


def _forest(name, n):
    if name == "two_disks":  # one root, one refined patch over each of two disks
        return Forest(n, [0, 1, 1], [(0, 0), (0, n // 2), (n, n // 2)], -1.0, -1.0, 2.0 / n)
    if name == "tiles":  # six root tiles, one refined patch over each of two disks
        org = [(0, 0), (n, 0), (0, n), (n, n), (0, 2 * n), (n, 2 * n), (n // 2, 5 * n // 2), (5 * n // 2, 5 * n // 2)]
        return Forest(n, [0] * 6 + [1, 1], org, -1.0, -1.5, 1.0 / n)
    raise ValueError(name)


def _geometry(case):
    if case.get("forest"):
        return _forest(case["forest"], case["n"])
    return Nest(case["n"], case["levels"], case.get("cx", 0.0), case.get("cy", 0.0))


def _batch_nests(case):
    out = []
    for part in case["shapes"].split():
        n, levels, count = (int(v) for v in part.split("x"))
        out += [Nest(n, levels)] * count
    return out


def _cells(case):
    if case["kind"] == "batch":
        return sum(g.levels * g.n * g.n for g in _batch_nests(case))
    g = _geometry(case)
    return g.levels * g.n * g.n


# --------------------------------------------------------------------- cases
def _case(name, kind, n, levels, precision, **more):
    c = {"name": name, "kind": kind, "n": n, "levels": levels, "precision": precision, "zero_rim": False,
         "cx": 0.0, "cy": 0.0}
    c.update(more)
    return c


def listed():
    return [
        # the smallest call: a verification run of one small disk in double precision
        _case("disk64_fp64", "force", 64, 1, "fp64"),
        # a simulation step on a small nest that follows an off-centre clump
        _case("nest256x3_fp32", "force", 256, 3, "fp32", cx=0.3),
        # a disk resolved on a large root grid with two refinements at its centre
        _case("nest1024x3_fp32", "force", 1024, 3, "fp32"),
        # a deep nest, as a request of the serving mix in its other precision
        _case("nest512x4_bf16x", "force", 512, 4, "bf16x"),
        # a large grid with one refinement over an off-centre planet
        _case("nest2048x2_fp32", "force", 2048, 2, "fp32", cx=0.3, cy=-0.2),
        # a grid size that is no power of two, refined once
        _case("ragged600x2_fp32", "force", 600, 2, "fp32"),
        # one uniform grid whose mass reaches the edges
        _case("uniform1024_fp32", "force", 1024, 1, "fp32"),
        # the largest grid: one level, nothing on the rim
        _case("uniform4096_zero_rim_fp32", "force", 4096, 1, "fp32", zero_rim=True),
        # the mid-plane potential for an energy budget, on a grid with a refinement
        _case("potential1024x2_fp32", "potential", 1024, 2, "fp32"),
        # two binary disks: several patches per level
        _case("forest_tiles256_fp32", "force", 256, 8, "fp32", forest="tiles"),
        # a parameter study: independent nests of uneven size and depth in one call
        _case("batch20_fp32", "batch", 0, 0, "fp32",
              shapes="128x1x2 128x2x3 128x3x2 256x1x2 256x2x3 256x3x2 512x1x1 512x2x2 512x3x2 1024x2x1"),
        # host arrays in and out, as a CPU code calls it once per step
        _case("host1024x2_fp32", "host", 1024, 2, "fp32"),
    ]


def _even_log(rng, lo, hi):
    """An even number of [lo, hi], uniform in its logarithm."""
    return min(hi, max(lo, 2 * int(round(0.5 * math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _centre(rng):
    r, t = 0.4 * math.sqrt(rng.random()), 2.0 * math.pi * rng.random()
    return {"cx": round(r * math.cos(t), 3), "cy": round(r * math.sin(t), 3)}


def draw(rng):
    kind = rng.choice(["nest", "nest", "nest", "uniform", "uniform", "potential", "forest", "batch", "host"])
    if kind == "nest":
        precision = rng.choice(["fp32", "fp32", "fp32", "bf16x", "fp64"])
        levels = rng.choice([2, 2, 3, 3, 4])
        hi = {2: 2048, 3: 1024, 4: 512}[levels] if precision != "fp64" else {2: 512, 3: 256, 4: 128}[levels]
        n = 2 ** rng.randint(5, int(math.log2(hi))) if rng.random() < 0.6 else _even_log(rng, 32, hi)
        return _case(None, "force", n, levels, precision, **(_centre(rng) if rng.random() < 0.5 else {}))
    if kind == "uniform":
        precision = rng.choice(["fp32", "fp32", "fp32", "bf16x", "fp64"])
        hi = 1024 if precision == "fp64" else 2048 if precision == "bf16x" else 4096
        n = 2 ** rng.randint(6, int(math.log2(hi))) if rng.random() < 0.6 else _even_log(rng, 64, hi)
        return _case(None, "force", n, 1, precision, zero_rim=n >= 96 and rng.random() < 0.5)
    if kind == "potential":
        levels = rng.choice([1, 2])
        n = 2 ** rng.randint(6, 11 if levels == 1 else 10)
        return _case(None, "potential", n, levels, "fp32", zero_rim=levels == 1 and n >= 128 and rng.random() < 0.5)
    if kind == "forest":
        name = rng.choice(["two_disks", "tiles"])
        n = 2 ** rng.randint(5, 8) if rng.random() < 0.6 else _even_log(rng, 32, 256) // 4 * 4
        return _case(None, "force", n, 3 if name == "two_disks" else 8, "fp32", forest=name)
    if kind == "batch":
        shapes = {}
        for _ in range(rng.randint(3, 10)):
            n, levels = rng.choice([64, 128, 256, 512]), rng.randint(1, 3)
            shapes[(n, levels)] = shapes.get((n, levels), 0) + rng.randint(1, 2)
        return _case(None, "batch", 0, 0, "fp32", shapes=" ".join("%dx%dx%d" % (n, l, c) for (n, l), c in shapes.items()))
    return _case(None, "host", _even_log(rng, 64, 1400), rng.choice([1, 2]), "fp32")


# -------------------------------------------------------------------- inputs
def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _density(geom, seed, zero_rim, dtype):
    """Per patch: a disk with a smooth edge, up to three clumps, lognormal noise per cell."""
    dev = _device()
    g = torch.Generator(device=dev).manual_seed(seed)
    r = np.random.Generator(np.random.PCG64(seed))
    radius = r.uniform(0.6, 0.95) if zero_rim else r.uniform(0.7, 1.3)  # the larger disks are cut by the edges
    clumps = [(r.uniform(-0.5, 0.5), r.uniform(-0.5, 0.5), r.uniform(1.0, 5.0), r.uniform(0.02, 0.1))
              for _ in range(int(r.integers(0, 4)))]
    out = []
    for level, px, py in geom.patches():
        h = geom.h0 / (1 << level)
        c = torch.arange(geom.n, device=dev, dtype=torch.float64) + 0.5
        x, y = (geom.x0 + (px + c) * h)[None, :], (geom.y0 + (py + c) * h)[:, None]
        s = torch.clamp(1.0 - (x * x + y * y) / radius ** 2, min=0.0).sqrt_()
        for qx, qy, peak, w in clumps:
            s = s + peak * torch.exp(-((x - qx) ** 2 + (y - qy) ** 2) / (2.0 * w * w))
        s = s * torch.exp(0.3 * torch.randn(geom.n, geom.n, device=dev, generator=g, dtype=torch.float32)).double()
        if zero_rim:
            s[:2], s[-2:], s[:, :2], s[:, -2:] = 0.0, 0.0, 0.0, 0.0
        out.append(s.to(dtype).contiguous())
    return out


def _dtype(case):
    return torch.float64 if case["precision"] == "fp64" else torch.float32


def _inputs(case, seed):
    if case["kind"] == "batch":
        return [_density(g, seed * 1000 + k, False, _dtype(case)) for k, g in enumerate(_batch_nests(case))]
    return _density(_geometry(case), seed, case["zero_rim"], _dtype(case))


def prepare(case, seed):
    """The plan (tuned once, as a program that solves many steps does), the densities, the output arrays."""
    sigma = _inputs(case, seed)
    st = {"kind": case["kind"], "sigma": sigma}
    if case["kind"] == "batch":
        base, plans = {}, []
        for g in _batch_nests(case):
            key = (g.n, g.levels)
            if key not in base:  # plans of one shape share its spectra
                base[key] = sgf.Plan(g, case["precision"])
                base[key].autotune(reps=2)
                plans.append(base[key])
            else:
                plans.append(base[key].share())
        st["plan"] = sgf.Batch(plans)
        for out in ("fx", "fy"):  # one array of all levels per nest
            st[out] = [torch.empty((len(lst),) + tuple(lst[0].shape), dtype=lst[0].dtype, device=lst[0].device)
                       for lst in sigma]
            st[out + "_levels"] = [list(t) for t in st[out]]
        return st
    plan = sgf.Plan(_geometry(case), case["precision"], zero_rim=case["zero_rim"], potential=case["kind"] == "potential")
    plan.autotune(reps=5)
    st["plan"] = plan
    if case["kind"] == "host":
        st["sigma"] = [s.cpu().numpy() for s in sigma]
        st["fx"] = [np.empty_like(s) for s in st["sigma"]]
        st["fy"] = [np.empty_like(s) for s in st["sigma"]]
    else:
        st["fx"] = [torch.empty_like(s) for s in sigma]
        if case["kind"] == "force":
            st["fy"] = [torch.empty_like(s) for s in sigma]
    return st


def run(state):
    if state["kind"] == "potential":
        return {"phi": state["plan"].solve_potential(state["sigma"], state["fx"])}
    if state["kind"] == "batch":
        state["plan"].solve(state["sigma"], state["fx_levels"], state["fy_levels"])
        return {"fx": state["fx"], "fy": state["fy"]}
    if state["kind"] == "host":
        fx, fy = state["plan"].solve_host(state["sigma"], state["fx"], state["fy"])
    else:
        fx, fy = state["plan"].solve(state["sigma"], state["fx"], state["fy"])
    return {"fx": fx, "fy": fy}


def work(case):
    """Densities read once and results written once; the real transforms of every patch's zero-padded
    2n x 2n grid, one in and one out per result component."""
    size = 8 if case["precision"] == "fp64" else 4
    comps = 1 if case["kind"] == "potential" else 2
    geoms = _batch_nests(case) if case["kind"] == "batch" else [_geometry(case)]
    flops = 0.0
    for g in geoms:
        p2 = 4.0 * g.n * g.n
        flops += g.levels * (1 + comps) * 2.5 * p2 * math.log2(p2)
    return {"bytes": (1 + comps) * size * _cells(case), "flops": flops}


# ------------------------------------------------ the results in 64 bits
def _corner(u, v, pot):
    """Antiderivatives at cell corners (u: columns, v: rows): force integrals of u/r^3, v/r^3, u^2/r^3,
    uv/r^3, v^2/r^3, or potential integrals of 1/r, u/r, v/r; terms of one variable alone cancel."""
    au, av = u.abs(), v.abs()
    zu, zv = au == 0.0, av == 0.0
    a = torch.asinh(v / torch.where(zu, 1.0, au)).masked_fill_(zu.expand(v.shape[0], u.shape[1]), 0.0)
    b = torch.asinh(u / torch.where(zv, 1.0, av)).masked_fill_(zv.expand(v.shape[0], u.shape[1]), 0.0)
    r = torch.hypot(u.expand(a.shape), v.expand(a.shape))
    if pot:
        lu, lv = u * a, v * b
        return [lu + lv, 0.5 * (v * r + u * lu), 0.5 * (u * r + v * lv)]
    lu = torch.where(zu, torch.where(zv, 0.0, torch.sign(v) * torch.log(torch.where(zv, 1.0, av))), 0.0)
    lv = torch.where(zv, torch.where(zu, 0.0, torch.sign(u) * torch.log(torch.where(zu, 1.0, au))), 0.0)
    return [-a - lu, -b - lv, v * b, -r, u * a]


def _tables(lox, loy, w, scale, pot, h):
    """Kernel tables of source cells with lower edges lox (columns), loy (rows) and width w, target at 0."""
    x0, y0 = lox[None, :], loy[:, None]
    c = [_corner(x0 + w, y0 + w, pot), _corner(x0, y0 + w, pot), _corner(x0 + w, y0, pot), _corner(x0, y0, pot)]
    i = [(c[0][k] - c[1][k]) - (c[2][k] - c[3][k]) for k in range(len(c[0]))]
    uc, vc = x0 + 0.5 * w, y0 + 0.5 * w
    if pot:
        return [[-h * i[0], -h * scale * (i[1] - uc * i[0]), -h * scale * (i[2] - vc * i[0])]]
    return [[i[0], scale * (i[2] - uc * i[0]), scale * (i[3] - vc * i[0])],
            [i[1], scale * (i[3] - uc * i[1]), scale * (i[4] - vc * i[1])]]


def _fast_len(k):
    best = 1 << (k - 1).bit_length()
    for odd in (3, 5, 9, 15):
        p = odd
        while p < k:
            p *= 2
        best = min(best, p)
    return best


def _fields(geom, sigma):
    """Per patch: density, x and y differences per cell, zero under the finer patches."""
    n, half = geom.n, geom.n // 2
    pat = geom.patches()
    full = [s.double().clone() for s in sigma]
    cover = [torch.zeros(n, n, dtype=torch.bool, device=sigma[0].device) for _ in pat]
    for s in sorted(range(len(pat)), key=lambda k: -pat[k][0]):
        for q in range(len(pat)):
            if pat[q][0] != pat[s][0] + 1:
                continue
            fx, fy = pat[q][1] // 2 - pat[s][1], pat[q][2] // 2 - pat[s][2]
            x0, x1, y0, y1 = max(fx, 0), min(fx + half, n), max(fy, 0), min(fy + half, n)
            if x0 >= x1 or y0 >= y1:
                continue
            mean = full[q].reshape(half, 2, half, 2).mean(dim=(1, 3))
            full[s][y0:y1, x0:x1] = mean[y0 - fy:y1 - fy, x0 - fx:x1 - fx]
            cover[s][y0:y1, x0:x1] = True
    out = []
    for f, c in zip(full, cover):
        dx, dy = torch.empty_like(f), torch.empty_like(f)
        dx[:, 1:-1], dx[:, 0], dx[:, -1] = 0.5 * (f[:, 2:] - f[:, :-2]), f[:, 1] - f[:, 0], f[:, -1] - f[:, -2]
        dy[1:-1], dy[0], dy[-1] = 0.5 * (f[2:] - f[:-2]), f[1] - f[0], f[-1] - f[-2]
        out.append([t.masked_fill(c, 0.0) for t in (f, dx, dy)])
    return out, cover


def _solve64(geom, sigma, pot):
    fields, cover = _fields(geom, sigma)
    n, pat = geom.n, geom.patches()
    dev = sigma[0].device
    comps = 1 if pot else 2
    out = [[torch.zeros(n, n, dtype=torch.float64, device=dev) for _ in range(comps)] for _ in pat]
    spectra = {}  # pairs of one relative position have the same tables

    def convolve(key, edges, w, scale, h, src, nt):
        ns = src[0].shape[0]
        p = _fast_len(ns + nt - 1)
        if key not in spectra:
            d = torch.arange(p, device=dev, dtype=torch.float64)
            d = torch.where(d <= nt - 1, d, d - p)
            tabs = _tables(edges(d, 0), edges(d, 1), w, scale, pot, h)
            spectra[key] = [[torch.fft.rfft2(t) for t in row] for row in tabs]
            if p > 4096 or len(spectra) > 64:  # keep little of what is used again
                k = spectra.pop(key)
            else:
                k = spectra[key]
        else:
            k = spectra[key]
        hat = [torch.fft.rfft2(f, s=(p, p)) for f in src]
        res = []
        for row in k:
            acc = row[0] * hat[0]
            acc += row[1] * hat[1]
            acc += row[2] * hat[2]
            res.append(torch.fft.irfft2(acc, s=(p, p))[:nt, :nt])
        return res

    for s, (ls, sx, sy) in enumerate(pat):
        for t, (lt, tx, ty) in enumerate(pat):
            m = 1 << abs(ls - lt)
            h = geom.h0 / (1 << max(ls, lt))
            if ls == lt:
                off = (sx - tx, sy - ty)
                res = convolve((1, off, h), lambda d, a: -d - 0.5 + off[a], 1.0, 1.0, h, fields[s], n)
                for c in range(comps):
                    out[t][c] += res[c]
                continue
            off = (sx - m * tx, sy - m * ty) if ls > lt else (tx - m * sx, ty - m * sy)
            for py in range(m):
                for px in range(m):
                    ph = (px, py)
                    if ls > lt:  # a finer source: its cells split into m x m phases
                        res = convolve((2, m, ph, off, h), lambda d, a: -m * d + ph[a] - 0.5 * m + off[a], 1.0, 1.0, h,
                                       [f[py::m, px::m] for f in fields[s]], n)
                        for c in range(comps):
                            out[t][c] += res[c]
                    else:  # a coarser source: the target's cells split into phases
                        res = convolve((3, m, ph, off, h), lambda d, a: -m * d - ph[a] - off[a] - 0.5, float(m), 1.0 / m,
                                       h, fields[s], -(-n // m))
                        for c in range(comps):
                            view = out[t][c][py::m, px::m]
                            view += res[c][:view.shape[0], :view.shape[1]]
    return [[o.masked_fill(c, 0.0) for o in lst] for lst, c in zip(out, cover)]


def exact(case, seed):
    """The same sums in 64 bits: closed-form kernel tables, every pair of patches by torch.fft."""
    sigma = _inputs(case, seed)
    pot = case["kind"] == "potential"
    if case["kind"] == "batch":
        res = [_solve64(g, s, False) for g, s in zip(_batch_nests(case), sigma)]
        return {"fx": [torch.stack([o[0] for o in lst]) for lst in res],
                "fy": [torch.stack([o[1] for o in lst]) for lst in res]}
    res = _solve64(_geometry(case), sigma, pot)
    if pot:
        return {"phi": [o[0] for o in res]}
    if case["kind"] == "host":
        return {"fx": [o[0].cpu().numpy() for o in res], "fy": [o[1].cpu().numpy() for o in res]}
    return {"fx": [o[0] for o in res], "fy": [o[1] for o in res]}
