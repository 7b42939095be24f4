"""What this tracer's users have it do, as cases that can be timed and checked.

Every case goes through the package's public entry points: columns of a cube
or of an adaptive octree, in either arithmetic form, from every leaf centre or
from scattered points; the same with a gradient (autograd, walked or replayed
from a record); the fused per-source epilogues; a batch of clouds; a source
grid turned into an octree and traced; and the call on host buffers.  Clouds
are lognormal turbulent fields (power spectrum k^-4) drawn from the seed, as in
the benchmark and the tests.

exact() is an independent FP64 evaluation in plain torch: a vectorised walk
over the sorted keys, or on a cube with a source in every leaf the shifted sum
that the translation invariance of the paths allows.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2605_09882_gb300 as rt

D = 21                                        # depth of the Morton lattice
FRACTIONS = (1.0, 0.4, 1.0e-4, 2.0e-4, 0.1, 3.0e-3, 1.0e-5, 0.05)  # species per total density
PDR_WEIGHTS = (1.0, 2.0)                      # N_H = n(H) + 2 n(H2)
AV, GAMMA = 1.6, 3.02                         # extinction per unit column, A_V,eff exponent


def listed():
    f32 = dict(mode="f32k", dens="f32")
    f64 = dict(mode="fp64", dens="f64")
    return [
        # the benchmark: a 512^3 cloud, four species, all twelve base rays of every cell
        dict(name="cube512", path="columns", grid="cube", base=512, sources="centres", n_src=0, nside=1, species=4, **f32),
        # the smallest whole cloud in the reference form: launch and latency count
        dict(name="cube32_fp64", path="columns", grid="cube", base=32, sources="centres", n_src=0, nside=1, species=1, **f64),
        # an adaptive cloud traced from a million mass-weighted points (Lagrangian tracers, off the cell centres)
        dict(name="amr128", path="columns", grid="amr", base=128, refine=2, pct=90.0, sources="mass", n_src=1000000, nside=2, species=4, **f32),
        # the bitwise FP64 form on an adaptive cloud, single-precision densities as simulations store them
        dict(name="amr64_fp64", path="columns", grid="amr", base=64, refine=1, pct=85.0, sources="centres", n_src=0, nside=1, species=2, mode="fp64", dens="f32"),
        # a sky map: one observer, many directions, a box that is no power of two, an odd species count
        dict(name="skymap", path="columns", grid="amr", base=96, refine=2, pct=85.0, sources="mass", n_src=1, nside=32, species=3, **f32),
        # a training step on an adaptive cloud: columns and the gradient of the densities
        dict(name="step_amr64", path="step", grid="amr", base=64, refine=1, pct=85.0, sources="centres", n_src=0, nside=2, species=1, **f32),
        # the same on a cube with four species
        dict(name="step_cube256", path="step", grid="cube", base=256, sources="centres", n_src=0, nside=1, species=4, **f32),
        # an optimisation loop over one geometry: forward and backward replayed from the recorded paths
        dict(name="replay_amr48", path="replay", grid="amr", base=48, refine=2, pct=85.0, sources="mass", n_src=100003, nside=2, species=2, **f32),
        # chemistry coupling: the effective visual extinction of every cell, no columns written
        dict(name="aveff_amr64", path="av_eff", grid="amr", base=64, refine=2, pct=85.0, sources="centres", n_src=0, nside=2, species=2, **f32),
        # many small clouds of uneven size and depth in one launch (a parameter study)
        dict(name="batch24", path="batch", grid="amr", base=48, refine=2, pct=80.0, sources="centres", n_src=0, nside=2, species=2, clouds=24, **f32),
        # a simulation snapshot: build the contribution grid, index it, trace it
        dict(name="grid256", path="build", grid="build", base=256, sources="mass", n_src=300000, nside=1, species=2, **f32),
        # a host program's whole call: octree, densities and sources up, columns down
        dict(name="host_cube128", path="host", grid="cube", base=128, sources="centres", n_src=0, nside=1, species=4, **f32),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    path = rng.choice(["columns", "columns", "columns", "skymap", "step", "step", "replay", "av_eff", "beta", "batch", "build", "host"])
    c = dict(path="columns" if path == "skymap" else path)
    fp64 = path not in ("batch", "build", "host") and rng.random() < 0.3
    c["mode"] = "fp64" if fp64 else "f32k"
    c["dens"] = "f64" if fp64 and rng.random() < 0.5 else "f32"
    c["species"] = rng.choice([1, 2, 2, 3, 4, 4, 4, 5, 8])
    c["nside"] = rng.choice([1, 1, 2, 2, 4])
    if path == "build":
        c.update(grid="build", base=rng.choice([64, 128, 256]), sources="mass", n_src=_log_int(rng, 3000, 500000))
        c["nside"] = min(c["nside"], 2)
    elif rng.random() < (0.0 if path in ("batch", "skymap") else 0.4):
        c.update(grid="cube", base=rng.choice([16, 32, 64, 128] + ([] if fp64 else [256])))
    else:
        c.update(grid="amr", base=_log_int(rng, 16, 96), refine=rng.randint(0, 3), pct=round(rng.uniform(80.0, 93.0), 1))
    if path == "batch":
        c["clouds"] = _log_int(rng, 3, 48)
    if path == "skymap":
        c.update(sources="mass", n_src=rng.randint(1, 20), nside=rng.choice([8, 16, 32, 64]))
    elif c["grid"] != "build":
        c["sources"] = rng.choice(["centres", "mass"])
        c["n_src"] = _log_int(rng, 40, 400000) if c["sources"] == "mass" else 0
    # well below the largest listed case: the FP64 form runs at about a tenth of
    # the FP32 rate, a gradient takes an FP64 atomic per segment and species, a
    # record takes eight bytes a segment, and host buffers are pinned
    most = 2.0e9 if fp64 else {"step": 4.0e9, "replay": 2.0e9, "host": 1.0e9}.get(path, 1.0e10)
    while _segments(c) > most:
        if c["nside"] > 1 and path != "skymap":
            c["nside"] //= 2
        elif c["n_src"] > 1000:
            c["n_src"] //= 2
        elif c.get("refine"):
            c["refine"] -= 1
        else:
            c["base"] //= 2
    return c


# ------------------------------------------------------------------ sizes

def _leaves(c):
    if c["grid"] == "cube":
        return float(c["base"]) ** 3
    if c["grid"] == "build":
        return 0.5 * float(c["base"]) ** 3
    f, n, total = 1.0 - c["pct"] / 100.0, float(c["base"]) ** 3, 0.0
    for _ in range(c["refine"]):
        total += (1.0 - f) * n
        n *= 8.0 * f
    return total + n


def _sources(c):
    return float(c["n_src"] or _leaves(c))


def _rays(c):
    n = _sources(c) * 12 * c["nside"] ** 2
    return n * (0.12 * c["clouds"] if c["path"] == "batch" else 1.0)  # clouds are smaller, shallower and half of them at Nside 1


def _segments(c):
    """About how many (ray, leaf) pairs a pass visits: half the cloud's leaves per axis, as measured."""
    return _rays(c) * (0.512 if c["grid"] == "cube" else 0.62) * _leaves(c) ** (1.0 / 3.0)


def work(case):
    c = case
    S, rays, leaves, segs = c["species"], _rays(c), _leaves(c), _segments(c)
    o = 8 if c["mode"] == "fp64" else 4
    d = 8 if c["dens"] == "f64" else 4
    n = 0.2 * c["clouds"] if c["path"] == "batch" else 1.0
    octree = n * leaves * (9 + d * S)
    src = 24 * n * _sources(c)
    if c["path"] in ("av_eff", "beta"):
        return {"bytes": octree + src + 8 * _sources(c), "flops": segs * 2 * S}
    if c["path"] in ("step", "replay"):  # columns out, their gradient in, the densities' gradient out
        return {"bytes": octree + src + 2 * rays * S * o + leaves * S * d, "flops": segs * 4 * S}
    if c["path"] == "build":
        cells = float(c["base"]) ** 3
        return {"bytes": cells * 4 * (1 + S) + 2 * octree + src + rays * S * o, "flops": segs * 2 * S}
    return {"bytes": octree + src + rays * S * o, "flops": segs * 2 * S}


# ----------------------------------------------------------------- inputs

def _spread(v):
    v = v & 0x1FFFFF
    v = (v | (v << 32)) & 0x1F00000000FFFF
    v = (v | (v << 16)) & 0x1F0000FF0000FF
    v = (v | (v << 8)) & 0x100F00F00F00F00F
    v = (v | (v << 4)) & 0x10C30C30C30C30C3
    return (v | (v << 2)) & 0x1249249249249249


def _compact(v):
    v = v & 0x1249249249249249
    v = (v | (v >> 2)) & 0x10C30C30C30C30C3
    v = (v | (v >> 4)) & 0x100F00F00F00F00F
    v = (v | (v >> 8)) & 0x1F0000FF0000FF
    v = (v | (v >> 16)) & 0x1F00000000FFFF
    return (v | (v >> 32)) & 0x1FFFFF


def _corner(keys):
    return torch.stack([_compact(keys), _compact(keys >> 1), _compact(keys >> 2)], dim=1)


def _field(n, gen):
    """Lognormal field exp(g) on an n^3 grid [z][y][x], g of power spectrum k^-4 and deviation 1.5."""
    dev = torch.device("cuda")
    w = torch.fft.rfftn(torch.randn((n, n, n), generator=gen, device=dev))
    k = torch.fft.fftfreq(n, device=dev) * n
    kx = torch.fft.rfftfreq(n, device=dev) * n
    k2 = k[:, None, None] ** 2 + k[None, :, None] ** 2 + kx[None, None, :] ** 2
    k2[0, 0, 0] = 1.0
    w /= k2
    w[0, 0, 0] = 0
    del k2
    g = torch.fft.irfftn(w, s=(n, n, n))
    g *= 1.5 / g.std()
    return g.exp_()


def _morton_grid(level):
    """Morton index of every cell of a 2^level cube, laid out [z][y][x]."""
    s = _spread(torch.arange(1 << level, device="cuda"))
    return (s[None, None, :] | (s[None, :, None] << 1) | (s[:, None, None] << 2)).reshape(-1)


def _cube(n, gen):
    """Keys, levels and total density of n^3 equal leaves."""
    level = n.bit_length() - 1
    field = _field(n, gen)
    total = torch.empty(n ** 3, device="cuda")
    total[_morton_grid(level)] = field.reshape(-1)
    keys = torch.arange(n ** 3, device="cuda") << (3 * (D - level))
    return keys, torch.full((n ** 3,), level, device="cuda", dtype=torch.uint8), total, None


def _amr(base, refine, pct, gen):
    """base^3 leaves, those above the pct-th percentile of their level split into eight, refine times over."""
    root = (base - 1).bit_length()
    deep = refine
    while (base << deep) > 256 and deep > 0:  # the field's grid; leaves below it take their parent's value
        deep -= 1
    field = _field(base << deep, gen)
    g = torch.arange(base, device="cuda")
    cur = torch.stack(torch.meshgrid(g, g, g, indexing="ij")[::-1], dim=-1).reshape(-1, 3)
    off = torch.tensor([[x, y, z] for z in (0, 1) for y in (0, 1) for x in (0, 1)], device="cuda")
    keys, levels, total = [], [], []
    for r in range(refine + 1):
        up = max(0, r - deep)
        f = 1 << max(0, deep - r)
        mean = torch.nn.functional.avg_pool3d(field[None, None], f)[0, 0] if f > 1 else field
        p = cur >> up
        d = mean[p[:, 2], p[:, 1], p[:, 0]]
        split = torch.zeros_like(d, dtype=torch.bool)
        if r < refine:
            split[torch.sort(d, stable=True).indices[int(pct / 100.0 * d.numel()):]] = True
        c = cur[~split] << (D - root - r)
        keys.append(_spread(c[:, 0]) | (_spread(c[:, 1]) << 1) | (_spread(c[:, 2]) << 2))
        levels.append(torch.full((c.shape[0],), root + r, device="cuda", dtype=torch.uint8))
        total.append(d[~split])
        cur = (2 * cur[split][:, None, :] + off[None]).reshape(-1, 3)
    keys, order = torch.sort(torch.cat(keys))
    ext = None if base == 1 << root else (base << (D - root),) * 3
    return keys, torch.cat(levels)[order], torch.cat(total)[order], ext


def _species(total, count, dtype, gen):
    dens = torch.empty((total.numel(), count), device="cuda", dtype=dtype)
    for k in range(count):
        u = torch.rand(total.numel(), generator=gen, device="cuda") * 0.4 + 0.8
        dens[:, k] = (FRACTIONS[k] * total * u).to(dtype)
    return dens


def _centres(keys, levels):
    half = torch.ldexp(torch.ones(levels.numel(), device="cuda", dtype=torch.float64), D - 1 - levels.to(torch.int64))
    return ((_corner(keys).to(torch.float64) + half[:, None]) * 2.0 ** -D).contiguous()


def _mass_weighted(keys, levels, total, n, gen):
    """n points, leaf by mass and uniform within the leaf, in the order of the leaves."""
    w = torch.ldexp(total.to(torch.float64), 3 * (12 - levels.to(torch.int64)))
    w = (w * (2.0 ** 60 / (float(w.max()) * w.numel()))).to(torch.int64)  # whole numbers: the same sums every time
    cdf = torch.cumsum(w, 0)
    u = (torch.rand(n, generator=gen, device="cuda", dtype=torch.float64) * float(cdf[-1])).to(torch.int64)
    j = torch.sort(torch.searchsorted(cdf, u, right=True).clamp_(max=keys.numel() - 1)).values
    span = (1 << (D - levels[j].to(torch.int64))) << 32
    at = (torch.rand((n, 3), generator=gen, device="cuda", dtype=torch.float64) * span[:, None].to(torch.float64)).to(torch.int64)
    q = (_corner(keys[j]) << 32) + torch.minimum(at, span[:, None] - 1)
    return q.to(torch.float64) * 2.0 ** -53


def _cloud(c, base, refine, n_src, gen):
    dtype = torch.float64 if c["dens"] == "f64" else torch.float32
    if c["grid"] == "cube":
        keys, levels, total, ext = _cube(base, gen)
    else:
        keys, levels, total, ext = _amr(base, refine, c["pct"], gen)
    src = _centres(keys, levels) if c["sources"] == "centres" else _mass_weighted(keys, levels, total, n_src, gen)
    return dict(keys=keys, levels=levels, ext=ext, dens=_species(total, c["species"], dtype, gen), src=src, nside=c["nside"])


def _inputs(c, seed):
    """The arrays of a case, before any handle is made."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    if c["path"] == "batch":
        pick = np.random.default_rng(3)
        out = []
        for i in range(c["clouds"]):  # sizes from a quarter of the largest up, of any depth to the deepest, the same for every seed
            base = c["base"] if i == 0 else max(8, int(c["base"] * pick.uniform(0.25, 1.0)))
            one = _cloud(c, base, int(pick.integers(0, c["refine"] + 1)), c["n_src"], gen)
            out.append(dict(one, nside=c["nside"] if i % 2 == 0 else 1))
        return dict(clouds=out)
    if c["grid"] == "build":
        level = c["base"].bit_length() - 1
        # one field in a random orientation, so that every seed has as many leaves
        field = _field(c["base"], torch.Generator(device="cuda").manual_seed(11))
        pick = np.random.default_rng(seed)
        field = field.permute(*pick.permutation(3).tolist()).flip(np.flatnonzero(pick.integers(0, 2, 3)).tolist())
        nref = torch.empty(c["base"] ** 3, device="cuda")
        nref[_morton_grid(level)] = field.reshape(-1)
        keys = torch.arange(nref.numel(), device="cuda") << (3 * (D - level))
        levels = torch.full((nref.numel(),), level, device="cuda", dtype=torch.uint8)
        src = _mass_weighted(keys, levels, nref, c["n_src"], gen)
        return dict(nref=nref, vals=_species(nref, c["species"], torch.float32, gen), src=src, nside=c["nside"])
    x = _cloud(c, c["base"], c.get("refine", 0), c["n_src"], gen)
    if c["path"] in ("step", "replay"):
        odt = torch.float64 if c["mode"] == "fp64" else torch.float32
        x["g"] = torch.rand((x["src"].shape[0], 12 * c["nside"] ** 2, c["species"]), generator=gen, device="cuda", dtype=odt)
        x["g"] += 0.5  # weights of a loss's residuals, of one sign
    if c["path"] == "beta":
        x["coef"] = 0.1 + torch.rand(x["src"].shape[0], generator=gen, device="cuda", dtype=torch.float64)
    return x


def _weights(c):
    return [PDR_WEIGHTS[k] if k < 2 else 0.0 for k in range(c["species"])]


def prepare(case, seed):
    c = case
    x = dict(_inputs(c, seed), case=c)
    if c["path"] == "batch":
        trees = [rt.Octree(y["keys"], y["levels"], extent=y["ext"]) for y in x["clouds"]]
        x["batch"] = rt.Batch([(t, y["src"], y["nside"], y["dens"]) for t, y in zip(trees, x["clouds"])], mode=c["mode"])
        del x["clouds"]
    elif c["path"] == "host":
        for k in ("keys", "levels", "src", "dens"):
            x[k] = x[k].cpu().pin_memory()
        x["out"] = torch.empty((x["src"].shape[0], 12 * c["nside"] ** 2, c["species"]), dtype=torch.float32, pin_memory=True)
    elif c["path"] != "build":
        x["tree"] = rt.Octree(x["keys"], x["levels"], extent=x["ext"])
        if c["path"] in ("step", "replay"):
            x["dens"].requires_grad_()
        if c["path"] == "replay":
            x["paths"] = rt.Paths(x["tree"], x["src"], c["nside"], c["mode"])
    return x


# -------------------------------------------------------------------- run

#: Split criterion of the contribution grid: density threshold and least relative variation (the paper's 1 %).
N_PDR, REL_VAR = 1.0, 0.01


def run(state):
    x, c = state, state["case"]
    if c["path"] == "columns":
        return rt.trace_columns(x["tree"], x["src"], c["nside"], x["dens"], c["mode"])
    if c["path"] in ("step", "replay"):
        out = rt.Columns.apply(x["dens"], x["tree"], x["src"], c["nside"], c["mode"], x.get("paths"))
        grad, = torch.autograd.grad(out, x["dens"], x["g"])
        return {"columns": out, "grad": grad}
    if c["path"] in ("av_eff", "beta"):
        return rt.trace_epilogue(x["tree"], x["src"], c["nside"], x["dens"], c["path"], _weights(c), AV, gamma=GAMMA, coef=x.get("coef"), mode=c["mode"])
    if c["path"] == "batch":
        return x["batch"].launch()
    if c["path"] == "build":
        keys, levels, vals = rt.build_amr(x["nref"], x["vals"], n_pdr=N_PDR, rel_var=REL_VAR)
        out = rt.trace_columns(rt.Octree(keys, levels), x["src"], c["nside"], vals, c["mode"])
        return {"keys": keys, "levels": levels, "vals": vals, "columns": out}
    out, _ = rt.trace_columns_host(x["keys"], x["levels"], x["src"], c["nside"], x["dens"], c["mode"], out=x["out"], extent=x["ext"])
    return out


def tolerance(case):
    """Against exact(), FP32 columns are 2.6e-8 to 3.5e-8 off (a rounding of the
    result, and of each segment's length), and their gradient, which sums the
    same lengths and is returned in the densities' type, 2.5e-8: four times
    that, and ten roundings for a single value.  The FP64 form is 3e-16 to 7e-16
    off, from the order of the sums and the direction's reciprocal."""
    if case["mode"] == "fp64" and not (case["path"] in ("step", "replay") and case["dens"] == "f32"):
        return {"rel": 3e-15, "max": 1e-12}
    return {"rel": 1.4e-7, "max": 1e-6}


# ------------------------------------------------------------------ exact

def _healpix(nside):
    """Pixel centres in ring order (Gorski et al. 2005, equations 2 to 9)."""
    out = []
    for i in range(1, 4 * nside):
        cap = min(i, 4 * nside - i)
        if cap < nside:
            h = cap * cap / (3.0 * nside * nside)
            z, st, n = (1.0 - h) * (1 if i < nside else -1), math.sqrt(h * (2.0 - h)), 4 * cap
            phi = (np.arange(1, n + 1) - 0.5) * (math.pi / (2 * cap))
        else:
            z, n = (2 * nside - i) * 2.0 / (3 * nside), 4 * nside
            st = math.sqrt((1.0 - z) * (1.0 + z))
            phi = (np.arange(n) + 0.5 * ((i - nside + 1) % 2)) * (math.pi / (2 * nside))
        out.append(np.stack([st * np.cos(phi), st * np.sin(phi), np.full(n, z)], axis=1))
    m = np.concatenate(out)
    m[np.abs(m) < 1e-15] = 0.0
    return m


def _walk(keys, levels, ext, src, dirs, visit):
    """All rays of (src, dirs) leaf by leaf: visit(ray index, leaf, length) for every step."""
    dev = src.device
    nd = dirs.shape[0]
    ext = torch.tensor(ext or (1 << D,) * 3, device=dev)
    m_all = torch.from_numpy(dirs).to(dev)
    step = max(1, (1 << 25) // nd)
    for s0 in range(0, src.shape[0], step):
        Q = src[s0:s0 + step].repeat_interleave(nd, 0)
        n = Q.shape[0]
        ray = torch.arange(n, device=dev) + s0 * nd
        m = m_all.repeat(n // nd, 1)
        c = torch.floor(Q * 2.0 ** D).to(torch.int64)
        t = torch.zeros(n, device=dev, dtype=torch.float64)
        while ray.numel():
            M = _spread(c[:, 0]) | (_spread(c[:, 1]) << 1) | (_spread(c[:, 2]) << 2)
            j = torch.searchsorted(keys, M, right=True) - 1
            size = 1 << (D - levels[j].to(torch.int64))
            lo = c & ~(size - 1)[:, None]
            F = (lo + size[:, None] * (m > 0)).to(torch.float64) * 2.0 ** -D
            tb = torch.where(m == 0, float("inf"), (F - Q) / torch.where(m == 0, 1.0, m))
            t1 = tb.min(1).values
            visit(ray, j, t1 - t)
            P = torch.floor((Q + t1[:, None] * m) * 2.0 ** D).to(torch.int64)
            P = torch.maximum(torch.minimum(P, lo + size[:, None] - 1), lo)
            c = torch.where(tb == t1[:, None], torch.where(m > 0, lo + size[:, None], lo - 1), P)
            t = t1
            on = ((c >= 0) & (c < ext)).all(1)
            ray, Q, m, c, t = ray[on], Q[on], m[on], c[on], t[on]


def _exact_walk(keys, levels, ext, src, dens, nside, g=None):
    """Columns and, for a gradient g of them, the densities' gradient."""
    nd = 12 * nside * nside
    dens = dens.detach().to(torch.float64)
    out = torch.zeros((src.shape[0] * nd, dens.shape[1]), device=src.device, dtype=torch.float64)
    grad = torch.zeros_like(dens) if g is not None else None
    g = g.to(torch.float64).reshape(out.shape) if g is not None else None

    def visit(ray, j, ds):
        out[ray] += dens[j] * ds[:, None]
        if g is not None:
            grad.index_add_(0, j, g[ray] * ds[:, None])

    _walk(keys, levels, ext, src, _healpix(nside), visit)
    return out.reshape(src.shape[0], nd, -1), grad


def _exact_cube(n, dens, nside, g=None):
    """The same for a source at the centre of every leaf of an n^3 cube: along
    a direction every source takes the same steps of the same lengths, so the
    columns are a sum of shifted copies of the density."""
    morton = _morton_grid(n.bit_length() - 1)
    S = dens.shape[1]
    nd = 12 * nside * nside
    a = dens.detach()[morton].to(torch.float64).reshape(n, n, n, S)
    out = torch.empty((n ** 3, nd, S), device=a.device, dtype=torch.float64)
    grad = torch.zeros_like(a) if g is not None else None
    for q, m in enumerate(_healpix(nside)):
        col = torch.zeros_like(a)
        gq = g[morton, q].to(torch.float64).reshape(n, n, n, S) if g is not None else None
        cell, t = [0, 0, 0], 0.0
        while max(abs(v) for v in cell) < n:
            tb = [((abs(cell[b]) + 0.5) / n / abs(m[b])) if m[b] else math.inf for b in range(3)]
            t1 = min(tb)
            here, there = [], []  # the sources that reach this step, and the cells they are in
            for b in (2, 1, 0):
                o = cell[b]
                here.append(slice(max(0, -o), n - max(0, o)))
                there.append(slice(max(0, o), n - max(0, -o)))
            col[tuple(here)] += a[tuple(there)] * (t1 - t)
            if g is not None:
                grad[tuple(there)] += gq[tuple(here)] * (t1 - t)
            for b in range(3):
                if tb[b] <= t1 * (1 + 1e-14):
                    cell[b] += 1 if m[b] > 0 else -1
            t = t1
        out[morton, q] = col.reshape(-1, S)
    if g is None:
        return out, None
    back = torch.empty((n ** 3, S), device=a.device, dtype=torch.float64)
    back[morton] = grad.reshape(-1, S)
    return out, back


def _exact_build(nref, vals):
    """Leaves of the split criterion, finest first: keys, levels and means."""
    L = (nref.numel().bit_length() - 1) // 3
    lo = hi = nref.to(torch.float64)
    mean = vals.to(torch.float64)
    means, splits = [mean], []
    for _ in range(L):
        lo, hi, mean = lo.reshape(-1, 8).amin(1), hi.reshape(-1, 8).amax(1), mean.reshape(-1, 8, mean.shape[1]).mean(1)
        splits.insert(0, (hi >= N_PDR) & ((hi - lo) / hi >= REL_VAR))
        means.insert(0, mean)
    open_ = torch.zeros(1, device=nref.device, dtype=torch.int64)
    keys, levels, out = [], [], []
    for l in range(L + 1):
        s = splits[l][open_] if l < L else torch.zeros_like(open_, dtype=torch.bool)
        leaf = open_[~s]
        keys.append(leaf << (3 * (D - l)))
        levels.append(torch.full_like(leaf, l, dtype=torch.uint8))
        out.append(means[l][leaf])
        open_ = (8 * open_[s][:, None] + torch.arange(8, device=nref.device)).reshape(-1)
    keys, order = torch.sort(torch.cat(keys))
    return keys, torch.cat(levels)[order], torch.cat(out)[order]


def exact(case, seed):
    c = case
    if _segments(c) > 6.0e10 or (_segments(c) > 8.0e9 and not (c["grid"] == "cube" and c["sources"] == "centres")):
        return None  # over twenty seconds
    x = _inputs(c, seed)
    if c["path"] == "batch":
        return [_exact_walk(y["keys"], y["levels"], y["ext"], y["src"], y["dens"], y["nside"])[0] for y in x["clouds"]]
    if c["path"] == "build":
        keys, levels, vals = _exact_build(x["nref"], x["vals"])
        out, _ = _exact_walk(keys, levels, None, x["src"], vals.to(torch.float32), c["nside"])
        return {"keys": keys, "levels": levels, "vals": vals, "columns": out}
    if c["grid"] == "cube" and c["sources"] == "centres":
        out, grad = _exact_cube(c["base"], x["dens"], c["nside"], x.get("g"))
    else:
        out, grad = _exact_walk(x["keys"], x["levels"], x["ext"], x["src"], x["dens"], c["nside"], x.get("g"))
    if c["path"] in ("step", "replay"):
        return {"columns": out, "grad": grad}
    if c["path"] in ("av_eff", "beta"):
        N = (out * torch.tensor(_weights(c), device=out.device, dtype=torch.float64)).sum(-1)
        if c["path"] == "av_eff":
            return -torch.log(torch.exp(-GAMMA * AV * N).mean(1)) / GAMMA
        tau = x["coef"][:, None] * N
        return torch.where(tau == 0, 1.0, -torch.expm1(-tau) / torch.where(tau == 0, 1.0, tau)).mean(1)
    return out
