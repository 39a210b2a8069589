"""The work that users of this library have it do, as cases that can be timed and checked.

A case is a plain dict.  ``prepare`` makes what a program has in hand before the call (fields on the GPU, the
LGF table, the mesh, a captured batch), ``run`` is one pass through the public entry points of
``paper_2010_13213_gb300.lgf``, ``work`` what such a pass cannot do without, and ``exact`` the same outputs from
plain torch in 64 bits on dense boxes.

Kinds: ``box`` a single-level Poisson solve; ``amr`` a composite-mesh Poisson solve (FLGF-AMR); ``heat`` an
integrating-factor apply (FIF-AMR); ``refresh`` the velocity from the vorticity; ``projection`` the pressure
projection of a Runge-Kutta stage; ``batch`` captured stages (Poisson and heat) of many uneven instances.
"""
from __future__ import annotations

import functools
import math
import weakref

import numpy as np
import torch

import paper_2010_13213_gb300.lgf as L

PREC = {"fp64": L.LGF_PREC_FP64, "fp32": L.LGF_PREC_FP32, "df32": L.LGF_PREC_DF32}
STORE = {"f64": (L.LGF_F64, torch.float64, 8), "f32": (L.LGF_F32, torch.float32, 4)}


def listed():
    return [
        # the smallest call: 32^3 cells in eight blocks, one scalar, as in the smoke check (launch latency)
        dict(name="random32_fp64", kind="box", block=16, nx=2, ny=2, nz=2, ncomp=1, precision="fp64", storage="f64",
             field="random", fill=1.0),
        # an irregular set of small blocks, two scalars: a sparse source region on a coarse octree level
        dict(name="sparse_b8_df32", kind="box", block=8, nx=5, ny=7, nz=3, ncomp=2, precision="df32", storage="f64",
             field="random", fill=0.6),
        # the vector solve of one vortex ring on 96x96x48 cells, mixed precision: the everyday single-level solve
        dict(name="ring96_df32", kind="box", block=16, nx=6, ny=6, nz=3, ncomp=3, precision="df32", storage="f64",
             field="ring", fill=1.0),
        # the same ring in native double (reference runs, acceptance checks)
        dict(name="ring96_fp64", kind="box", block=16, nx=6, ny=6, nz=3, ncomp=3, precision="fp64", storage="f64",
             field="ring", fill=1.0),
        # two coaxial rings on 96x96x112 cells, single precision fields and arithmetic (previews, preconditioning)
        dict(name="tworings_fp32", kind="box", block=16, nx=6, ny=6, nz=7, ncomp=3, precision="fp32", storage="f32",
             field="tworing", fill=1.0),
        # the two rings in mixed precision
        dict(name="tworings_df32", kind="box", block=16, nx=6, ny=6, nz=7, ncomp=3, precision="df32", storage="f64",
             field="tworing", fill=1.0),
        # the adaptive ring on three levels (h = R/16, R/32, R/64): one composite solve of a time step
        dict(name="ring3level_df32", kind="amr", levels=3, nxy=192, nz=96, res=64, sigma=0.2, n_ext=16,
             precision="df32"),
        # a two-level ring in double with the paper's 14-cell extension: the acceptance run of a small mesh
        dict(name="ring2level_fp64", kind="amr", levels=2, nxy=80, nz=48, res=22, sigma=0.2, n_ext=14,
             precision="fp64"),
        # the integrating factor of the viscous term on the three-level mesh
        dict(name="heat3level_df32", kind="heat", levels=3, nxy=192, nz=96, res=64, sigma=0.2, n_ext=16, alpha=0.1,
             precision="df32"),
        # velocity from vorticity after every time step
        dict(name="refresh96_df32", kind="refresh", block=16, nx=6, ny=6, nz=3, precision="df32", storage="f64"),
        # the pressure projection of a Runge-Kutta stage on two levels
        dict(name="projection2level_df32", kind="projection", levels=2, nxy=128, nz=64, res=36, sigma=0.2, n_ext=16,
             alpha=0.1, precision="df32"),
        # one Runge-Kutta stage (vector Poisson solve and heat apply) of sixteen uneven instances as one graph
        dict(name="batch16_df32", kind="batch", first=0, count=16, alpha=0.1, precision="df32"),
    ]


def draw(rng):
    kind = rng.choice(["box", "box", "box", "amr", "amr", "heat", "refresh", "projection", "batch"])
    if kind == "box" or kind == "refresh":
        block = rng.choice([8, 16, 16])
        cells = int(math.exp(rng.uniform(math.log(2 * block ** 3), math.log(1.0e6))))
        blocks = max(1, cells // block ** 3)
        top = 12 if block == 8 else 8
        nx = max(1, min(top, int(round(blocks ** (1 / 3) * rng.uniform(0.7, 1.5)))))
        ny = max(1, min(top, int(round(math.sqrt(blocks / nx) * rng.uniform(0.7, 1.4)))))
        nz = max(1, min(top, blocks // (nx * ny)))
        precision = rng.choice(["df32", "df32", "df32", "fp64", "fp32"])
        storage = "f32" if precision == "fp32" else "f64"
        c = dict(kind=kind, block=block, nx=nx, ny=ny, nz=nz, precision=precision, storage=storage)
        if kind == "box":
            field = rng.choice(["random", "ring"])
            c.update(ncomp=3 if field == "ring" else rng.choice([1, 2, 3, 4]), field=field,
                     fill=rng.choice([1.0, round(rng.uniform(0.4, 0.9), 2)]))
        return c
    if kind == "batch":
        return dict(kind=kind, first=rng.randrange(100, 5000), count=rng.randint(2, 6),
                    alpha=round(rng.uniform(0.03, 0.3), 3), precision="df32")
    levels = rng.choice([2, 3]) if kind == "amr" else rng.choice([1, 2, 3])
    precision = rng.choice(["df32", "df32", "df32", "fp64", "fp32"])
    nxy = 16 * rng.randint(2, 7 if precision == "fp64" else 10)
    nz = 16 * max(2, round(nxy / 32 * rng.uniform(0.9, 1.3)))
    sigma = round(rng.uniform(0.1, 0.25), 3)
    c = dict(kind=kind, levels=levels, nxy=nxy, nz=nz, res=max(4, int(nxy / (2 + 8 * sigma))), sigma=sigma,
             n_ext=rng.choice([8, 14, 16]), precision=precision)
    if kind != "amr":
        c["alpha"] = round(math.exp(rng.uniform(math.log(0.02), math.log(0.6))), 3)
    return c


# ------------------------------------------------------------------ meshes and fields
def _box_blocks(nx, ny, nz):
    z, y, x = np.meshgrid(np.arange(nz), np.arange(ny), np.arange(nx), indexing="ij")
    return np.stack([x.ravel(), y.ravel(), z.ravel()], 1).astype(np.int32)


def _near_ring(n, h, origin, B, R, limit):
    """Blocks of a level grid of n cells holding a cell centre within s^2 < limit of the ring's core circle."""
    x, y, z = (origin[a] + (np.arange(n[a]) + 0.5) * h for a in range(3))
    d = (np.sqrt(x[None, :] ** 2 + y[:, None] ** 2) - R) ** 2
    d = d.reshape(n[1] // B, B, n[0] // B, B).min(axis=(1, 3))
    bz, by, bx = np.nonzero((z ** 2).reshape(n[2] // B, B).min(axis=1)[:, None, None] + d[None] < limit)
    return np.stack([bx, by, bz], 1).astype(np.int32)


def _ring_mesh(levels, nxy, nz, R, sigma, h_fine, B=16):
    """Block lists per level and spacings and origins of the Gaussian-core ring's composite mesh: level 0 the support box
    dilated by a block, level 1 of 3 the blocks above 1e-3 of the peak and the parents of level 2, the finest level
    those above 1e-2."""
    h = [h_fine * 2 ** (levels - 1 - k) for k in range(levels)]
    n0 = [int(math.ceil(n / 2 ** (levels - 1) / B)) * B + (2 * B if levels > 1 else 0) for n in (nxy, nxy, nz)]
    origin = [-n * h[0] / 2 for n in n0]
    blocks = [_box_blocks(*(n // B for n in n0))]

    def above(k, rel):
        return _near_ring([n * 2 ** k for n in n0], h[k], origin, B, R, -sigma * sigma * math.log(rel))

    if levels >= 2:
        fine = above(levels - 1, 1e-2)
        if levels == 3:
            blocks.append(np.unique(np.concatenate([above(1, 1e-3), fine // 2]), axis=0).astype(np.int32))
        blocks.append(fine)
    return blocks, h, origin


def _ring_field(blocks, B, h, origin, R, sigma, seed, centres=(0.0,)):
    """Vorticity [3][nblk][B][B][B] of wavy Gaussian-core rings: the core circle of each is displaced radially and
    axially by a few per cent with random modes and phases."""
    rng = np.random.default_rng(seed)
    b = torch.from_numpy(np.asarray(blocks)).cuda().double()
    loc = (torch.arange(B, device="cuda", dtype=torch.float64) + 0.5) * h
    x, y, z = (origin[a] + b[:, a, None] * (B * h) + loc for a in range(3))
    x, y, z = x[:, None, None, :], y[:, None, :, None], z[:, :, None, None]
    r, th = torch.sqrt(x * x + y * y), torch.atan2(y, x)
    out = torch.zeros(3, len(b), B, B, B, device="cuda", dtype=torch.float64)
    for zc in centres:
        gamma = rng.uniform(0.8, 1.2)
        m1, m2 = (int(v) for v in rng.integers(2, 6, 2))
        p1, p2 = rng.uniform(0, 2 * math.pi, 2)
        e1, e2 = rng.uniform(0.01, 0.03, 2)
        rc, drc = R * (1 + e1 * torch.cos(m1 * th + p1)), -e1 * m1 * torch.sin(m1 * th + p1)
        zr, dzr = zc + e2 * R * torch.cos(m2 * th + p2), -e2 * m2 * torch.sin(m2 * th + p2)
        w = gamma / (math.pi * sigma ** 2) * torch.exp(-((z - zr) ** 2 + (r - rc) ** 2) / sigma ** 2)
        out[0] += w * (drc * torch.cos(th) - torch.sin(th))
        out[1] += w * (drc * torch.sin(th) + torch.cos(th))
        out[2] += w * dzr
    return out


def _geometry(c):
    """What the sizes of a case give without its values: levels of blocks, spacings, origin, roles, ring."""
    if c["kind"] in ("box", "refresh"):
        n, B = (c["nx"], c["ny"], c["nz"]), c["block"]
        blocks = _box_blocks(*n)
        field = c.get("field", "ring")
        if c.get("fill", 1.0) < 1.0:  # an irregular part of the box, the same one for the same sizes
            keep = np.random.default_rng(sum(n) + 100 * B).permutation(len(blocks))
            blocks = blocks[np.sort(keep[:max(1, int(c["fill"] * len(blocks)))])]
        roles, R, sigma, h, origin = None, 1.0, 0.2, 1.0, [0.0] * 3
        if field != "random":
            sigma = 0.2 if field == "ring" else 0.15
            h = 1.0 / 32 if n[0] * B >= 96 else 3.0 / (n[0] * B)
            origin = [-n[a] * B * h / 2 for a in range(3)]
            if field == "ring" and c["kind"] == "box":  # sources where the vorticity is above 1e-6 of its peak
                src = {tuple(b) for b in _near_ring([n[a] * B for a in range(3)], h, origin, B, R,
                                                    -sigma * sigma * math.log(1e-6))}
                roles = np.array([3 if tuple(b) in src else 2 for b in blocks], np.uint8)
                roles = None if roles.max() < 3 else roles
        return dict(B=B, levels=[blocks], h=[h], origin=origin, roles=roles, R=R, sigma=sigma, n_ext=16,
                    centres=(-1.0, 1.0) if field == "tworing" else (0.0,))
    blocks, h, origin = _ring_mesh(c["levels"], c["nxy"], c["nz"], 1.0, c["sigma"], 1.0 / c["res"])
    return dict(B=16, levels=blocks, h=h, origin=origin, roles=None, R=1.0, sigma=c["sigma"], n_ext=c["n_ext"],
                centres=(0.0,))


def _instances(c):
    """The uneven ring problems of a batch: radius, core, level count and resolution drawn per instance."""
    out = []
    for i in range(c["count"]):
        rng = np.random.default_rng(1000 + c["first"] + i)
        R = float(rng.uniform(0.5, 1.5))
        sigma = float(rng.uniform(0.1, 0.25)) * R
        levels = int(rng.integers(1, 4))
        nxy = int(rng.choice(np.arange(32, 193, 16)))
        nz = max(32, 16 * int(math.ceil(nxy / 32)))
        blocks, h, origin = _ring_mesh(levels, nxy, nz, R, sigma, (2 * R + 8 * sigma) / nxy)
        out.append(dict(B=16, levels=blocks, h=h, origin=origin, roles=None, R=R, sigma=sigma, n_ext=16,
                        centres=(0.0,)))
    return out


def _values(c, g, seed):
    """The input field [ncomp][all blocks][B][B][B] in 64 bits."""
    if c.get("field") == "random":
        gen = torch.Generator(device="cuda").manual_seed(seed)
        return torch.randn(c["ncomp"], len(g["levels"][0]), g["B"], g["B"], g["B"], generator=gen, device="cuda",
                           dtype=torch.float64)
    return torch.cat([_ring_field(b, g["B"], h, g["origin"], g["R"], g["sigma"], seed, g["centres"])
                      for b, h in zip(g["levels"], g["h"])], 1).contiguous()


# ------------------------------------------------------------------ what a program keeps
class _Table:
    """An LGF table and its release."""

    def __init__(self, block, reach, flags):
        self.h = L.lgf_table_create(block, reach, flags)

    def __del__(self):
        try:
            L.lgf_table_destroy(self.h)
        except Exception:
            pass


_tables = weakref.WeakValueDictionary()  # one table per geometry, as a program has, while a state holds it


def _table(block, reach, flags):
    key = (block, tuple(reach), flags)
    t = _tables.get(key)
    if t is None:
        t = _tables[key] = _Table(*key)
    return t


def _table_for(c, gs):
    ext = [max(int(b[:, a].max() - b[:, a].min()) + 1 for g in gs for b in g["levels"]) for a in range(3)]
    if c["kind"] == "box" and int(np.prod(ext)) <= 64:  # small boxes: the pair spectra as well
        flags = {"fp64": L.LGF_TBL_FP64, "fp32": L.LGF_TBL_FP32, "df32": L.LGF_TBL_DF32}[c["precision"]]
        return _table(gs[0]["B"], [max(0, e - 1) for e in ext], flags)
    more = 0 if c["kind"] == "box" else (1 if c["kind"] == "refresh" else 4)
    return _table(gs[0]["B"], [e - 1 + more for e in ext], L.LGF_TBL_BOX_ONLY)


def prepare(case, seed):
    c = case
    if c["kind"] == "batch":
        gs = _instances(c)
        st = torch.cuda.Stream()
        f = [_values(c, g, seed + 7919 * i) for i, g in enumerate(gs)]
        phi, heat = [torch.zeros_like(v) for v in f], [torch.zeros_like(v) for v in f]
        table = _table_for(c, gs)
        meshes = [L.Mesh(g["levels"], 16, g["h"][0], n_ext=g["n_ext"]) for g in gs]
        b = L.Batch(table.h, meshes, 3, L.LGF_F64, alpha=[c["alpha"]] * len(gs),
                    opts=L.make_opts(precision=PREC[c["precision"]]), nstreams=2)
        torch.cuda.synchronize()
        b.graph_create(1, [v.data_ptr() for v in f], [v.data_ptr() for v in phi], [v.data_ptr() for v in heat], None,
                       st.cuda_stream)
        return dict(case=c, batch=b, table=table, f=f, phi=phi, g=heat, stream=st)
    g = _geometry(c)
    code, dtype, _ = STORE[c.get("storage", "f64")]
    s = dict(case=c, table=_table_for(c, [g]), code=code,
             mesh=L.Mesh(g["levels"], g["B"], g["h"][0], n_ext=g["n_ext"], roles=g["roles"]),
             opts=L.make_opts(precision=PREC[c["precision"]]), f=_values(c, g, seed).to(dtype).contiguous())
    s["out"] = torch.zeros_like(s["f"])
    if c["kind"] in ("box", "amr"):
        L.lgf_table_prepare(s["table"].h, s["mesh"], s["f"].shape[0], code, s["opts"],
                            torch.cuda.current_stream().cuda_stream)
    if c["kind"] == "projection":
        s["p"] = torch.zeros_like(s["f"][:1])
    return s


def run(state):
    s, c = state, state["case"]
    if c["kind"] == "batch":
        s["batch"].graph_launch(s["stream"].cuda_stream)
        return {"phi": s["phi"], "g": s["g"]}
    st, t, f, out = torch.cuda.current_stream().cuda_stream, s["table"].h, s["f"], s["out"]
    if c["kind"] in ("box", "amr"):
        L.lgf_poisson_solve(t, s["mesh"], f.shape[0], f.data_ptr(), out.data_ptr(), s["code"], s["opts"], None, st)
    elif c["kind"] == "heat":
        L.lgf_heat_apply(t, s["mesh"], f.shape[0], f.data_ptr(), out.data_ptr(), s["code"], c["alpha"], s["opts"],
                         None, st)
    elif c["kind"] == "refresh":
        L.lgf_velocity_refresh(t, s["mesh"], f.data_ptr(), out.data_ptr(), s["code"], s["opts"], None, st)
    else:
        L.lgf_stage_projection(t, s["mesh"], f.data_ptr(), out.data_ptr(), s["p"].data_ptr(), s["code"], c["alpha"],
                               s["opts"], None, st)
        return {"u": out, "p": s["p"]}
    return out


# ------------------------------------------------------------------ what a pass cannot do without
def _poisson_flops(B, blocks, ncomp):
    """Two zero-padded real FFTs over the box around the blocks, per component."""
    m = 8.0 * float(np.prod(blocks.max(0) - blocks.min(0) + 1)) * B ** 3
    return ncomp * 2 * 2.5 * m * math.log2(m)


def work(case):
    c = case
    gs = _instances(c) if c["kind"] == "batch" else [_geometry(c)]
    size = STORE[c.get("storage", "f64")][2]
    total = {"bytes": 0.0, "flops": 0.0}
    for g in gs:
        B, nl = g["B"], len(g["levels"])
        ncomp = c.get("ncomp", 3)
        cells = [(len(b) - (len(g["levels"][k + 1]) / 8 if k + 1 < nl else 0)) * B ** 3
                 for k, b in enumerate(g["levels"])]  # the cells that carry the solution
        poisson = sum(_poisson_flops(B, b, 1 if c["kind"] == "projection" else ncomp) for b in g["levels"])
        heat = 0.0
        if c["kind"] in ("heat", "projection", "batch"):  # three line sums of the symmetric kernel per cell
            for k in range(nl):
                r = len(_heat_weights(c["alpha"] * 4.0 ** (k + 1 - nl))) - 1
                heat += 3 * ncomp * cells[k] * (3 * r + 1)
        fields = {"box": 2, "amr": 2, "heat": 2, "refresh": 2, "projection": 2 + 1 / 3, "batch": 3}[c["kind"]]
        total["bytes"] += fields * ncomp * sum(cells) * size
        total["flops"] += heat + (0.0 if c["kind"] == "heat" else poisson)
    return total


# ------------------------------------------------------------------ the same in 64 bits on dense boxes
def _scaled_bessel(x, n):
    """e^-x I_0..n(x) for a tensor x > 0: below 1e6 by the backward recurrence of the ratios I_{k+1} / I_k (a
    contraction), scaled by e^-x I_0(x); above by the large-argument series."""
    m = n + 60 + int(math.sqrt(40.0 * min(float(x.max()), 1e6)))
    lo = torch.clamp(x, max=1e6)
    ratio = lo / (2 * m + 2 + lo)
    rs = torch.zeros(n, len(x), dtype=torch.float64, device=x.device)
    for k in range(m, 0, -1):
        ratio = 1.0 / (2.0 * k / lo + ratio)
        if k <= n:
            rs[k - 1] = ratio
    i0 = torch.special.i0e(lo)
    small = torch.cat([i0[None], i0 * torch.cumprod(rs, 0)]) if n else i0[None]
    big = torch.clamp(x, min=1e6)
    mu = 4.0 * torch.arange(n + 1, dtype=torch.float64, device=x.device)[:, None] ** 2
    term = torch.ones(n + 1, len(x), dtype=torch.float64, device=x.device)
    series = term.clone()
    for j in range(1, 25):
        term = -term * (mu - (2 * j - 1) ** 2) / (j * 8.0 * big)
        series += term
    return torch.where(x <= 1e6, small, series / torch.sqrt(2 * math.pi * big))


@functools.lru_cache(maxsize=4)
def _lgf(n):
    """G on [0, n]^3: -int_0^inf prod e^-2t I_{n_a}(2t) dt by the trapezoidal rule in ln t."""
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    step = 1.0 / 16
    u = torch.arange(-42.0, 92.0, step, dtype=torch.float64, device=dev)
    t = torch.exp(u)
    e = _scaled_bessel(2 * t, n)
    w = -step * t
    return torch.stack([(e * (w * e[c])) @ e.T for c in range(n + 1)])


def _convolve(src, h):
    """h^2 G * src on the box of src [ncomp][nz][ny][nx]."""
    shape = src.shape[1:]
    G = _lgf(16 * int(math.ceil(max(shape) / 16)))
    idx = []
    for n in shape:
        i = torch.arange(2 * n, device=src.device)
        idx.append(torch.where(i <= n, i, 2 * n - i))
    K = torch.fft.rfftn(G[idx[0]][:, idx[1]][:, :, idx[2]].contiguous())
    pad = tuple(2 * n for n in shape)
    return torch.stack([h * h * torch.fft.irfftn(torch.fft.rfftn(s, s=pad) * K, s=pad)[:shape[0], :shape[1], :shape[2]]
                        for s in src])


@functools.lru_cache(maxsize=64)
def _heat_weights(alpha):
    w = _scaled_bessel(torch.tensor([2.0 * alpha], dtype=torch.float64), 79)[:, 0]
    r = int((w >= 1e-18).sum())
    return tuple(float(v) for v in w[:max(r, 1)])


def _along(a, axis, d):
    """a[n + d] along an axis, zero beyond the box."""
    out = torch.zeros_like(a)
    n = a.shape[axis]
    if abs(d) < n:
        out.narrow(axis, max(0, -d), n - abs(d)).copy_(a.narrow(axis, max(0, d), n - abs(d)))
    return out


def _heat_box(f, alpha):
    for axis in (1, 2, 3):
        acc = torch.zeros_like(f)
        for d, w in reversed(list(enumerate(_heat_weights(alpha)))):
            acc += w * (f if d == 0 else _along(f, axis, d) + _along(f, axis, -d))
        f = acc
    return f


class _Dense:
    """A level's dense box: its lowest cell (x, y, z), its shape [nz][ny][nx] and the cells of its blocks."""

    def __init__(self, blocks, B, h, pad):
        self.blocks, self.B, self.h = blocks, B, h
        lo, hi = (blocks.min(0) * B - pad), ((blocks.max(0) + 1) * B + pad)
        self.lo = [int(v) - int(v) % 2 for v in lo]
        self.shape = tuple(int(hi[a]) + int(hi[a]) % 2 - self.lo[a] for a in (2, 1, 0))
        cell = torch.arange(B)
        b = torch.from_numpy(np.asarray(blocks)).long() * B - torch.tensor(self.lo)
        x, y, z = (b[:, a, None] + cell for a in range(3))
        flat = (z[:, :, None, None] * self.shape[1] + y[:, None, :, None]) * self.shape[2] + x[:, None, None, :]
        self.flat = flat.reshape(-1).cuda()
        self.user = self.dense(torch.ones(1, len(blocks), B, B, B, device="cuda"))[0] > 0

    def dense(self, v):
        out = torch.zeros(v.shape[0], int(np.prod(self.shape)), dtype=v.dtype, device=v.device)
        out[:, self.flat] = v.reshape(v.shape[0], -1)
        return out.reshape(v.shape[0], *self.shape)

    def gather(self, a):
        n = a.shape[0]
        return a.reshape(n, -1)[:, self.flat].reshape(n, len(self.blocks), self.B, self.B, self.B)


def _levels(g, extra):
    pads, K = [0] * len(g["levels"]), len(g["levels"])
    for k in range(K - 1, -1, -1):
        pads[k] = g["n_ext"] + 10 + extra if k == K - 1 else max(g["n_ext"] + 10 + extra, (pads[k + 1] + 1) // 2 + 8)
    lv = [_Dense(b, g["B"], g["h"][k], pads[k]) for k, b in enumerate(g["levels"])]
    for k, l in enumerate(lv):
        l.omega = l.user & ~(_coarsen(lv[k + 1].user[None].double(), lv[k + 1], l)[0] > 0) if k + 1 < K else l.user
    return lv


def _coarsen(a, fine, coarse):
    """The mean of the eight children, on the coarse box."""
    m = a.reshape(a.shape[0], a.shape[1] // 2, 2, a.shape[2] // 2, 2, a.shape[3] // 2, 2).mean(dim=(2, 4, 6))
    o = [fine.lo[i] // 2 - coarse.lo[i] for i in (2, 1, 0)]
    out = torch.zeros(a.shape[0], *coarse.shape, dtype=a.dtype, device=a.device)
    out[:, o[0]:o[0] + m.shape[1], o[1]:o[1] + m.shape[2], o[2]:o[2] + m.shape[3]] = m
    return out


def _interp(a, coarse, fine):
    """Tensor-product linear interpolation: 3/4 of the parent, 1/4 of its neighbour towards the child, per axis."""
    for axis in (1, 2, 3):
        gl = fine.lo[3 - axis] + torch.arange(fine.shape[axis - 1], device=a.device)
        p = torch.div(gl, 2, rounding_mode="floor")
        q = torch.where(gl % 2 == 0, p - 1, p + 1)
        p, q = p - coarse.lo[3 - axis], q - coarse.lo[3 - axis]
        a = 0.75 * a.index_select(axis, p) + 0.25 * a.index_select(axis, q)
    return a


def _laplacian(a, h):
    s = -6.0 * a
    for axis in (1, 2, 3):
        s = s + _along(a, axis, 1) + _along(a, axis, -1)
    return s / (h * h)


def _dilate(mask, r):
    m = mask[None, None].float()
    for k in ((r, 0, 0), (0, r, 0), (0, 0, r)):
        m = torch.nn.functional.max_pool3d(m, tuple(2 * v + 1 for v in k), stride=1, padding=k)
    return m[0, 0] > 0


def _cumulative(lv, f):
    F = [None] * len(lv)
    for k in range(len(lv) - 1, -1, -1):
        F[k] = f[k] if k + 1 == len(lv) else f[k] + _coarsen(F[k + 1], lv[k + 1], lv[k])
    return F


def _flgf(lv, f, n_ext):
    """FLGF-AMR: phi on the boxes of all levels from the sources f[k] (zero off Omega_k)."""
    F, psi, out = _cumulative(lv, f), None, []
    for k, l in enumerate(lv):
        A, c = f[k], 0.0
        if k:
            up = lv[k - 1]
            c = _interp(psi, up, l)
            s = _interp(_laplacian(psi, up.h), up, l) - _laplacian(c, l.h)
            A = A + torch.where(_dilate(l.omega, n_ext), s, torch.zeros_like(s))
        rest = F[k] - f[k]
        psi = c + _convolve(A, l.h)
        out.append((psi + _convolve(rest, l.h) if k + 1 < len(lv) else psi) * l.omega)
    return out


def _reconstruct(lv, f):
    F, T = _cumulative(lv, f), []
    for k, l in enumerate(lv):
        T.append(F[0] if k == 0 else torch.where(l.user, F[k], _interp(T[k - 1], lv[k - 1], l)))
    return T


def _heat_levels(lv, f, alpha):
    T = _reconstruct(lv, f)
    return [_heat_box(T[k], alpha * 4.0 ** (k + 1 - len(lv))) * l.omega for k, l in enumerate(lv)]


def _split(g, v):
    at = np.cumsum([0] + [len(b) for b in g["levels"]])
    return [v[:, at[k]:at[k + 1]] for k in range(len(g["levels"]))]


def _gather(lv, a):
    return torch.cat([l.gather(x) for l, x in zip(lv, a)], 1)


def exact(case, seed):
    c = case
    if c["kind"] == "batch":
        phi, heat = [], []
        for i, g in enumerate(_instances(c)):
            lv = _levels(g, len(_heat_weights(c["alpha"])))
            f = [l.dense(v) * l.omega for l, v in zip(lv, _split(g, _values(c, g, seed + 7919 * i)))]
            phi.append(_gather(lv, _flgf(lv, f, g["n_ext"])))
            heat.append(_gather(lv, _heat_levels(lv, f, c["alpha"])))
        return {"phi": phi, "g": heat}
    g = _geometry(c)
    v = _values(c, g, seed).to(STORE[c.get("storage", "f64")][1]).double()
    if c["kind"] in ("box", "refresh"):
        l = _Dense(g["levels"][0], g["B"], g["h"][0], 0 if c["kind"] == "box" else 2)
        if g["roles"] is not None:
            v = v * torch.from_numpy((g["roles"] & 1).astype(np.float64)).cuda()[None, :, None, None, None]
        p = _convolve(l.dense(v), l.h)
        if c["kind"] == "refresh":  # u = -C^T psi, backward differences
            def back(a, comp):
                return a - _along(a[None], 3 - comp, -1)[0]
            p = -torch.stack([back(p[(a + 2) % 3], (a + 1) % 3) - back(p[(a + 1) % 3], (a + 2) % 3)
                              for a in range(3)]) / l.h
        return l.gather(p)
    lv = _levels(g, len(_heat_weights(c["alpha"])) if "alpha" in c else 0)
    f = [l.dense(x) * l.omega for l, x in zip(lv, _split(g, v))]
    if c["kind"] == "amr":
        return _gather(lv, _flgf(lv, f, g["n_ext"]))
    if c["kind"] == "heat":
        return _gather(lv, _heat_levels(lv, f, c["alpha"]))
    # the projection: L p = D r, u = E (r - G p), D backward and G forward differences of the reconstructions
    T = _reconstruct(lv, f)
    d = [(sum(T[k][a] - _along(T[k][a:a + 1], 3 - a, -1)[0] for a in range(3)) / l.h)[None] * l.omega
         for k, l in enumerate(lv)]
    p = _flgf(lv, d, g["n_ext"])
    P = _reconstruct(lv, p)
    w = [(f[k] - torch.stack([(_along(P[k], 3 - a, 1) - P[k])[0] for a in range(3)]) / l.h) * l.omega
         for k, l in enumerate(lv)]
    return {"u": _gather(lv, _heat_levels(lv, w, c["alpha"])), "p": _gather(lv, p)}
