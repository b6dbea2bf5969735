"""The workloads whose speed matters to a user of this package, as cases.

A case is a dict of plain values: an operation (``op``), a shape as text
("100x500x500", last extent varying fastest), a dtype and the options that the
public entry point takes.  ``prepare`` makes what a program has in hand before
the call, ``run`` is the call, ``exact`` states its result in 64 bits with
plain torch.  Fields are seeded Gaussian random fields with a power-law
spectrum, sums of Gaussian bumps, or fronts and vortex tubes over a smooth
background; all are drawn on the GPU from the seed alone.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

import paper_2609_00205_gb300 as bm

DEV = "cuda"
F32, F64 = "f32", "f64"


# ---------------------------------------------------------------------------
# The cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # A small diagnostic field compressed inside a simulation's loop:
        # latency and launches count.  8 bumps and a little noise, an absolute
        # bound, every level inside the block.
        dict(name="compress_65", op="compress", shape="65x65x65", dtype=F32, field="bumps", tol=1e-3, mode="abs",
             block=9, levels=3, global_levels=0, roi="none"),
        # ... and read back.
        dict(name="decompress_65", op="decompress", shape="65x65x65", dtype=F32, field="bumps", tol=1e-3, mode="abs",
             block=9, levels=3, global_levels=0, roi="none"),
        # A weather-model slab (the shape of the hurricane data sets), ragged
        # in every dimension, at a tight bound: symbols spread over the whole
        # dictionary.
        dict(name="compress_slab", op="compress", shape="100x500x500", dtype=F32, field="grf", tol=1e-4, mode="rel",
             block=17, levels=2, global_levels=2, roi="none"),
        # A wider slab read back at a medium bound.
        dict(name="decompress_slab", op="decompress", shape="98x1200x1200", dtype=F32, field="grf", tol=1e-3,
             mode="rel", block=17, levels=2, global_levels=2, roi="none"),
        # The benchmark's field at a medium bound ...
        dict(name="compress_513", op="compress", shape="513x513x513", dtype=F32, field="grf", tol=1e-3, mode="rel",
             block=17, levels=2, global_levels=2, roi="none"),
        # ... at its tightest, where most codes leave the dictionary ...
        dict(name="compress_513_tight", op="compress", shape="513x513x513", dtype=F32, field="grf", tol=1e-5,
             mode="rel", block=17, levels=2, global_levels=2, roi="none"),
        # ... and read back in between.
        dict(name="decompress_513", op="decompress", shape="513x513x513", dtype=F32, field="grf", tol=1e-4, mode="rel",
             block=17, levels=2, global_levels=2, roi="none"),
        # Region-of-interest control on a double-precision field of fronts and
        # vortices: blocks with strong gradients at 1e-5, the others at 1e-2.
        dict(name="compress_roi_f64", op="compress", shape="385x385x257", dtype=F64, field="fronts", tol=1e-2,
             mode="rel", block=9, levels=2, global_levels=2, roi="gradient"),
        dict(name="decompress_roi_f64", op="decompress", shape="385x385x257", dtype=F64, field="fronts", tol=1e-2,
             mode="rel", block=9, levels=2, global_levels=2, roi="gradient"),
        # One horizontal level of a model: a 2-D field.
        dict(name="compress_plane", op="compress", shape="1535x2049", dtype=F32, field="grf", tol=1e-3, mode="rel",
             block=17, levels=2, global_levels=2, roi="none"),
        # Many uneven fields of both precisions with their own bounds and
        # region maps, as one checkpoint of a multi-variable code.
        dict(name="batch_64", op="batch", fields=64, layout=64, block=17, levels=2, global_levels=2),
        # A training step through the differentiable recomposition: the field
        # from its coefficients, then the coefficients' gradient.
        dict(name="recompose_grad_257", op="recompose_grad", shape="257x257x257", dtype=F32, field="grf", block=17,
             levels=2, global_levels=2),
    ]


def draw(rng: random.Random):
    op = rng.choices(["compress", "decompress", "batch", "recompose_grad", "decompose_grad"], [35, 30, 8, 16, 11])[0]
    if op == "batch":
        return dict(op="batch", fields=rng.randint(4, 64), layout=rng.randrange(1 << 20), block=rng.choice([9, 17]),
                    levels=rng.choice([1, 2]), global_levels=2)
    dtype = rng.choices([F32, F64], [3, 1])[0]
    block = rng.choice([9, 17])
    case = dict(op=op, dtype=dtype, block=block, levels=rng.randint(1, 3), global_levels=rng.randint(0, 3))
    grad = op.endswith("_grad")
    if not grad and rng.random() < 0.2:
        most = 5.0e6
        v = math.exp(rng.uniform(math.log(1.0e4), math.log(most)))
        a = math.exp(rng.uniform(-0.8, 0.8))
        shape = [math.sqrt(v) * a, math.sqrt(v) / a]
    else:
        most = (1.7e7 if grad else 1.3e8) / (1 if dtype == F32 else 4)
        v = math.exp(rng.uniform(math.log(3.0e4), math.log(most)))
        a, b = math.exp(rng.uniform(-0.6, 0.6)), math.exp(rng.uniform(-0.6, 0.6))
        e = v ** (1.0 / 3.0)
        shape = [e * a, e * b, e / (a * b)]
    case["shape"] = "x".join(str(max(12, int(n))) for n in shape)
    case["field"] = "bumps" if v < 3.0e5 and rng.random() < 0.5 else "grf"
    if not grad:
        case.update(tol=10.0 ** rng.uniform(-5, -2), mode="rel", roi=rng.choices(["none", "random"], [7, 3])[0])
    return case


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _shape(case):
    return tuple(int(n) for n in case["shape"].split("x"))


def _dtype(case):
    return torch.float64 if case["dtype"] == F64 else torch.float32


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed) % (1 << 62))


def _smooth(n):
    """The least number >= n with no prime factor above 5 (FFT lengths)."""
    while True:
        m = n
        for p in (2, 3, 5):
            while m % p == 0:
                m //= p
        if m == 1:
            return n
        n += 1


def _grf(shape, exponent, seed, dtype):
    """Gaussian random field with the shell spectrum k^exponent and unit
    variance: the corner of a periodic one on FFT-friendly extents."""
    big = [_smooth(n) for n in shape]
    spec = torch.fft.rfftn(torch.randn(big, generator=_gen(seed), device=DEV, dtype=dtype))
    k2 = torch.zeros((), device=DEV, dtype=torch.float64)
    for d, n in enumerate(big):
        k = torch.fft.rfftfreq(n, d=1.0 / n, device=DEV) if d == len(big) - 1 else torch.fft.fftfreq(n, d=1.0 / n,
                                                                                                    device=DEV)
        k2 = k2 + (k.double() ** 2).view([-1 if i == d else 1 for i in range(len(big))])
    p = (exponent - (len(big) - 1)) / 4.0
    spec.mul_(torch.where(k2 > 0, k2.clamp_min(1e-30) ** p, torch.zeros_like(k2)).to(dtype))
    u = torch.fft.irfftn(spec, s=big)[tuple(slice(0, n) for n in shape)]
    del spec, k2
    return ((u - u.mean()) / u.std()).contiguous()


def _axes(shape):
    return [torch.arange(n, device=DEV, dtype=torch.float64).view([-1 if i == d else 1 for i in range(len(shape))])
            for d, n in enumerate(shape)]


def _bumps(shape, seed, dtype):
    """8 Gaussian bumps (amplitudes U[0.5, 2], widths U[4, 12] cells) and
    N(0, 1e-3) noise."""
    rng = np.random.default_rng(seed)
    u = torch.randn(shape, generator=_gen(seed), device=DEV, dtype=torch.float64) * 1e-3
    X = _axes(shape)
    for _ in range(8):
        c = [rng.uniform(0, n - 1) for n in shape]
        amp, width = rng.uniform(0.5, 2.0), rng.uniform(4.0, 12.0)
        u += amp * torch.exp(-sum((x - a) ** 2 for x, a in zip(X, c)) / (2.0 * width * width))
    return u.to(dtype)


def _fronts(shape, seed, dtype):
    """A smooth k^-3 background, 12 tanh fronts two cells thick and 6 Gaussian
    vortex tubes."""
    rng = np.random.default_rng(seed)
    u = _grf(shape, -3.0, seed + 1, torch.float64)
    X = _axes(shape)
    box = np.array(shape) - 1.0
    for _ in range(12):
        n = rng.normal(size=3)
        n /= np.linalg.norm(n)
        p, amp = rng.uniform(0, 1, size=3) * box, rng.uniform(0.5, 2.0)
        u += amp * torch.tanh((sum(x * a for x, a in zip(X, n)) - float(n @ p)) / 2.0)
    for _ in range(6):
        t = rng.normal(size=3)
        t /= np.linalg.norm(t)
        p, amp, width = rng.uniform(0, 1, size=3) * box, rng.uniform(0.5, 2.0), rng.uniform(2.0, 6.0)
        dx = [x - a for x, a in zip(X, p)]
        along = sum(d * a for d, a in zip(dx, t))
        r2 = sum(d * d for d in dx) - along * along
        u += amp * torch.exp(-r2.clamp_min(0.0) / (2.0 * width * width))
    return u.to(dtype)


def _field(case, seed):
    shape, dtype = _shape(case), _dtype(case)
    if case["field"] == "bumps":
        return _bumps(shape, seed, dtype)
    if case["field"] == "fronts":
        return _fronts(shape, seed, dtype)
    return _grf(shape, -5.0 / 3.0, seed, dtype)


def _random_roi(shape, block, tol, seed):
    """10 % of the blocks at a ten times tighter bound."""
    n = math.prod(-(-s // block) for s in shape)
    r = np.full(n, tol)
    r[np.random.default_rng(seed).choice(n, size=max(1, n // 10), replace=False)] = tol / 10
    return r


def _gradient_roi(u, block, tol, tight):
    """The tight bound where a block's largest gradient exceeds the field's
    95th percentile."""
    mag = sum(g * g for g in torch.gradient(u))
    sample = mag.flatten()[:: max(1, mag.numel() // 1000003)]
    thr = sample.kthvalue(int(0.95 * sample.numel())).values
    nb = [-(-n // block) for n in u.shape]
    pad = [v for n, b in zip(reversed(u.shape), reversed(nb)) for v in (0, b * block - n)]
    m = torch.nn.functional.pad(mag, pad, value=-math.inf).view(nb[0], block, nb[1], block, nb[2], block)
    hot = (m.amax(dim=(1, 3, 5)) > thr).flatten().cpu().numpy()
    return np.where(hot, tight, tol)


def _batch_specs(case):
    """Shapes, dtypes, spectra and bounds of a batch, from the case alone: of
    64 fields 24 planes with sides U[100, 2049], 32 boxes with sides
    U[33, 257] and 8 FP64 cubes of 129."""
    rng = random.Random(case["layout"])
    n = case["fields"]
    flat, cubes = max(1, n * 3 // 8), max(1, n // 8)
    out = []
    for i in range(n):
        if i < flat:
            shape, dt = tuple(rng.randint(100, 2049) for _ in range(2)), torch.float32
        elif i < n - cubes:
            shape, dt = tuple(rng.randint(33, 257) for _ in range(3)), torch.float32
        else:
            shape, dt = (129, 129, 129), torch.float64
        out.append((shape, dt, rng.uniform(-4.0, -1.5), 10.0 ** rng.uniform(-5, -2)))
    return out


def _params(case):
    return dict(block=case["block"], levels=case["levels"], global_levels=case["global_levels"])


def prepare(case, seed):
    op, p = case["op"], _params(case)
    if op == "batch":
        us, tols, rois = [], [], []
        for i, (shape, dt, exponent, tol) in enumerate(_batch_specs(case)):
            us.append(_grf(shape, exponent, seed * 1000 + i, dt))
            tols.append(tol)
            rois.append(_random_roi(shape, case["block"], tol, seed * 1000 + i))
        # one buffer, each stream at a 256-byte boundary of it
        at = [0]
        for u in us:
            at.append(at[-1] + -(-bm.compress_bound(u.shape, u.dtype) // 256) * 256)
        out = torch.zeros(at[-1], dtype=torch.uint8, device=DEV)
        return dict(op=op, params=p, fields=us, tols=tols, rois=rois, out=out,
                    outs=[out[a:b] for a, b in zip(at, at[1:])])
    u = _field(case, seed)
    if op in ("compress", "decompress"):
        tol = case["tol"]
        if case["mode"] == "abs":
            tol *= float(u.max() - u.min())
        roi = None
        if case["roi"] == "random":
            roi = _random_roi(u.shape, case["block"], tol, seed)
        elif case["roi"] == "gradient":
            roi = _gradient_roi(u, case["block"], tol, tol / 1000)
        kw = dict(p, mode=case["mode"], roi=roi)
        if op == "compress":
            # the output buffer that a program which compresses step after step keeps
            out = torch.zeros(bm.compress_bound(u.shape, u.dtype), dtype=torch.uint8, device=DEV)
            return dict(op=op, params=kw, field=u, tol=tol, out=out)
        return dict(op=op, stream=bm.compress(u, tol, **kw).clone())
    if op == "recompose_grad":
        c = bm.decompose(u, **p)
        g = torch.randn(u.shape, generator=_gen(seed + 7), device=DEV, dtype=u.dtype)
        return dict(op=op, params=p, shape=tuple(u.shape), coeffs=c.requires_grad_(True), grad=g)
    n = bm.coeff_count(u.shape, **p)
    g = torch.randn(n, generator=_gen(seed + 7), device=DEV, dtype=u.dtype)
    return dict(op=op, params=p, field=u.requires_grad_(True), grad=g)


def run(state):
    op = state["op"]
    if op == "compress":
        s = bm.compress(state["field"], state["tol"], out=state["out"], **state["params"])
        return [state["out"], s.numel()]
    if op == "decompress":
        return bm.decompress(state["stream"])
    if op == "batch":
        s = bm.compress_batch(state["fields"], state["tols"], rois=state["rois"], outs=state["outs"], **state["params"])
        return [state["out"], np.array([v.numel() for v in s])]
    if op == "recompose_grad":
        u = bm.recompose_ad(state["coeffs"], state["shape"], **state["params"])
        (g,) = torch.autograd.grad(u, state["coeffs"], state["grad"])
        return [u.detach(), g]
    c = bm.decompose_ad(state["field"], **state["params"])
    (g,) = torch.autograd.grad(c, state["field"], state["grad"])
    return [c.detach(), g]


# ---------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------
def _ratio(tol, dtype):
    """Rough compression ratio (the 513^3 FP32 benchmark field: 3.84, 2.72,
    2.11 and 1.16 at 1e-2 .. 1e-5; twice that in double precision)."""
    x = min(5.0, max(2.0, -math.log10(tol)))
    r = np.interp(x, [2, 3, 4, 5], [3.84, 2.72, 2.11, 1.16])
    return float(r) * (2 if dtype in (F64, torch.float64) else 1)


def _transform_flops(shape, block, levels):
    """In-cache levels: the interpolation and the three line passes (band of
    five, forward and backward substitution) of every block."""
    nd = len(shape)
    blocks = math.prod(-(-n // block) for n in shape)
    total, n = 0.0, block
    for _ in range(levels):
        c = (n + 1) // 2
        lines = sum(n ** (nd - 1 - d) * c ** d for d in range(nd))
        total += lines * 15 * c + n ** (nd - 1) * (4 * c + 3 * n)
        n = c
    return blocks * total


def work(case):
    op, block, levels = case["op"], case["block"], case["levels"]
    if op == "batch":
        b = f = 0.0
        for shape, dt, _, tol in _batch_specs(case):
            size = math.prod(shape) * (8 if dt == torch.float64 else 4)
            b += size + size / _ratio(tol, dt)
            f += _transform_flops(shape, block, levels)
        return {"bytes": b, "flops": f}
    shape = _shape(case)
    size = math.prod(shape) * (8 if case["dtype"] == F64 else 4)
    flops = _transform_flops(shape, block, levels)
    if op in ("compress", "decompress"):
        ratio = 7.7 if case["roi"] == "gradient" else _ratio(case["tol"], case["dtype"])
        return {"bytes": size + size / ratio, "flops": flops}
    # coefficients in and field out, then the field's gradient in and the
    # coefficients' out (or the other way round)
    coeffs = bm.coeff_count(shape, **_params(case)) * (8 if case["dtype"] == F64 else 4)
    return {"bytes": 2.0 * (size + coeffs), "flops": 2.0 * flops}


def tolerance(case):
    if case["op"] in ("compress", "batch"):
        return "exact"  # streams are bytes
    # four times the distance from exact() over the listed and drawn cases
    # (FP32: 1.1e-7 and, for gradients, 4.6e-6 at the worst value; FP64: 2.3e-16
    # and 3.6e-15)
    if case["dtype"] == F64:
        return {"rel": 1e-15, "max": 1.5e-14}
    return {"rel": 5e-7, "max": 2e-5}


# ---------------------------------------------------------------------------
# 64-bit statement of the computed outputs (plain torch)
# ---------------------------------------------------------------------------
def _coarse(n):
    return list(range(0, n, 2)) + ([n - 1] if n % 2 == 0 else [])


def _operators(x):
    """Interpolation I (n x c) and projection P = M_c^-1 I^T M_f (c x n) of the
    piecewise-linear level on nodes x."""
    x = np.asarray(x, dtype=np.float64)
    n = len(x)
    ci = _coarse(n)
    interp = np.zeros((n, len(ci)))
    for J, i in enumerate(ci):
        interp[i, J] = 1.0
    for i in range(n):
        if i not in set(ci):
            lo, hi = ci.index(i - 1), ci.index(i + 1)
            w = (x[i] - x[i - 1]) / (x[i + 1] - x[i - 1])
            interp[i, lo], interp[i, hi] = 1.0 - w, w

    def mass(y):
        m = np.zeros((len(y), len(y)))
        for i in range(len(y) - 1):
            h = y[i + 1] - y[i]
            m[i:i + 2, i:i + 2] += h / 6.0 * np.array([[2.0, 1.0], [1.0, 2.0]])
        return m if len(y) > 1 else np.ones((1, 1))

    proj = np.linalg.solve(mass(x[ci]), interp.T @ mass(x)) if n > 1 else np.ones((1, 1))
    t = dict(device=DEV, dtype=torch.float64)
    return ci, torch.tensor(interp, **t), torch.tensor(proj, **t)


def _apply(mats, u):
    """The matrices along the last three dimensions of u."""
    for d, m in enumerate(mats):
        u = torch.movedim(torch.tensordot(u, m, dims=([u.dim() - 3 + d], [1])), -1, u.dim() - 3 + d)
    return u


class _Hierarchy:
    """Levels of one (shape, B, K, M): blocks of B nodes per dimension (one
    node along an extent of 1), then M global levels on the gathered coarse
    values at their physical coordinates."""

    def __init__(self, shape, B, K, M):
        self.shape = (1,) * (3 - len(shape)) + tuple(shape)
        self.edge = [1 if n == 1 else B for n in self.shape]
        self.nb = [-(-n // e) for n, e in zip(self.shape, self.edge)]
        self.local, self.glob = [], []
        x = [list(range(e)) for e in self.edge]
        for _ in range(K):
            x = self._level(x, self.local)
        self.m = [len(v) for v in x]
        x = [[b * e + v for b in range(nb) for v in xs] for nb, e, xs in zip(self.nb, self.edge, x)]
        for _ in range(M):
            x = self._level(x, self.glob)
        self.coarsest = [len(v) for v in x]
        self.blocks = math.prod(self.nb)
        self.counts = [len(lv["fine"]) for lv in self.local]
        self.per_block = sum(self.counts)

    @staticmethod
    def _level(x, out):
        ops = [_operators(v) for v in x]
        n = [len(v) for v in x]
        c = torch.zeros(n, dtype=torch.bool, device=DEV)
        c[np.ix_(*[o[0] for o in ops])] = True
        out.append(dict(n=n, c=[len(o[0]) for o in ops], I=[o[1] for o in ops], P=[o[2] for o in ops],
                        fine=torch.nonzero(~c.flatten()).flatten(), coarse=torch.nonzero(c.flatten()).flatten()))
        return [[v[i] for i in o[0]] for v, o in zip(x, ops)]

    @staticmethod
    def _down(lv, u):
        """Values (..., n) -> (coefficients, coarse values)."""
        flat = u.reshape(-1, math.prod(lv["n"]))
        uc = flat[:, lv["coarse"]].view(-1, *lv["c"])
        d = u.reshape(-1, *lv["n"]) - _apply(lv["I"], uc)
        df = d.reshape(flat.shape)[:, lv["fine"]]
        d0 = torch.zeros_like(flat).index_copy(1, lv["fine"], df).view(d.shape)
        return df, uc + _apply(lv["P"], d0)

    @staticmethod
    def _up(lv, df, c):
        d = torch.zeros(df.shape[0], math.prod(lv["n"]), device=DEV, dtype=df.dtype)
        d = d.index_copy(1, lv["fine"], df).view(-1, *lv["n"])
        return _apply(lv["I"], c.reshape(-1, *lv["c"]) - _apply(lv["P"], d)) + d

    def _to_blocks(self, g, e):
        nb = self.nb
        return g.reshape(nb[0], e[0], nb[1], e[1], nb[2], e[2]).permute(0, 2, 4, 1, 3, 5).reshape(-1, *e)

    def _from_blocks(self, b, e):
        nb = self.nb
        return b.reshape(*nb, *e).permute(0, 3, 1, 4, 2, 5).reshape([k * v for k, v in zip(nb, e)])

    def decompose(self, u):
        u = u.reshape(self.shape)
        pad = [v for n, k, e in zip(reversed(self.shape), reversed(self.nb), reversed(self.edge)) for v in (0, k * e - n)]
        b = self._to_blocks(torch.nn.functional.pad(u, pad), self.edge)
        parts = []
        for lv in self.local:
            d, b = self._down(lv, b)
            parts.append(d)
        parts = [torch.cat(parts, dim=1).flatten()]
        g = self._from_blocks(b, self.m)
        for lv in self.glob:
            d, g = self._down(lv, g)
            parts.append(d.flatten())
        return torch.cat(parts + [g.flatten()])

    def recompose(self, c):
        pos = self.blocks * self.per_block
        blk, rest = c[:pos].view(self.blocks, self.per_block), c[pos:]
        sizes = [len(lv["fine"]) for lv in self.glob] + [math.prod(self.coarsest)]
        parts = torch.split(rest, sizes)
        g = parts[-1].view(1, *self.coarsest)
        for lv, d in zip(reversed(self.glob), reversed(parts[:-1])):
            g = self._up(lv, d.view(1, -1), g)
        b = self._to_blocks(g.reshape([k * v for k, v in zip(self.nb, self.m)]), self.m)
        for lv, d in zip(reversed(self.local), reversed(torch.split(blk, self.counts, dim=1))):
            b = self._up(lv, d, b)
        u = self._from_blocks(b, self.edge)
        return u[tuple(slice(0, n) for n in self.shape)]


def _stream_values(buf):
    """The dequantised coefficients of a (non-raw) stream, its shape and its
    hierarchy parameters: chunked canonical Huffman codes decoded one symbol of
    every chunk at a time."""
    h = buf.cpu().numpy()
    u16 = lambda o: int(h[o:o + 2].view("<u2")[0])
    i32 = lambda o: int(h[o:o + 4].view("<i4")[0])
    u64 = lambda o: int(h[o:o + 8].view("<u8")[0])
    if u16(6) & 1:
        return None
    ndim, B, K, M, chunk, radius, tiers = i32(8), i32(12), i32(40), i32(44), i32(48), i32(52), i32(56)
    shape = [int(v) for v in h[16:40].view("<i8")][3 - ndim:]
    n, chunks, outliers, words = u64(96), u64(104), u64(112), u64(120)
    q = torch.tensor(h[u64(136):][: 8 * (tiers * K + M + 1)].view("<f8").copy(), device=DEV)
    lens = np.zeros(2 * radius, dtype=np.int64)
    pos, end = u64(160), u64(160) + int(h[192:196].view("<u4")[0])
    for _ in range(int(h[196:200].view("<u4")[0])):
        first, count = int(h[pos:pos + 4].view("<u4")[0]), int(h[pos + 4:pos + 8].view("<u4")[0])
        lens[first:first + count] = h[pos + 8:pos + 8 + count]
        pos += 8 + (count + 3) // 4 * 4
    assert pos <= end
    present = np.flatnonzero(lens)
    order = present[np.argsort(lens[present], kind="stable")]
    limit, base, used, code, at = [], [], [], 0, 0
    for length in range(1, 33):
        cnt = int((lens == length).sum())
        if cnt:
            used.append(length)
            base.append(at - code)
            limit.append((code + cnt) << (32 - length))
            at += cnt
            code += cnt
        code <<= 1
    t = lambda v: torch.tensor(v, device=DEV, dtype=torch.int64)
    limit, base, used, order = t(limit), t(base), t(used), t(order)
    w = torch.zeros(words + 2, device=DEV, dtype=torch.int64)
    w[:words] = t(h[u64(168):][: 4 * words].view("<u4").astype(np.int64))
    cw = t(h[u64(152):][: 4 * chunks].view("<u4").astype(np.int64))
    bit = (torch.cumsum(cw, 0) - cw) * 32
    sym = torch.zeros(chunks, chunk, device=DEV, dtype=torch.int32)
    last = n - (chunks - 1) * chunk
    for s in range(min(chunk, n)):
        i, off = bit >> 5, bit & 31
        v = ((w[i] << off) & 0xFFFFFFFF) | (w[i + 1] >> (32 - off))
        k = torch.searchsorted(limit, v, right=True).clamp_max(len(used) - 1)
        ln = used[k]
        sym[:, s] = order[(base[k] + (v >> (32 - ln))).clamp(0, len(order) - 1)].int()
        step = ln
        if s >= last:
            step = ln.clone()
            step[-1] = 0
        bit = (bit + step).clamp_max(32 * words)
    sym = sym.flatten()[:n]
    codes = (sym - radius).double()
    esc = torch.nonzero(sym == 0).flatten()
    assert len(esc) == outliers
    if outliers:
        codes[esc] = torch.tensor(h[u64(176):][: 4 * outliers].view("<i4").astype(np.float64), device=DEV)
    H = _Hierarchy(shape, B, K, M)
    nblk = H.blocks * H.per_block
    tier = torch.zeros(H.blocks, device=DEV, dtype=torch.int64)
    if tiers > 1:
        tier = t(h[u64(144):][: H.blocks].astype(np.int64))
    at = 0
    blk = codes[:nblk].view(H.blocks, H.per_block)
    for l, cnt in enumerate(H.counts):
        blk[:, at:at + cnt] *= q[tier * K + l].unsqueeze(1)
        at += cnt
    at = nblk
    for l, cnt in enumerate([len(lv["fine"]) for lv in H.glob] + [math.prod(H.coarsest)]):
        codes[at:at + cnt] *= q[tiers * K + l]
        at += cnt
    return codes, H, shape


def exact(case, seed):
    if case["op"] in ("compress", "batch"):
        return None
    state = prepare(case, seed)
    if case["op"] == "decompress":
        values = _stream_values(state["stream"])
        if values is None:
            return None
        c, H, shape = values
        return H.recompose(c).reshape(shape)
    H = _Hierarchy(_shape(case), case["block"], case["levels"], case["global_levels"])
    f, x = (H.recompose, state["coeffs"]) if case["op"] == "recompose_grad" else (H.decompose, state["field"])
    x = x.detach().double().requires_grad_(True)
    y = f(x)
    (g,) = torch.autograd.grad(y, x, state["grad"].double().reshape(y.shape))
    return [y.detach(), g]
