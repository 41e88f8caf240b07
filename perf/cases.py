"""The work that programs have this library do, as measurable cases.

A case is a dict of plain values.  Its "kind" is the entry point:

  tend     PW.tendencies: su, sv, sw once per model timestep
  step     PW.step: a short forecast, nsteps fused Euler steps from a saved state
  batch    Batch.tendencies: many grids of uneven sizes in one launch
  adjoint  PW.adjoint: one transposed evaluation, as data assimilation needs it
  rollout  autograd.rollout: a checkpointed forecast and its gradient

Sizes follow the package's own workloads (64^3, 512^2 x 64, 2048^2 x 64, the
batch recipe of widths 32..384 and depths 32..128, the 20-step rollout), plus
widths and heights that are odd or no multiple of a tile.
"""
import math
import random

import numpy as np
import torch

import paper_2301_13016_gb300 as pw
from paper_2301_13016_gb300.autograd import rollout

TORCH = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}
# FP16 storage of winds up to 64 m/s: physical = stored * 2^-8, and source
# terms (at most 512 m/s^2 for such winds on these levels) stored as 64 times
# their value.  BF16 and FP32 need no scaling.
F16_SCALE = (2.0 ** -8, 2.0 ** -8, 2.0 ** -8, 64.0, 64.0, 64.0)
MAX_CELLS = 2048 * 2048 * 64
LINE = 64   # a grid's slice of a batch buffer starts at a multiple of this many elements (128 bytes or more)


def listed():
    return [
        # a small column ensemble member or a unit test: one call is mostly launch
        {"name": "tend_f32_64", "kind": "tend", "dtype": "f32", "nx": 64, "ny": 64, "nz": 64},
        # a large-eddy domain on one GPU
        {"name": "tend_f32_512", "kind": "tend", "dtype": "f32", "nx": 512, "ny": 512, "nz": 64},
        # the largest domain of the package's workloads, bound by HBM
        {"name": "tend_f32_2048", "kind": "tend", "dtype": "f32", "nx": 2048, "ny": 2048, "nz": 64},
        # a domain whose width is what the user's region gave it: odd in x and y
        {"name": "tend_f32_odd", "kind": "tend", "dtype": "f32", "nx": 1021, "ny": 1023, "nz": 61},
        # 16-bit storage of the largest domain (half the bytes of a memory-bound path)
        {"name": "tend_bf16_2048", "kind": "tend", "dtype": "bf16", "nx": 2048, "ny": 2048, "nz": 64},
        # FP16 storage with its scales, a width that fills no whole vector of 8, ragged rows
        {"name": "tend_f16_ragged", "kind": "tend", "dtype": "f16", "nx": 1020, "ny": 765, "nz": 70},
        # a short forecast between two outputs, odd number of steps
        {"name": "step_f32_512", "kind": "step", "dtype": "f32", "nx": 512, "ny": 512, "nz": 64, "nsteps": 5},
        # a long-running large forecast in BF16 storage, a stretch of its steps
        {"name": "step_bf16_2048", "kind": "step", "dtype": "bf16", "nx": 2048, "ny": 2048, "nz": 64, "nsteps": 10},
        # an ensemble of limited-area domains of uneven sizes
        {"name": "batch_f32", "kind": "batch", "dtype": "f32", "grids": 96, "lo": 32, "hi": 384, "shapes": 2304},
        # the same kind of ensemble in 16-bit storage
        {"name": "batch_bf16", "kind": "batch", "dtype": "bf16", "grids": 64, "lo": 32, "hi": 384, "shapes": 2305},
        # data assimilation on a limited-area domain: boundary values are inputs of their own
        {"name": "adjoint_open", "kind": "adjoint", "nx": 384, "ny": 320, "nz": 64, "periodic": False, "add": False},
        # the gradient of a 20-step forecast on a doubly periodic domain, checkpoint every 5 steps
        {"name": "rollout_512", "kind": "rollout", "nx": 512, "ny": 512, "nz": 64, "nsteps": 20, "every": 5},
    ]


def _size(rng, lo, hi):
    """A size between lo and hi, spread over its logarithm: whole tiles, multiples of 4, or any."""
    n = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    m = rng.choice((1, 1, 4, 4, 64))
    return int(min(hi, max(lo, round(n / m) * m)))


def draw(rng):
    kind = rng.choice(("tend", "tend", "tend", "step", "step", "batch", "adjoint", "rollout"))
    if kind == "batch":
        return {"kind": "batch", "dtype": rng.choice(("f32", "f32", "bf16", "f16")), "grids": _size(rng, 4, 80), "lo": 32,
                "hi": rng.choice((128, 256, 384)), "shapes": rng.randrange(1 << 20)}
    big = {"tend": 2048, "step": 1536, "adjoint": 512, "rollout": 512}[kind]
    c = {"kind": kind, "nx": _size(rng, 32, big), "ny": _size(rng, 32, big),
         "nz": rng.randint(16, 96) if kind == "tend" else rng.randint(16, 64)}
    while c["nx"] * c["ny"] * c["nz"] > MAX_CELLS:
        c["nz"] -= 1
    if kind in ("tend", "step"):
        c["dtype"] = rng.choice(("f32", "f32", "bf16", "f16"))
    if kind == "step":
        c["nsteps"] = rng.randint(1, 10)
    if kind == "adjoint":
        c["periodic"] = rng.random() < 0.5
        c["add"] = rng.random() < 0.5
    if kind == "rollout":
        c["nsteps"] = rng.randint(3, 20)
        c["every"] = rng.choice((1, 2, 5))
    return c


def _shapes(case):
    """The batch's grids: widths and heights multiples of 4, depths 32..128."""
    r = random.Random(case["shapes"])
    side = lambda: 4 * r.randint(case["lo"] // 4, case["hi"] // 4)
    return [(side(), side(), r.randint(32, 128)) for _ in range(case["grids"])]


# ---------------------------------------------------------------------------
# Inputs (from the seed alone; nothing of the library)

def _column(nz):
    """dx = dy = 100 m, levels stretched 20 -> 200 m: {tcx, tcy, tzc1, tzc2, tzd1, tzd2} in float64, and an
    anelastic weighting so that the two flux coefficients of a level differ."""
    zw = np.zeros(nz + 2)
    for k in range(2, nz + 1):
        zw[k] = zw[k - 1] + 20.0 + 180.0 * (k - 2) / (nz - 2)
    zw[0], zw[nz + 1] = -zw[2], 2 * zw[nz] - zw[nz - 1]
    zu = np.zeros(nz + 2)
    zu[1:] = 0.5 * (zw[:-1] + zw[1:])
    ru, rw = np.exp(-zu / 8000.0), np.exp(-zw / 8000.0)
    c = {n: np.zeros(nz + 2) for n in ("tzc1", "tzc2", "tzd1", "tzd2")}
    for k in range(2, nz + 1):
        d = 4.0 * ru[k] * (zw[k] - zw[k - 1])
        c["tzc1"][k], c["tzc2"][k] = rw[k - 1] / d, rw[k] / d
    for k in range(2, nz):
        d = 4.0 * rw[k] * (zu[k + 1] - zu[k])
        c["tzd1"][k], c["tzd2"][k] = ru[k] / d, ru[k + 1] / d
    c["tcx"] = c["tcy"] = 0.0025
    return c


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _wrap(f):
    """Periodic images in the one-cell lateral halo of a dense (nz+2, ny+2, nx+2) field."""
    f[:, :, 0], f[:, :, -1] = f[:, :, -2], f[:, :, 1]
    f[:, 0], f[:, -1] = f[:, -2], f[:, 1]
    return f


def _turbulent(nx, ny, nz, seed, wrap=True):
    """u, v, w = 10 N(0, 1) m/s, w = 0 at the surface and the lid."""
    out = []
    for q in range(3):
        f = torch.randn((nz + 2, ny + 2, nx + 2), generator=_generator(8 * seed + q), device="cuda").mul_(10.0)
        f[0] = f[-1] = 0.0
        if q == 2:
            f[1] = f[-2] = 0.0
        out.append(_wrap(f) if wrap else f)
    return out


def _smooth(nx, ny, nz, seed):
    """u, v, w as sums of 4 sine modes, at most about 10 (w: 1) m/s, w = 0 at the surface and the lid."""
    r = random.Random(seed)
    x = torch.arange(nx, device="cuda", dtype=torch.float64) * (2 * math.pi / nx)
    y = torch.arange(ny, device="cuda", dtype=torch.float64) * (2 * math.pi / ny)
    z = torch.arange(nz, device="cuda", dtype=torch.float64) * (math.pi / (nz - 1))
    out = []
    for q in range(3):
        f = torch.zeros((nz + 2, ny + 2, nx + 2), device="cuda")
        for _ in range(4):
            a, kz = r.uniform(1.0, 2.5) * (0.1 if q == 2 else 1.0), r.randint(1, 2)
            h = torch.sin(r.randint(1, 4) * x[None, :] + r.randint(1, 4) * y[:, None] + r.uniform(0, 2 * math.pi))
            v = torch.sin(kz * z) if q == 2 else torch.cos(kz * z)
            f[1:-1, 1:-1, 1:-1].add_((a * v).float()[:, None, None] * h.float()[None])
        if q == 2:
            f[1] = f[-2] = 0.0
        out.append(_wrap(f))
    return out


def _stored(f, dtype, scale=1.0):
    """The field as it sits in storage, in float64 physical values."""
    return (f / scale).to(TORCH[dtype]).double() * scale


def _scales(case):
    return F16_SCALE if case.get("dtype") == "f16" else None


# ---------------------------------------------------------------------------
# What a program holds before the call, and the call

def _inner(g, t):
    """The interior of a field, levels 1..nz."""
    h = g.halo
    return g.view(t)[1:-1, h:h + g.ny, h:h + g.nx]


def _whole(g, t):
    """Levels 1..nz with the one-cell lateral halo."""
    h = g.halo
    return g.view(t)[1:-1, h - 1:h + g.ny + 1, h - 1:h + g.nx + 1]


def _prepare_batch(case, seed):
    """All grids of a batch in one allocation per field, each grid's part a slice of it."""
    shapes = _shapes(case)
    grids = [pw.Grid(*s, dtype=case["dtype"]) for s in shapes]
    starts, total = [], 0
    for g in grids:
        starts.append(total)
        total += -(-g.alloc_elems // LINE) * LINE
    bufs = [torch.zeros(total, dtype=TORCH[case["dtype"]], device="cuda") for _ in range(6)]
    parts = [[b[s:s + g.alloc_elems] for s, g in zip(starts, grids)] for b in bufs]
    scale = _scales(case)
    for n, (s, g) in enumerate(zip(shapes, grids)):
        for q, f in enumerate(_turbulent(*s, seed * 1000 + n)):
            _whole(g, parts[q][n]).copy_(f[1:-1] / (scale[q] if scale else 1.0))
    batch = pw.Batch(grids, [_column(s[2]) for s in shapes])
    return {"case": case, "batch": batch, "parts": parts, "bufs": bufs, "scale": scale}


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return _prepare_batch(case, seed)
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    dtype, scale = case.get("dtype", "f32"), _scales(case)
    g = pw.Grid(nx, ny, nz, dtype=dtype)
    h = pw.PW(g, _column(nz))
    s = {"case": case, "grid": g, "handle": h, "scale": scale}
    load = lambda fields: [g.from_dense(f, scale=scale[q] if scale else 1.0) for q, f in enumerate(fields)]
    if kind == "tend":
        s["q"] = load(_turbulent(nx, ny, nz, seed))
        s["out"] = [g.alloc() for _ in range(3)]
        s["result"] = [_inner(g, t) for t in s["out"]]
    elif kind == "step":
        s["start"] = load(_smooth(nx, ny, nz, seed))
        s["q"], s["tmp"] = [g.alloc() for _ in range(3)], [g.alloc() for _ in range(3)]
        s["result"] = [_whole(g, t) for t in s["q"]]
    elif kind == "adjoint":
        s["q"] = load(_turbulent(nx, ny, nz, seed, wrap=case["periodic"]))
        s["lam"] = load([f * 0.1 for f in _turbulent(nx, ny, nz, seed + (1 << 30), wrap=False)])
        s["out"] = [g.alloc() for _ in range(3)]
        s["result"] = [(_inner if case["periodic"] else _whole)(g, t) for t in s["out"]]
        s["flags"] = (pw.PW_ADJ_PERIODIC if case["periodic"] else 0) | (pw.PW_ADJ_ADD_LAMBDA if case["add"] else 0)
    else:
        s["q"] = [t.requires_grad_(True) for t in load(_smooth(nx, ny, nz, seed))]
        s["target"] = _smooth(nx, ny, nz, seed + (1 << 30))[0][1:-1, 1:-1, 1:-1].contiguous()
    return s


def run(state):
    s = state
    kind = s["case"]["kind"]
    if kind == "tend":
        s["handle"].tendencies(*s["q"], *s["out"], scale=s["scale"])
        return s["result"]
    if kind == "batch":
        s["batch"].tendencies(*s["parts"], scale=s["scale"])
        return s["bufs"][3:]
    if kind == "step":   # a forecast from the saved state
        for t, t0 in zip(s["q"], s["start"]):
            t.copy_(t0)
        s["handle"].step(*s["q"], *s["tmp"], 1.0, s["case"]["nsteps"], scale=s["scale"] and s["scale"][:3])
        return s["result"]
    if kind == "adjoint":
        s["handle"].adjoint(*s["q"], *s["lam"], *s["out"], alpha=1.0, flags=s["flags"])
        return s["result"]
    g = s["grid"]
    final = rollout(*s["q"], s["handle"], 1.0, s["case"]["nsteps"], s["case"]["every"])
    miss = _inner(g, final[0]) - s["target"]
    grads = torch.autograd.grad(0.5 * (miss * miss).sum(), s["q"])
    return [_inner(g, t.detach()) for t in final], [_inner(g, t) for t in grads]


def work(case):
    """Each input read once and each output written once; operations as the scheme is written: 63 a cell for the
    source terms (3 fields of 6 pair sums, 6 products and 9 differences and scalings), 6 for the update, and 3 for
    each of the adjoint's 50 terms."""
    kind = case["kind"]
    size = 4 if case.get("dtype", "f32") == "f32" else 2
    if kind == "batch":
        cells = sum(a * b * c for a, b, c in _shapes(case))
        return {"bytes": 6 * size * cells, "flops": 63 * cells}
    cells = case["nx"] * case["ny"] * case["nz"]
    if kind == "tend":
        return {"bytes": 6 * size * cells, "flops": 63 * cells}
    if kind == "step":
        return {"bytes": 6 * size * cells, "flops": 69 * cells * case["nsteps"]}
    if kind == "adjoint":
        return {"bytes": 9 * size * cells, "flops": 150 * cells}
    return {"bytes": 10 * size * cells, "flops": (69 + 156) * cells * case["nsteps"]}


# ---------------------------------------------------------------------------
# The same in 64 bits, plain torch on dense (nz+2, ny+2, nx+2) arrays

def _sources(slab, c, k, e, nz):
    """su, sv, sw of levels k..e from u, v, w of levels k-1..e+1: the scheme's formulas, zero where it has no term."""
    u, v, w = slab
    lev = np.arange(k, e + 1)
    col = lambda a, ok: torch.from_numpy(np.where(ok, a, 0.0)).to(u.device)[:, None, None]
    low, mid = lev >= 2, (lev >= 2) & (lev < nz)
    z1, z2 = col(c["tzc1"][k:e + 1], low), col(c["tzc2"][k:e + 1], mid)
    d1, d2 = col(c["tzd1"][k:e + 1], mid), col(c["tzd2"][k:e + 1], mid)
    on, onw = col(1.0, low), col(1.0, mid)
    tcx, tcy = c["tcx"], c["tcy"]

    def at(f, dk=0, dj=0, di=0):
        return f[1 + dk:1 + dk + e - k + 1, 1 + dj:f.shape[1] - 1 + dj, 1 + di:f.shape[2] - 1 + di]

    u0, v0, w0 = at(u), at(v), at(w)
    ue, uw, un, us, uu, ud = (at(u, di=1), at(u, di=-1), at(u, dj=1), at(u, dj=-1), at(u, dk=1), at(u, dk=-1))
    ve, vw, vn, vs, vu, vd = (at(v, di=1), at(v, di=-1), at(v, dj=1), at(v, dj=-1), at(v, dk=1), at(v, dk=-1))
    we, ww, wn, ws, wu, wd = (at(w, di=1), at(w, di=-1), at(w, dj=1), at(w, dj=-1), at(w, dk=1), at(w, dk=-1))
    su = on * (tcx * (uw * (u0 + uw) - ue * (u0 + ue)) + tcy * (us * (vs + at(v, 0, -1, 1)) - un * (v0 + ve)))
    su = su + z1 * (ud * (wd + at(w, -1, 0, 1))) - z2 * (uu * (w0 + we))
    sv = on * (tcx * (vw * (uw + at(u, 0, 1, -1)) - ve * (u0 + un)) + tcy * (vs * (v0 + vs) - vn * (v0 + vn)))
    sv = sv + z1 * (vd * (wd + at(w, -1, 1, 0))) - z2 * (vu * (w0 + wn))
    sw = onw * (tcx * (ww * (uw + at(u, 1, 0, -1)) - we * (u0 + uu)) + tcy * (ws * (vs + at(v, 1, -1, 0)) - wn * (v0 + vu)))
    sw = sw + d1 * (wd * (w0 + wd)) - d2 * (wu * (w0 + wu))
    return su, sv, sw


def _slabs(nz, n):
    return [(k, min(nz, k + n - 1)) for k in range(1, nz + 1, n)]


def _all_sources(q, c):
    nz = q[0].shape[0] - 2
    out = [torch.empty((nz,) + tuple(n - 2 for n in f.shape[1:]), dtype=torch.float64, device=f.device) for f in q]
    for k, e in _slabs(nz, 4):
        for t, s in zip(out, _sources([f[k - 1:e + 2] for f in q], c, k, e, nz)):
            t[k - 1:e] = s
    return out


def _euler(q, c):
    out = []
    for f, t in zip(q, _all_sources(q, c)):
        n = f.clone()
        n[1:-1, 1:-1, 1:-1] += t
        out.append(_wrap(n))
    return out


def _transposed(q, lam, c, periodic):
    """J(q)^T l for l given on the interior, dense arrays in and out; folded onto the interior when periodic."""
    nz = q[0].shape[0] - 2
    grads = [torch.zeros_like(f) for f in q]
    for k, e in _slabs(nz, 8):
        slab = [f[k - 1:e + 2].detach().clone().requires_grad_(True) for f in q]
        loss = sum((s * l[k - 1:e]).sum() for s, l in zip(_sources(slab, c, k, e, nz), lam))
        for g, d in zip(grads, torch.autograd.grad(loss, slab)):
            g[k - 1:e + 2] += d
    if periodic:
        for g in grads:   # the transpose of _wrap
            g[:, 1] += g[:, -1]
            g[:, -2] += g[:, 0]
            g[:, :, 1] += g[:, :, -1]
            g[:, :, -2] += g[:, :, 0]
    return grads


def _place(nx, ny, nz, dtype):
    """The default layout as its documentation gives it: (length, pitch_k, pitch_j, offset of i = 0) in elements.
    Interior rows start on 128-byte boundaries, rows are a multiple of 128 bytes long, one halo cell all round."""
    line = 128 // (4 if dtype == "f32" else 2)
    pj = -(-(line + nx + 1) // line) * line
    return pj * (ny + 2) * (nz + 2), pj * (ny + 2), pj, line - 1


def _exact_batch(case, seed):
    shapes, scale = _shapes(case), _scales(case) or (1.0,) * 6
    places = [_place(*s, case["dtype"]) for s in shapes]
    total = sum(-(-p[0] // LINE) * LINE for p in places)
    out = [torch.zeros(total, dtype=torch.float64, device="cuda") for _ in range(3)]
    start = 0
    for n, ((nx, ny, nz), (size, pk, pj, x0)) in enumerate(zip(shapes, places)):
        q = [_stored(f, case["dtype"], scale[i]) for i, f in enumerate(_turbulent(nx, ny, nz, seed * 1000 + n))]
        for o, t, f in zip(out, _all_sources(q, _column(nz)), scale[3:]):
            torch.as_strided(o, (nz, ny, nx), (pk, pj, 1), start + pk + pj + x0 + 1).copy_(t * f)
        start += -(-size // LINE) * LINE
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return _exact_batch(case, seed)
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    c, dtype, scale = _column(nz), case.get("dtype", "f32"), _scales(case) or (1.0,) * 6
    if kind == "tend":
        q = [_stored(f, dtype, s) for f, s in zip(_turbulent(nx, ny, nz, seed), scale)]
        return [t.mul_(s) for t, s in zip(_all_sources(q, c), scale[3:])]
    if kind == "step":
        q = [_stored(f, dtype, s) for f, s in zip(_smooth(nx, ny, nz, seed), scale)]
        for _ in range(case["nsteps"]):
            q = _euler(q, c)
        return [f[1:-1] / s for f, s in zip(q, scale)]
    if kind == "adjoint":
        q = [f.double() for f in _turbulent(nx, ny, nz, seed, wrap=case["periodic"])]
        lam = [(f * 0.1).double() for f in _turbulent(nx, ny, nz, seed + (1 << 30), wrap=False)]
        g = _transposed(q, [l[1:-1, 1:-1, 1:-1] for l in lam], c, case["periodic"])
        cut = (lambda f: f[1:-1, 1:-1, 1:-1]) if case["periodic"] else (lambda f: f[1:-1])
        return [cut(a + l) if case["add"] else cut(a) for a, l in zip(g, lam)]
    states = [[f.double() for f in _smooth(nx, ny, nz, seed)]]
    for _ in range(case["nsteps"]):
        states.append(_euler(states[-1], c))
    final = [f[1:-1, 1:-1, 1:-1].clone() for f in states.pop()]
    target = _smooth(nx, ny, nz, seed + (1 << 30))[0][1:-1, 1:-1, 1:-1].double()
    lam = [final[0] - target, torch.zeros_like(target), torch.zeros_like(target)]
    for q in reversed(states):
        g = _transposed(q, lam, c, True)
        lam = [l + t[1:-1, 1:-1, 1:-1] for l, t in zip(lam, g)]
    return final, lam
