"""Timed cases of the CG-DIR library: whole registrations, a batch, and the
steps that a caller's own loop runs, each through the public Python API.

Whole registrations are most of what a user asks for, from the 64 x 64 x 32
test volume to the 512 x 512 x 160 pelvic case; the step primitives are what a
program with its own iteration loop calls.  Inputs are layered ellipsoid
phantoms with CT values, edges half a voxel wide and Gaussian noise; the
moving image is the same anatomy displaced by a few Gaussian bumps.  The
displacement fields handed to the step primitives are such bumps plus the
small correlated fluctuation that the noise of the images leaves in a field
while it is being optimised.

`exact` restates Algorithm A of arXiv:1301.0970 in FP64 torch.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1301_0970_gb300 as cg

SPACING, MARGIN, OFFSET = (1.97, 1.97, 2.5), 10.0, 1000.0
DTYPES = {"f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}
BATCH = [(64, 128, 128, 2), (64, 128, 128, 4), (96, 256, 256, 3), (96, 256, 256, 5), (128, 384, 384, 7),
         (160, 512, 512, 6)]


def listed():
    return [
        # the smallest whole call: one level, two structures, as a test or a cropped organ
        {"name": "reg_phantom64", "do": "register", "nz": 32, "ny": 64, "nx": 64, "k": 2, "levels": 1, "iters": "100",
         "lam": 1.0, "dtype": "f32", "tuned": False, "auto_sign": True},
        # the paper's head-and-neck case HN4 with its two levels, in a program that calls register() and no tuner
        {"name": "reg_paper_hn4", "do": "register", "nz": 70, "ny": 160, "nx": 240, "k": 3, "levels": 2,
         "iters": "100,50", "lam": 1e-3, "dtype": "f32", "tuned": False, "auto_sign": True},
        # the head-and-neck workload on a tuned context (a clinic's server keeps one)
        {"name": "reg_headneck256", "do": "register", "nz": 96, "ny": 256, "nx": 256, "k": 5, "levels": 3,
         "iters": "100,50,25", "lam": 1e-3, "dtype": "f32", "tuned": True, "auto_sign": False},
        # the largest single registration, tuned
        {"name": "reg_pelvis512", "do": "register", "nz": 160, "ny": 512, "nx": 512, "k": 6, "levels": 3,
         "iters": "100,50,25", "lam": 1e-3, "dtype": "f32", "tuned": True, "auto_sign": False},
        # 16-bit image storage with the most structures, signs decided by the library
        {"name": "reg_384_f16", "do": "register", "nz": 128, "ny": 384, "nx": 384, "k": 8, "levels": 3,
         "iters": "100,50,25", "lam": 1e-3, "dtype": "f16", "tuned": False, "auto_sign": True},
        # a cropped volume of odd sizes: no vector width divides a row
        {"name": "reg_odd_bf16", "do": "register", "nz": 67, "ny": 141, "nx": 189, "k": 4, "levels": 2,
         "iters": "60,30", "lam": 1e-3, "dtype": "bf16", "tuned": False, "auto_sign": True},
        # many patients at once: uneven sizes in one call, 16-bit images
        {"name": "batch_mix_f16", "do": "batch", "cases": 6, "levels": 3, "iters": "100,50,25", "lam": 1e-3,
         "dtype": "f16"},
        # a caller's own loop at full size: one iteration with structure terms
        {"name": "iterate_pelvis512", "do": "iterate", "nz": 160, "ny": 512, "nx": 512, "k": 6, "contour": True},
        # the same loop at a coarse level: plain demons, where launches count
        {"name": "iterate_demons128", "do": "iterate", "nz": 64, "ny": 128, "nx": 128, "k": 0, "contour": False},
        # the moving-vector step alone, with the stopping metric
        {"name": "force_256", "do": "force", "nz": 96, "ny": 256, "nx": 256, "k": 5, "contour": True},
        # fluid smoothing and composite update of an odd-sized field
        {"name": "smooth_compose_odd", "do": "smooth_compose", "nz": 91, "ny": 217, "nx": 181, "sigma": 1.0},
        # everything a program prepares before its own loop, and the metric after it
        {"name": "setup_256", "do": "setup", "nz": 96, "ny": 256, "nx": 256, "k": 5},
    ]


def draw(rng):
    def size(lo, hi, odd=0.3):
        v = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
        return v | 1 if rng.random() < odd else max(lo, v // 8 * 8)

    kind = rng.choice(["register", "register", "register", "iterate", "iterate", "force", "smooth_compose", "setup",
                       "batch"])
    nz, ny, nx = size(24, 144), size(48, 448), size(48, 448)
    k = rng.randint(1, 8)
    if kind == "register":
        levels = rng.randint(1, 3)
        iters = ",".join(str(rng.choice([100, 60, 40]) // 2 ** l) for l in range(levels))
        return {"do": kind, "nz": nz, "ny": ny, "nx": nx, "k": k, "levels": levels, "iters": iters,
                "lam": rng.choice([1e-3, 1.0]), "dtype": rng.choice(["f32", "f32", "f16", "bf16"]),
                "tuned": rng.random() < 0.4, "auto_sign": rng.random() < 0.5}
    if kind == "batch":
        return {"do": kind, "cases": rng.randint(2, 5), "levels": rng.randint(2, 3),
                "iters": rng.choice(["100,50,25", "60,30,15", "40,20,10"]), "lam": 1e-3,
                "dtype": rng.choice(["f32", "f16", "bf16"])}
    if kind in ("iterate", "force"):
        contour = rng.random() < 0.7
        return {"do": kind, "nz": nz, "ny": ny, "nx": nx, "k": k if contour else 0, "contour": contour}
    if kind == "smooth_compose":
        return {"do": kind, "nz": nz, "ny": ny, "nx": nx, "sigma": rng.choice([1.0, 1.0, 0.6, 1.5])}
    return {"do": kind, "nz": nz, "ny": ny, "nx": nx, "k": k}


# ---- inputs -----------------------------------------------------------------
def _grid(shape, dtype=torch.float32):
    nz, ny, nx = shape
    ax = [torch.arange(n, device="cuda", dtype=dtype) for n in (nx, ny, nz)]
    return ax[0].view(1, 1, nx), ax[1].view(1, ny, 1), ax[2].view(nz, 1, 1)


def _bumps(shape, rng, count=6):
    """A smooth displacement [3][nz][ny][nx]: Gaussian bumps of at most 8 voxels, gradient at most about 0.4."""
    nz, ny, nx = shape
    x, y, z = _grid(shape)
    u = torch.zeros((3,) + tuple(shape), device="cuda")
    for _ in range(count):
        c = rng.uniform(0.25, 0.75, 3) * (nx, ny, nz)
        s = rng.uniform(0.12, 0.25) * min(nx, ny, max(nz, 24))
        amp = rng.uniform(-1, 1, 3) * min(4.0, 0.25 * s)
        g = torch.exp(-((x - c[0]) ** 2 + (y - c[1]) ** 2) / (2 * s * s)) * torch.exp(-(z - c[2]) ** 2 / (2 * s * s))
        for a in range(3):
            u[a] += float(amp[a]) * g
    return u


def _anatomy(shape, d, k, rng, gen):
    """CT volume and k masks of the phantom seen at x - d(x) (d None: at x), with noise."""
    nz, ny, nx = shape
    x, y, z = _grid(shape)
    if d is not None:
        x, y, z = x - d[0], y - d[1], z - d[2]

    def occ(c, r):
        q = torch.sqrt(((x - c[0] * nx) / (r[0] * nx)) ** 2 + ((y - c[1] * ny) / (r[1] * ny)) ** 2 +
                       ((z - c[2] * nz) / (r[2] * nz)) ** 2 + 1e-12)
        dist = (1 - q) * min(r[0] * nx, r[1] * ny, r[2] * nz)
        return torch.sigmoid(dist / 0.5), dist > 0

    img = torch.full(shape, -1000.0, device="cuda")
    body, _ = occ((0.5, 0.5, 0.5), (0.44, 0.40, 0.60))
    img += body * 950.0
    outer, _ = occ((0.5, 0.5, 0.5), (0.30, 0.27, 0.45))
    inner, _ = occ((0.5, 0.5, 0.5), (0.26, 0.23, 0.40))
    img += (outer - inner) * 750.0
    del body, outer, inner
    masks = []
    for j in range(k):
        a = 2 * math.pi * j / max(k, 1) + float(rng.uniform(-0.2, 0.2))
        c = (0.5 + 0.15 * math.cos(a), 0.5 + 0.14 * math.sin(a), 0.5 + float(rng.uniform(-0.08, 0.08)))
        r = tuple(float(v) for v in rng.uniform(0.045, 0.075, 2)) + (float(rng.uniform(0.10, 0.16)),)
        o, m = occ(c, r)
        img += o * (45.0 if j % 2 == 0 else -40.0)
        masks.append(m.to(torch.uint8).contiguous())
    img += 25.0 * torch.randn(shape, device="cuda", generator=gen)
    return img, masks


def _pair(shape, k, dtype, seed):
    """Static and moving volume with their masks."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    d = _bumps(shape, np.random.default_rng(seed))
    static, sm = _anatomy(shape, None, k, np.random.default_rng(seed + 1), gen)
    moving, mm = _anatomy(shape, d, k, np.random.default_rng(seed + 1), gen)
    return static.to(DTYPES[dtype]), moving.to(DTYPES[dtype]), sm, mm


def _field(shape, seed, scale=1.0):
    """A displacement field as an iteration meets it: bumps and correlated noise of about 0.1 voxel."""
    gen = torch.Generator(device="cuda").manual_seed(seed + 7)
    u = _bumps(shape, np.random.default_rng(seed + 7))
    for a in range(3):
        n = torch.randn((1, 1) + tuple(shape), device="cuda", generator=gen)
        for _ in range(2):
            n = torch.nn.functional.avg_pool3d(n, 3, 1, 1, count_include_pad=False)
        u[a] += 1.2 * n[0, 0]
    return (scale * u).contiguous()


def _shape(case):
    return case["nz"], case["ny"], case["nx"]


def _iters(case):
    return [int(v) for v in case["iters"].split(",")][-case["levels"]:]


def _batch_specs(case):
    return [BATCH[i] for i in (range(len(BATCH)) if case["cases"] >= len(BATCH) else range(case["cases"]))]


def _signs(k):
    return [1 if j % 2 == 0 else -1 for j in range(k)]


def _reg_kw(case, k):
    return dict(levels=case["levels"], iters=_iters(case), lam=[case["lam"]] * k, spacing_mm=SPACING,
                margin_mm=MARGIN, sign=None if case.get("auto_sign", True) else _signs(k),
                stop_mode=cg.CGDIR_STOP_FIXED)


def prepare(case, seed):
    do = case["do"]
    ctx = cg.Context(0)
    st = {"case": case, "ctx": ctx}
    if do == "batch":
        st["cases"] = []
        for i, (nz, ny, nx, k) in enumerate(_batch_specs(case)):
            s, m, sm, mm = _pair((nz, ny, nx), k, case["dtype"], seed * 64 + i)
            st["cases"].append(dict(static=s, moving=m, static_masks=sm, moving_masks=mm, **_reg_kw(case, k)))
        return st
    shape = _shape(case)
    if do == "smooth_compose":
        st.update(u=_field(shape, seed), du=_field(shape, seed + 1, 0.3),
                  out=torch.empty((3,) + shape, device="cuda"))
        return st
    k = case["k"]
    st["pair"] = s, m, sm, mm = _pair(shape, k, case.get("dtype", "f32"), seed)
    if do == "register":
        if case["tuned"]:
            ctx.autotune(shape, k, case["levels"],
                         storage_dtype={"f32": cg.CGDIR_F32, "f16": cg.CGDIR_F16, "bf16": cg.CGDIR_BF16}[case["dtype"]])
        return st
    st["u"] = _field(shape, seed)
    if do == "setup":
        half = tuple((n + 1) // 2 for n in shape)
        st["uc"] = _field(half, seed + 3)
        return st
    if k:
        st["sbits"], st["mbits"] = ctx.pack_masks(sm), ctx.pack_masks(mm)
        st["uroi"] = ctx.uroi(st["sbits"], k, SPACING, MARGIN)
    else:
        st["sbits"] = st["mbits"] = st["uroi"] = None
    st["out"] = torch.empty((3,) + shape, device="cuda")
    return st


def run(st):
    case, ctx = st["case"], st["ctx"]
    do = case["do"]
    if do == "batch":
        return [_answer(r) for r in ctx.register_batch(st["cases"])]
    if do == "register":
        s, m, sm, mm = st["pair"]
        return _answer(ctx.register(s, m, sm, mm, **_reg_kw(case, case["k"])))
    if do == "smooth_compose":
        return ctx.smooth_compose(st["du"], st["u"], sigma=case["sigma"], out=st["out"])
    s, m, sm, mm = st["pair"]
    k = case["k"]
    if do == "iterate":
        return ctx.iterate(m, s, st["mbits"], st["sbits"], [1e-3] * k, _signs(k), st["u"], offset=OFFSET,
                           contour=case["contour"], uroi=st["uroi"], out=st["out"])
    if do == "force":
        du, stats = ctx.force(m, s, st["mbits"], st["sbits"], [1e-3] * k, _signs(k), st["u"], offset=OFFSET,
                              contour=case["contour"], uroi=st["uroi"], du=st["out"], want_stats=True)
        return du, np.array(stats)
    sb, mb = ctx.pack_masks(sm), ctx.pack_masks(mm)
    uroi = ctx.uroi(sb, k, SPACING, MARGIN)
    signs = ctx.auto_sign(s, sb, k)
    coarse = [ctx.restrict_image(s), ctx.restrict_image(m), ctx.restrict_bits(sb), ctx.restrict_bits(mb)]
    u = ctx.prolong(st["uc"], _shape(case))
    rms, count = ctx.rms_id(m, s, u, uroi)
    return {"bits": [sb, mb], "uroi": uroi, "signs": np.array(signs), "coarse": coarse, "u": u,
            "rms": rms, "count": count}


def _answer(r):
    dvf, stats = r
    return {"dvf": dvf, "iters": np.array([s["iters_run"] for s in stats]),
            "rms": [np.array(s["rms_id"]) for s in stats]}


# ---- what a pass cannot do without --------------------------------------------
_FLOPS = {"force": 110, "smooth": 3 * 3 * 14, "compose": 60}


def _work_reg(shape, k, levels, iters, esz):
    n = shape[0] * shape[1] * shape[2]
    b, f = n * (2 * esz + 2 * k + 12), 0
    dims = list(shape)
    for it in reversed(iters):
        v = dims[0] * dims[1] * dims[2]
        # an iteration reads and writes u and reads both images, the packed masks and the UROI
        b += it * v * (24 + 2 * esz + 3)
        f += it * v * (_FLOPS["force"] + 2 * _FLOPS["smooth"] + _FLOPS["compose"])
        dims = [(d + 1) // 2 for d in dims]
        esz = 4
    return b, f


def work(case):
    do = case["do"]
    if do == "batch":
        w = [_work_reg(s[:3], s[3], case["levels"], _iters(case), 4 if case["dtype"] == "f32" else 2)
             for s in _batch_specs(case)]
        return {"bytes": sum(v[0] for v in w), "flops": sum(v[1] for v in w)}
    shape = _shape(case)
    n = shape[0] * shape[1] * shape[2]
    if do == "register":
        b, f = _work_reg(shape, case["k"], case["levels"], _iters(case), 4 if case["dtype"] == "f32" else 2)
        return {"bytes": b, "flops": f}
    if do == "smooth_compose":
        return {"bytes": 36 * n, "flops": n * (_FLOPS["smooth"] + _FLOPS["compose"])}
    masks = 3 if case["k"] and do != "setup" else 0
    if do == "iterate":
        return {"bytes": n * (32 + masks), "flops": n * (_FLOPS["force"] + 2 * _FLOPS["smooth"] + _FLOPS["compose"])}
    if do == "force":
        return {"bytes": n * (32 + masks), "flops": n * _FLOPS["force"]}
    # setup: images, masks and the coarse field in; bits, UROI, coarse images and bits, the field out
    return {"bytes": n * (8 + 2 * case["k"] + 12 / 8 + 3 + 10 / 8 + 12), "flops": n * 80}


# ---- FP64 restatement -----------------------------------------------------------
def _taps(sigma):
    r = math.ceil(3 * sigma - 1e-9)
    w = np.exp(-np.arange(-r, r + 1) ** 2 / (2.0 * sigma * sigma))
    return r, w / w.sum()


def _smooth(f, sigma):
    r, w = _taps(sigma)
    for axis in (-1, -2, -3):
        n = f.shape[axis]
        g = torch.zeros_like(f)
        for j in range(-r, r + 1):
            i = (torch.arange(n, device=f.device) + j).clamp(0, n - 1)
            g += float(w[j + r]) * f.index_select(axis % f.dim(), i)
        f = g
    return f


def _corners(u):
    """Flat corner indices and weights of the points x + u(x)."""
    shape = u.shape[1:]
    nz, ny, nx = shape
    lo, hi, fr = [], [], []
    for p, n in zip((g + v for g, v in zip(_grid(shape, torch.float64), u)), (nx, ny, nz)):
        p = p.clamp(0, n - 1)
        f = p.floor()
        lo.append(f.to(torch.int64))
        hi.append((lo[-1] + 1).clamp(max=n - 1))
        fr.append(p - f)
    out = []
    for q in range(8):
        i = [(hi if q >> a & 1 else lo)[a] for a in range(3)]
        w = [(fr[a] if q >> a & 1 else 1 - fr[a]) for a in range(3)]
        out.append(((i[2] * ny + i[1]) * nx + i[0], w[0] * w[1] * w[2]))
    return out


def _at(f, corners):
    f = f.reshape(-1)
    return sum(w * f[i].to(torch.float64) for i, w in corners)


def _grad(f):
    out = []
    for axis in (2, 1, 0):
        n = f.shape[axis]
        i = torch.arange(n, device=f.device)
        out.append(0.5 * (f.index_select(axis, (i + 1).clamp(max=n - 1)) - f.index_select(axis, (i - 1).clamp(min=0))))
    return out


def _force64(i0, t0, mm, sm, lam, sign, u, uroi):
    """Eq. 7 and the UROI sums: du, sum of squares, count."""
    c = _corners(u)
    w0 = _at(i0, c)
    g = _grad(w0)
    r0 = t0 - w0
    g2 = g[0] ** 2 + g[1] ** 2 + g[2] ** 2
    gn = g2.sqrt()
    inv = torch.where(g2 > 0, 1 / gn.clamp(min=1e-300), torch.zeros_like(gn))
    n = [v * inv for v in g]
    num, den = gn * r0, g2.clone()
    for j in range(len(lam)):
        mi = _at((1 + 0.5 * sign[j] * mm[j].to(torch.float64)) * (i0 + OFFSET), c)
        gm = _grad(mi)
        a = gm[0] * n[0] + gm[1] * n[1] + gm[2] * n[2]
        r = (1 + 0.5 * sign[j] * sm[j].to(torch.float64)) * (t0 + OFFSET) - mi
        num += lam[j] * a * r
        den += lam[j] * a * a
    den += r0 * r0
    v = torch.where(den > 0, num / den.clamp(min=1e-300), torch.zeros_like(den))
    sq = r0 * r0
    return (torch.stack([v * x for x in n]), float(sq.sum() if uroi is None else sq[uroi].sum()),
            float(sq.numel() if uroi is None else uroi.sum()))


def _compose64(u, du):
    c = _corners(du)
    return torch.stack([du[a] + _at(u[a], c) for a in range(3)])


def _restrict64(f):
    for axis in range(3):
        n = f.shape[axis]
        i = torch.arange((n + 1) // 2, device=f.device) * 2
        f = 0.5 * (f.index_select(axis, i) + f.index_select(axis, (i + 1).clamp(max=n - 1)))
    return f


def _prolong64(uc, shape):
    for a, n in zip((3, 2, 1), reversed(shape)):
        c = uc.shape[a]
        p = ((torch.arange(n, device="cuda", dtype=torch.float64) + 0.5) / 2 - 0.5).clamp(0, c - 1)
        lo = p.floor().to(torch.int64)
        w = (p - lo).view([-1 if d == a else 1 for d in range(4)])
        uc = (1 - w) * uc.index_select(a, lo) + w * uc.index_select(a, (lo + 1).clamp(max=c - 1))
    return 2 * uc


def _uroi64(sm, spacing, margin):
    """Union of the masks dilated by the ellipsoid of `margin` mm."""
    m = torch.stack([v.bool() for v in sm]).any(0)
    nz, ny, nx = m.shape
    r = [int(margin / s) for s in spacing]
    pad = torch.nn.functional.pad(m, (r[0], r[0], r[1], r[1], r[2], r[2]))
    out = torch.zeros_like(m)
    for dz in range(-r[2], r[2] + 1):
        for dy in range(-r[1], r[1] + 1):
            for dx in range(-r[0], r[0] + 1):
                if (dx * spacing[0]) ** 2 + (dy * spacing[1]) ** 2 + (dz * spacing[2]) ** 2 <= margin ** 2:
                    out |= pad[r[2] + dz:r[2] + dz + nz, r[1] + dy:r[1] + dy + ny, r[0] + dx:r[0] + dx + nx]
    return out


def _signs64(t0, sm):
    out = []
    for m in sm:
        m = m.bool()
        shell = torch.nn.functional.max_pool3d(m[None, None].float(), 5, 1, 2)[0, 0].bool() & ~m
        ok = bool(m.any()) and bool(shell.any())
        out.append(1 if not ok or float(t0[m].mean()) >= float(t0[shell].mean()) else -1)
    return out


def _register64(static, moving, sm, mm, case):
    iters, L = _iters(case), case["levels"]
    t, i = [static.double()], [moving.double()]
    sml, mml = [sm], [mm]
    for _ in range(L - 1):
        t.insert(0, _restrict64(t[0]))
        i.insert(0, _restrict64(i[0]))
        sml.insert(0, [(_restrict64(m.double()) >= 0.5).to(torch.uint8) for m in sml[0]])
    signs = _signs64(t[-1], sm) if case.get("auto_sign", True) else _signs(len(sm))
    u, hist = torch.zeros((3,) + t[0].shape, device="cuda", dtype=torch.float64), []
    for l in range(L):
        if l:
            u = _prolong64(u, t[l].shape)
        f = 2.0 ** (L - 1 - l)
        uroi = _uroi64(sml[l], [s * f for s in SPACING], MARGIN)
        fine = l == L - 1
        h = []
        for _ in range(iters[l]):
            du, s, c = _force64(i[l], t[l], mm if fine else [], sm if fine else [], [case["lam"]] * (len(sm) * fine),
                                signs, u, uroi)
            h.append(math.sqrt(s / c) if c else 0.0)
            u = _smooth(_compose64(u, _smooth(du, 1.0)), 1.0)
        r = (t[l] - _at(i[l], _corners(u)))[uroi]
        h.append(float((r * r).mean().sqrt()) if r.numel() else 0.0)
        hist.append(np.array(h))
    return {"dvf": u, "iters": np.array(iters), "rms": hist}


def exact(case, seed):
    st = prepare(dict(case, tuned=False) if "tuned" in case else case, seed)
    do = case["do"]
    if do == "batch":
        return [_register64(c["static"], c["moving"], c["static_masks"], c["moving_masks"], case) for c in st["cases"]]
    if do == "register":
        return _register64(*st["pair"], case)
    if do == "smooth_compose":
        return _compose64(st["u"].double(), _smooth(st["du"].double(), case["sigma"]))
    s, m, sm, mm = st["pair"]
    s, m, u, k = s.double(), m.double(), st["u"].double(), case["k"]
    if do == "setup":
        u = _prolong64(st["uc"].double(), _shape(case))
        uroi = _uroi64(sm, SPACING, MARGIN)
        r = (s - _at(m, _corners(u)))[uroi]

        def pack(masks):
            return sum(v.to(torch.uint8) << j for j, v in enumerate(masks))
        return {"bits": [pack(sm), pack(mm)], "uroi": uroi.to(torch.uint8), "signs": np.array(_signs64(s, sm)),
                "coarse": [_restrict64(s), _restrict64(m)] +
                          [pack([(_restrict64(v.double()) >= 0.5).to(torch.uint8) for v in w]) for w in (sm, mm)],
                "u": u, "rms": float((r * r).mean().sqrt()) if r.numel() else 0.0, "count": int(uroi.sum())}
    uroi = None if st["uroi"] is None else st["uroi"].bool()
    du, ssd, count = _force64(m, s, mm, sm, [1e-3] * k, _signs(k), u, uroi)
    if do == "force":
        return du, np.array([ssd, count, float((du * du).sum(0).max().sqrt())])
    return _smooth(_compose64(u, _smooth(du, 1.0)), 1.0)
