"""Kernels that march along z and keep values between planes, at the sizes and
displacements where that can go wrong, against the FP64 oracle.

Tolerance: as in the parity tests, 1e-5 of the reference's scale for values
that a few dozen FP32 operations form (about 6e-8 relative rounding each).
"""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - CPU container
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1301_0970_gb300 as cg  # noqa: E402

DEV = torch.device("cuda:0")


@pytest.fixture(scope="module")
def ctx():
    with cg.Context(0) as c:
        yield c


def field(kind, shape, rng):
    """Displacements [3][nz][ny][nx]: slowly varying (the cell moves up by one
    plane from voxel to voxel), jumping (it does not), or beyond the border."""
    nz, ny, nx = shape
    z, y, x = np.meshgrid(np.arange(nz), np.arange(ny), np.arange(nx), indexing="ij")
    if kind == "smooth":
        u = np.stack([1.3 * np.sin(0.21 * x + 0.13 * z), 0.9 * np.cos(0.17 * y) + 0.4, -0.7 + 0.05 * z])
    elif kind == "jumping":
        u = rng.uniform(-2.5, 2.5, (3, nz, ny, nx))
    else:
        u = np.stack([np.full(shape, 2.0 * nx), np.full(shape, -3.0), np.where(z % 2 == 0, 1.5 * nz, -1.5 * nz)])
    return u.astype(np.float32)


@pytest.mark.parametrize("kind", ["smooth", "jumping", "outside"])
@pytest.mark.parametrize("shape", [(1, 5, 36), (2, 9, 33), (3, 8, 32), (9, 10, 65), (70, 6, 40)])
def test_force_warp_pass(ctx, shape, kind):
    """I0~ of the force step (its `warped` output), structure terms on and off."""
    rng = np.random.default_rng(hash_of(shape))
    img = rng.uniform(-1000, 700, shape).astype(np.float32)
    u = field(kind, shape, rng)
    bits = rng.integers(0, 4, shape, dtype=np.uint8)
    ref = oracle.warp(img, u)
    d = [torch.from_numpy(a).to(DEV) for a in (img, u, bits)]
    for contour in (False, True):
        out = torch.empty_like(d[0])
        ctx.force(d[0], d[0], d[2], d[2], [1e-3] * 2, [1, -1], d[1], contour=contour, warped=out)
        torch.cuda.synchronize()
        err = np.abs(out.cpu().numpy().astype(np.float64) - ref).max()
        assert err <= 1e-5 * np.abs(img).max(), (contour, err)


def smooth_ctx(variant):
    import os
    old = os.environ.get("CGDIR_SMOOTH")
    os.environ["CGDIR_SMOOTH"] = variant
    try:
        return cg.Context(0)
    finally:
        if old is None:
            del os.environ["CGDIR_SMOOTH"]
        else:
            os.environ["CGDIR_SMOOTH"] = old


@pytest.mark.parametrize("sigma", [0.3, 0.6, 1.0, 1.3, 1.6, 2.0])      # radii 1 .. 6
@pytest.mark.parametrize("shape", [(1, 1, 1), (3, 2, 4), (2, 33, 12), (9, 32, 32), (5, 65, 36), (17, 31, 64),
                                   (40, 70, 100), (9, 34, 33), (23, 67, 45), (6, 5, 130)])
def test_smooth_march_equals_tile_kernel(shape, sigma):
    """The z-march (32 x 32 and 32 x 16 tiles; TMA where nx % 4 == 0, else
    4-byte copies) has the tile kernel's order of operations, so the same
    bits: partial tiles in every axis, volumes thinner than the filter, one
    component and three, and a field that is not 16-byte aligned."""
    rng = np.random.default_rng(hash_of(shape))
    f = torch.from_numpy(rng.normal(0, 3, (3,) + shape).astype(np.float32)).to(DEV)
    off = torch.empty(f.numel() + 1, device=DEV)[1:].view(f.shape)
    off.copy_(f)
    got = {}
    for variant in ("tile", "march", "march32"):
        with smooth_ctx(variant) as c:
            got[variant] = [c.smooth(f, sigma), c.smooth(f[1].contiguous(), sigma), c.smooth(off, sigma)]
            c.sync()
    for variant in ("march", "march32"):
        for a, b in zip(got["tile"], got[variant]):
            assert torch.equal(a, b)


def hash_of(shape):
    return shape[0] * 10007 + shape[1] * 101 + shape[2]


@pytest.mark.parametrize("dtype", [torch.float32, torch.float16])
@pytest.mark.parametrize("shape", [(1, 3, 4), (9, 21, 44), (30, 40, 64), (33, 50, 200), (70, 90, 128), (13, 22, 45), (21, 30, 70)])
def test_small_level_schedule_keeps_histories(shape, dtype, monkeypatch):
    """The untuned schedule of small levels (narrow threads, short chunks, the
    sums' chains taken up by other threads, the fused tile kernels) against the
    four-voxel / per-step one: DVF and RMS-ID histories bit for bit, structure
    terms on, over the schedule's size classes and a width that is no multiple
    of four."""
    rng = np.random.default_rng(hash_of(shape))
    img = rng.normal(0, 300, shape).astype(np.float32)
    mov = torch.from_numpy(img + rng.normal(0, 40, shape).astype(np.float32)).to(DEV, dtype)
    img = torch.from_numpy(img).to(DEV, dtype)
    masks = [torch.from_numpy((rng.random(shape) < p).astype(np.uint8)).to(DEV) for p in (0.02, 0.5)]
    kw = dict(levels=1, iters=[4], lam=[1e-3, 0.5], sign=[1, -1], stop_mode=cg.CGDIR_STOP_FIXED)
    out = []
    for env in ({}, {"CGDIR_SMOOTH": "march"}, {"CGDIR_SMOOTH": "tile", "CGDIR_FORCE_ZCHUNK": str(default_zchunk(shape))}):
        for name, v in env.items():
            monkeypatch.setenv(name, v)
        with cg.Context(0) as c:
            out.append(c.register(img, mov, masks, masks, **kw))
        for name in env:
            monkeypatch.delenv(name)
    for dvf, stats in out[1:]:
        assert torch.equal(dvf, out[0][0])
        assert stats[0]["rms_id"] == out[0][1][0]["rms_id"]


def default_zchunk(shape):
    """The chunk of the widest thread's pass: two CTAs per SM and four waves of
    128-wide tiles (at least 4 planes), or four and two of 32-wide ones."""
    nz, ny, nx = shape
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    tiles = -(-(nx // 4 if nx % 4 == 0 else nx) // 32) * -(-ny // 8)
    chunks = max(1, min(nz, -(-8 * sms // tiles)))
    zc = -(-nz // chunks)
    return max(min(4, nz), zc) if nx % 4 == 0 else zc


@pytest.mark.parametrize("shape", [(5, 7, 9), (24, 59, 53), (33, 65, 67), (40, 91, 107)])
@pytest.mark.parametrize("sigma", [0.5, 1.0, 2.0])
def test_rows_without_tma_take_the_split_kernels_with_the_same_bits(monkeypatch, shape, sigma):
    """The default for nx % 4 != 0 (split kernels where there is a scratch
    field, tiles or the z-march without one) against the z-march: every
    variant sums its taps in one order, so the results are equal."""
    torch.manual_seed(3)
    du = torch.randn((3,) + shape, device="cuda")
    u = 2 * torch.randn((3,) + shape, device="cuda")
    got = []
    for forced in (None, "march"):
        if forced:
            monkeypatch.setenv("CGDIR_SMOOTH", forced)
        with cg.Context(0) as ctx:
            got.append([ctx.smooth_compose(du, u, sigma=sigma), ctx.smooth(du, sigma),
                        ctx.smooth(du[0].contiguous(), sigma)])
            ctx.sync()
    for a, b in zip(*got):
        assert torch.equal(a, b)


@pytest.mark.parametrize("limit_us", [200, 1000])
def test_march_reports_a_plane_that_never_arrives(limit_us):
    """Every plane's wait is reported, also in the last turn of the plane loop
    (the self-test withholds the first, a middle and the last plane of chunks of
    1 and 20 planes, by TMA and by asynchronous copies), and the context and its
    smoothing work afterwards."""
    f = torch.randn(3, 20, 32, 32, device=DEV)
    with cg.Context(0, mem_budget_bytes=1) as c:      # nothing of it counts as the context's memory
        want = c.smooth(f, 1.0)
        assert c.selftest_wait_timeout(limit_us) == cg.CGDIR_ETIMEDOUT
        got = c.smooth(f, 1.0)
        c.sync()
    assert torch.equal(got, want)


@pytest.mark.parametrize("shape", [(100000, 1, 1), (90000, 9, 9), (200000, 1, 1), (270000, 1, 4)])
def test_volumes_deeper_than_a_grid_of_slabs(shape, monkeypatch):
    """Thin volumes of more z slabs than a grid's z extent holds run, with the
    z-march's bits, in every step that smooths, and so do their force steps."""
    torch.manual_seed(1)
    du = torch.randn((3,) + shape, device=DEV)
    u = torch.randn((3,) + shape, device=DEV)
    img = torch.randn(shape, device=DEV)
    bits = torch.randint(0, 2, shape, device=DEV, dtype=torch.uint8)
    got = []
    for forced in (None, "split", "march"):
        if forced:
            monkeypatch.setenv("CGDIR_SMOOTH", forced)
        with cg.Context(0) as c:
            got.append([c.smooth_compose(du, u, sigma=1.0), c.smooth(du, 1.0),
                        c.iterate(img, img, bits, bits, [1e-3], [1], u, contour=True)])
            c.sync()
    for other in got[:2]:
        for a, b in zip(other, got[2]):
            assert torch.equal(a, b)


@pytest.mark.parametrize("shape", [(21, 33, 63), (43, 61, 127)])
def test_unaligned_coarse_level_keeps_its_history(shape, monkeypatch):
    """A coarse level with whole quads in fields that start at no quad's
    boundary (the finest level has an odd number of voxels): its RMS-ID history
    with structure terms is the one of the default chunk."""
    rng = np.random.default_rng(hash_of(shape))
    img = rng.normal(0, 300, shape).astype(np.float32)
    mov = torch.from_numpy(img + rng.normal(0, 40, shape).astype(np.float32)).to(DEV)
    img = torch.from_numpy(img).to(DEV)
    masks = [torch.from_numpy((rng.random(shape) < 0.3).astype(np.uint8)).to(DEV)]
    kw = dict(levels=2, iters=[4, 1], lam=[1e-3], sign=[1], contour_level_mask=3, stop_mode=cg.CGDIR_STOP_FIXED)
    coarse = tuple((n + 1) // 2 for n in shape)
    got = []
    for zc in (None, default_zchunk(coarse)):
        if zc:
            monkeypatch.setenv("CGDIR_FORCE_ZCHUNK", str(zc))
        with cg.Context(0) as c:
            got.append(c.register(img, mov, masks, masks, **kw))
    assert torch.equal(got[0][0], got[1][0])
    assert got[0][1][0]["rms_id"] == got[1][1][0]["rms_id"]


@pytest.mark.parametrize("nx", [6, 32, 34])
@pytest.mark.parametrize("which", ["T0", "du", "uroi", "sbits"])
def test_force_on_views_that_start_at_an_odd_element(ctx, nx, which):
    """Force fields that are views one element into their storage (no pair of
    voxels is aligned): the same du and the same count as for aligned copies,
    the RMS sum to the rounding of its FP32 parts (a few dozen terms each)."""
    shape = (7, 9, nx)
    gen = torch.Generator(device=DEV).manual_seed(nx)
    img, mov = (300 * torch.randn(shape, device=DEV, generator=gen) for _ in range(2))
    bits = torch.randint(0, 4, shape, device=DEV, dtype=torch.uint8, generator=gen)
    uroi = torch.randint(0, 2, shape, device=DEV, dtype=torch.uint8, generator=gen)
    u = torch.randn((3,) + shape, device=DEV, generator=gen)

    def run(odd):
        a = {"T0": img, "du": torch.empty_like(u), "uroi": uroi, "sbits": bits}
        if odd:
            t = torch.empty(a[which].numel() + 1, device=DEV, dtype=a[which].dtype)[1:].view(a[which].shape)
            a[which] = t.copy_(a[which])
        return ctx.force(mov, a["T0"], bits, a["sbits"], [1e-3] * 2, [1, -1], u, uroi=a["uroi"], du=a["du"],
                         want_stats=True)

    (du, st), (want, wst) = run(True), run(False)
    assert torch.equal(du, want)
    assert st[1] == wst[1] and st[2] == wst[2]
    assert abs(st[0] - wst[0]) <= 64 * 2.0 ** -24 * wst[0]


@pytest.mark.parametrize("kernels", ["plain", "fused"])
@pytest.mark.parametrize("shape", [(9, 21, 44), (30, 40, 64), (13, 22, 45)])
def test_other_kernel_families_keep_the_default_chunk(shape, kernels, monkeypatch):
    """The plain and the one-pass force kernels run small levels with the
    default chunk: histories and statistics bit for bit."""
    rng = np.random.default_rng(hash_of(shape))
    img = rng.normal(0, 300, shape).astype(np.float32)
    mov = torch.from_numpy(img + rng.normal(0, 40, shape).astype(np.float32)).to(DEV)
    img = torch.from_numpy(img).to(DEV)
    masks = [torch.from_numpy((rng.random(shape) < 0.3).astype(np.uint8)).to(DEV)]
    u = torch.from_numpy(rng.normal(0, 1, (3,) + shape).astype(np.float32)).to(DEV)
    monkeypatch.setenv("CGDIR_KERNELS", kernels)
    got = []
    for zc in (None, default_zchunk(shape)):
        if zc:
            monkeypatch.setenv("CGDIR_FORCE_ZCHUNK", str(zc))
        with cg.Context(0) as c:
            dvf, st = c.register(img, mov, masks, masks, levels=1, iters=[4], lam=[1e-3], sign=[1],
                                 stop_mode=cg.CGDIR_STOP_FIXED)
            _, stats = c.force(mov, img, masks[0], masks[0], [1e-3], [1], u, want_stats=True)
            got.append((dvf, st[0]["rms_id"], stats))
    assert torch.equal(got[0][0], got[1][0])
    assert got[0][1:] == got[1][1:]


def test_unaligned_coarse_level_takes_the_split_kernels():
    """A coarse level with nx % 4 == 0 whose fields are not 16-byte aligned (the
    finest level has an odd number of voxels) cannot load them by TMA: six
    kernels an iteration (two force passes, two smoothings in two) and not the
    fused tiles' three."""
    shape = (67, 71, 127)
    img = torch.randn(shape, device=DEV)
    with cg.Context(0) as c:
        count = []
        for n in (10, 30):
            kw = dict(levels=2, iters=[n, 1], lam=[], sign=[], stop_mode=cg.CGDIR_STOP_FIXED)
            c.register(img, img, [], [], **kw)
            before = cg.launch_count()
            c.register(img, img, [], [], **kw)
            count.append(cg.launch_count() - before)
    assert count[1] - count[0] == 20 * 6


@pytest.mark.parametrize("shape", [(16, 94, 72), (30, 40, 64), (40, 64, 128)])
def test_largest_step_does_not_depend_on_the_pass(shape, monkeypatch):
    """max |du| of the force step with structure terms on small levels, whose
    threads are narrower than the four-voxel ones they stand for: equal to that
    pass's, bit for bit."""
    got = []
    for zc in (None, default_zchunk(shape)):
        if zc:
            monkeypatch.setenv("CGDIR_FORCE_ZCHUNK", str(zc))
        with cg.Context(0) as c:
            for seed in range(40):
                gen = torch.Generator(device=DEV).manual_seed(seed)
                img, mov = (300 * torch.randn(shape, device=DEV, generator=gen) for _ in range(2))
                bits = torch.randint(0, 2, shape, device=DEV, dtype=torch.uint8, generator=gen)
                u = torch.randn((3,) + shape, device=DEV, generator=gen)
                got.append(c.force(mov, img, bits, bits, [1e-3], [1], u, want_stats=True)[1])
    assert got[:40] == got[40:]
