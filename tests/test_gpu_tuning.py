"""The tuner's choices and the sums that go with them."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - CPU container
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1301_0970_gb300 as cg  # noqa: E402

DEV = torch.device("cuda:0")


def pair(shape, seed=5, p=(0.02, 0.3)):
    """Static and moving image and the masks of len(p) structures."""
    rng = np.random.default_rng(seed)
    img = rng.normal(0, 300, shape).astype(np.float32)
    mov = img + rng.normal(0, 40, shape).astype(np.float32)
    masks = [torch.from_numpy((rng.random(shape) < q).astype(np.uint8)).to(DEV) for q in p]
    return torch.from_numpy(img).to(DEV), torch.from_numpy(mov).to(DEV), masks


def register(ctx, data, **more):
    img, mov, masks = data
    kw = dict(levels=1, iters=[6], lam=[1e-3] * len(masks), sign=([1, -1] * 4)[:len(masks)],
              stop_mode=cg.CGDIR_STOP_FIXED)
    kw.update(more)
    return ctx.register(img, mov, masks, masks, **kw)


def test_tuned_histories_do_not_follow_timing_noise():
    """A level without structure terms whose chunks of 4 (the default) and 8
    planes are 5 % apart as a registration runs them, and tie when each launch
    waits for the host: every tuning keeps the default, and with it the untuned
    sums, bit for bit."""
    data = pair((40, 128, 128))
    with cg.Context(0) as c:
        dvf, st = register(c, data, contour_level_mask=0)
    for _ in range(3):
        with cg.Context(0) as c:
            c.autotune((40, 128, 128), 2, 1, contour_level_mask=0)
            got, gst = register(c, data, contour_level_mask=0)
        assert torch.equal(got, dvf)
        assert gst[0]["rms_id"] == st[0]["rms_id"]


def test_a_table_fixes_the_histories():
    """One table gives one history, in any context and with any smoothing."""
    shape = (12, 48, 64)
    data = pair(shape)
    with cg.Context(0) as c:
        tab = c.autotune(shape, 2, 1)
        want = register(c, data)
    for smooth in ("march", "tile", "fused"):
        with cg.Context(0) as c:
            c.load_tuning([dict(t, smooth=smooth, smooth_zchunk=0) for t in tab])
            got = register(c, data)
        assert torch.equal(got[0], want[0])
        assert got[1][0]["rms_id"] == want[1][0]["rms_id"]


@pytest.mark.parametrize("shape", [(12, 48, 48), (24, 64, 64), (30, 60, 100), (24, 62, 54), (34, 71, 95), (40, 96, 160)])
@pytest.mark.parametrize("k", [0, 2])
def test_no_choice_is_slower_than_the_untuned_one(shape, k):
    """By the tuner's own times, with and without structure terms, on levels
    whose untuned schedule is the fused one, the split kernels or narrow force
    threads."""
    with cg.Context(0) as c:
        for t in c.autotune(shape, k, 1):
            assert t["smooth_ms"] + t["force_ms"] <= (t["default_smooth_ms"] + t["default_force_ms"]) * 1.0001 + 1e-6


@pytest.mark.parametrize("fluid, diff, kernels", [(1.0, 1.0, 3), (1.0, 0.0, 4), (0.0, 1.0, 5), (0.0, 0.0, 5)])
def test_small_levels_without_one_smoothing(fluid, diff, kernels, monkeypatch):
    """Kernels per iteration of a small level: the fused schedule's three; two
    force passes, smoothing with update in one tile kernel and a copy; two
    passes, a copy, the update and a smoothing or copy.  Same field as with the
    z-march."""
    data = pair((16, 32, 48))
    kw = dict(sigma_fluid=fluid, sigma_diff=diff)
    with cg.Context(0) as c:
        count = []
        for n in (4, 24):
            register(c, data, iters=[n], **kw)
            before = cg.launch_count()
            got = register(c, data, iters=[n], **kw)
            count.append(cg.launch_count() - before)
    assert count[1] - count[0] == 20 * kernels
    monkeypatch.setenv("CGDIR_SMOOTH", "march")
    with cg.Context(0) as c:
        assert torch.equal(register(c, data, iters=[24], **kw)[0], got[0])
