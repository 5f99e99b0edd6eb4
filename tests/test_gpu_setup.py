"""Set-up kernels (UROI on bit rows, automatic signs) at row lengths and
margins where words, vectors and borders can go wrong, against the oracle;
all of it exact."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - CPU container
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import paper_1301_0970_gb300 as cg  # noqa: E402

DEV = torch.device("cuda:0")
SHAPES = [(1, 1, 1), (5, 7, 3), (4, 9, 31), (6, 5, 32), (3, 11, 33), (9, 6, 48), (17, 12, 64), (20, 10, 100),
          (35, 4, 130)]


@pytest.fixture(scope="module")
def ctx():
    with cg.Context(0) as c:
        yield c


def sparse_masks(shape, k, rng):
    """k masks of a few voxels and boxes each, some on the volume's border."""
    m = np.zeros((k,) + shape, np.uint8)
    for j in range(k):
        for _ in range(3):
            lo = [int(rng.integers(0, n)) for n in shape]
            hi = [min(n, a + int(rng.integers(1, 4))) for a, n in zip(lo, shape)]
            m[j, lo[0]:hi[0], lo[1]:hi[1], lo[2]:hi[2]] = 1
    return m


def packed(m, offset=0):
    b = np.zeros(m.shape[1:], np.uint8)
    for j in range(m.shape[0]):
        b |= m[j] << j
    t = torch.empty(b.size + offset, dtype=torch.uint8, device=DEV)[offset:].view(b.shape)
    t.copy_(torch.from_numpy(b))
    return t


@pytest.mark.parametrize("spacing,margin", [((1.97, 1.97, 2.5), 10.0), ((1.0, 1.0, 1.0), 15.0), ((1.0, 2.0, 0.7), 4.0),
                                            ((3.0, 3.0, 3.0), 0.0)])
@pytest.mark.parametrize("shape", SHAPES)
def test_uroi_bit_rows(ctx, shape, spacing, margin):
    rng = np.random.default_rng(sum(shape))
    m = sparse_masks(shape, 2, rng)
    ref = oracle.uroi(m, shape, spacing, margin)
    for offset in (0, 1):                         # 16-byte aligned mask bytes or not
        got = ctx.uroi(packed(m, offset), 2, spacing, margin)
        torch.cuda.synchronize()
        assert np.array_equal(got.cpu().numpy(), ref)
    none = ctx.uroi(packed(np.zeros_like(m)), 2, spacing, margin)
    assert int(none.sum()) == 0


@pytest.mark.parametrize("k", [1, 3, 8])
@pytest.mark.parametrize("shape", SHAPES)
def test_auto_sign_over_shapes(ctx, shape, k):
    """T0 is well above zero inside the structures of even index and below
    elsewhere (or the other way round), so the means differ; empty
    structures and empty shells (the whole volume) included."""
    rng = np.random.default_rng(sum(shape) + k)
    m = sparse_masks(shape, k, rng)
    if k == 3:
        m[1] = 0
        m[2] = 1
    T = rng.normal(0, 5, shape)
    for j in range(k):
        T = T + np.where(m[j] != 0, 300.0 * (j + 1) * (1 if j % 2 == 0 else -1), 0.0)
    T = T.astype(np.float32)
    ref = oracle.auto_sign(T.astype(np.float64), m)
    for offset in (0, 1):
        assert ctx.auto_sign(torch.from_numpy(T).to(DEV), packed(m, offset), k) == ref


@pytest.mark.parametrize("shape", SHAPES + [(3, 5, 8), (9, 4, 24)])
def test_restrict_and_pack_vectors(ctx, shape):
    """Restriction of images and bits and mask packing: the vector forms
    (aligned rows) and the general ones on the same data, shifted by one
    element in memory, give the same values; bits equal the oracle's."""
    rng = np.random.default_rng(sum(shape))
    m = (rng.random((8,) + shape) < 0.5).astype(np.uint8)
    img = rng.normal(0, 500, shape).astype(np.float32)
    b0, b1 = packed(m), packed(m, 1)
    t = [torch.from_numpy(v).to(DEV) for v in m]
    assert torch.equal(ctx.pack_masks(t), b0)
    off = []
    for v in t:                                   # mask bytes that are not 4-byte aligned
        o = torch.empty(v.numel() + 1, dtype=torch.uint8, device=DEV)[1:].view(v.shape)
        off.append(o.copy_(v))
    assert torch.equal(ctx.pack_masks(off), b0)
    r0, r1 = ctx.restrict_bits(b0), ctx.restrict_bits(b1)
    ref = np.zeros(r0.shape, np.uint8)
    for j in range(8):
        ref |= (oracle.restrict_mask(m[j]) != 0).astype(np.uint8) << j
    assert np.array_equal(r0.cpu().numpy(), ref) and np.array_equal(r1.cpu().numpy(), ref)
    i0 = torch.from_numpy(img).to(DEV)
    i1 = torch.empty(img.size + 1, device=DEV)[1:].view(img.shape).copy_(i0)
    assert torch.equal(ctx.restrict_image(i0), ctx.restrict_image(i1))


@pytest.mark.parametrize("fine", [(1, 1, 1), (2, 3, 5), (8, 8, 64), (9, 17, 66), (16, 15, 63), (5, 9, 130), (7, 30, 128)])
def test_prolong_tiles(ctx, fine):
    """Every border of the tiles and of the volume, against the oracle at
    1e-6 of the field's scale (the weights are exact, eight products are
    added: about 8 roundings of 6e-8)."""
    rng = np.random.default_rng(sum(fine))
    uc = rng.normal(0, 3, (3,) + tuple((n + 1) // 2 for n in fine)).astype(np.float32)
    got = ctx.prolong(torch.from_numpy(uc).to(DEV), fine)
    torch.cuda.synchronize()
    ref = oracle.prolong(uc, fine)
    assert np.abs(got.cpu().numpy() - ref).max() <= 1e-6 * np.abs(ref).max()


@pytest.mark.parametrize("shape", [(17, 12, 64), (20, 10, 33)])
def test_auto_sign_of_sums_beyond_float(ctx, shape):
    """Values whose sum over a few voxels overflows a float have a mean all the
    same; an infinite or NaN voxel decides as it does in FP64."""
    m = np.zeros((1,) + shape, np.uint8)
    m[0, 4:14, 3:9, 8:24] = 1
    for inside, shell in ((2.0e38, 1.0e38), (1.0e38, 2.0e38), (-2.0e38, -1.0e38), (3.0e38, 3.4028235e38)):
        for odd in (None, np.inf, -np.inf, np.nan):
            T = np.where(m[0] != 0, inside, shell).astype(np.float32)
            if odd is not None:
                T[6, 5, 12] = odd
            with np.errstate(invalid="ignore"):
                want = oracle.auto_sign(T.astype(np.float64), m)
            assert ctx.auto_sign(torch.from_numpy(T).to(DEV), packed(m), 1) == want


@pytest.mark.parametrize("shape", [(16, 12, 64), (16, 12, 33)])
def test_auto_sign_keeps_what_fp64_keeps(ctx, shape):
    """A column of 2^48, 2^24, 1, -2^48, -2^24, 0, 0, 0 has mean 1/8 in FP64 and
    0 in a sum of 48 bits; its shell's value lies between."""
    m = np.zeros((1,) + shape, np.uint8)
    m[0, 4:12, 6, 17] = 1
    T = np.full(shape, 0.0625, np.float32)
    T[4:12, 6, 17] = [2.0 ** 48, 2.0 ** 24, 1, -2.0 ** 48, -2.0 ** 24, 0, 0, 0]
    want = oracle.auto_sign(T.astype(np.float64), m)
    assert ctx.auto_sign(torch.from_numpy(T).to(DEV), packed(m), 1) == want
    T[6, 6, 17] = 0
    assert ctx.auto_sign(torch.from_numpy(T).to(DEV), packed(m), 1) == [-s for s in want]


@pytest.mark.parametrize("fine", [(2, 3, 5), (8, 8, 64), (9, 17, 66), (1, 2, 130)])
def test_prolong_of_values_that_are_not_finite(ctx, fine):
    """Every corner enters with its weight, also with weight 0 at the borders: an
    infinite or NaN coarse value spoils the fine voxels that the oracle's does."""
    coarse = tuple((n + 1) // 2 for n in fine)
    at = {(min(a, coarse[0] - 1), min(b, coarse[1] - 1), min(c, coarse[2] - 1))
          for a in (0, 1, 99) for b in (0, 1, 99) for c in (0, 1, 99)}
    for place in sorted(at):
        for value in (np.inf, -np.inf, np.nan):
            uc = np.ones((3,) + coarse, np.float32)
            uc[(slice(None),) + place] = value
            got = ctx.prolong(torch.from_numpy(uc).to(DEV), fine).cpu().numpy()
            with np.errstate(invalid="ignore"):
                ref = oracle.prolong(uc, fine)
            assert np.array_equal(np.isnan(got), np.isnan(ref)) and np.array_equal(np.isinf(got), np.isinf(ref)), place


@pytest.mark.parametrize("nx, spacing, margin", [(1, 2.5, 10.0), (4, 2.5, 10.0), (5, 2.5, 10.0), (8, 1.0, 15.0),
                                                 (13, 1.0, 15.0), (14, 1.0, 15.0), (33, 1.0, 15.0)])
def test_uroi_scratch_of_narrow_volumes(nx, spacing, margin):
    """The UROI of a context whose budget holds 5 bytes of scratch per voxel:
    word rows where they fit, rows dilated in place where they do not."""
    shape = (100, 700, nx)                        # 2 MB is the unit of the budget
    m = np.zeros((1,) + shape, np.uint8)
    m[0, 40:50, 300:340, nx // 2] = 1
    m[0, 0, 0, 0] = m[0, -1, -1, -1] = 1
    unit = 1 << 21
    budget = -(-(m.size * 5 + 3) // unit) * unit
    with cg.Context(0, mem_budget_bytes=budget) as c:
        got = c.uroi(packed(m), 1, (spacing,) * 3, margin)
        torch.cuda.synchronize()
    assert np.array_equal(got.cpu().numpy(), oracle.uroi(m, shape, (spacing,) * 3, margin))


@pytest.mark.parametrize("shape", [(300000, 1, 1), (1, 300000, 1), (1, 1, 300000), (40000, 5, 3), (75000, 1, 4)])
def test_auto_sign_of_thin_volumes(shape):
    """Volumes of few columns or few planes: the signs, in scratch of two buffers
    of a byte per voxel (allocated in units of 2 MB)."""
    rng = np.random.default_rng(shape[0])
    m = np.zeros((8,) + shape, np.uint8)
    for j in range(8):
        for _ in range(4):
            at = [int(rng.integers(0, n)) for n in shape]
            m[j][tuple(slice(a, a + 9) for a in at)] = 1
    T = rng.normal(0, 5, shape)
    for j in range(8):
        T = T + np.where(m[j] != 0, 300.0 * (j + 1) * (1 if j % 2 == 0 else -1), 0.0)
    T = T.astype(np.float32)
    want = oracle.auto_sign(T.astype(np.float64), m)
    with cg.Context(0, mem_budget_bytes=2 << 21) as c:
        assert c.auto_sign(torch.from_numpy(T).to(DEV), packed(m), 8) == want
