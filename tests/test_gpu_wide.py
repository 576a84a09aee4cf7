"""The integer form of the weighted sum (csrc/wide.cuh) and the kernels that
only it has: sizes at the edges of their tiles, unaligned grids, and the values
at which it hands over to the FMA chain."""
from fractions import Fraction

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu
PERIODIC, DIRICHLET = 1, 0
EPS = 2.0 ** -53


@pytest.fixture(scope="module")
def st():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2303_08365_gb300 import build
    build.build()
    import paper_2303_08365_gb300 as st
    return st


def weights(kind, ndim, radius, seed=5):
    side = 2 * radius + 1
    w = np.random.default_rng(seed).random((side,) * ndim) + 0.01
    if kind == "star":
        off = np.stack(np.meshgrid(*[np.arange(-radius, radius + 1)] * ndim, indexing="ij"))
        w[(off != 0).sum(axis=0) > 1] = 0.0
    return w / w.sum()


def run(st, u0, w, radius, boundary, T, tuning=(0, 0), offset=0):
    """Sweeps a copy of u0 placed `offset` elements past a 256-byte boundary, between canaries."""
    import torch
    n = u0.size
    buf = torch.full((n + 128,), 7.0, dtype=torch.float64, device="cuda")
    g = buf[64 + offset:64 + offset + n].view(u0.shape)
    g.copy_(torch.from_numpy(u0))
    p = st.Plan(u0.shape, radius, w, boundary)
    p.set_tuning(*tuning)
    p.run(g, T)
    assert p.status() == 0
    out = g.cpu().numpy().copy()
    g.fill_(7.0)
    assert bool((buf == 7.0).all())
    p.close()
    return out


# planes of one row or column more or fewer than a tile, one tile in all, rows
# that start on and off 16 bytes, a grid that ends half-way through 16 bytes
SHAPES3D = [(1, 8, 32), (2, 17, 33), (3, 16, 64), (5, 15, 65), (7, 33, 63), (4, 18, 129), (9, 31, 191), (40, 9, 130)]


# the smallest that are streamed (2^17 and 2^21 cells), a last tile of one column and
# one row, of 63 and 15
SHAPES3D += [(17, 97, 129), (15, 95, 127), (130, 129, 129)]


@pytest.mark.parametrize("kind", ["star", "box"])
@pytest.mark.parametrize("boundary", [DIRICHLET, PERIODIC])
@pytest.mark.parametrize("shape", SHAPES3D)
def test_streaming_any_shape_3d(st, shape, boundary, kind):
    w = weights(kind, 3, 1)
    u0 = synth.normal(31, shape)
    T, taps = 3, int(np.count_nonzero(w))
    ref = oracle.run(u0, w, 1, boundary, T, nthreads=0)
    # two roundings per tap and step in the oracle, fewer on the GPU; the sums do not expand
    tol = T * (2 * taps + 2) * EPS * np.abs(u0).max()
    for offset in (0, 1):
        got = run(st, u0, w, 1, boundary, T, (1, st.VARIANT_DIRECT), offset)
        assert np.abs(got - ref).max() <= tol, offset


SHAPES2D = [(8, 33), (17, 64), (90, 1460), (1025, 129), (1009, 191), (481, 449), (480, 448), (20, 6593)]


@pytest.mark.parametrize("kind,radius", [("star", 2), ("box", 2)])
@pytest.mark.parametrize("boundary", [DIRICHLET, PERIODIC])
@pytest.mark.parametrize("shape", SHAPES2D)
def test_streaming_any_shape_2d(st, shape, boundary, kind, radius):
    w = weights(kind, 2, radius)
    u0 = synth.normal(32, shape)
    T, taps = 3, int(np.count_nonzero(w))
    ref = oracle.run(u0, w, radius, boundary, T, nthreads=0)
    tol = T * (2 * taps + 2) * EPS * np.abs(u0).max()
    for variant, offset in ((st.VARIANT_DIRECT, 0), (st.VARIANT_DIRECT, 1), (0, 0)):
        got = run(st, u0, w, radius, boundary, T, (1, variant), offset)
        assert np.abs(got - ref).max() <= tol, (variant, offset)


def exact_sum(u, w, at, radius):
    """(sum, largest |product|) of one cell over the reals, zeros outside."""
    total, top = Fraction(0), Fraction(0)
    for o in np.ndindex(*w.shape):
        i = tuple(a + k - radius for a, k in zip(at, o))
        if w[o] != 0 and all(0 <= a < n for a, n in zip(i, u.shape)):
            p = Fraction(float(w[o])) * Fraction(float(u[i]))
            total += p
            top = max(top, abs(p))
    return total, top


WIDE_RANGE = [((6, 9, 33), "star", 1), ((4, 9, 34), "box", 1), ((19, 70), "star", 2), ((19, 70), "box", 2)]


@pytest.mark.parametrize("spread", [0, 8, 60, 300])
@pytest.mark.parametrize("shape,kind,radius", WIDE_RANGE)
def test_one_step_against_exact_arithmetic(st, shape, kind, radius, spread):
    """Values of both signs whose exponents are spread, with zeros among them:
    one rounding of the result and 2^-55 of the largest product."""
    rng = np.random.default_rng(spread)
    u0 = rng.standard_normal(shape) * 2.0 ** rng.integers(-spread, spread + 1, shape)
    u0[rng.random(shape) < 0.1] = 0.0
    w = weights(kind, len(shape), radius)
    got = run(st, u0, w, radius, DIRICHLET, 1)
    for at in np.ndindex(*shape):
        want, top = exact_sum(u0, w, at, radius)
        err = abs(Fraction(float(got[at])) - want)
        assert err <= abs(want) * Fraction(EPS) + top * Fraction(2.0 ** -55), at


@pytest.mark.parametrize("shape,kind,radius", WIDE_RANGE)
def test_values_outside_the_integer_range(st, shape, kind, radius):
    """Infinities, NaN, the largest and the smallest doubles, and all-zero
    neighbourhoods take the FMA chain: as the oracle has them."""
    rng = np.random.default_rng(9)
    w = weights(kind, len(shape), radius)
    for values in ([np.inf, 1.0], [np.nan, 1.0], [-np.inf, np.inf, 0.0], [1.7e308, -1.2e308, 3.0],
                   [5e-324, -3e-310, 0.0], [2.3e-308, 0.0], [1e-290, 1e-292], [0.0, -0.0]):
        u0 = np.zeros(shape)
        mask = rng.random(shape) < 0.05
        u0[mask] = rng.choice(values, int(mask.sum()))
        with np.errstate(all="ignore"):
            ref = oracle.run(u0, w, radius, DIRICHLET, 1, nthreads=1)
            got = run(st, u0, w, radius, DIRICHLET, 1)
            assert np.array_equal(np.isnan(got), np.isnan(ref)), values
            fine = np.isfinite(ref)
            assert np.array_equal(got[~fine & ~np.isnan(ref)], ref[~fine & ~np.isnan(ref)]), values
            # 27 roundings at most of sums no larger than the largest value; below the
            # normal range each is half of the smallest subnormal
            top = np.abs(u0[np.isfinite(u0)]).max() if np.isfinite(u0).any() else 0.0
            assert np.abs(got[fine] - ref[fine]).max(initial=0.0) <= max(60 * EPS * top, 60 * 5e-324), values


@pytest.mark.parametrize("kind", ["heat", "star", "box"])
@pytest.mark.parametrize("boundary", [DIRICHLET, PERIODIC])
@pytest.mark.parametrize("shape", SHAPES2D)
def test_streaming_any_shape_2d_radius_1(st, shape, boundary, kind):
    w = synth.heat_weights(2, 0.2) if kind == "heat" else weights(kind, 2, 1)
    u0 = synth.normal(33, shape)
    T, taps = 3, int(np.count_nonzero(w))
    ref = oracle.run(u0, w, 1, boundary, T, nthreads=0)
    tol = T * (2 * taps + 2) * EPS * np.abs(u0).max()
    for tb, variant, offset in ((1, st.VARIANT_DIRECT, 0), (1, st.VARIANT_DIRECT, 1), (0, 0, 0)):
        got = run(st, u0, w, 1, boundary, T, (tb, variant), offset)
        assert np.abs(got - ref).max() <= tol, (tb, variant, offset)


@pytest.mark.parametrize("spread", [0, 60])
@pytest.mark.parametrize("kind", ["heat", "star", "box"])
def test_one_step_against_exact_arithmetic_2d_radius_1(st, kind, spread):
    rng = np.random.default_rng(spread)
    u0 = rng.standard_normal((19, 70)) * 2.0 ** rng.integers(-spread, spread + 1, (19, 70))
    u0[rng.random(u0.shape) < 0.1] = 0.0
    w = synth.heat_weights(2, 0.2) if kind == "heat" else weights(kind, 2, 1)
    for tuning in ((1, st.VARIANT_DIRECT), (4, st.VARIANT_PERSISTENT)):
        got = run(st, u0, w, 1, DIRICHLET, 1, tuning)
        for at in np.ndindex(*u0.shape):
            want, top = exact_sum(u0, w, at, 1)
            assert abs(Fraction(float(got[at])) - want) <= abs(want) * Fraction(EPS) + top * Fraction(2.0 ** -55), at


# at least 200 tiles of 64 x 16: one column of tiles, one and a half rows of them, ragged
# last ones, more than one tile for every CTA
TILED = [(3200, 64), (23, 6500), (1009, 250), (833, 512), (1500, 1501)]


def same(a, b):
    """Equal bits, any NaN for another (which one depends on the order of the sum)."""
    return np.array_equal(np.isnan(a), np.isnan(b)) and np.array_equal(a[~np.isnan(a)], b[~np.isnan(b)])


@pytest.mark.parametrize("kind", ["heat", "star"])
@pytest.mark.parametrize("boundary", [DIRICHLET, PERIODIC])
@pytest.mark.parametrize("shape", TILED)
def test_persistent_tiles_equal_single_steps(st, shape, boundary, kind):
    """The integer form's result depends on a cell's values alone: all steps in one
    launch give the bits of one launch a step, also where cells take the FMA chain."""
    w = synth.heat_weights(2, 0.2) if kind == "heat" else weights(kind, 2, 1)
    rng = np.random.default_rng(3)
    u0 = synth.normal(34, shape)
    for T in (1, 2, 31):
        want = run(st, u0, w, 1, boundary, T, (1, st.VARIANT_DIRECT), 1)
        assert same(run(st, u0, w, 1, boundary, T, (1, st.VARIANT_PERSISTENT), 1), want), T
    mask = rng.random(shape) < 1e-4
    u0[mask] = rng.choice([np.inf, -np.inf, np.nan, 1.7e308, 5e-324, 1e-300], int(mask.sum()))
    want = run(st, u0, w, 1, boundary, 3, (1, st.VARIANT_DIRECT))
    assert same(run(st, u0, w, 1, boundary, 3, (1, st.VARIANT_PERSISTENT)), want)


# (cells per side, items): cells per thread, small tiles' share too low; tiles of many
# grids; tiles of a few large ones
BATCHES = [((20, 90), 30), ((150, 700), 40), ((900, 1400), 5)]


@pytest.mark.parametrize("boundary", [DIRICHLET, PERIODIC])
@pytest.mark.parametrize("sides,n", BATCHES)
def test_batch_equals_plans(st, sides, n, boundary):
    import torch
    rng = np.random.default_rng(n)
    shapes = [tuple(int(k) for k in rng.integers(sides[0], sides[1], 2)) for _ in range(n)]
    steps = [int(rng.integers(0, 40)) for _ in range(n)]
    alphas = [float(rng.uniform(0.05, 0.24)) for _ in range(n)]
    u0 = [synth.normal(200 + i, s) for i, s in enumerate(shapes)]
    grids = [torch.from_numpy(u.copy()).cuda() for u in u0]
    with st.Batch(grids, alphas, steps, boundary) as b:
        for tuning in ((1, 0, 0), (1, 1, 0), (1, 4, 0), (4, 0, 0)):
            for g, u in zip(grids, u0):
                g.copy_(torch.from_numpy(u))
            b.set_tuning(*tuning)
            b.run()
            assert b.status() == 0
            for g, u, a, T in zip(grids, u0, alphas, steps):
                want = run(st, u, synth.heat_weights(2, a), 1, boundary, T, (1, st.VARIANT_DIRECT)) if T else u
                assert np.array_equal(g.cpu().numpy(), want), (tuning, u.shape, a, T)


# TMA tiles, bulk copies with a last tile of 45 and of one column, both directions' ragged
# tiles; persistent tiles; 16 x 32 tiles
ZEROS = [((20, 64, 128), "heat", 1, (0, 0)), ((18, 127, 1005), "heat", 1, (1, 1)), ((17, 97, 129), "box", 1, (1, 1)),
         ((16, 64, 64), "box", 1, (0, 0)), ((320, 512), "heat", 1, (1, 2)), ((411, 557), "box", 2, (1, 1)),
         ((411, 557), "star", 1, (1, 1)), ((833, 513), "heat", 1, (1, 4)), ((90, 130), "heat", 1, (4, 4)),
         ((20, 64, 128), "heat", 1, (4, 5))]


@pytest.mark.parametrize("boundary", [DIRICHLET, PERIODIC])
@pytest.mark.parametrize("shape,kind,radius,tuning", ZEROS)
def test_a_few_values_among_zeros(st, shape, kind, radius, tuning, boundary):
    """Zeros of either sign stay zeros where nothing else reaches; tiny values beside them."""
    if tuning[0] == 0 and boundary == PERIODIC and shape[-1] % 64:
        pytest.skip("no streamed form")
    rng = np.random.default_rng(12)
    w = synth.heat_weights(len(shape), 0.12) if kind == "heat" else weights(kind, len(shape), radius)
    u0 = np.where(rng.random(shape) < 0.5, 0.0, -0.0)
    at = rng.integers(0, u0.size, 40)
    u0.reshape(-1)[at] = rng.standard_normal(40) * 10.0 ** rng.integers(-320, 5, 40)
    T = 4
    ref = oracle.run(u0, w, radius, boundary, T, nthreads=0)
    got = run(st, u0, w, radius, boundary, T, tuning)
    taps = int(np.count_nonzero(w))
    assert np.array_equal(got == 0.0, ref == 0.0) or np.abs(got[(got == 0.0) != (ref == 0.0)]).max() <= 1e-320
    # relative to what a cell's neighbourhood holds: the largest value that reaches it
    top = oracle.run(np.abs(u0), (w > 0).astype(float), radius, boundary, T, nthreads=0)
    assert (np.abs(got - ref) <= T * (2 * taps + 2) * EPS * top + 60 * T * 5e-324).all()


# axes of one, two and three cells (shorter than the radius and as long), and of a block and one more
SHORT = [(1,), (2,), (257,), (1, 1), (2, 33), (9, 2), (3, 65), (1, 1, 1), (2, 1, 33), (1, 9, 2), (3, 2, 3), (4, 9, 33)]


@pytest.mark.parametrize("kind", ["star", "box"])
@pytest.mark.parametrize("boundary", [DIRICHLET, PERIODIC])
@pytest.mark.parametrize("shape", SHORT)
def test_cell_by_cell_on_short_axes(st, shape, boundary, kind):
    for radius in (1, 2):
        w = weights(kind, len(shape), radius)
        u0 = synth.normal(34, shape)
        T, taps = 3, int(np.count_nonzero(w))
        ref = oracle.run(u0, w, radius, boundary, T, nthreads=0)
        tol = T * (2 * taps + 2) * EPS * np.abs(u0).max()
        got = run(st, u0, w, radius, boundary, T, (1, st.VARIANT_DIRECT))
        assert np.abs(got - ref).max() <= tol, radius


# the smallest that are streamed since, and the first with tiles of 16 rows
@pytest.mark.parametrize("boundary", [DIRICHLET, PERIODIC])
@pytest.mark.parametrize("shape,kind,radius", [((257, 129, 127), "star", 1), ((101, 103, 101), "box", 1),
                                               ((257, 256), "star", 2), ((331, 297), "box", 2)])
def test_smallest_streamed(st, shape, boundary, kind, radius):
    w = weights(kind, len(shape), radius)
    u0 = synth.normal(35, shape)
    T, taps = 2, int(np.count_nonzero(w))
    ref = oracle.run(u0, w, radius, boundary, T, nthreads=0)
    got = run(st, u0, w, radius, boundary, T, (1, st.VARIANT_DIRECT))
    assert np.abs(got - ref).max() <= T * (2 * taps + 2) * EPS * np.abs(u0).max()


def equal_weights(ndim, radius):
    return np.full((2 * radius + 1,) * ndim, 1.0 / (2 * radius + 1) ** ndim)


@pytest.mark.parametrize("spread", [0, 3, 60])
@pytest.mark.parametrize("radius", [1, 2])
def test_equal_box_against_exact_arithmetic(st, radius, spread):
    """The equal-weight boxes align the values of four cells to one exponent, at most 3 (2)
    above a cell's own: 8 (24) units of 2^-55 and half a unit of the product, 2^-52, of the
    cell's largest product, and one rounding of the result."""
    rng = np.random.default_rng(spread + radius)
    u0 = rng.standard_normal((19, 70)) * 2.0 ** rng.integers(-spread, spread + 1, (19, 70))
    u0[rng.random(u0.shape) < 0.1] = 0.0
    w = equal_weights(2, radius)
    got = run(st, u0, w, radius, DIRICHLET, 1, (1, st.VARIANT_STREAM))
    slack = Fraction((8 if radius == 1 else 24) * 2.0 ** -55 + 2.0 ** -52)
    for at in np.ndindex(*u0.shape):
        want, top = exact_sum(u0, w, at, radius)
        assert abs(Fraction(float(got[at])) - want) <= abs(want) * Fraction(EPS) + top * slack, at


@pytest.mark.parametrize("shape,boundary", [((1, 2), DIRICHLET), ((17, 66), DIRICHLET), ((15, 62), DIRICHLET),
                                            ((16, 64), PERIODIC), ((48, 192), PERIODIC), ((643, 1286), DIRICHLET)])
@pytest.mark.parametrize("radius", [1, 2])
def test_equal_box_tiles(st, shape, boundary, radius):
    w = equal_weights(2, radius)
    taps, T = w.size, 3
    for u0 in (synth.normal(36, shape), np.where(synth.uniform(37, shape) < 0.003, synth.normal(38, shape), 0.0)):
        ref = oracle.run(u0, w, radius, boundary, T, nthreads=0)
        got = run(st, u0, w, radius, boundary, T, (1, st.VARIANT_STREAM))
        assert np.abs(got - ref).max() <= T * (2 * taps + 2) * EPS * np.abs(u0).max()
        assert np.array_equal(got == 0.0, ref == 0.0)


@pytest.mark.parametrize("radius", [1, 2])
def test_equal_box_values_outside_the_integer_range(st, radius):
    rng = np.random.default_rng(10)
    w = equal_weights(2, radius)
    for values in ([np.inf, 1.0], [np.nan, 1.0], [-np.inf, np.inf, 0.0], [1.7e308, -1.2e308, 3.0],
                   [5e-324, -3e-310, 0.0], [2.3e-308, 0.0], [0.0, -0.0]):
        u0 = np.zeros((19, 70))
        mask = rng.random(u0.shape) < 0.05
        u0[mask] = rng.choice(values, int(mask.sum()))
        with np.errstate(all="ignore"):
            ref = oracle.run(u0, w, radius, DIRICHLET, 1, nthreads=1)
            got = run(st, u0, w, radius, DIRICHLET, 1, (1, st.VARIANT_STREAM))
            assert np.array_equal(np.isnan(got), np.isnan(ref)), values
            fine = np.isfinite(ref)
            assert np.array_equal(got[~fine & ~np.isnan(ref)], ref[~fine & ~np.isnan(ref)]), values
            top = np.abs(u0[np.isfinite(u0)]).max() if np.isfinite(u0).any() else 0.0
            assert np.abs(got[fine] - ref[fine]).max(initial=0.0) <= max(60 * EPS * top, 60 * 5e-324), values


@pytest.mark.parametrize("n", [1, 2, 3, 31, 47, 48, 49, 385, 65535, 65537, 65536 + 7 * 8 * 112, (1 << 20) - 1, (1 << 20) + 12345])
@pytest.mark.parametrize("boundary", [DIRICHLET, PERIODIC])
def test_fused_1d_equals_single_steps(st, n, boundary):
    """Warps of 64, 128 and 256 cells, the last one ragged; 11 steps as 8 and 3."""
    for radius, w in ((1, synth.heat_weights(1, 0.2)), (1, weights("star", 1, 1)), (2, weights("star", 1, 2))):
        u0 = synth.normal(39, (n,))
        got = run(st, u0, w, radius, boundary, 11)
        assert np.array_equal(got, run(st, u0, w, radius, boundary, 11, (1, st.VARIANT_DIRECT))), radius
        ref = oracle.run(u0, w, radius, boundary, 11, nthreads=0)
        assert np.abs(got - ref).max() <= 11 * (2 * w.size + 2) * EPS * np.abs(u0).max(), radius


@pytest.mark.parametrize("values", [[np.inf, 1.0], [np.nan, 1.0], [-np.inf, np.inf, 0.0], [1.7e308, -1.2e308, 3.0],
                                    [5e-324, -3e-310, 0.0], [2.3e-308, 0.0], [0.0, -0.0]])
def test_fused_1d_values_outside_the_integer_range(st, values):
    rng = np.random.default_rng(11)
    for radius in (1, 2):
        w = weights("star", 1, radius)
        u0 = np.zeros(1500)
        mask = rng.random(u0.shape) < 0.02
        u0[mask] = rng.choice(values, int(mask.sum()))
        for T in (1, 8):
            got = run(st, u0, w, radius, DIRICHLET, T)
            assert same(got, run(st, u0, w, radius, DIRICHLET, T, (1, st.VARIANT_DIRECT))), (radius, T)
        with np.errstate(all="ignore"):
            ref = oracle.run(u0, w, radius, DIRICHLET, 1, nthreads=1)
            got = run(st, u0, w, radius, DIRICHLET, 1)
            assert np.array_equal(np.isnan(got), np.isnan(ref))
            fine = np.isfinite(ref)
            assert np.array_equal(got[~fine & ~np.isnan(ref)], ref[~fine & ~np.isnan(ref)])
            top = np.abs(u0[np.isfinite(u0)]).max() if np.isfinite(u0).any() else 0.0
            assert np.abs(got[fine] - ref[fine]).max(initial=0.0) <= max(60 * EPS * top, 60 * 5e-324)


# one brick of 32 x 8 x 16 cells and less, bricks of unequal sizes, every depth (2 to 16), the
# largest cuts that are taken in one launch (152 bricks) and one beyond
BRICKS = [(1, 1, 1), (1, 1, 2), (2, 3, 4), (3, 9, 33), (16, 8, 32), (17, 8, 32), (5, 17, 65), (64, 64, 64), (65, 65, 65),
          (33, 47, 61), (40, 150, 127), (299, 16, 31), (70, 80, 90), (113, 28, 118)]


@pytest.mark.parametrize("kind", ["heat", "star"])
@pytest.mark.parametrize("boundary", [DIRICHLET, PERIODIC])
@pytest.mark.parametrize("shape", BRICKS)
def test_persistent_bricks_equal_single_steps(st, shape, boundary, kind):
    w = synth.heat_weights(3, 0.12) if kind == "heat" else weights("star", 3, 1)
    u0 = synth.normal(40, shape)
    for T in (3, 8, 31):
        want = run(st, u0, w, 1, boundary, T, (1, st.VARIANT_DIRECT))
        for offset in (0, 1):
            assert np.array_equal(run(st, u0, w, 1, boundary, T, (0, 0), offset), want), (T, offset)


@pytest.mark.parametrize("values", [[np.inf, 1.0], [np.nan, 1.0], [-np.inf, np.inf, 0.0], [1.7e308, -1.2e308, 3.0],
                                    [5e-324, -3e-310, 0.0], [2.3e-308, 0.0], [0.0, -0.0], [1.0, 0.0]])
def test_persistent_bricks_values_outside_the_integer_range(st, values):
    rng = np.random.default_rng(12)
    w = weights("star", 3, 1)
    u0 = np.zeros((11, 13, 40))
    mask = rng.random(u0.shape) < 0.01
    u0[mask] = rng.choice(values, int(mask.sum()))
    for T in (3, 4):
        got = run(st, u0, w, 1, DIRICHLET, T)
        assert same(got, run(st, u0, w, 1, DIRICHLET, T, (1, st.VARIANT_DIRECT))), T


def test_persistent_bricks_under_capture(st):
    """A graph captured after a run, replayed on new data; and one captured before there was any."""
    import torch
    w = synth.heat_weights(3, 0.12)
    fields = [synth.uniform(41 + k, (33, 20, 40)) for k in range(2)]
    g = torch.from_numpy(fields[0].copy()).cuda()
    p = st.Plan(fields[0].shape, 1, w, PERIODIC)
    p.run(g, 1)
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        p.run(g, 9)
    for u in fields:
        g.copy_(torch.from_numpy(u))
        graph.replay()
        torch.cuda.synchronize()
        assert np.array_equal(g.cpu().numpy(), run(st, u, w, 1, PERIODIC, 9, (1, st.VARIANT_DIRECT)))
    assert p.status() == 0
    p.close()


@pytest.mark.parametrize("spread", [0, 3, 60])
def test_equal_box_against_exact_arithmetic_3d(st, spread):
    """As in two dimensions, at most 2 exponents apart: 26 units of 2^-55 and half a unit of
    the product, 2^-52, of the cell's largest product, and one rounding of the result."""
    rng = np.random.default_rng(spread + 7)
    u0 = rng.standard_normal((4, 11, 34)) * 2.0 ** rng.integers(-spread, spread + 1, (4, 11, 34))
    u0[rng.random(u0.shape) < 0.1] = 0.0
    w = equal_weights(3, 1)
    got = run(st, u0, w, 1, DIRICHLET, 1, (1, st.VARIANT_STREAM))
    slack = Fraction(26 * 2.0 ** -55 + 2.0 ** -52)
    for at in np.ndindex(*u0.shape):
        want, top = exact_sum(u0, w, at, 1)
        assert abs(Fraction(float(got[at])) - want) <= abs(want) * Fraction(EPS) + top * slack, at


@pytest.mark.parametrize("shape,boundary,tile", [((1, 1, 2), DIRICHLET, 16), ((3, 17, 66), DIRICHLET, 16),
                                                 ((5, 15, 62), DIRICHLET, 8), ((4, 16, 64), PERIODIC, 16),
                                                 ((9, 24, 192), PERIODIC, 8), ((61, 97, 130), DIRICHLET, 16)])
def test_equal_box_tiles_3d(st, shape, boundary, tile):
    w = equal_weights(3, 1)
    T = 3
    for u0 in (synth.normal(44, shape), np.where(synth.uniform(45, shape) < 0.001, synth.normal(46, shape), 0.0),
               np.where(synth.uniform(47, shape) < 0.001, np.inf, 1.0)):
        with np.errstate(all="ignore"):
            ref = oracle.run(u0, w, 1, boundary, T, nthreads=0)
        import torch
        g = torch.from_numpy(u0.copy()).cuda()
        p = st.Plan(shape, 1, w, boundary)
        p.set_tuning(1, st.VARIANT_STREAM)
        p.set_tile(64, tile)
        p.run(g, T)
        assert p.status() == 0
        p.close()
        got = g.cpu().numpy()
        fine = np.isfinite(ref)
        assert np.array_equal(fine, np.isfinite(got))
        top = np.abs(u0[np.isfinite(u0)]).max()
        assert np.abs(got[fine] - ref[fine]).max(initial=0.0) <= T * (2 * w.size + 2) * EPS * top
        assert np.array_equal(got == 0.0, ref == 0.0)


@pytest.mark.parametrize("ndim,radius,shape", [(2, 1, (64, 128)), (2, 2, (64, 128)), (3, 1, (16, 32, 64))])
def test_equal_boxes_lean_to_no_side(st, ndim, radius, shape):
    """A field and its negative over many steps: sums that lose or gain a unit of 2^-58 a value and
    step on one side would end 160 of them apart, 5e-16; roundings to nearest differ cell by
    cell at most, which the mean of some thousand cells does not show."""
    w, T = equal_weights(ndim, radius), 160
    u0 = synth.uniform(48, shape)
    a, b = (run(st, sign * u0, w, radius, PERIODIC, T, (1, st.VARIANT_STREAM)) for sign in (1.0, -1.0))
    total = sum(Fraction(float(x)) for x in a.flat)
    assert abs(total + sum(Fraction(float(x)) for x in b.flat)) <= total * Fraction(EPS) / 2


# more cells than the temporal kernel takes, rows that TMA does not take: one row or column more
# than a tile, tiles four fifths full and a little less
@pytest.mark.parametrize("boundary", [DIRICHLET, PERIODIC])
@pytest.mark.parametrize("shape", [(513, 513), (600, 602), (331, 1101), (4097, 65), (2600, 103), (2600, 102)])
def test_stars_by_default_equal_the_persistent_kernel(st, shape, boundary):
    w = synth.heat_weights(2, 0.2)
    u0 = synth.normal(49, shape)
    for T in (1, 6):
        for offset in (0, 1):
            got = run(st, u0, w, 1, boundary, T, (0, 0), offset)
            assert np.array_equal(got, run(st, u0, w, 1, boundary, T, (1, st.VARIANT_PERSISTENT), offset)), (T, offset)


def equal_box_fields(shape):
    """Values of one binade, of many, at the ends of the binades that share an alignment, and among
    zeros and values that the integer form does not take."""
    rng = np.random.default_rng(50)
    yield synth.uniform(51, shape)
    yield rng.uniform(1.0, 4.0, shape) * rng.choice([1.0, -1.0], shape)
    yield rng.uniform(0.02, 4.0, shape)
    yield rng.standard_normal(shape) * 2.0 ** rng.integers(-4, 5, shape)
    yield rng.choice([2.0, np.nextafter(2.0, 0), -2.0, 0.125, 0.0, -0.0], shape)
    u0 = rng.standard_normal(shape) * 2.0 ** rng.integers(-60, 61, shape)
    u0[rng.random(shape) < 0.3] = 0.0
    mask = rng.random(shape) < 1e-3
    u0[mask] = rng.choice([np.inf, -np.inf, np.nan, 1.7e308, 5e-324, 1e-300], int(mask.sum()))
    yield u0


# cell by cell against tiles (TMA; tiles of 8, 16 and 32 rows), Tb steps on the chip and handed over
# between CTAs; and as many cells as bulk copies take (3D: 8 and 16 rows)
EQUAL_BOXES = [((64, 128), 1, ["direct", "persistent", "stream"]), ((512, 320), 1, ["direct", "persistent", "stream"]),
               ((64, 192), 2, ["direct", "stream"]), ((512, 256), 2, ["direct", "stream"]),
               ((5, 32, 128), 1, ["direct", "stream", "temporal", "exchange"]),
               ((34, 64, 64), 1, ["direct", "stream"]), ((260, 64, 64), 1, ["direct", "stream"])]


@pytest.mark.parametrize("boundary", [DIRICHLET, PERIODIC])
@pytest.mark.parametrize("shape,radius,kernels", EQUAL_BOXES)
def test_equal_boxes_have_the_same_bits_in_every_kernel(st, shape, radius, kernels, boundary):
    import torch
    w, T = equal_weights(len(shape), radius), 4
    for u0 in equal_box_fields(shape):
        want = run(st, u0, w, radius, boundary, T, (1, st.VARIANT_DIRECT), 1)
        ways = [("direct", 1, 0), *(("stream", 1, ty) for ty in ((0, 8, 16, 32) if len(shape) == 3 else (0,))),
                *((k, Tb, 0) for k in ("persistent", "temporal", "exchange") for Tb in (2, 4))]
        for kernel, Tb, tile in ways:
            if kernel not in kernels:
                continue
            g = torch.from_numpy(u0.copy()).cuda()
            p = st.Plan(shape, radius, w, boundary)
            p.set_tuning(Tb, getattr(st, "VARIANT_" + kernel.upper()))
            if tile:
                p.set_tile(64, tile)
            p.run(g, T)
            assert p.status() == 0
            p.close()
            assert same(g.cpu().numpy(), want), (kernel, Tb, tile)


@pytest.mark.parametrize("radius", [1, 2])
def test_equal_boxes_have_the_same_bits_in_a_part_of_the_grid(st, radius):
    """Rows that start at any row and columns that start at any column of the whole grid."""
    w = equal_weights(2, radius)
    for u0 in equal_box_fields((48, 130)):
        want = run(st, u0, w, radius, DIRICHLET, 1, (1, st.VARIANT_STREAM))
        for y, x in ((1, 0), (3, 1), (4, 2), (7, 5)):
            part = np.ascontiguousarray(u0[y:y + 33, x:x + 100])
            got = run(st, part, w, radius, DIRICHLET, 1, (1, st.VARIANT_STREAM))
            inner = (slice(radius, -radius),) * 2
            assert same(got[inner], want[y:y + 33, x:x + 100][inner]), (y, x)


def test_batch_runs_the_kernel_that_is_asked_for(st):
    """Tiles by default where the grids fill them; the cells per thread and blocks per SM that a
    caller names otherwise, the default ones among them.  The same bits; what is reported can be set."""
    import torch
    u0 = [synth.uniform(60 + i, s) for i, s in enumerate([(900, 1300), (1024, 640), (700, 900)])]
    grids = [torch.from_numpy(u.copy()).cuda() for u in u0]
    with st.Batch(grids, [0.1, 0.2, 0.15], [7, 12, 3]) as b:
        assert b.get_tuning() == (1, 0, 0)
        b.run()
        assert b.status() == 0
        want = [g.cpu().numpy().copy() for g in grids]
        for tuning in ((1, 2, 4), (1, 2, 0), (1, 0, 4), (1, 4, 2), (1, 0, 0)):
            for g, u in zip(grids, u0):
                g.copy_(torch.from_numpy(u))
            b.set_tuning(*tuning)
            got = b.get_tuning()
            assert got == tuning if tuning in ((1, 2, 4), (1, 4, 2), (1, 0, 0)) else got[1] > 0 and got[2] > 0, tuning
            b.set_tuning(*got)
            assert b.get_tuning() == got
            b.run()
            assert b.status() == 0
            assert all(np.array_equal(g.cpu().numpy(), w) for g, w in zip(grids, want)), tuning


def test_autotune_keeps_a_default_that_no_variant_names(st):
    """A small 3D star runs all its steps in one launch, by default alone: the tuner times that too, and
    what it records serves other plans of the key.  20 steps of one launch each take more than twice as long."""
    import torch
    shape, w = (64, 64, 64), synth.heat_weights(3, 0.11)
    g = torch.from_numpy(synth.uniform(70, shape)).cuda()
    with st.Plan(shape, 1, w, PERIODIC) as a, st.Plan(shape, 1, w, PERIODIC) as b:
        a.autotune(g.clone(), 20)
        for p in (a, b):
            before = st.stencil_launch_count()
            p.run(g, 20)
            assert st.stencil_launch_count() - before == 1
            assert p.status() == 0


# (kernel of the self-test, a grid that it takes, its variant)
STARVED = [(0, (8, 32, 128), 2), (1, (64, 128), 2), (2, (512, 640), 4), (3, (8, 32, 128), 0)]


@pytest.mark.parametrize("kernel,shape,variant", STARVED)
def test_waits_that_run_out_report_it_and_the_context_survives(st, kernel, shape, variant):
    """Every bounded wait of the kernels for positive weights: copies that never come, steps that a
    neighbour never publishes.  They end by their limit of 20 ms, and the next sweep is right."""
    import time
    t0 = time.perf_counter()
    assert st.stencil_selftest_wide_timeout(kernel, 20.0) == st.ERR_TIMEOUT
    assert time.perf_counter() - t0 < 5.0
    w, u0 = synth.heat_weights(len(shape), 0.1), synth.normal(71, shape)
    got = run(st, u0, w, 1, PERIODIC, 5, (1, variant) if variant else (0, 0))
    assert np.array_equal(got, run(st, u0, w, 1, PERIODIC, 5, (1, st.VARIANT_DIRECT), 1))
    with pytest.raises(st.StencilError):
        st._check(st.lib().stencil_selftest_wide_timeout(4, 20.0, None))


@pytest.mark.parametrize("radius,shape", [(2, (40, 100)), (1, (6, 20, 34))])
def test_equal_boxes_of_spread_values_lean_by_what_the_alignment_cuts(st, radius, shape):
    """Positive values from e^-4 to e^4.  A value more than 2^9 below the alignment, the largest exponent
    field rounded up to 4 n + 3, is cut by half a unit of 2^-61 of it on average, and the rounding to
    nearest leans to no side: its mean over some 4000 cells is within four times 0.5 / sqrt(n) of 2^-53."""
    w = equal_weights(len(shape), radius)
    u0 = np.exp(np.random.default_rng(72).uniform(-4.0, 4.0, shape))
    got = run(st, u0, w, radius, DIRICHLET, 1, (1, st.VARIANT_STREAM))
    field = np.frexp(u0)[1] + 1022
    lean, cut = [], []
    for at in np.ndindex(*shape):
        want, _ = exact_sum(u0, w, at, radius)
        lean.append(float((Fraction(float(got[at])) - want) / want) / EPS)
        box = field[tuple(slice(max(0, a - radius), a + radius + 1) for a in at)]
        top = int(box.max()) | 3
        unit = w.flat[0] * 2.0 ** (top - 1084)
        cut.append(0.5 * unit * int((box < top - 9).sum()) / float(want) / EPS)
    assert abs(np.mean(lean)) <= np.mean(cut) + 4 * 0.5 / np.sqrt(got.size)
