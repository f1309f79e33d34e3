"""FP64 half-sweeps of lines of 64 .. 1024 steps (sliced integer products on the tensor cores,
FP64 sums where the lines are few) against sums in extended precision.

Bounds, against S = sum |k| |b| of a value (b the gathered line, k the inverse column):
  * sliced: b keeps 59 bits below its largest operand, the dropped products are below
    2^-59 (largest |k|) (largest |b|), the total is rounded once: 4e-16 of the largest S and b.
  * FP64 sums: b rounded five times, at most M / 16 products a thread in a chain of sums, eight
    sums of the chains' results and two of what is left: (M / 16 + 15) * 2^-53.
"""
import numpy as np
import pytest

from paper_1608_05400_gb300 import inputs
from paper_1608_05400_gb300 import mgwr as G

pytestmark = pytest.mark.gpu
Q = np.longdouble


def _sums(lines, M):  # the rule that takes few lines to the FP64 sums
    return lines * M * M // 2 <= (1 << 21) + (1 << 13) * M


def _bound(lines, M):
    return (M / 16 + 15) * 2.0 ** -53 if _sums(lines, M) else 4e-16


@pytest.fixture(scope="module", autouse=True)
def _lib():
    G.load()


def _points(d, n, colour):
    if d == 1:
        return [i for i in range(n) if i % 2 == (1 if colour == G.MGWR_RED else 0)]
    return [i + n * j for j in range(n) for i in range(n) if (i + j) % 2 == colour]


def _gathered(u, f, p, d, n):
    i, j = (p, 0) if d == 1 else (p % n, p // n)
    s = np.zeros(u.shape[1], dtype=Q)
    for ok, q in ((i > 0, p - 1), (i < n - 1, p + 1), (d == 2 and j > 0, p - n),
                  (d == 2 and j < n - 1, p + n)):
        if ok:
            s = s + u[q].astype(Q)
    return f[p].astype(Q) + Q(float((n + 1) ** 2)) * s


def _check(s, d, n, M, colour, u, f, batch, sample, bound):
    l = s.num_levels() - 1
    shape = (batch, n ** d, M) if batch > 1 else (n ** d, M)
    s.field_set(G.MGWR_H64, l, G.MGWR_U, u.reshape(shape))
    s.field_set(G.MGWR_H64, l, G.MGWR_F, f.reshape(shape))
    s.smooth(G.MGWR_H64, l, colour)
    got = s.field_get(G.MGWR_H64, l, G.MGWR_U).reshape(batch, n ** d, M)
    k = s.inverse_column(l).reshape(batch, M)
    pts = _points(d, n, colour)
    others = np.setdiff1d(np.arange(n ** d), pts)
    np.testing.assert_array_equal(got[:, others], u[:, others])
    for b in range(batch):
        kq = k[b].astype(Q)
        for p in sorted({pts[int(x * (len(pts) - 1))] for x in sample}):
            line = _gathered(u[b], f[b], p, d, n)
            want = np.array([np.dot(kq[:m + 1][::-1], line[:m + 1]) for m in range(M)])
            scale = np.array([np.dot(abs(kq[:m + 1][::-1]), abs(line[:m + 1])) for m in range(M)])
            err = np.abs(got[b, p].astype(Q) - want)
            assert float(err.max()) <= bound * float(scale.max()), (b, p, float(err.max() / scale.max()))


# (d, n, M, batch): the two forms on both sides of their boundary, groups of 16
# and of 32 lines, partly filled groups, several slabs, the shortest and the longest lines, and
# instances with columns of their own
@pytest.mark.parametrize("d,n,M,batch", [
    (1, 1, 64, 1), (1, 63, 64, 1), (2, 15, 128, 1), (1, 31, 1024, 1),       # sums
    (2, 63, 64, 3), (1, 1023, 128, 1), (2, 15, 256, 3), (1, 127, 512, 1), (2, 7, 1024, 2),
    (2, 127, 256, 1), (2, 127, 1024, 1)])                                    # sliced
@pytest.mark.parametrize("data", ["random", "smooth", "wide"])
def test_half_sweep_against_extended_sums(d, n, M, batch, data):
    if data != "random" and n == 127 and d == 2:
        pytest.skip("one kind of data at the large sizes")
    rng = np.random.default_rng(d + n + M)
    N = n ** d
    t = np.arange(1, M + 1) / M
    if data == "random":
        u, f = rng.uniform(-1, 1, (batch, N, M)), rng.uniform(-1, 1, (batch, N, M)) * (n + 1) ** 2
    elif data == "smooth":
        x = np.sin(np.pi * np.arange(1, N + 1) / (N + 1))[None, :, None]
        u, f = x * t ** 0.3 * np.ones((batch, 1, 1)), x * (1 + 20 * t) * np.ones((batch, 1, 1))
    else:  # twelve orders of magnitude within a line
        u, f = (rng.uniform(-1, 1, (batch, N, M)) * 10.0 ** rng.uniform(-12, 0, (batch, N, M))
                for _ in range(2))
    lines = len(_points(d, n, G.MGWR_BLACK if n == 1 and d == 1 else G.MGWR_RED)) * batch
    bound = _bound(lines, M)
    alphas = 0.45 if batch == 1 else list(np.linspace(0.15, 0.95, batch))
    with G.Solver(d, n, M, 1.0, alphas) as s:
        colour = G.MGWR_RED
        if n == 1:  # the one point is colour 0 whatever the call names
            s.field_set(G.MGWR_H64, 0, G.MGWR_F, f[0])
            s.coarsest(G.MGWR_H64)
            got, k = s.field_get(G.MGWR_H64, 0, G.MGWR_U)[0], s.inverse_column(0).astype(Q)
            want = np.array([np.dot(k[:m + 1][::-1], f[0, 0, :m + 1].astype(Q)) for m in range(M)])
            assert float(np.abs(got - want).max()) <= bound * float(np.abs(k).sum() * np.abs(f).max())
            return
        _check(s, d, n, M, colour, u, f, batch, (0.0, 0.37, 0.5, 1.0), bound)


@pytest.mark.parametrize("scale", [1e-290, 1e290])
def test_half_sweep_scales_exactly(scale):
    # a power of two in f and u scales the half-sweep exactly, to the ends of FP64's range
    d, n, M = 1, 255, 256
    two = 2.0 ** round(np.log2(scale))
    u, f = inputs.random_field(n, M, 1), inputs.random_field(n, M, 2, scale=(n + 1.0) ** 2)
    out = []
    for c in (1.0, two):
        with G.Solver(d, n, M, 1.0, 0.5) as s:
            l = s.num_levels() - 1
            s.field_set(G.MGWR_H64, l, G.MGWR_U, c * u)
            s.field_set(G.MGWR_H64, l, G.MGWR_F, c * f)
            s.smooth(G.MGWR_H64, l, G.MGWR_RED)
            out.append(s.field_get(G.MGWR_H64, l, G.MGWR_U))
    np.testing.assert_array_equal(out[1], two * out[0])


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_infinities_and_nan_reach_the_solver(bad):
    for d, n, M in ((1, 255, 256), (1, 31, 64)):  # sliced and sums
        f = inputs.random_field(n, M, 3)
        f[n // 2, M // 3] = bad
        with G.Solver(d, n, M, 1.0, 0.5) as s:
            s.set_rhs(f)
            with pytest.raises(G.MGWRError) as e:
                s.solve(1, 1, 1, tol=1e-10, max_cycles=5)
            assert e.value.status == G.MGWR_E_NUMERIC
            l = s.num_levels() - 1
            s.field_set(G.MGWR_H64, l, G.MGWR_F, f)
            s.field_set(G.MGWR_H64, l, G.MGWR_U, np.zeros_like(f))
            s.smooth(G.MGWR_H64, l, G.MGWR_RED)
            assert not np.isfinite(s.field_get(G.MGWR_H64, l, G.MGWR_U)[n // 2]).all()


# one, three and the most lines of the FP64 sums, which take tiles of 8, 16 and 32 steps between
# them; f alone (u = 0) so that the reference is a plain convolution
@pytest.mark.parametrize("M", [64, 128, 256, 512, 1024])
def test_sums_at_the_edges_of_their_tiles(M):
    sizes = [3, 7, 15, 31, 63, 127, 255, 511, 1023]
    few = [n for n in sizes if _sums(n // 2, M)]
    for n in (few[0], few[1], few[2], few[-2], few[-1]):
        f = inputs.random_field(n, M, n)
        with G.Solver(1, n, M, 1.0, 0.35) as s:
            _check(s, 1, n, M, G.MGWR_RED, np.zeros((1, n, M)), f[None], 1, (0.0, 0.5, 1.0),
                   _bound(n // 2, M))


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("n,M", [(4095, 64), (511, 256), (127, 1024)])
def test_non_finite_values_stay_in_their_line_of_a_sliced_sweep(n, M, bad):
    assert not _sums(n // 2, M)
    f = inputs.random_field(n, M, 5)
    hit = n // 2 | 1
    f[hit, M // 3] = bad
    with G.Solver(1, n, M, 1.0, 0.5) as s:
        l = s.num_levels() - 1
        s.field_set(G.MGWR_H64, l, G.MGWR_F, f)
        s.field_set(G.MGWR_H64, l, G.MGWR_U, np.zeros_like(f))
        s.smooth(G.MGWR_H64, l, G.MGWR_RED)
        got = s.field_get(G.MGWR_H64, l, G.MGWR_U)
        assert not np.isfinite(got[hit]).all()
        assert np.isfinite(np.delete(got, hit, axis=0)).all()
        with pytest.raises(G.MGWRError) as e:
            s.set_rhs(f)
            s.solve(1, 1, 1, tol=1e-10, max_cycles=5)
        assert e.value.status == G.MGWR_E_NUMERIC


# every launch sums the same whole numbers: the bits of a half-sweep, its changes and a defect
# repeat, and lines with the same data agree with one another (each line length, groups of 16
# and of 32 lines, columns with and without slices that vanish at far lags)
@pytest.mark.parametrize("n,M", [(4095, 64), (1023, 128), (511, 256), (127, 512), (511, 512),
                                 (127, 1024), (1023, 1024)])
def test_sliced_products_repeat_their_bits(n, M):
    assert not _sums(n // 2, M)
    line = inputs.random_field(1, M, 6, scale=(n + 1.0) ** 2)[0]
    f = np.tile(line, (n, 1))
    with G.Solver(1, n, M, 1.0, 0.4) as s:
        l = s.num_levels() - 1
        s.field_set(G.MGWR_H64, l, G.MGWR_F, f)
        seen = []
        for _ in range(25):
            s.field_set(G.MGWR_H64, l, G.MGWR_U, np.zeros_like(f))
            s.smooth(G.MGWR_H64, l, G.MGWR_RED)
            u = s.field_get(G.MGWR_H64, l, G.MGWR_U)
            s.defect(G.MGWR_H64, l)
            seen.append((u, s.field_get(G.MGWR_H64, l, G.MGWR_R)))
    for u, r in seen:
        np.testing.assert_array_equal(u, seen[0][0])
        np.testing.assert_array_equal(r, seen[0][1])
    red = seen[0][0][1::2]
    np.testing.assert_array_equal(red, np.tile(red[0], (len(red), 1)))


# a line with an infinity or NaN in it: NaN throughout where it is sliced, unchanged values before
# that step and none finite from it on where it is summed
@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("n,M", [(4095, 64), (511, 256), (127, 1024), (31, 64), (15, 1024)])
def test_a_line_with_a_non_finite_value(n, M, bad):
    f = inputs.random_field(n, M, 8)
    hit, step = n // 2 | 1, M // 3
    out = []
    for g in (f, f.copy()):
        if g is not f:
            g[hit, step] = bad
        with G.Solver(1, n, M, 1.0, 0.5) as s:
            l = s.num_levels() - 1
            s.field_set(G.MGWR_H64, l, G.MGWR_F, g)
            s.field_set(G.MGWR_H64, l, G.MGWR_U, np.zeros_like(f))
            s.smooth(G.MGWR_H64, l, G.MGWR_RED)
            out.append(s.field_get(G.MGWR_H64, l, G.MGWR_U))
    if _sums(n // 2, M):
        np.testing.assert_array_equal(out[1][hit, :step], out[0][hit, :step])
        assert not np.isfinite(out[1][hit, step:]).any()
    else:
        assert np.isnan(out[1][hit]).all()
    np.testing.assert_array_equal(np.delete(out[1], hit, axis=0), np.delete(out[0], hit, axis=0))


SWEEP64 = G.KERNEL_CLASSES.index("sweep64")


def _solved(s, f):
    s.set_rhs(f)
    st = s.solve(1, 1, 1, tol=1e-10, max_cycles=40)
    return s.solution(), st.cycles


# a split that was set runs the transform it names (half-sweeps, one-point solve, whole solves with
# their zero starts, graphs and device loops), on one level or on all
@pytest.mark.parametrize("d,n,M,batch", [(1, 63, 64, 1), (2, 15, 256, 3), (2, 31, 1024, 1)])
def test_a_set_split_runs_the_transform(d, n, M, batch):
    alphas = 0.45 if batch == 1 else list(np.linspace(0.15, 0.95, batch))
    shape = (n ** d, M) if batch == 1 else (batch, n ** d, M)
    f = np.random.default_rng(9).uniform(-1, 1, shape)
    out = []
    for split, level in ((None, 0), (1, -1), (2, -1), (1, 1)):
        with G.Solver(d, n, M, 1.0, alphas) as s:
            if split is not None:
                s.set_engine_split(SWEEP64, split, level=level)
            out.append(_solved(s, f)[0])
    sliced, one, two, mixed = out
    np.testing.assert_array_equal(one, two)  # E moves butterflies between threads only
    scale = np.abs(sliced).max()
    # each form solves to 1e-10 of the defect, which bounds the difference of the solutions
    for u in (one, mixed):
        assert not np.array_equal(u, sliced)
        assert np.abs(u - sliced).max() <= 1e-9 * scale


# without memory for the bands and digits a handle runs the transforms, and the sliced products as
# soon as there is some
def test_sliced_products_come_back_with_the_memory():
    d, n, M = 2, 31, 256
    f = inputs.random_field(n ** d, M, 10)
    with G.Solver(d, n, M, 1.0, 0.5) as s:
        sliced = _solved(s, f)
    with G.Solver(d, n, M, 1.0, 0.5) as s:
        s.set_engine_split(SWEEP64, 1)
        transform = _solved(s, f)
        s.inject_nomem(1)
        s.autotune()  # no split is set any more
        s.inject_nomem(1)
        short = _solved(s, f)
        again = _solved(s, f)
    np.testing.assert_array_equal(short[0], transform[0])
    np.testing.assert_array_equal(again[0], sliced[0])
    assert not np.array_equal(sliced[0], transform[0])


# batches of few lines an instance, on both sides of the line to the transform (its rounding:
# log2(2M) stages of a few half-ulps of the norms of k and b, 1e-12 of the largest S as for every
# transform), every instance with a column of its own; and the one-point solve
@pytest.mark.parametrize("d,n,M,batch", [(1, 3, 1024, 64), (1, 7, 1024, 64), (2, 3, 1024, 48),
                                         (1, 7, 512, 64), (1, 15, 512, 64), (1, 3, 256, 96)])
def test_batches_of_few_lines_an_instance(d, n, M, batch):
    rng = np.random.default_rng(11)
    N = n ** d
    u, f = rng.uniform(-1, 1, (batch, N, M)), rng.uniform(-1, 1, (batch, N, M)) * (n + 1) ** 2
    with G.Solver(d, n, M, 1.0, list(np.linspace(0.15, 0.95, batch))) as s:
        _check(s, d, n, M, G.MGWR_RED, u, f, batch, (0.0, 1.0), 1e-12)
        s.field_set(G.MGWR_H64, 0, G.MGWR_F, f[:, :1])
        s.coarsest(G.MGWR_H64)
        got, k = s.field_get(G.MGWR_H64, 0, G.MGWR_U), s.inverse_column(0)
        for b in (0, batch - 1):
            line, kq = f[b, 0].astype(Q), k[b].astype(Q)
            want = np.array([np.dot(kq[:m + 1][::-1], line[:m + 1]) for m in range(M)])
            scale = float(np.abs(kq).sum() * np.abs(line).max())
            assert float(np.abs(got[b].reshape(M) - want).max()) <= 1e-12 * scale


# the defect with a sliced time term against extended sums.  Bound of a value, with S the largest
# sum |T| |u| of its line and A = h^-2 sum over the neighbours (|u_p| + |u_q|): the product 4e-16 S;
# the differences, at most three sums and the two subtractions from f one rounding each.
@pytest.mark.parametrize("d,n,M,batch", [(2, 63, 64, 1), (1, 1023, 128, 1), (2, 15, 256, 3),
                                         (1, 63, 512, 2), (1, 127, 1024, 1)])
@pytest.mark.parametrize("data", ["random", "wide"])
def test_sliced_defect_against_extended_sums(d, n, M, batch, data):
    rng = np.random.default_rng(12)
    N = n ** d
    assert N * batch * M * M // 2 > 1 << 22
    u, f = rng.uniform(-1, 1, (batch, N, M)), rng.uniform(-1, 1, (batch, N, M)) * (n + 1) ** 2
    if data == "wide":
        u, f = (x * 10.0 ** rng.uniform(-12, 0, (batch, N, M)) for x in (u, f))
    shape = (N, M) if batch == 1 else (batch, N, M)
    hinv2, eps = float((n + 1) ** 2), 2.0 ** -53
    alphas = 0.45 if batch == 1 else list(np.linspace(0.15, 0.95, batch))
    with G.Solver(d, n, M, 1.0, alphas) as s:
        l = s.num_levels() - 1
        s.field_set(G.MGWR_H64, l, G.MGWR_U, u.reshape(shape))
        s.field_set(G.MGWR_H64, l, G.MGWR_F, f.reshape(shape))
        norm = s.defect(G.MGWR_H64, l)
        got = s.field_get(G.MGWR_H64, l, G.MGWR_R).reshape(batch, N, M)
        r = s.toeplitz_column().reshape(batch, M)
    assert norm == np.abs(got).max()
    for b in range(batch):
        rq = r[b].astype(Q)
        for p in sorted({int(x * (N - 1)) for x in (0.0, 0.37, 0.5, 1.0)}):
            i, j = (p, 0) if d == 1 else (p % n, p // n)
            v = u[b, p].astype(Q)
            lap, A = np.zeros(M, dtype=Q), np.zeros(M)
            for ok, q in ((i > 0, p - 1), (i < n - 1, p + 1), (j > 0, p - n), (j < n - 1, p + n))[:2 * d]:
                w = u[b, q].astype(Q) if ok else 0 * v
                lap, A = lap + (v - w), A + hinv2 * np.abs(u[b, p]) + hinv2 * np.abs(w).astype(float)
            y = np.array([np.dot(rq[:m + 1][::-1], v[:m + 1]) for m in range(M)])
            S = max(np.dot(np.abs(r[b][:m + 1][::-1]), np.abs(u[b, p][:m + 1])) for m in range(M))
            want = f[b, p].astype(Q) - y - Q(hinv2) * lap
            bound = 4e-16 * S + eps * (2 * np.abs(f[b, p]) + 2 * S + 6 * A)
            err = np.abs(got[b, p].astype(Q) - want).astype(float)
            assert (err <= bound).all(), (b, p, float((err / bound).max()))
