"""The dense bin (rows counted in windows of packed counters): counter widths
at their largest value, window edges, every list of tails it keeps."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import hypergen as hg  # noqa: E402
import oracle  # noqa: E402
import paper_2010_11448_gb300 as slg  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2010_11448_gb300 import build_lib
    build_lib.build()
    slg.load()


def hub_rows(k, m, n=700, seed=3):
    """Row 0 holds vertices 0 .. k-1 and so do the last two rows (weights k:
    the largest a counter of the row has to hold); the rows between hold 1 to
    4 random vertices, so that row 0's far ends cover ids up to m."""
    rng = np.random.default_rng(seed + k)
    size = rng.integers(1, 5, m - 3)
    r = np.concatenate([np.zeros(k, np.int64), np.repeat(np.arange(1, m - 2), size),
                        np.full(k, m - 2), np.full(k, m - 1)])
    hub = np.arange(k)
    c = np.concatenate([hub, rng.integers(0, n, int(size.sum())), hub, hub])
    return hg.from_pairs(r, c, m, n)


def as_np(t):
    return np.stack([x.cpu().numpy() for x in t], 1).astype(np.int64)


# 4-, 8- and 16-bit counters at both ends of their range; 600 tails: the list
# beyond shared memory.  120,000 ids cross a window of every width.
@pytest.mark.parametrize("k,m", [(15, 120_000), (16, 120_000), (255, 60_000), (256, 120_000),
                                 (600, 110_000), (15, 3_001)])
def test_counter_widths_and_windows(k, m):
    h = hub_rows(k, m)
    dh = slg.to_device(h)
    for s in (1, 2, 3, k):
        want = oracle.canonical(*oracle.line_graph_of(h, s, threads=8))
        got = as_np(slg.build(dh, s))
        st = slg.last_stats()
        if m > 10_000 and s <= 2:  # (fewer far ends are left at larger s)
            assert st["rows_bin"][3] > 0
        assert np.array_equal(got, want), s
        assert (0, m - 1, k) in map(tuple, got[got[:, 0] == 0])
        i, j, w = slg.build(dh, s, unweighted=True)
        assert w is None and np.array_equal(
            np.stack([i.cpu().numpy(), j.cpu().numpy()], 1), want[:, :2])
        assert slg.count(dh, s) == want.shape[0]


def test_long_tails_are_cut():
    # two tails of 60,000 entries in one window: each is swept as several
    m = 60_000
    rng = np.random.default_rng(1)
    r = np.concatenate([np.arange(m), np.arange(m), np.arange(m)])
    c = np.concatenate([np.zeros(m, np.int64), np.ones(m, np.int64),
                        rng.integers(2, 5_000, m)])
    keep = (r < 3) | (rng.random(r.shape[0]) < 0.6)
    h = hg.from_pairs(r[keep], c[keep], m, 5_000)
    rows = np.array([0, 1, 2, 777, 30_000, m - 2], np.int32)
    mm, n, off, idx = oracle.side(h, False)
    for s in (1, 2):
        want = oracle.canonical(*oracle.line_graph(mm, n, off, idx, s, rows=rows, threads=8))
        ptr = slg.row_offsets(slg.to_device(h), s).cpu().numpy()
        for e in rows:
            n_e = int(ptr[e + 1] - ptr[e])
            i, j, w = slg.build_rows(slg.to_device(h), s, int(e), int(e) + 1,
                                     capacity=max(n_e, 1))
            assert np.array_equal(as_np((i, j, w)), want[want[:, 0] == e]), (s, e)


# the longest tails are split over the warps in blocks of 32 entries: one block
# less, exactly and more than a round of all warps, alone, with others beside
# them and with the whole length in one window or spread over all
@pytest.mark.parametrize("tails", [(2_049,), (4_000, 4_000), (1_023, 1_025, 2_080, 40),
                                   (1_500,) * 15, (1_500,) * 17, (3_000, 255, 256, 257, 31, 33)])
@pytest.mark.parametrize("spread", [True, False])
def test_split_tails(tails, spread):
    m, n = 100_000, 50_000
    rng = np.random.default_rng(len(tails))
    r, c = [np.zeros(len(tails), np.int64)], [np.arange(len(tails))]
    for v, deg in enumerate(tails):
        far = rng.choice(np.arange(1, m) if spread else np.arange(90_000, 95_000), deg, False)
        r.append(far)
        c.append(np.full(deg, v))
    size = rng.integers(1, 4, m - 1)
    r.append(np.repeat(np.arange(1, m), size))
    c.append(rng.integers(100, n, int(size.sum())))
    h = hg.from_pairs(np.concatenate(r), np.concatenate(c), m, n)
    dh = slg.to_device(h)
    for s in (1, 2, 3):
        want = oracle.canonical(*oracle.line_graph_of(h, s, threads=8))
        assert np.array_equal(as_np(slg.build(dh, s)), want), s
        assert slg.count(dh, s) == want.shape[0]


def test_more_tails_than_wedges_per_window():
    """Row 0 has 20,000 vertices and 21 windows of 96K ids.  With tails of 3 far
    ends a window has a seventh of a wedge per visited tail, and the row is counted
    elsewhere although it has 2,000 wedges per window; with tails of 60 it is dense."""
    m, k = 2_000_000, 20_000
    for tail, dense in ((3, False), (60, True)):
        rng = np.random.default_rng(tail)
        r = np.concatenate([np.zeros(k, np.int64), rng.integers(1, m, k * tail)])
        c = np.concatenate([np.arange(k), np.repeat(np.arange(k), tail)])
        extra = rng.integers(k, k + 50_000, 2 * k * tail)  # far ends of three vertices
        h = hg.from_pairs(np.concatenate([r, np.repeat(r[k:], 2)]), np.concatenate([c, extra]),
                          m, k + 50_000)
        dh = slg.to_device(h)
        n, nv, off, idx = oracle.side(h, False)
        for s in (2, 3):
            want = oracle.canonical(*oracle.line_graph(n, nv, off, idx, s,
                                                       rows=np.zeros(1, np.int32), threads=8))
            pairs = int(slg.row_offsets(dh, s)[1])
            i, j, w = slg.build_rows(dh, s, 0, 1, capacity=max(pairs, 1))
            st = slg.last_stats()
            assert (st["giant_cycles"][3] > 0) == dense, (tail, s)
            assert np.array_equal(as_np((i, j, w)), want), (tail, s)


# 16-bit counters at their largest value, and 32-bit ones, on a side above the
# short path's 16,384 rows: weights of the row's size
@pytest.mark.parametrize("k", [65_535, 65_536, 70_000])
def test_widest_counters(k):
    h = hub_rows(k, 20_000, n=k + 100)
    dh = slg.to_device(h)
    for s in (1, 2, k):
        want = oracle.canonical(*oracle.line_graph_of(h, s, threads=8))
        got = as_np(slg.build(dh, s))
        assert slg.last_stats()["giant_cycles"][3] > 0
        assert np.array_equal(got, want), s
        assert (0, 19_999, k) in map(tuple, got[got[:, 0] == 0])
        i, j, w = slg.build(dh, s, unweighted=True)
        assert w is None and np.array_equal(
            np.stack([i.cpu().numpy(), j.cpu().numpy()], 1), want[:, :2])
        assert slg.count(dh, s) == want.shape[0]


# the large-window instance splits its longest tails (1,024 entries per window and
# more than a sixteenth of the row) over 32 warps: a round of all warps is 1,024
# entries, a step two rounds.  One entry less and more than a round and a step, 15
# tails and one too many, in one window and in two, all in a part of the window and
# spread
@pytest.mark.parametrize("tails", [(1_025,), (2_047, 2_048), (2_049, 4_097, 3_072, 1_024),
                                   (30_000,), (33_000, 33_025), (2_000,) * 15, (2_000,) * 17])
@pytest.mark.parametrize("m,spread", [(90_000, True), (150_000, False)])
def test_split_tails_of_the_large_windows(tails, m, spread):
    n, few = 50_000, 300
    rng = np.random.default_rng(len(tails) + m)
    r, c = [np.zeros(len(tails) + few, np.int64)], [np.arange(len(tails) + few)]
    lo, hi = (1, m) if spread else (m // 2, m // 2 + 40_000)
    for v, deg in enumerate(tails):
        r.append(rng.choice(np.arange(lo, hi), deg, replace=False))
        c.append(np.full(deg, v))
    r.append(rng.integers(1, m, 3 * few))  # short tails beside them
    c.append(np.repeat(len(tails) + np.arange(few), 3))
    size = rng.integers(1, 4, m - 1)
    r.append(np.repeat(np.arange(1, m), size))
    c.append(rng.integers(1_000, n, int(size.sum())))
    h = hg.from_pairs(np.concatenate(r), np.concatenate(c), m, n)
    dh = slg.to_device(h)
    mm, nn, off, idx = oracle.side(h, False)
    for s in (1, 2, 3):
        want = oracle.canonical(*oracle.line_graph(mm, nn, off, idx, s, rows=np.zeros(1, np.int32),
                                                   threads=8))
        got = as_np(slg.build_rows(dh, s, 0, 1, capacity=max(want.shape[0], 1)))
        if sum(tails) > 2 * 2_000 and s <= 2:
            assert slg.last_stats()["giant_cycles"][3] > 0
        assert np.array_equal(got, want), s
