"""The sparse bin (rows of 1,025 to 16,384 wedges with s >= 2, above the CTA
bins only when their far ends are sparse in their id span): a first pass
marks far ends seen twice in a Bloom filter and claims them as candidates
in a shared table, a second pass counts the candidates' wedges exactly.
Rows above 8,192 wedges run in the kernel instance with the larger table,
the others in the one with the smaller table; a row whose candidates or
survivors do not fit its table is handed to the giant bin.  Every case is
compared with the CPU oracle element by element."""
import numpy as np
import pytest

import hypergen as hg
import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
slg = pytest.importorskip("paper_2010_11448_gb300")


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2010_11448_gb300 import build_lib
    build_lib.build()
    slg.load()


def as_np(t):
    i, j, w = t
    cols = [i.cpu().numpy(), j.cpu().numpy()]
    cols.append(w.cpu().numpy() if w is not None else np.zeros_like(cols[0]))
    return np.stack(cols, 1).astype(np.int64) if cols[0].shape[0] else np.zeros((0, 3), np.int64)


def many_repeats(m=100_000, n=20_000, k=3, shared=3000, seed=4):
    """Hyperedge 0 holds vertices 0..k-1; hyperedges 10000 .. 10000+shared-1
    hold all of them too (plus a few random vertices), so row 0 has k x
    shared wedges and `shared` distinct far ends that each repeat k times:
    more repeated far ends than one window of the sparse bin's table holds.
    The rest are small random hyperedges over the other vertices."""
    rng = np.random.default_rng(seed)
    rows = []
    for e in range(m):
        if e == 0:
            rows.append(np.arange(k))
        elif 10_000 <= e < 10_000 + shared:
            extra = rng.choice(np.arange(k, n), 3, replace=False)
            rows.append(np.concatenate([np.arange(k), np.sort(extra)]))
        else:
            rows.append(np.sort(rng.choice(np.arange(k, n), int(rng.integers(1, 6)),
                                           replace=False)))
    return hg.from_rows(rows, n)


@pytest.mark.parametrize("k", [2, 3])
def test_window_overflow_split(k):
    h = many_repeats(k=k)
    dh = slg.to_device(h)
    for s in (2, k):
        got = as_np(slg.build(dh, s))
        st = slg.last_stats()
        assert st["rows_bin"][4] >= 1, "row 0 did not take the sparse bin"
        assert np.array_equal(got, oracle.canonical(*oracle.line_graph_of(h, s, threads=8)))
        # the short-circuit gives the same pairs
        i, j, w = slg.build(dh, s, unweighted=True)
        assert w is None
        assert np.array_equal(np.stack([i.cpu().numpy(), j.cpu().numpy()], 1), got[:, :2])
        assert slg.count(dh, s) == got.shape[0]


def test_rows_across_two_windows():
    # The dual of a Chung-Lu hypergraph with 1.5M vertices: long rows whose
    # far ends spread over an id span of up to 1.5M (a Bloom filter of at
    # most 2^17 bits per row), on both sides of the 8,192-wedge split.
    h = hg.chung_lu(200_000, 1_500_000, seed=33, size_cap=10_000)
    dh = slg.to_device(h)
    m, n, off, idx = oracle.side(h, True)
    deg = np.diff(off)
    heavy = np.argsort(-deg, kind="stable")[:2000]
    rows = np.unique(np.concatenate([heavy, np.arange(0, m, 211)])).astype(np.int32)
    want2 = oracle.canonical(*oracle.line_graph(m, n, off, idx, 2, rows=rows, threads=16))
    rows_t = torch.from_numpy(rows).cuda()
    for s in (2, 3, 5):
        i, j, w = slg.build(dh, s, dual=True)
        st = slg.last_stats()
        assert st["rows_bin"][4] > 100
        sel = torch.isin(i, rows_t)
        got = np.stack([i[sel].cpu().numpy(), j[sel].cpu().numpy(), w[sel].cpu().numpy()],
                       1).astype(np.int64)
        assert np.array_equal(got, want2[want2[:, 2] >= s]), s
        key = i.long() * m + j.long()
        assert bool(torch.all(key[1:] > key[:-1])) and bool(torch.all(w >= s))
        assert i.shape[0] == slg.count(dh, s, dual=True)


def split_rows(m=200_000, n=400_000, seed=8):
    """Small random hyperedges (1 to 4 of vertices 1000 .. n-1) plus hubs:
    row 0 holds hubs 0..19, each also in 640 random hyperedges (about
    12,800 wedges at s = 2, 9,900 at s = 3: the larger-table instance); row
    1 holds hubs 20..29, each in 500 (about 5,000: the smaller-table
    instance); row 2 holds hubs 30 and 31, both in the same 3,000 random
    hyperedges, so that row 2 has 3,000 far ends of two wedges each, more
    distinct candidates than a 2,048-slot table holds, and every one of
    those 3,000 rows meets the others in two vertices.  All far ends spread
    over ids up to m: the rows are sparse in their span."""
    rng = np.random.default_rng(seed)
    size = rng.integers(1, 5, m)
    r = [np.repeat(np.arange(m), size), np.zeros(20, np.int64), np.ones(10, np.int64),
         np.full(2, 2)]
    c = [rng.integers(1000, n, int(size.sum())), np.arange(20), np.arange(20, 30),
         np.array([30, 31])]
    for hub in range(30):
        f = rng.choice(np.arange(3, m), 640 if hub < 20 else 500, replace=False)
        r.append(f)
        c.append(np.full(f.shape[0], hub))
    f = rng.choice(np.arange(3, m), 3000, replace=False)
    r += [f, f]
    c += [np.full(3000, 30), np.full(3000, 31)]
    return hg.from_pairs(np.concatenate(r), np.concatenate(c), m, n)


@pytest.mark.parametrize("s", [2, 3])
def test_two_instances_and_hand_off(s):
    from test_shard_cpu import row_work_by_definition
    h = split_rows()
    work = row_work_by_definition(h, s, False)
    assert work[0] > 8192 and 1024 < work[1] <= 8192 and 1024 < work[2] <= 8192
    dh = slg.to_device(h)
    want = oracle.canonical(*oracle.line_graph_of(h, s, threads=8))
    got = as_np(slg.build(dh, s))
    st = slg.last_stats()
    assert st["rows_bin"][4] >= 3, "rows 0, 1 and 2 take the sparse bin"
    # row 2's 3,000 candidates cannot fit the smaller table: handed over
    assert st["rows_bin"][3] >= 1, "no sparse row was handed to the giant bin"
    assert np.array_equal(got, want)
    i, j, w = slg.build(dh, s, unweighted=True)
    assert w is None
    assert np.array_equal(np.stack([i.cpu().numpy(), j.cpu().numpy()], 1), want[:, :2])
    assert slg.count(dh, s) == want.shape[0]


def aside_rows(m=500_000, n=900_000, seed=15, small=(1, 4)):
    """Three rows sparse in 500,000 ids, the other rows of small[0] to
    small[1] - 1 random vertices.  Row 0: two vertices with the same
    6,000 other hyperedges (more survivors than one range can order) and 18
    rare ones.  Row 1: 600 vertices of 40 hyperedges (more tails than a batch
    holds, nothing set aside), 100 hyperedges holding seven of them.  Row 2:
    12 vertices of 100 to 4,000 hyperedges (all but a few of its wedges are in
    the longest tails), 50 hyperedges holding nine of them."""
    rng = np.random.default_rng(seed)
    size = rng.integers(*small, m)
    r = [np.repeat(np.arange(m), size)]
    c = [rng.integers(10_000, n, int(size.sum()))]

    def add(row, col):
        r.append(np.broadcast_to(row, np.broadcast(row, col).shape).ravel())
        c.append(np.broadcast_to(col, np.broadcast(row, col).shape).ravel())

    f = rng.choice(np.arange(3, m), 6_000, replace=False)
    add(f, 0)
    add(f, 1)
    add(0, np.arange(20))
    for v in range(600):
        add(rng.choice(np.arange(3, m), 40, replace=False), 1_000 + v)
    add(1, np.arange(1_000, 1_600))
    for x in rng.choice(np.arange(3, m), 100, replace=False):
        add(x, 1_000 + rng.choice(600, 7, replace=False))
    for v in range(12):
        add(rng.choice(np.arange(3, m), 100 if v < 6 else 4_000, replace=False), 3_000 + v)
    add(2, np.arange(3_000, 3_012))
    for x in rng.choice(np.arange(3, m), 50, replace=False):
        add(x, 3_000 + rng.choice(12, 9, replace=False))
    return hg.from_pairs(np.concatenate(r), np.concatenate(c), m, n)


@pytest.fixture(scope="module")
def aside():
    h = aside_rows()
    return h, slg.to_device(h)


@pytest.mark.parametrize("s", [2, 3, 4, 5, 6, 9, 12])
def test_tails_set_aside_and_split_ranges(aside, s):
    h, dh = aside
    want = oracle.canonical(*oracle.line_graph_of(h, s, threads=8))
    got = as_np(slg.build(dh, s))
    if s <= 3:  # (the small rows leave at larger s)
        assert slg.last_stats()["rows_bin"][4] > 0
    assert np.array_equal(got, want)
    i, j, w = slg.build(dh, s, unweighted=True)
    assert w is None and np.array_equal(
        np.stack([i.cpu().numpy(), j.cpu().numpy()], 1), want[:, :2])
    assert slg.count(dh, s) == want.shape[0]


@pytest.fixture(scope="module")
def aside_large():
    h = aside_rows(small=(12, 15))
    return h, slg.to_device(h)


@pytest.mark.parametrize("s", [4, 6, 9, 12])
def test_tails_set_aside_large_rows(aside_large, s):
    # rows of 12 and more vertices: the far ends stay at these thresholds
    h, dh = aside_large
    rows = np.unique(np.concatenate([np.arange(3), np.arange(0, h.m, 53)])).astype(np.int32)
    m, n, off, idx = oracle.side(h, False)
    want = oracle.canonical(*oracle.line_graph(m, n, off, idx, s, rows=rows, threads=8))
    got = as_np(slg.build(dh, s))
    assert slg.last_stats()["rows_bin"][4] > 0
    assert np.array_equal(got[np.isin(got[:, 0], rows)], want)
    assert slg.count(dh, s) == got.shape[0]


# the rows bin: one batch of 32 tails and one more, wedges up to its limit of
# 1,024, more far ends of two wedges than its table of 256 holds (handed over)
@pytest.mark.parametrize("k,deg", [(2, 500), (2, 512), (31, 33), (32, 32), (33, 31), (40, 25),
                                   (3, 120)])
def test_short_rows(k, deg):
    rng = np.random.default_rng(k * deg)
    m, n, hubs = 60_000, 200_000, 40
    r, c = [], []
    for hub in range(hubs):  # row `hub`: k vertices of `deg` other hyperedges each
        v = 1_000 + hub * k + np.arange(k)
        r.append(np.full(k, hub))
        c.append(v)
        far = rng.choice(np.arange(hubs, m), deg, replace=False)
        for x in range(k):  # the same far ends for the first two vertices
            f = far if x < 2 else rng.choice(np.arange(hubs, m), deg, replace=False)
            r.append(f)
            c.append(np.full(deg, v[x]))
    size = rng.integers(4, 8, m)
    r.append(np.repeat(np.arange(m), size))
    c.append(rng.integers(10_000, n, int(size.sum())))
    h = hg.from_pairs(np.concatenate(r), np.concatenate(c), m, n)
    dh = slg.to_device(h)
    for s in (2, 3, 4, 6):
        want = oracle.canonical(*oracle.line_graph_of(h, s, threads=8))
        assert np.array_equal(as_np(slg.build(dh, s)), want), s
        i, j, w = slg.build(dh, s, unweighted=True)
        assert w is None and np.array_equal(
            np.stack([i.cpu().numpy(), j.cpu().numpy()], 1), want[:, :2])
        assert slg.count(dh, s) == want.shape[0]


# the flat bin: rows of more than 48 vertices with less than 32 far ends per tail
# on average, 1,025 to 16,384 wedges, above 8,192 in the instance with the larger
# table.  Both sides of each of these limits, one batch of tails (256) and more,
# more survivors than it orders (992: handed over), tails of no far end
@pytest.mark.parametrize("k,lens,repeat", [
    (48, (31, 32), 3), (49, (31,), 3), (49, (32,), 3), (49, (0, 62), 3), (256, (1, 7, 8, 9), 3),
    (257, (0, 1, 8, 9, 31, 32, 33), 3), (300, (4,), 3), (512, (16,), 3), (513, (16, 17), 3),
    (512, (16,), 8), (1_024, (16,), 3), (1_025, (16,), 4), (1_000, (0, 1, 30), 2),
    (600, (25,), 15)])
@pytest.mark.parametrize("mixed", [False, True])
def test_short_tails(k, lens, repeat, mixed):
    m, n = 2_000_000, 120_000
    rng = np.random.default_rng(k + repeat)
    total = sum(lens[v % len(lens)] for v in range(k))
    r, c = [np.zeros(k, np.int64)], [np.arange(k)]
    pool = rng.choice(np.arange(10, m), max(total // repeat, 100), replace=False)
    for v in range(k):  # far ends from a pool: most occur in several tails
        d = lens[v % len(lens)]
        r.append(rng.choice(pool, d, replace=False))
        c.append(np.full(d, v))
    r.append(np.repeat(pool, 3))
    c.append(rng.integers(10_000, n, 3 * pool.size))
    if mixed:  # more wedges in a row of long tails: the sparse bin takes both rows
        for v in range(9):
            f = rng.choice(pool, pool.size // 2, replace=False) if v < 2 else \
                rng.choice(np.arange(10, m), 5_000, replace=False)
            r += [f, np.ones(1, np.int64)]
            c += [np.full(f.size, 5_000 + v), np.full(1, 5_000 + v)]
    h = hg.from_pairs(np.concatenate(r), np.concatenate(c), m, n)
    dh = slg.to_device(h)
    for s in (2, 3, 4, 6):
        want = oracle.canonical(*oracle.line_graph_of(h, s, threads=8))
        got = as_np(slg.build(dh, s))
        assert np.array_equal(got, want), s
        i, j, w = slg.build(dh, s, unweighted=True)
        assert w is None and np.array_equal(
            np.stack([i.cpu().numpy(), j.cpu().numpy()], 1), want[:, :2])
        assert slg.count(dh, s) == want.shape[0]
        if s == 3:
            plan = slg.Plan([dh], [s])
            plan.execute()
            assert np.array_equal(as_np(plan.results()[0]), want)


def test_short_tails_do_not_take_a_warp_each():
    """100,000 rows of 250 vertices with a mean of 13 rows per vertex: nothing
    but short tails.  A warp per tail and a rank among all tails took 58 CTA cycles
    per wedge, flattened tails 11."""
    m, n = 100_000, 1_900_000
    gen = torch.Generator(device="cuda").manual_seed(1)
    rows = torch.arange(m, device="cuda").repeat_interleave(250)
    cols = torch.randint(0, n, rows.shape, generator=gen, device="cuda")
    key = torch.unique(rows * n + cols)
    rows, cols = key // n, key % n
    by = torch.argsort(cols, stable=True)
    off = lambda x, k: torch.nn.functional.pad(torch.bincount(x, minlength=k).cumsum(0),
                                               (1, 0)).int()
    dh = slg.DeviceHypergraph(m, n, off(rows, m), cols.int(), off(cols, n), rows[by].int())
    slg.count(dh, 2)
    st = slg.last_stats()
    assert st["rows_bin"][4] > 30_000
    assert sum(st["sparse_cycles"]) < 25 * st["wedges_bin"][4]


def hubs(k, count, m=40_000, shared=500, seed=7):
    """`count` rows with late ids of `k` vertices each, of which `shared` draws are
    in one later row: many tails, almost all of them empty."""
    rng = np.random.default_rng(seed)
    base = np.repeat(np.arange(m - 2 * count), 3)
    hub = np.arange(count)
    r = [base, np.repeat(m - 2 * count + hub, k), np.repeat(m - count + hub, shared)]
    c = [rng.integers(0, 50_000, base.size),
         50_000 + (hub[:, None] * k + np.arange(k)).ravel(),
         50_000 + (hub[:, None] * k + rng.integers(0, k, (count, shared))).ravel()]
    return hg.from_pairs(np.concatenate(r), np.concatenate(c), m, 50_000 + count * k)


# on both sides of the 16,384 vertices up to which a warp takes a row
@pytest.mark.parametrize("k", [16_383, 16_384, 16_385, 40_000])
def test_rows_of_many_vertices_and_few_wedges(k):
    h = hubs(k, 10)
    dh = slg.to_device(h)
    for s in (2, 3, 50):
        want = oracle.canonical(*oracle.line_graph_of(h, s, threads=8))
        assert np.array_equal(as_np(slg.build(dh, s)), want), s
        assert slg.count(dh, s) == want.shape[0]
        i, j, w = slg.build(dh, s, unweighted=True)
        assert w is None and np.array_equal(
            np.stack([i.cpu().numpy(), j.cpu().numpy()], 1), want[:, :2])


def test_rows_of_many_vertices_are_not_left_to_a_warp():
    """At s = 1 a CTA walks such a row; a warp took three times as long."""
    dh = slg.to_device(hubs(100_000, 4))
    slg.set_profiling(True)
    try:
        ms = {}
        for s in (1, 2):
            got = []
            for _ in range(5):
                slg.count(dh, s)
                got.append(slg.last_stats()["ms_walk"][1])
            ms[s] = sorted(got)[2]
    finally:
        slg.set_profiling(False)
    assert ms[2] < 1.7 * ms[1], ms


# tails alike (the longest no eighth of the row) of 32 to 127 far ends on average, in
# rows of more than 32 vertices; a longest tail at, below and above that share; above
# 16,384 wedges
@pytest.mark.parametrize("k,lens,repeat", [
    (32, (40,), 3), (33, (40,), 3), (34, (100, 127), 4), (40, (128,), 4), (64, (127,), 5),
    (33, (60, 60, 60, 60, 60, 60, 60, 60, 60, 60, 267), 3),
    (33, (60, 60, 60, 60, 60, 60, 60, 60, 60, 60, 600), 3),
    (130, (126,), 8), (131, (126,), 8), (300, (64,), 10)])
@pytest.mark.parametrize("mixed", [False, True])
def test_tails_alike(k, lens, repeat, mixed):
    test_short_tails(k, lens, repeat, mixed)
