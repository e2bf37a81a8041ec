"""Planning: the CSR -> CSC map, by incidences dealt out evenly or, where the rows are
long and none lasts long beside the whole, by rows."""
import time

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


def rows_alike(m, size, n, hub=0):
    """m rows of `size` random vertices, the first of at least `hub`, on the GPU."""
    gen = torch.Generator(device="cuda").manual_seed(m + hub)
    rows = torch.arange(m, device="cuda").repeat_interleave(size)
    cols = torch.randint(0, n, rows.shape, generator=gen, device="cuda")
    if hub:
        rows = torch.cat([rows, torch.zeros(hub, dtype=torch.int64, device="cuda")])
        cols = torch.cat([cols, torch.arange(hub, device="cuda") * (n // hub)])
    key = torch.unique(rows * n + cols)
    rows, cols = key // n, key % n
    by = torch.argsort(cols, stable=True)
    off = lambda x, k: torch.nn.functional.pad(torch.bincount(x, minlength=k).cumsum(0),
                                               (1, 0)).int()
    return off(rows, m), cols.int(), off(cols, n), rows[by].int()


# rows of 127, 128 and 129 vertices on average (by rows from 128 on), a longest row
# on both sides of a five-thousandth of the incidences, rows of no vertex
@pytest.mark.parametrize("m,size,n,hub", [(20_000, 126, 400_000, 0), (20_000, 140, 400_000, 0),
                                          (20_000, 140, 400_000, 400), (20_000, 140, 400_000, 700),
                                          (17_000, 1_000, 6_000_000, 0)])
def test_both_ways_of_making_the_map(m, size, n, hub):
    a = [x.cpu().numpy() for x in rows_alike(m, size, n, hub)]
    extra = np.concatenate([a[0], np.full(5, a[0][-1], a[0].dtype)])  # five empty rows
    h = hg.Hypergraph(m + 5, n, extra, *a[1:])
    dh = slg.to_device(h)
    for s in (1, 2):
        want = oracle.canonical(*oracle.line_graph_of(h, s, threads=8))
        with slg.Graph(dh) as g:
            for got in (slg.build(dh, s), g.build(s)):
                assert np.array_equal(np.stack([x.cpu().numpy() for x in got], 1), want)
    # another id in the last row of the CSC half: not the same incidence
    bad = [x.copy() for x in a]
    c = int(np.flatnonzero(np.diff(bad[2]) == 1)[-1])
    bad[3][bad[2][c]] = (bad[3][bad[2][c]] + 1) % m
    with pytest.raises(slg.SlgError) as ei:
        slg.count(slg.to_device(hg.Hypergraph(m + 5, n, extra, bad[1], bad[2], bad[3])), 1)
    assert ei.value.status == 1


def test_long_rows_pass_through_the_columns_together():
    """100,000 rows of 800 of 20M columns, with and without a row of 40,000: with it
    the incidences are dealt out evenly, and the columns that the warps look up at
    a time lie far apart."""
    took = {}
    for hub in (0, 40_000):
        dh = slg.DeviceHypergraph(100_000, 20_000_000, *rows_alike(100_000, 800, 20_000_000, hub))
        got = []
        for _ in range(5):
            torch.cuda.synchronize()
            t = time.perf_counter()
            slg.Graph(dh).close()
            torch.cuda.synchronize()
            got.append(time.perf_counter() - t)
        took[hub] = sorted(got)[1]
        del dh
        torch.cuda.empty_cache()
    assert took[0] < 0.85 * took[40_000], took
