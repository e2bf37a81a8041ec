"""Sides of at most 16,384 rows (the short path): every entry point that takes
it, against the oracle, at its largest side and one row beyond."""
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


def as_np(t):
    return np.stack([x.cpu().numpy() for x in t], 1).astype(np.int64)


def check(h, s, dual):
    dh = slg.to_device(h)
    want = oracle.canonical(*oracle.line_graph_of(h, s, dual=dual, threads=8))
    got = as_np(slg.build(dh, s, dual=dual))
    assert np.array_equal(got, want)
    assert slg.last_stats()["wedges"] == oracle.wedges(*oracle.side(h, dual), s)
    assert slg.count(dh, s, dual) == want.shape[0]
    i, j, w = slg.build(dh, s, dual=dual, unweighted=True)
    assert w is None and np.array_equal(
        np.stack([i.cpu().numpy(), j.cpu().numpy()], 1), want[:, :2])
    R = dh.rows(dual)
    ptr = np.concatenate([[0], np.cumsum(np.bincount(want[:, 0], minlength=R))])
    p, j, w = slg.build_csr(dh, s, dual)
    assert np.array_equal(p.cpu().numpy(), ptr) and np.array_equal(j.cpu().numpy(), want[:, 1])
    assert np.array_equal(slg.row_offsets(dh, s, dual).cpu().numpy(), ptr)
    with slg.Graph(dh) as g:
        assert np.array_equal(as_np(g.build(s, dual)), want)
        assert g.count(s, dual) == want.shape[0]
    a, b = R // 3, (2 * R + 2) // 3
    part = want[(want[:, 0] >= a) & (want[:, 0] < b)]
    got = slg.build_rows(dh, s, a, b, dual, capacity=max(part.shape[0], 1))
    assert np.array_equal(as_np(got), part)
    if want.shape[0] > 1:
        with pytest.raises(slg.SlgError) as ei:
            slg.build(dh, s, dual, capacity=want.shape[0] - 1)
        assert ei.value.status == 2 and ei.value.needed == want.shape[0]


@pytest.mark.parametrize("m,n", [(16_384, 3_001), (16_385, 3_001), (33, 70), (31, 16_384)])
@pytest.mark.parametrize("s", [1, 2, 5])
def test_short_path(m, n, s):
    h = hg.chung_lu(m, n, seed=m + s, size_cap=600)
    for dual in (False, True):
        check(h, s, dual)


def test_wide_counters_and_many_tails():
    # 70,000 shared vertices: counts above 16 bits, rows of many batches of
    # tails; a hub vertex in every hyperedge: a tail for whole warps
    rows = [list(range(70_000)), list(range(1, 70_001)), [0, 1, 2]]
    rows += [[0, 70_002 + k] for k in range(300)]
    h = hg.from_rows(rows, 70_400)
    for s in (1, 2, 69_999, 70_000):
        check(h, s, False)


@pytest.mark.parametrize("rows", [[], [[]], [[], []], [[0]], [[0], [0]], [[1], []]])
def test_tiny(rows):
    h = hg.from_rows(rows, 2)
    for dual in (False, True):
        check(h, 1, dual)
