"""Malformed incidences are error statuses on every path: the short one (sides of
at most 16,384 rows), the general one and a graph handle; in short rows and in rows
of more than 128 ids, which whole warps read; in either half of the input."""
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


@pytest.fixture(scope="module")
def inputs():
    """Both sides below the short path's limit, and both above; hyperedge 7 and
    vertex 7 have several hundred ids."""
    out = {}
    for m in (500, 20_000):
        rng = np.random.default_rng(m)
        size = rng.integers(3, 12, m)
        r = [np.repeat(np.arange(m), size), np.full(400, 7), rng.choice(m, 400, replace=False)]
        c = [rng.integers(0, m, int(size.sum())), rng.choice(m, 400, replace=False),
             np.full(400, 7)]
        out[m] = hg.from_pairs(np.concatenate(r), np.concatenate(c), m, m)
    return out


def corrupt(h, half, what, where):
    a = {"e_off": h.e_off.copy(), "e_idx": h.e_idx.copy(), "v_off": h.v_off.copy(),
         "v_idx": h.v_idx.copy()}
    off, idx = a[half + "_off"], a[half + "_idx"]
    row = 7 if where >= 0 else int(np.argmax(np.diff(off) >= 3))
    k = int(off[row]) + max(where, 0)
    if what == "unsorted":
        idx[k], idx[k + 1] = idx[k + 1], idx[k]
    elif what == "twice":
        idx[k + 1] = idx[k]
    elif what == "too_large":
        idx[off[row + 1] - 1] = h.m + 3
    elif what == "negative":
        idx[off[row]] = -1
    elif what == "first_offset":
        off[0] = 1
    elif what == "last_offset":
        off[-1] += 10
    elif what == "descending_offsets":
        off[row + 1] = off[row] - 1 if row else -1
    elif what == "offset_beyond":
        off[row + 1] = h.nnz + 5
    elif what == "mismatch":  # ascending and in range, but another id
        lo, hi = int(off[row]), int(off[row + 1])
        idx[lo:hi] = np.sort(np.append(np.delete(idx[lo:hi], max(where, 0)),
                                       np.setdiff1d(np.arange(h.m), idx[lo:hi])[-1]))
    return hg.Hypergraph(h.m, h.n, **a)


CASES = [("unsorted", -1), ("unsorted", 0), ("unsorted", 31), ("unsorted", 127), ("unsorted", 128),
         ("unsorted", 255), ("unsorted", 398), ("twice", -1), ("twice", 200), ("too_large", -1),
         ("too_large", 0), ("negative", -1), ("negative", 0), ("first_offset", -1),
         ("last_offset", -1), ("descending_offsets", -1), ("descending_offsets", 0),
         ("offset_beyond", -1), ("offset_beyond", 0), ("mismatch", -1), ("mismatch", 300)]


@pytest.mark.parametrize("m", [500, 20_000])
@pytest.mark.parametrize("half", ["e", "v"])
@pytest.mark.parametrize("what,where", CASES)
def test_malformed(inputs, m, half, what, where):
    h = inputs[m]
    dh = slg.to_device(corrupt(h, half, what, where))
    calls = [lambda: slg.count(dh, 2), lambda: slg.count(dh, 1, dual=True),
             lambda: slg.build(dh, 2), lambda: slg.Graph(dh), lambda: slg.row_work(dh, 2)]
    for call in calls:
        with pytest.raises(slg.SlgError) as ei:
            call()
        assert ei.value.status == 1


@pytest.mark.parametrize("m", [500, 20_000])
def test_the_library_goes_on(inputs, m):
    h = inputs[m]
    with pytest.raises(slg.SlgError):
        slg.count(slg.to_device(corrupt(h, "v", "mismatch", 300)), 2)
    dh = slg.to_device(h)
    for dual in (False, True):
        want = oracle.canonical(*oracle.line_graph_of(h, 2, dual=dual, threads=8))
        got = slg.build(dh, 2, dual=dual)
        assert np.array_equal(np.stack([x.cpu().numpy() for x in got], 1), want)
