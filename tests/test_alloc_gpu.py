"""Builds that allocate their outputs by the pair count (one walk): equal to a
build into arrays of that size, also when the walk's staging area turns out
too small (short path: walked again; general path: walked again straight to
the output, through every bin)."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import hypergen as hg  # noqa: E402
import paper_2010_11448_gb300 as slg  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2010_11448_gb300 import build_lib
    build_lib.build()
    slg.load()


def same(h, s, dual=False):
    dh = slg.to_device(h)
    ref = slg.build(dh, s, dual, capacity=max(slg.count(dh, s, dual), 1))
    rows = dh.rows(dual)
    ptr = torch.zeros(rows + 1, dtype=torch.int64, device="cuda")
    ptr[1:] = torch.bincount(ref[0].long(), minlength=rows).cumsum(0)
    with slg.Graph(dh) as g:
        for got in (slg.build(dh, s, dual), g.build(s, dual)):
            assert all(torch.equal(a, b) for a, b in zip(got, ref))
        for got in (slg.build(dh, s, dual, unweighted=True), g.build(s, dual, unweighted=True)):
            assert got[2] is None and all(torch.equal(a, b) for a, b in zip(got[:2], ref))
    p, j, w = slg.build_csr(dh, s, dual)
    assert torch.equal(p, ptr) and torch.equal(j, ref[1]) and torch.equal(w, ref[2])
    return int(ref[0].numel())


def groups(count, size, k, extra):
    """`count` groups of `size` equal hyperedges of k vertices, dealt out over
    the ids, and `extra` empty ones: every wedge belongs to a pair of weight k."""
    m = count * size + extra
    rng = np.random.default_rng(count)
    ids = rng.permutation(m)[: count * size].reshape(count, size)
    r = np.repeat(ids.ravel(), k)
    c = np.repeat(np.arange(count) * k, size)[:, None] + np.arange(k)
    return hg.from_pairs(r, c.ravel(), m, count * k)


def test_outputs_by_count():
    for m, n in ((900, 2_000), (30_000, 60_000)):
        h = hg.chung_lu(m, n, seed=m, size_cap=3000)
        for dual in (False, True):
            for s in (1, 2, 6, 10_000):
                same(h, s, dual)


# short path; warp, CTA-S, dense and sparse bins
@pytest.mark.parametrize("count,size,k,extra", [
    (20, 800, 2, 0), (20_000, 24, 2, 0), (400, 200, 2, 0), (10, 3_000, 2, 0),
    (10, 3_000, 2, 500_000), (6, 3_000, 20, 500_000)])
def test_lists_longer_than_the_staging_area(count, size, k, extra):
    h = groups(count, size, k, extra)
    pairs = count * size * (size - 1) // 2
    assert same(h, 2) == pairs


def test_refused():
    lib = slg.load()
    dh = slg.to_device(hg.uniform(50, 80, 1, 5, seed=2))
    n = ctypes.c_int64(0)
    cb = slg._AllocFn(lambda *a: 1)
    args = (ctypes.byref(dh.struct), 1)
    tail = (None, cb, None, ctypes.byref(n), None)
    assert lib.slg_build_alloc(*args, slg.SLG_ALGO_PLAIN, *tail) == 6
    assert lib.slg_build_alloc(*args, slg.SLG_RELABEL_ASC, *tail) == 6
    assert lib.slg_build_alloc(*args, 0, *tail) == 3  # no memory
    nothing = slg._AllocFn(lambda *a: 0)  # no arrays given
    assert lib.slg_build_alloc(*args, 0, None, nothing, None, ctypes.byref(n), None) == 1
    with pytest.raises(slg.SlgError) as ei:
        slg.build(dh, 0)
    assert ei.value.status == 1


# the short path and the general one, lists that fit the staging area and longer ones
@pytest.mark.parametrize("count,size,extra", [(20, 30, 0), (20, 800, 0), (20, 30, 20_000),
                                              (20_000, 24, 0)])
def test_the_callback_may_call_the_library(count, size, extra):
    h = groups(count, size, 2, extra)
    dh = slg.to_device(h)
    other = [slg.to_device(hg.uniform(m, 2 * m, 1, 20, seed=4)) for m in (300, 30_000)]
    want = [slg.count(x, 1) for x in other]
    ref = slg.build(dh, 2, capacity=slg.count(dh, 2))
    stats = slg.last_stats()
    out, seen = [], []

    def alloc(_, n, oi, oj, ow):
        seen.extend(slg.count(x, 1) for x in other)
        out.extend(torch.full((n,), -1, dtype=torch.int32, device="cuda") for _ in range(3))
        for p, t in zip((oi, oj, ow), out):
            p[0] = t.data_ptr()
        return 0

    n = ctypes.c_int64(0)
    rc = slg.load().slg_build_alloc(ctypes.byref(dh.struct), 2, 0, None, slg._AllocFn(alloc), None,
                                    ctypes.byref(n), None)
    torch.cuda.synchronize()
    assert rc == 0 and seen == want and n.value == ref[0].numel()
    assert all(torch.equal(a, b) for a, b in zip(out, ref))
    got = slg.last_stats()
    assert all(got[k] == stats[k] for k in ("wedges", "pairs", "rows_active", "rows_bin"))


def test_statistics_of_a_list_walked_twice():
    # warp-sized rows; rows of the dense and the sparse bin
    for args in ((20_000, 24, 2, 0), (10, 3_000, 2, 0), (10, 3_000, 2, 500_000)):
        dh = slg.to_device(groups(*args))
        once = slg.build(dh, 2, capacity=slg.count(dh, 2))
        want = slg.last_stats()
        got = slg.build(dh, 2)
        st = slg.last_stats()
        assert st["pairs"] == got[0].numel() == once[0].numel()
        assert sum(st["pairs_bin"]) == st["pairs"] and st["pairs_bin"] == want["pairs_bin"]
        assert st["rows_bin"] == want["rows_bin"]


def test_far_more_wedges_than_pairs():
    """400 rows with the same 40,000 vertices: 3.2e9 wedges, 79,800 pairs.  The
    staging area does not grow with the wedges."""
    m, rows, k = 20_000, 400, 40_000
    ids = torch.arange(rows, device="cuda", dtype=torch.int32) * 50
    e_off = torch.zeros(m + 1, dtype=torch.int64, device="cuda")
    e_off[ids.long() + 1] = k
    dh = slg.DeviceHypergraph(
        m, k, e_off.cumsum(0).int(), torch.arange(k, device="cuda", dtype=torch.int32).repeat(rows),
        torch.arange(k + 1, device="cuda", dtype=torch.int32) * rows, ids.repeat(k))
    want = torch.triu_indices(rows, rows, 1, device="cuda") * 50
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    slg.release_memory()
    free = torch.cuda.mem_get_info()[0]
    for s in (1, 2, k):
        i, j, w = slg.build(dh, s)
        assert torch.equal(i, want[0].int()) and torch.equal(j, want[1].int())
        assert bool((w == k).all())
    torch.cuda.synchronize()
    assert free - torch.cuda.mem_get_info()[0] < 5 << 30
    slg.release_memory()


@pytest.mark.parametrize("form", ["build", "graph", "csr"])
def test_outputs_that_cannot_be_had_beside_the_walk(form, monkeypatch):
    """torch's allocator refuses while the walk's memory is held: the library's
    memory is given back before the build is done over, counting first."""
    h = groups(200, 24, 2, 20_000)
    dh = slg.to_device(h)
    want = slg.build(dh, 2, capacity=slg.count(dh, 2))
    real_out, real_release, log = slg._outputs, slg.release_memory, []

    def outputs(n, unweighted, device):
        log.append("outputs")
        if len(log) == 1:
            raise torch.cuda.OutOfMemoryError("no memory")
        return real_out(n, unweighted, device)

    def release():
        log.append("release")
        real_release()

    monkeypatch.setattr(slg, "_outputs", outputs)
    monkeypatch.setattr(slg, "release_memory", release)
    if form == "csr":
        got = slg.build_csr(dh, 2)[1:]
    elif form == "graph":
        with slg.Graph(dh) as g:
            got = g.build(2)[1:]
    else:
        got = slg.build(dh, 2)[1:]
    assert log == ["outputs", "release", "outputs"]
    assert all(torch.equal(a, b) for a, b in zip(got, want[1:]))


def test_no_memory_in_the_library(monkeypatch):
    released = []
    monkeypatch.setattr(slg, "release_memory", lambda: released.append(1))
    got = slg._build_alloc(lambda *a: 3, "slg_build", None, 2, 0, False, "cuda", None)
    assert got is None and released == [1]
