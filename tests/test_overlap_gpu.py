"""The bins' kernels of one build run on two streams beside the caller's: many
builds at once (host threads, each with its own stream or two in turn) give the
oracle's list, and so do a plan and a build under per-bin timing, where the
kernels follow one another."""
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import hypergen as hg  # noqa: E402
import paper_2010_11448_gb300 as slg  # noqa: E402
import oracle  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2010_11448_gb300 import build_lib
    build_lib.build()
    slg.load()


@pytest.fixture(scope="module")
def case():
    h = hg.chung_lu(60_000, 120_000, seed=8, size_cap=6000)
    return slg.to_device(h), {s: oracle.canonical(*oracle.line_graph_of(h, s, threads=8))
                              for s in (2, 4, 8)}


def as_np(x):
    return np.stack([t.cpu().numpy() for t in x], 1)


def test_every_group_has_rows(case):
    dh, want = case
    for s in want:
        slg.set_profiling(True)
        try:
            assert np.array_equal(as_np(slg.build(dh, s)), want[s])
            rows = slg.last_stats()["rows_bin"]
        finally:
            slg.set_profiling(False)
        assert rows[1] > 0 and rows[3] > 0 and rows[4] > 0, rows


@pytest.mark.parametrize("threads,streams", [(1, 1), (1, 2), (4, 1), (4, 2)])
def test_many_at_once(case, threads, streams):
    dh, want = case
    bad = []

    def work(k):
        try:
            own = [torch.cuda.Stream() for _ in range(streams)]
            for rep in range(6):
                s = (2, 4, 8)[(rep + k) % 3]
                st = own[rep % streams]
                with torch.cuda.stream(st):
                    got = slg.build(dh, s, stream=st)
                    n = slg.count(dh, s, stream=st)
                st.synchronize()
                if n != want[s].shape[0] or not np.array_equal(as_np(got), want[s]):
                    bad.append((k, rep, s))
        except Exception as e:  # noqa: BLE001
            bad.append((k, repr(e)))

    ts = [threading.Thread(target=work, args=(k,)) for k in range(threads)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not bad


def test_plan(case):
    dh, want = case
    p = slg.Plan([dh, dh], [2, 8])
    for _ in range(3):
        p.execute()
        for got, s in zip(p.results(), (2, 8)):
            assert np.array_equal(as_np(got), want[s])
