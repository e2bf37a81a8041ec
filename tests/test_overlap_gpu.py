"""The bins' kernels of one build run on two streams beside the caller's: many
builds at once (host threads, each with its own stream or two in turn) give the
oracle's list, and so do a plan and a build under per-bin timing, where the
kernels follow one another."""
import threading
import time

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


def test_side_streams_have_the_priority_of_the_callers():
    """A count on a stream of the highest priority does not wait for a kernel of
    the default one that fills the device: its bins' kernels, on the call's side
    streams too, go before the blocks still to come."""
    dh = slg.to_device(hg.chung_lu(100_000, 200_000, seed=8, size_cap=6000))
    want = slg.count(dh, 4)
    st = slg.last_stats()
    assert st["giant_cycles"][3] > 0 and st["rows_bin"][1] > 0  # it forks
    high = torch.cuda.Stream(priority=-5)
    assert slg.count(dh, 4, stream=high) == want
    x = torch.rand(1 << 28, dtype=torch.float64, device="cuda") + 1.5
    out = torch.empty_like(x)
    done = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
    torch.cuda.synchronize()
    done[0].record()
    torch.special.zeta(x, x, out=out)  # one kernel of a million blocks
    done[1].record()
    t = time.perf_counter()
    got = slg.count(dh, 4, stream=high)
    waited = (time.perf_counter() - t) * 1e3
    torch.cuda.synchronize()
    assert got == want
    busy = done[0].elapsed_time(done[1])
    assert busy > 150 and waited < 0.3 * busy, (waited, busy)  # 10 of 616 ms; was 615
