"""Id spaces far above the grids that kernels are capped at."""
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


# 2^20 blocks of 256 columns end at id 268,435,456
@pytest.mark.parametrize("n", [268_435_455, 268_435_456, 300_000_000])
def test_columns_above_a_capped_grid(n):
    """A few vertices spread over a large id space, at both its ends and
    around 2^28: L_s does not depend on the vertices' names."""
    h = hg.uniform(20_000, 30_000, 1, 20, seed=5)
    edge = [x for x in range(268_435_400, 268_435_500) if x < n - 40]
    ids = np.unique(np.concatenate([np.arange(40), edge, np.arange(n - 40, n)]))
    rest = np.random.default_rng(n).choice(n - 1_000_000, 2 * h.n, replace=False) + 500_000
    rest = np.setdiff1d(rest, ids)
    ids = np.sort(np.concatenate([ids, rest[:h.n - ids.size]]))
    assert ids.size == h.n
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    v_off = torch.zeros(n + 1, dtype=torch.int32, device="cuda")
    v_off[t(ids) + 1] = t(np.diff(h.v_off).astype(np.int32))
    v_off = v_off.cumsum(0, dtype=torch.int32)
    dh = slg.DeviceHypergraph(h.m, n, t(h.e_off), t(ids.astype(np.int32)[h.e_idx]), v_off,
                              t(h.v_idx))
    for s in (1, 2):
        got = np.stack([x.cpu().numpy() for x in slg.build(dh, s)], 1)
        assert np.array_equal(got, oracle.canonical(*oracle.line_graph_of(h, s, threads=8))), s
