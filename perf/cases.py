"""The work that the framework is timed on: what its users have it do, from
one small query to the full-size build, through the public entry points.

A case names a call, a seeded hypergraph and the call's options:

  call    build    slg.build into the caller's arrays
          query    slg.build(h, s): the list sized by the call itself
          offsets  slg.row_offsets: the counting pass, every row's place in the list
          csr      slg.build_csr into the caller's arrays
          step     one slg.Graph handle and four builds through it (both sides, s and s2)
          sweep    slg.build_sweep, thresholds s, s + 1, s + 2, s + 4, ... into the caller's arrays
          filter   slg.filter_pairs of an L_s list at s2, as the query server answers from its base list
          post     squeeze, adjacency and components of an L_s list
          batch    slg.Plan.execute and its results
          host     slg.build_host_many: pinned host arrays in, row form with 16-bit weights out
  shape   uniform   sizes U{1..2 mean - 1}, uniform vertices (hypergen.uniform)
          chung_lu  power-law sizes (exponent 2.1, at most 10,000) and vertex weights (2.3) (hypergen.chung_lu)
          web       lognormal(2, 1.5) sizes, uniform vertices, a planted 4,096-hyperedge core (hypergen.lognormal_web)

The inputs follow the recipes of ``hypergen`` but are drawn on the GPU, so
that a full-size one takes a fraction of a second (duplicates of a row are
merged and not drawn again).  A case's incidence is the same up to the names
of its hyperedges and vertices, which the seed shuffles: the lists of two
seeds differ in every id and have the same length.
"""
import math
import types

import numpy as np
import torch

import paper_2010_11448_gb300 as slg

DEV = "cuda"
EXACT_WEDGES = 1_500_000_000  # above this, the 64-bit answer takes too long


def _case(name, call, shape, m, n, mean, s, dual=False, **more):
    c = {"name": name, "call": call, "shape": shape, "m": m, "n": n, "mean": mean, "s": s,
         "s2": 0, "dual": dual, "weighted": True, "tensor": False, "members": 1}
    c.update(more)
    return c


def listed():
    return [
        # one interactive query on a small hypergraph (the uniform_2k configuration): latency
        _case("small_build", "build", "uniform", 2_000, 4_000, 10.5, 2),
        # the call as a first-time user writes it, on a mid-size dual
        _case("query_dual", "query", "chung_lu", 30_011, 60_029, 20.0, 3, True),
        # the counting pass before a streamed build: every row's place, no list
        _case("offsets_h", "offsets", "chung_lu", 120_000, 240_000, 20.0, 4),
        # the benchmark's step: chung_lu_1m, L_2 and L_8 of H and H* through one handle
        _case("step_1m", "step", "chung_lu", 1_000_000, 2_000_000, 20.0, 2, s2=8),
        # a strong-overlap list of a large dual
        _case("build_dual_s8", "build", "chung_lu", 300_007, 600_011, 20.0, 8, True),
        # the adjacency pattern alone, in row form, for graph analytics
        _case("csr_pattern", "csr", "chung_lu", 500_009, 1_000_003, 20.0, 3, weighted=False),
        # the full line graph (s = 1): every pair that shares a vertex
        _case("line_graph_s1", "build", "chung_lu", 100_003, 200_017, 20.0, 1),
        # a study over thresholds: L_2 and the larger ones from one walk
        _case("sweep_dual", "sweep", "chung_lu", 150_000, 300_000, 20.0, 2, True),
        # the query server's answer from its base list
        _case("filter_l2", "filter", "chung_lu", 200_000, 400_000, 20.0, 2, True, s2=6),
        # what follows the list: squeezed ids, adjacency, s-connected components
        _case("post_l2", "post", "chung_lu", 250_000, 500_000, 20.0, 2),
        # many hypergraphs of log-uniform size, each with its own s, in one plan
        _case("batch_16", "batch", "chung_lu", 100_000, 200_000, 20.0, 2, members=16),
        # end to end from host memory: upload, two builds, copies back
        _case("host_many", "host", "chung_lu", 200_000, 400_000, 20.0, 2, s2=8),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["build"] * 4 + ["query"] * 2 + ["offsets"] * 2 + ["csr"] * 2 +
                      ["step", "sweep", "filter", "post", "batch", "host"])
    shape, tensor = "chung_lu", False
    dual = rng.random() < 0.5
    weighted = call not in ("build", "query", "csr") or rng.random() < 0.75
    s = 1 if call in ("build", "csr") and rng.random() < 0.12 else _log(rng, 2, 8 if dual else 16)
    hi = {"query": 200_000, "step": 400_000, "sweep": 150_000, "filter": 200_000,
          "post": 300_000, "batch": 60_000, "host": 200_000}.get(call, 600_000)
    if s == 1:
        hi = 100_000
    m = _log(rng, 1_000, hi)
    n = int(m * rng.uniform(1.0, 3.0)) + rng.randrange(2)
    mean = round(rng.uniform(12.0, 22.0), 1)
    kind = rng.random()
    if call in ("build", "offsets") and kind < 0.2:
        shape, s = "uniform", 2  # larger overlaps are rare between uniform sets
    elif call == "build" and kind < 0.35:
        # the dense-core option on a web-shaped input
        shape, tensor, weighted, s = "web", True, True, max(s, 2)
        m, n = _log(rng, 100_000, 600_000), _log(rng, 400_000, 1_500_000)
    return _case("", call, shape, m, n, mean, s, dual, weighted=weighted, tensor=tensor,
                 s2=s + _log(rng, 1, 4 if call == "filter" else 12), members=rng.randint(4, 20))


# ------------------------------------------------------------------ inputs --

def _sizes(m, mean, cap, rng):
    """Discrete power law of exponent 2.1 on [kmin, cap], mean about `mean`."""
    p = np.arange(1, cap + 1, dtype=np.float64) ** -2.1
    kp, sp = (p * np.arange(1, cap + 1))[::-1].cumsum()[::-1], p[::-1].cumsum()[::-1]
    kmin = int(np.argmin(np.abs(kp[:200] / sp[:200] - mean))) + 1
    cdf = np.cumsum(p[kmin - 1:])
    return np.searchsorted(cdf, rng.random(m) * cdf[-1], side="right") + kmin


def _offsets(ids, count):
    off = torch.zeros(count + 1, dtype=torch.int64, device=DEV)
    off[1:] = torch.bincount(ids, minlength=count).cumsum(0)
    return off.int()


def _hypergraph(shape, m, n, mean, seed):
    """(e_off, e_idx, v_off, v_idx), int32 on the GPU: the incidence of these
    sizes, its ids shuffled by the seed."""
    rng = np.random.default_rng([m, n])
    gen = torch.Generator(device=DEV).manual_seed(m + n)
    weights = None
    if shape == "uniform":
        sizes = rng.integers(1, int(2 * mean), size=m)
    elif shape == "web":
        sizes = np.clip(np.rint(rng.lognormal(2.0, 1.5, size=m)), 1, 100_000).astype(np.int64)
    else:
        sizes = np.minimum(_sizes(m, mean, 10_000, rng), n)
        total = int(sizes.sum())
        weights = rng.pareto(1.3, size=n) + 1.0
        weights *= (total / n) / weights.mean()
        weights = np.minimum(weights, max(total / int(sizes.max()), 1.0))
    sizes = torch.from_numpy(sizes).to(DEV)
    rows = torch.repeat_interleave(torch.arange(m, device=DEV), sizes)
    if weights is None:
        cols = torch.randint(0, n, rows.shape, generator=gen, device=DEV)
    else:
        cdf = torch.from_numpy(np.cumsum(weights)).to(DEV)
        u = torch.rand(rows.shape, generator=gen, device=DEV, dtype=torch.float64) * cdf[-1]
        cols = torch.searchsorted(cdf, u, right=True).clamp_(max=n - 1)
    if shape == "web":
        core_e = torch.from_numpy(rng.choice(m, size=min(4096, m), replace=False)).to(DEV)
        core_v = torch.from_numpy(rng.choice(n, size=min(4096, n), replace=False)).to(DEV)
        hit = torch.rand(core_e.numel(), core_v.numel(), generator=gen, device=DEV) < 0.3
        ri, ci = hit.nonzero(as_tuple=True)
        rows, cols = torch.cat([rows, core_e[ri]]), torch.cat([cols, core_v[ci]])
    names = torch.Generator(device=DEV).manual_seed(seed)
    e_name = torch.randperm(m, generator=names, device=DEV)
    v_name = torch.randperm(n, generator=names, device=DEV)
    key = torch.unique(e_name[rows] * n + v_name[cols])
    rows, cols = key // n, key % n
    by_col = torch.argsort(cols, stable=True)
    return _offsets(rows, m), cols.int(), _offsets(cols, n), rows[by_col].int()


def _graph(shape, m, n, mean, seed):
    return slg.DeviceHypergraph(m, n, *_hypergraph(shape, m, n, mean, seed))


def _members(case):
    """Log-uniform member sizes up to the case's m (hypergen.batch), each with its s."""
    rng = np.random.default_rng([case["m"], case["n"]])
    ms = np.exp(rng.uniform(np.log(1_000), np.log(max(case["m"], 1_001)), case["members"]))
    return [(int(x), max(int(x * case["n"] / case["m"]), 1), int(s))
            for x, s in zip(ms, rng.integers(case["s"], case["s"] + 31, case["members"]))]


def _thresholds(case):
    return [case["s"] + x for x in (0, 1, 2, 4, 6, 10, 14)]


def _jobs(case):
    return [(dual, s) for dual in (False, True) for s in (case["s"], case["s2"])]


def _pinned(t):
    return torch.empty(t.shape, dtype=t.dtype, pin_memory=True).copy_(t)


def prepare(case, seed):
    call, dual, s = case["call"], case["dual"], case["s"]
    st = types.SimpleNamespace(case=case)
    shape = (case["shape"], case["m"], case["n"], case["mean"])
    if call == "batch":
        st.graphs, st.s = [], []
        for k, (m, n, sk) in enumerate(_members(case)):
            st.graphs.append(_graph("chung_lu", m, n, case["mean"], seed * 1000 + k))
            st.s.append(sk)
        st.plan = slg.Plan(st.graphs, st.s, dual)
        return st
    h = st.h = _graph(*shape, seed)
    weighted = case["weighted"]
    if call == "build":
        st.out = slg.alloc_outputs(slg.count(h, s, dual, tensor=case["tensor"]), not weighted)
    elif call == "csr":
        _, j, w = slg.alloc_outputs(slg.count(h, s, dual), not weighted)
        st.out = (torch.empty(h.rows(dual) + 1, dtype=torch.int64, device=DEV), j, w)
    elif call == "step":
        with slg.Graph(h) as g:
            st.outs = [slg.alloc_outputs(g.count(s, d)) for d, s in _jobs(case)]
    elif call == "sweep":
        st.outs = [slg.alloc_outputs(slg.count(h, x, dual)) for x in _thresholds(case)]
    elif call in ("filter", "post"):
        st.base = slg.build(h, s, dual)
    elif call == "host":
        st.host = types.SimpleNamespace(m=h.m, n=h.n, **{
            k: _pinned(getattr(h, k)) for k in ("e_off", "e_idx", "v_off", "v_idx")})
        st.queries = []
        for x in (s, case["s2"]):
            cap = slg.count(h, x, dual)
            st.queries.append({
                "s": x, "dual": dual, "w16": True, "capacity": cap,
                "row_ptr": torch.empty(h.rows(dual) + 1, dtype=torch.int64, pin_memory=True),
                "out_j": torch.empty(max(cap, 1), dtype=torch.int32, pin_memory=True),
                "out_w": torch.empty(max(cap, 1), dtype=torch.int16, pin_memory=True)})
    return st


def run(state):
    c = state.case
    call, dual, s = c["call"], c["dual"], c["s"]
    if call == "build":
        return slg.build(state.h, s, dual, not c["weighted"], out=state.out, tensor=c["tensor"])
    if call == "query":
        return slg.build(state.h, s, dual, not c["weighted"])
    if call == "offsets":
        return slg.row_offsets(state.h, s, dual)
    if call == "csr":
        return slg.build_csr(state.h, s, dual, not c["weighted"], out=state.out)
    if call == "step":
        with slg.Graph(state.h) as g:
            return [g.build(x, d, out=o) for (d, x), o in zip(_jobs(c), state.outs)]
    if call == "sweep":
        return slg.build_sweep(state.h, _thresholds(c), dual, outs=state.outs)
    if call == "filter":
        return slg.filter_pairs(*state.base, c["s2"])
    if call == "post":
        i, j, w = state.base
        rows = state.h.rows(dual)
        return {"squeeze": slg.squeeze(i, j, rows), "adjacency": slg.adjacency(i, j, w, rows),
                "components": slg.components(i, j, rows)}
    if call == "batch":
        state.plan.execute()
        return state.plan.results()
    done = slg.build_host_many(state.host, state.queries)
    return [{"status": rc, "row_ptr": q["row_ptr"], "j": q["out_j"][:p], "w": q["out_w"][:p]}
            for (rc, p), q in zip(done, state.queries)]


# ------------------------------------------------------------- what is due --

def _tensors(v):
    if isinstance(v, torch.Tensor):
        yield v
    elif isinstance(v, dict):
        for x in v.values():
            yield from _tensors(x)
    elif isinstance(v, (list, tuple)):
        for x in v:
            yield from _tensors(x)


def work(case):
    """Bytes: the incidence (or the list) read once and the outputs written
    once.  Operations: one add per wedge of the lists that are built (two
    compares per triple for calls on a list)."""
    st = prepare(case, 1)
    size = lambda v: sum(t.numel() * t.element_size() for t in _tensors(v))
    call, dual = case["call"], case["dual"]
    if call in ("filter", "post"):
        read, flops = size(st.base), 2 * int(st.base[0].numel())
    else:
        graphs = st.graphs if call == "batch" else [st.h]
        read = sum(size([h.e_off, h.e_idx, h.v_off, h.v_idx]) for h in graphs)
        jobs = {"step": lambda: [(st.h, x, d) for d, x in _jobs(case)],
                "host": lambda: [(st.h, x, dual) for x in (case["s"], case["s2"])],
                "batch": lambda: [(h, x, dual) for h, x in zip(st.graphs, st.s)]}
        flops = sum(slg.wedges(h, x, d)
                    for h, x, d in jobs.get(call, lambda: [(st.h, case["s"], dual)])())
    return {"bytes": read + size(run(st)), "flops": flops}


def _list(h, s, dual):
    """L_s in 64 bits with torch alone: (i, j, w), or None if it is too much.

    The wedges (i, j), i < j, of every column are expanded in chunks of rows
    and counted by sorting."""
    r_off, _, c_off, c_idx = ((h[2], h[3], h[0], h[1]) if dual else h)
    c_off, c_idx = c_off.long(), c_idx.long()
    R = r_off.numel() - 1
    q = torch.arange(c_idx.numel(), device=DEV)
    tail = torch.repeat_interleave(c_off[1:], c_off.diff()) - q - 1
    order = torch.argsort(c_idx, stable=True)
    c_row, q, tail = c_idx[order], q[order], tail[order]
    total = tail.cumsum(0)
    if not total.numel() or int(total[-1]) > EXACT_WEDGES:
        return None if total.numel() else (torch.zeros(0, dtype=torch.int64, device=DEV),) * 3
    ends = torch.searchsorted(c_row, torch.arange(1, R + 1, device=DEV))  # past each row
    row_total = torch.where(ends > 0, total[(ends - 1).clamp(min=0)], 0).cpu().numpy()
    ends = ends.cpu().numpy()
    got, r, a = [], 0, 0
    while r < R:
        done = row_total[r - 1] if r else 0
        r = max(r + 1, int(np.searchsorted(row_total, done + 150_000_000, side="right")))
        b = int(ends[r - 1])
        t = tail[a:b]
        start = torch.repeat_interleave(q[a:b] + 1 - (t.cumsum(0) - t), t)
        far = c_idx[start + torch.arange(start.numel(), device=DEV)]
        key = torch.repeat_interleave(c_row[a:b], t) * R + far
        key, w = torch.unique_consecutive(key.sort().values, return_counts=True)
        got.append(torch.stack([key[w >= s], w[w >= s]]))
        a = b
    key, w = torch.cat(got, 1)
    return key // R, key % R, w


def _row_form(lst, rows):
    ptr = torch.zeros(rows + 1, dtype=torch.int64, device=DEV)
    ptr[1:] = torch.bincount(lst[0], minlength=rows).cumsum(0)
    return ptr, lst[1], lst[2]


def _post(lst, rows):
    i, j, w = lst
    old = torch.unique(torch.cat([i, j]))
    new = torch.zeros(rows, dtype=torch.int64, device=DEV)
    new[old] = torch.arange(old.numel(), device=DEV)
    a, b = torch.cat([i, j]), torch.cat([j, i])
    order = torch.argsort(a * rows + b)
    off = torch.zeros(rows + 1, dtype=torch.int64, device=DEV)
    off[1:] = torch.bincount(a, minlength=rows).cumsum(0)
    label = torch.arange(rows, device=DEV)
    while True:  # the smallest label among the neighbours, then its label's label
        low = label.clone().scatter_reduce_(0, a, label[b], "amin")
        low = low[low]
        if torch.equal(low, label):
            break
        label = low
    return {"squeeze": (new[i], new[j], old),
            "adjacency": (off, b[order], torch.cat([w, w])[order]),
            "components": (label, int(torch.unique(label[old]).numel()))}


def exact(case, seed):
    call, dual, s = case["call"], case["dual"], case["s"]
    shape = (case["shape"], case["m"], case["n"], case["mean"])
    if call == "step" or case["shape"] == "web":
        return None
    if call == "batch":
        got = [_list(_hypergraph("chung_lu", m, n, case["mean"], seed * 1000 + k), sk, dual)
               for k, (m, n, sk) in enumerate(_members(case))]
        return None if any(x is None for x in got) else got
    h = _hypergraph(*shape, seed)
    rows = case["n"] if dual else case["m"]
    base = _list(h, s, dual)
    if base is None:
        return None
    at = lambda x: tuple(v[base[2] >= x] for v in base)
    if call in ("build", "query"):
        return base if case["weighted"] else (*base[:2], None)
    if call == "offsets":
        return _row_form(base, rows)[0]
    if call == "csr":
        out = _row_form(base, rows)
        return out if case["weighted"] else (*out[:2], None)
    if call == "sweep":
        return [at(x) for x in _thresholds(case)]
    if call == "filter":
        return at(case["s2"])
    if call == "post":
        return _post(base, rows)
    forms = [_row_form(at(x), rows) for x in (s, case["s2"])]
    return [{"status": 0, "row_ptr": p, "j": j, "w": w} for p, j, w in forms]
