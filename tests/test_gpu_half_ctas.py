"""Graphs whose hub sweep runs half CTAs (two per SM): no side above 2^17
vertices and no hub with more than four times a half CTA's mean share of the
hub wedges. The exported work of every pivot says which graphs these are."""
import time

import numpy as np
import pytest

import oracle
import paper_2609_21848_gb300 as dbbc

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)
    return torch


def _runs_half_ctas(g, torch):
    i = g.info
    ctas = 2 * torch.cuda.get_device_properties(0).multi_processor_count
    most = int(dbbc.dbbc_graph_export(g)["work"].max())
    return max(i["n_u"], i["n_v"]) <= 1 << 17 and most <= 4 * (i["wedges_hub"] // ctas)


def _edges(n_u, n_v, m, tail):
    """About m distinct edges; endpoints uniform, or (tail) by Pareto weights."""
    rng = np.random.default_rng(n_u + m)
    if tail:
        w = [rng.pareto(tail, n) + 1 for n in (n_u, n_v)]
        a, b = (rng.choice(n, m, p=x / x.sum()) for n, x in zip((n_u, n_v), w))
    else:
        a, b = rng.integers(0, n_u, m), rng.integers(0, n_v, m)
    key = np.unique(a.astype(np.int64) * n_v + b)
    u, v = (key // n_v).astype(np.int32), (key % n_v).astype(np.int32)
    return u, v, np.where(rng.random(u.shape[0]) < 0.7, 1, -1).astype(np.int8)


# sides at the limit and one past it (the second runs full CTAs); several half
# windows of 4-bit, 8-bit and 16-bit counters, and of mixed ones
GRAPHS = {
    "quarter": (131_072, 131_072, 1_500_000, None, 16, True),
    "quarter-full-ctas": (131_073, 131_072, 1_500_000, None, 16, False),
    "tiny": (131_072, 131_072, 3_200_000, None, 64, True),
    "narrow": (30_000, 120_000, 9_000_000, None, 4096, True),
    "mixed": (100_000, 90_000, 2_000_000, 4.0, 64, True),
    "mixed-tail": (131_072, 60_000, 2_000_000, 3.0, 64, True),
}


@pytest.mark.parametrize("name", sorted(GRAPHS))
def test_every_count_of_a_half_cta_graph(torch_cuda, name):
    """With cursors and with neighbour lists, each finalised per window and per
    wedge: the count, and what other entry points make of the same hub plan."""
    n_u, n_v, m, tail, medium, half = GRAPHS[name]
    u, v, s = _edges(n_u, n_v, m, tail)
    want = oracle.count(u, v, s, n_u, n_v, threads=16)[:2]
    base = dbbc.dbbc_get_tuning()
    try:
        for list_density in (0.0, 1e9):
            for finalize in (0, 2**64 - 1):
                dbbc.dbbc_set_tuning({"list_density": list_density, "finalize_window_wedges": finalize,
                                      "light_max_work": min(medium, 512), "medium_max_work": medium})
                with dbbc.dbbc_graph_from_coo(u, v, s, n_u, n_v) as g:
                    assert _runs_half_ctas(g, torch_cuda) == half
                    bal, unb, profile = dbbc.dbbc_count_profiled(g)
                    assert (bal, unb) == want
                    assert (profile["hub_list_visits"] > 0) == (list_density > 0)
                    with dbbc.dbbc_batch_create([g]) as b:
                        plan = dbbc.dbbc_batch_count(b)
                    assert [int(x[0]) for x in plan] == list(want)
                    parts = [dbbc.dbbc_count_partition(g, k, 3) for k in range(3)]
                    assert tuple(map(sum, zip(*parts))) == want
                    if finalize == 0:
                        vb, vu = dbbc.dbbc_count_vertices(g)
                        eb, eu = dbbc.dbbc_count_edges(g, u, v)
                        assert [int(x.sum(dtype=np.uint64)) for x in (vb, vu, eb, eu)] == [4 * x for x in want] * 2
    finally:
        dbbc.dbbc_set_tuning(base)


@pytest.mark.parametrize("list_density", [0.0, 1e9])
def test_union_on_half_ctas(torch_cuda, list_density):
    """A union's sides add up; its ranks are component-major, so hubs of the later
    components start inside a window."""
    graphs = [_edges(n_u, n_v, m, 4.0) + (n_u, n_v) for n_u, n_v, m in
              [(40_001, 30_003, 700_000), (29_999, 40_007, 500_000), (61_000, 60_000, 900_000)]]
    cat = [np.concatenate([g[i] for g in graphs]) for i in range(3)]
    off = np.concatenate([[0], np.cumsum([g[0].shape[0] for g in graphs])])
    want = [oracle.count(*g, threads=16)[:2] for g in graphs]
    base = dbbc.dbbc_get_tuning()
    try:
        dbbc.dbbc_set_tuning({"list_density": list_density, "light_max_work": 64, "medium_max_work": 64})
        with dbbc.dbbc_graph_from_coo_multi(*cat, off, [g[3] for g in graphs], [g[4] for g in graphs]) as g:
            assert _runs_half_ctas(g, torch_cuda)
            total = dbbc.dbbc_count(g)
            parts = dbbc.dbbc_count_components(g)
    finally:
        dbbc.dbbc_set_tuning(base)
    assert total == tuple(map(sum, zip(*want)))
    assert list(zip(*(x.tolist() for x in parts))) == want


def test_noalloc_with_scratch_for_few_half_ctas(torch_cuda):
    """400 hubs of about 27,000 lower neighbours each: the fixed scratch holds
    the cursors of about half the half CTAs. The count must equal the oracle's
    and take no longer than one whose scratch is allocated, give or take."""
    torch = torch_cuda
    rng = np.random.default_rng(3)
    u, v = (x.astype(np.int32) for x in np.nonzero(rng.random((400, 60_000)) < 0.45))
    s = np.where(rng.random(u.shape[0]) < 0.7, 1, -1).astype(np.int8)
    out = torch.zeros(2, dtype=torch.int64, device="cuda")

    def best(count):
        times = []
        for _ in range(10):
            torch.cuda.synchronize()
            t = time.perf_counter()
            count(g, out)
            torch.cuda.synchronize()
            times.append(time.perf_counter() - t)
        return min(times)

    with dbbc.dbbc_graph_from_coo(u, v, s, 400, 60_000) as g:
        assert _runs_half_ctas(g, torch)
        allocating = best(dbbc.dbbc_count_async)
        want = out.tolist()
        out.fill_(-1)
        fixed = best(dbbc.dbbc_count_noalloc)
        assert out.tolist() == want
    assert want == list(oracle.count(u, v, s, 400, 60_000, threads=16)[:2])
    assert fixed < 1.35 * allocating, (fixed, allocating)
