"""GPU parity of the graph build at the edges of its tiles: edge lists whose
length and vertex counts sit at, below and above the tiles of the sort, row and
pivot kernels, repeated pairs, and invalid edges at the end of a list. The
device CSR must equal one built on the host, the counts the oracle's."""
import numpy as np
import pytest

import oracle
import paper_2609_21848_gb300 as dbbc
from gpu_util import host_csr

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)
    dbbc.lib()


def _edges(seed, n_u, n_v, m, repeats):
    """m rows, `repeats` of them repeating an earlier pair, in random order."""
    rng = np.random.default_rng(seed)
    pairs = rng.choice(n_u * n_v, size=m - repeats, replace=False)
    pairs = np.concatenate([pairs, rng.choice(pairs, size=repeats)]) if repeats else pairs
    rng.shuffle(pairs)
    return (pairs // n_v).astype(np.int32), (pairs % n_v).astype(np.int32), \
        np.where(rng.random(m) < 0.5, 1, -1).astype(np.int8)


@pytest.mark.parametrize("n_u,n_v,m,repeats", [
    (1, 1, 1, 0), (1, 1, 50, 49),            # one pair, repeated past every degree a distinct list could have
    (3, 2, 120, 114), (2, 300, 599, 1),
    (100, 90, 4095, 0), (100, 90, 4096, 0), (100, 90, 4097, 0), (100, 90, 4097, 40),   # one and two sort tiles
    (700, 323, 8192, 0), (700, 324, 8193, 9), (701, 324, 12289, 0),                    # rows at a row tile's edge
    (1500, 548, 40_000, 0), (1500, 549, 40_961, 3_000), (60_000, 65_000, 300_007, 5),  # rows at a pivot tile's edge
])
def test_csr_and_counts_at_tile_edges(n_u, n_v, m, repeats):
    u, v, s = _edges(n_u * 7 + m, n_u, n_v, m, repeats)
    want = host_csr(u, v, s, n_u, n_v)
    with dbbc.dbbc_graph_from_coo(u, v, s, n_u, n_v) as g:
        got = dbbc.dbbc_graph_export(g)
        assert g.info["m"] == m - repeats and g.info["m_input"] == m
        for k in ("row_ptr", "col", "lower", "vertex"):
            assert np.array_equal(got[k].astype(np.int64), want[k].astype(np.int64)), k
        assert dbbc.dbbc_count(g) == oracle.count(u, v, s, n_u, n_v)[:2]


@pytest.mark.parametrize("m", [4096, 4097, 20_000])
@pytest.mark.parametrize("bad", ["u", "v", "sign"])
def test_an_invalid_last_edge_is_found(m, bad):
    u, v, s = _edges(m, 300, 200, m, 10)
    if bad == "u":
        u[-1] = 300
    elif bad == "v":
        v[-1] = -1
    else:
        s[-1] = 0
    with pytest.raises(dbbc.DbbcError) as ei:
        dbbc.dbbc_graph_from_coo(u, v, s, 300, 200)
    assert ei.value.status == dbbc.DBBC_EINVAL


@pytest.mark.parametrize("sizes", [[(5, 3, 0), (1, 1, 1), (300, 200, 4097), (4, 9, 0), (64, 64, 4096), (2, 2, 4)],
                                   [(3, 4, 12)] * 70, [(0, 0, 0), (40, 40, 800)]])
def test_union_components_of_uneven_sizes(sizes):
    parts = [_edges(i, *size, 0) if size[2] else tuple(np.zeros(0, t) for t in (np.int32, np.int32, np.int8))
             for i, size in enumerate(sizes)]
    off = np.concatenate([[0], np.cumsum([x[2] for x in sizes])])
    u, v, s = (np.concatenate([p[i] for p in parts]) for i in range(3))
    with dbbc.dbbc_graph_from_coo_multi(u, v, s, off, [x[0] for x in sizes], [x[1] for x in sizes]) as g:
        bal, unb = dbbc.dbbc_count_components(g)
    want = [oracle.count(*p, n_u, n_v)[:2] if m else (0, 0) for p, (n_u, n_v, m) in zip(parts, sizes)]
    assert list(zip(bal.tolist(), unb.tolist())) == want


@pytest.mark.parametrize("entry", ["count_async", "count_noalloc"])
def test_counts_can_be_captured_and_replayed(entry):
    """The tiers of a count overlap on the stream; captured into a CUDA graph
    they keep their order against what comes before and after."""
    import torch
    u, v, s = _edges(11, 900, 700, 60_000, 0)
    want = oracle.count(u, v, s, 900, 700)[:2]
    count = getattr(dbbc, f"dbbc_{entry}")
    with dbbc.dbbc_graph_from_coo(u, v, s, 900, 700) as g:
        info = g.info
        assert info["n_light"] and info["n_medium"] and info["n_hub"]
        d_out = torch.zeros(2, dtype=torch.int64, device="cuda")
        count(g, d_out)  # outside capture first
        copy = torch.zeros_like(d_out)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            count(g, d_out)
            copy.copy_(d_out)
        for _ in range(3):
            copy.fill_(-1)
            graph.replay()
            torch.cuda.synchronize()
            assert tuple(copy.tolist()) == want


@pytest.mark.parametrize("n_u", [3_300, 3_400, 6_700, 28_700, 57_300, 57_400])
@pytest.mark.parametrize("finalize", [0, 2**64 - 1])
def test_hub_windows_at_the_widths_that_fit(n_u, finalize):
    """Hubs whose endpoint ranks just fit, and just do not fit, one window of
    32-bit or 16-bit counters on a full and on a narrow CTA: counts of one
    graph, of a plan and per vertex."""
    rng = np.random.default_rng(n_u)
    hubs, n_v = 3, 400
    u = np.concatenate([rng.integers(0, n_u - hubs, 4 * n_u), np.repeat(np.arange(n_u - hubs, n_u), n_v)])
    v = np.concatenate([rng.integers(0, n_v, 4 * n_u), np.tile(np.arange(n_v), hubs)])
    key = np.unique(u.astype(np.int64) * n_v + v)
    u, v = (key // n_v).astype(np.int32), (key % n_v).astype(np.int32)
    s = np.where(rng.random(u.shape[0]) < 0.7, 1, -1).astype(np.int8)
    base = dbbc.dbbc_get_tuning()
    try:
        dbbc.dbbc_set_tuning({"finalize_window_wedges": finalize, "light_max_work": 64, "medium_max_work": 64})
        with dbbc.dbbc_graph_from_coo(u, v, s, n_u, n_v) as g:
            got = dbbc.dbbc_count(g)
            with dbbc.dbbc_batch_create([g]) as b:
                plan = tuple(int(x[0]) for x in dbbc.dbbc_batch_count(b))
            vb, vu = dbbc.dbbc_count_vertices(g)
    finally:
        dbbc.dbbc_set_tuning(base)
    want = oracle.count(u, v, s, n_u, n_v)[:2]
    assert got == want and plan == want
    assert (int(vb.sum(dtype=np.uint64)), int(vu.sum(dtype=np.uint64))) == (4 * want[0], 4 * want[1])


@pytest.mark.parametrize("n_u,n_v,m", [(131_072, 3_000, 600_000), (131_073, 3_000, 600_000), (30_000, 28_416, 900_000)])
@pytest.mark.parametrize("list_density", [0.0, 1e9])
def test_counts_on_whole_and_half_ctas(n_u, n_v, m, list_density):
    """Graphs on both sides of the size up to which the hub sweep runs half
    CTAs, with cursors and with neighbour lists."""
    rng = np.random.default_rng(n_u)
    w = rng.pareto(1.2, n_v) + 1
    key = np.unique(rng.integers(0, n_u, m).astype(np.int64) * n_v + rng.choice(n_v, m, p=w / w.sum()))
    u, v = (key // n_v).astype(np.int32), (key % n_v).astype(np.int32)
    s = np.where(rng.random(u.shape[0]) < 0.7, 1, -1).astype(np.int8)
    base = dbbc.dbbc_get_tuning()
    try:
        dbbc.dbbc_set_tuning({"list_density": list_density, "light_max_work": 32, "medium_max_work": 128})
        with dbbc.dbbc_graph_from_coo(u, v, s, n_u, n_v) as g:
            assert g.info["n_hub"] > 304
            got = dbbc.dbbc_count(g)
    finally:
        dbbc.dbbc_set_tuning(base)
    assert got == oracle.count(u, v, s, n_u, n_v, threads=8)[:2]
