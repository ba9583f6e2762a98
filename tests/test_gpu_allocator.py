"""Calls on an installed allocator: one whose memory is aligned to 8 bytes and no
more, on which every entry point that allocates must count as with the library's
own pool, and one that adds up what a build holds at once, which may not pass
the upper estimate that admission control goes by."""
import ctypes

import numpy as np
import pytest

import oracle
import paper_2609_21848_gb300 as dbbc

pytestmark = pytest.mark.gpu


@pytest.fixture
def eight_byte_allocator():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)
    live = {}

    def alloc(size, stream, ctx):
        block = torch.empty(size + 16, dtype=torch.uint8, device="cuda")
        assert block.data_ptr() % 16 == 0
        live[block.data_ptr() + 8] = block
        return block.data_ptr() + 8

    refs = (dbbc._ALLOC_FN(alloc), dbbc._FREE_FN(lambda p, stream, ctx: live.pop(int(p))))
    dbbc.lib().dbbc_set_allocator(ctypes.cast(refs[0], ctypes.c_void_p), ctypes.cast(refs[1], ctypes.c_void_p), None)
    yield
    torch.cuda.synchronize()
    dbbc.lib().dbbc_set_allocator(None, None, None)
    assert not live


@pytest.mark.parametrize("repeats", [0, 700])  # with repeated pairs the CSR is allocated twice
def test_counts_on_memory_aligned_to_eight_bytes(eight_byte_allocator, repeats):
    rng = np.random.default_rng(repeats)
    n_u, n_v, m = 901, 701, 60_000
    k = rng.choice(n_u * n_v, m - repeats, replace=False)
    k = np.concatenate([k, k[:repeats]])
    u, v = (k // n_v).astype(np.int32), (k % n_v).astype(np.int32)
    s = np.where(rng.random(m) < 0.6, 1, -1).astype(np.int8)
    want = oracle.count(u, v, s, n_u, n_v)[:2]
    base = dbbc.dbbc_get_tuning()
    try:
        dbbc.dbbc_set_tuning({"light_max_work": 256, "medium_max_work": 1024})
        with dbbc.dbbc_graph_from_coo(u, v, s, n_u, n_v) as g:
            assert g.info["n_light"] and g.info["n_medium"] and g.info["n_hub"]
            assert dbbc.dbbc_count(g) == want
            vb, vu = dbbc.dbbc_count_vertices(g)
            first = np.unique(k, return_index=True)[1]
            eb, eu = dbbc.dbbc_count_edges(g, u[first], v[first])
            with dbbc.dbbc_batch_create([g, g]) as b:
                plan = dbbc.dbbc_batch_count(b)
        with dbbc.dbbc_graph_from_coo_multi(np.tile(u, 2), np.tile(v, 2), np.tile(s, 2), [0, m, 2 * m], [n_u, n_u],
                                            [n_v, n_v]) as un:
            parts = dbbc.dbbc_count_components(un)
    finally:
        dbbc.dbbc_set_tuning(base)
    assert [int(x.sum(dtype=np.uint64)) for x in (vb, vu, eb, eu)] == [4 * want[0], 4 * want[1]] * 2
    assert [x.tolist() for x in plan] == [x.tolist() for x in parts] == [[want[0]] * 2, [want[1]] * 2]


@pytest.mark.parametrize("hubs", [False, True])  # True: every pivot that can close a butterfly is a hub
@pytest.mark.parametrize("n_u,n_v,m,repeats", [(3, 4, 5, 0), (3, 4, 9, 3), (60, 40, 700, 0), (1_000, 900, 20, 0),
                                               (2_000_000, 1_000_003, 10, 0), (40_000, 9_000, 600_000, 30_000),
                                               (3_000, 2_000, 400_000, 0)])
def test_builds_stay_within_the_estimate(n_u, n_v, m, repeats, hubs):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)
    rng = np.random.default_rng(m)
    k = np.unique(rng.integers(0, n_u * n_v, 2 * m)) if n_u * n_v > 100 * m else np.arange(n_u * n_v)
    k = rng.permutation(k)[:m - repeats]
    k = np.concatenate([k, k[:repeats]])
    u, v = (k // n_v).astype(np.int32), (k % n_v).astype(np.int32)
    s = np.where(rng.random(m) < 0.5, 1, -1).astype(np.int8)
    live, peak = {}, [0]

    def alloc(size, stream, ctx):
        block = torch.empty(size, dtype=torch.uint8, device="cuda")
        live[block.data_ptr()] = block
        peak[0] = max(peak[0], sum(b.numel() for b in live.values()))
        return block.data_ptr()

    refs = (dbbc._ALLOC_FN(alloc), dbbc._FREE_FN(lambda p, stream, ctx: live.pop(int(p))))
    base = dbbc.dbbc_get_tuning()
    dbbc.lib().dbbc_set_allocator(ctypes.cast(refs[0], ctypes.c_void_p), ctypes.cast(refs[1], ctypes.c_void_p), None)
    try:
        if hubs:
            dbbc.dbbc_set_tuning({"light_max_work": 1, "medium_max_work": 1})
        with dbbc.dbbc_graph_from_coo(u, v, s, n_u, n_v):
            pass
        torch.cuda.synchronize()
    finally:
        dbbc.lib().dbbc_set_allocator(None, None, None)
        dbbc.dbbc_set_tuning(base)
    assert 0 < peak[0] <= dbbc.dbbc_estimate_bytes(m, n_u, n_v), peak
