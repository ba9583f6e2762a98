"""GPU parity of the per-edge counts on both sides of the degree product 2^32,
below which both counts of an edge are accumulated in one 64-bit word."""
import numpy as np
import pytest

import oracle
import paper_2609_21848_gb300 as dbbc

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)
    dbbc.lib()


@pytest.mark.parametrize("deg_u,deg_v", [(65_536, 65_535), (65_536, 65_536), (70_001, 69_000)])
def test_edges_of_two_stars_and_a_dense_corner(deg_u, deg_v):
    """U vertex 0 and V vertex 0 have the two largest degrees; 40 x 50 further
    vertices form a dense corner with both."""
    rng = np.random.default_rng(deg_u)
    corner = rng.choice(40 * 50, 1500, replace=False)
    u = np.concatenate([np.zeros(deg_u), np.arange(1, deg_v), 1 + corner // 50]).astype(np.int32)
    v = np.concatenate([np.arange(deg_u), np.zeros(deg_v - 1), 1 + corner % 50]).astype(np.int32)
    s = np.where(rng.random(u.shape[0]) < 0.6, 1, -1).astype(np.int8)
    assert np.bincount(u).max() == deg_u and np.bincount(v).max() == deg_v
    want_b, want_u = oracle.count_per_edge(u, v, s, deg_v, deg_u, u, v)
    with dbbc.dbbc_graph_from_coo(u, v, s, deg_v, deg_u) as g:
        got_b, got_u = dbbc.dbbc_count_edges(g, u, v)
    assert np.array_equal(got_b, want_b) and np.array_equal(got_u, want_u)
    assert got_b.max() > 0 and got_u.max() > 0
