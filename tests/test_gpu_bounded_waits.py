"""What follows a bounded tile wait that gave up: the kernels after it must not
use what it left unwritten, the call returns DBBC_EINTERNAL, and the next call
works. Run on a checked variant of the library in which every tile that would
wait for an earlier one gives up before its first poll (-DDBBC_SPIN_LIMIT=0):
lists of a single tile build and count as ever, longer ones give up. Device
memory is filled with ones before the library gets it, so an index that was
never written is out of range and would be recorded."""
import os
import subprocess
import sys

import pytest

from paper_2609_21848_gb300 import buildlib

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import ctypes
import numpy as np, torch
import oracle
import paper_2609_21848_gb300 as dbbc

torch.cuda.set_device(0)
live = {}

def alloc(size, stream, ctx):
    t = torch.full((size,), 255, dtype=torch.uint8, device="cuda")
    live[t.data_ptr()] = t
    return t.data_ptr()

refs = (dbbc._ALLOC_FN(alloc), dbbc._FREE_FN(lambda p, stream, ctx: live.pop(int(p))))
dbbc.lib().dbbc_set_allocator(ctypes.cast(refs[0], ctypes.c_void_p), ctypes.cast(refs[1], ctypes.c_void_p), None)

def edges(seed, n_u, n_v, m, repeats=0):
    rng = np.random.default_rng(seed)
    k = rng.choice(n_u * n_v, m - repeats, replace=False)
    k = np.concatenate([k, k[:repeats]])
    return ((k // n_v).astype(np.int32), (k % n_v).astype(np.int32),
            np.where(rng.random(m) < 0.5, 1, -1).astype(np.int8), n_u, n_v)

def gives_up(f):
    try:
        f()
    except dbbc.DbbcError as e:
        assert e.status == dbbc.DBBC_EINTERNAL, e
    else:
        raise AssertionError("the call succeeded")
    torch.cuda.synchronize()
    assert dbbc.dbbc_checked_flags() == 0, "an index left its array"

# every pivot with a butterfly to close is a hub
dbbc.dbbc_set_tuning({"light_max_work": 1, "medium_max_work": 1})
assert dbbc.dbbc_is_checked()
small = [edges(i, 120, 120, 2_000) for i in range(30)]
want = [oracle.count(*g)[:2] for g in small]

def small_ones_count():
    graphs = [dbbc.dbbc_graph_from_coo(*g) for g in small]
    for g, w in zip(graphs, want):
        assert dbbc.dbbc_count(g) == w
    return graphs

graphs = small_ones_count()
items = [g.info["hub_items"] for g in graphs]
few = 8
assert sum(items[:few]) < 4096 < sum(items), items   # one and two tiles of the plan's sort
b, u = dbbc.dbbc_count_batch(graphs[:few])
assert list(zip(b.tolist(), u.tolist())) == want[:few]
gives_up(lambda: dbbc.dbbc_batch_create(graphs))
gives_up(lambda: dbbc.dbbc_count_batch(graphs))
for args in [edges(1, 700, 900, 3_000),          # row tiles
             edges(2, 200, 200, 20_000),         # tiles of the edge sorts
             edges(3, 100, 100, 3_000, 20),      # tiles of the repeats
             edges(4, 9_000, 8_000, 60_000),     # tiles of every kernel
             edges(5, 200, 200, 4_000)]:         # tiles of the hub plan
    gives_up(lambda: dbbc.dbbc_graph_from_coo(*args))
cat = [np.concatenate([g[i] for g in small]) for i in range(3)]
off = np.arange(len(small) + 1) * 2_000
gives_up(lambda: dbbc.dbbc_graph_from_coo_multi(*cat, off, [g[3] for g in small], [g[4] for g in small]))
for g in small_ones_count() + graphs:
    g.free()
torch.cuda.synchronize()
assert not live and dbbc.dbbc_checked_flags() == 0
print("ok")
"""


def test_calls_whose_tile_waits_give_up():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    lib = buildlib.build(extra_flags=["-DDBBC_CHECKED=1", "-DDBBC_SPIN_LIMIT=0"],
                         out_dir=os.path.join(buildlib.OUT_DIR, "no_waits"))
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, env=dict(os.environ, DBBC_LIBRARY=lib),
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.split()[-1:] == ["ok"], r.stdout + r.stderr
