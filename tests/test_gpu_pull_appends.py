"""A pull level that hands its finds to a push level as a queue.

A hub, its leaves, a thousand vertices behind them of which one has a long row,
and what lies behind those: the level of the leaves is pulled with few edges
left in the graph, and the level after it pushes from the queue that the pull
made, chunk units of the long row included.  Found vertices that fill words,
one to a word, and spread over the range.
"""
import ctypes

import numpy as np
import pytest

import graphgen
import oracle
import paper_2607_17106_gb300 as bg

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def _graph(n, ids):
    hub, a, b, c = 1, np.arange(2, 2002), np.arange(2002, 3002), np.arange(3002, 4002)
    more = np.arange(4002, 5102)  # the long row
    src = np.concatenate([[0], np.full(2000, hub), a[:1000], b, np.full(1100, b[7])])
    dst = np.concatenate([[hub], a, b, c, more])
    if ids == "apart":  # one found vertex a word
        return n, (src * 33 % n).astype(np.int32), (dst * 33 % n).astype(np.int32), 0
    if ids == "spread":
        p = graphgen.permutation(n, seed=3)
        return n, p[src].astype(np.int32), p[dst].astype(np.int32), int(p[0])
    return n, src.astype(np.int32), dst.astype(np.int32), 0


@pytest.mark.parametrize("ids", ["dense", "apart", "spread"])
@pytest.mark.parametrize("opt", [dict(), dict(chunk=64), dict(block_threads=512), dict(mode=bg.BFS_MODE_HOST_LOOP)])
def test_queue_of_a_sparse_pull(ids, opt):
    from paper_2607_17106_gb300 import build
    build.build()
    n, s, d, src = _graph((1 << 21) + 5, ids)
    adj = oracle.build_adjacency(n, s, d)
    ref, _ = oracle.bfs(adj, src, with_parent=False)
    g = bg.Graph.build(n, s, d)
    depth = torch.full((n,), -9, dtype=torch.int32, device="cuda")
    parent = torch.full((n,), -9, dtype=torch.int32, device="cuda")
    rec, lv = (bg.bfs_level_record * 16)(), ctypes.c_int32(0)
    o = bg.options(batch=0, level_log_cap=16, **opt)
    o.level_log, o.levels_out = ctypes.cast(rec, ctypes.POINTER(bg.bfs_level_record)), ctypes.pointer(lv)
    g.run(np.array([src], np.int32), depth, parent, o)
    g.sync()
    # the fifth level has no edge left to find: its form does not matter
    assert [(r.dir, r.f) for r in rec[:4]] == [(0, 1), (0, 1), (bg.BFS_DIR_PULL, 2000), (0, 1000)] and lv.value == 5
    assert np.array_equal(depth.cpu().numpy(), ref)
    assert oracle.validate(adj, src, ref, parent.cpu().numpy()) == 0
