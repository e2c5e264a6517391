"""Single-source searches at their last levels.

Connected graphs, whose last level is passed over because no unvisited vertex
has an edge; graphs with leftovers in small components, whose sparse pull levels
hand a queue to the push level after them, hubs with chunk units among it;
frontiers with less and with more than half of the edges (two forms of the pull
scan); unreached and isolated entries in dirty output rows off a 16-byte
boundary.  Depths and the level count against the oracle, parents validated,
several searches in one launch and one at a time, in the cluster (automatic
for graphs of this size) and grid-wide.
"""
import ctypes

import numpy as np
import pytest

import graphgen
import oracle
import paper_2607_17106_gb300 as bg

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def _late_hub(n, leaves):
    """An RMAT core; behind a chain from it, a hub whose leaves are one more level away."""
    _, s, d = graphgen.rmat(12, 16, seed=7)
    chain = np.concatenate([[int(s[0])], np.arange(n, n + 6)])
    hub = n + 6
    src = np.concatenate([s, chain, np.full(leaves, hub)])
    dst = np.concatenate([d, chain[1:], [hub], np.arange(hub + 1, hub + 1 + leaves)])
    return hub + 1 + leaves, src.astype(np.int32), dst.astype(np.int32)


def _case(kind):
    if kind == "rmat16":
        return graphgen.rmat(16, 16, seed=4)
    if kind == "er-connected":
        return graphgen.erdos_renyi(30011, 30011 * 12, seed=5)
    if kind == "er-sparse":
        return graphgen.erdos_renyi(50003, 60000, seed=6)
    if kind == "complete":
        a, b = np.triu_indices(67, 1)
        return 67, a.astype(np.int32), b.astype(np.int32)
    if kind == "late-hub":
        return _late_hub(1 << 12, 3000)
    return graphgen.barabasi_albert(20001, 4, seed=8)


@pytest.mark.parametrize("kind", ["rmat16", "er-connected", "er-sparse", "complete", "late-hub", "ba"])
@pytest.mark.parametrize("opt", [dict(), dict(small_levels=bg.BFS_SMALL_OFF), dict(small_levels=bg.BFS_SMALL_OFF, chunk=64), dict(chunk=64), dict(block_threads=512), dict(mode=bg.BFS_MODE_HOST_LOOP),
                                 dict(alpha=0.001, beta=1e9), dict(alpha=1e9, beta=1e-6)])
def test_last_levels(kind, opt):
    from paper_2607_17106_gb300 import build
    build.build()
    n, s, d = _case(kind)
    adj = oracle.build_adjacency(n, s, d)
    g = bg.Graph.build(n, s, d)
    deg = np.diff(adj.row_ptr)
    srcs = np.concatenate([np.random.default_rng(1).choice(np.flatnonzero(deg), 4), [int(np.argmin(deg)), n - 1]]).astype(np.int32)
    k = len(srcs)
    ref = [oracle.bfs(adj, int(v), with_parent=False)[0] for v in srcs]
    buf = torch.full((2 * k * n + 1,), -9, dtype=torch.int32, device="cuda")
    depth, parent = buf[1:1 + k * n].view(k, n), buf[1 + k * n:].view(k, n)
    g.run(srcs, depth, parent, bg.options(batch=0, **opt))
    g.sync()
    assert buf[0] == -9
    for j in range(k):
        assert np.array_equal(depth[j].cpu().numpy(), ref[j]), j
        assert oracle.validate(adj, int(srcs[j]), ref[j], parent[j].cpu().numpy()) == 0
        lv = ctypes.c_int32(0)
        o = bg.options(batch=0, **opt)
        o.levels_out = ctypes.pointer(lv)
        one = torch.full((n,), -9, dtype=torch.int32, device="cuda")
        g.run(srcs[j:j + 1], one, None, o)
        assert torch.equal(one, depth[j])
        assert lv.value == ref[j].max() + 1
