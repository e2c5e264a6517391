"""The cluster kernel for the small levels of low-degree graphs.

Its queue arithmetic (the k-th claim of a CTA goes to the next CTA in turn), the
hand-over of a frontier that outgrows the cluster, rows of up to 4 and of up to
8 neighbours, vertex counts around a bitmap word, and the options that send a
search through it.  Depths and parents against the oracle; the level log and
the level count against the same search without the cluster.
"""
import ctypes

import numpy as np
import pytest

import graphgen
import oracle
import paper_2607_17106_gb300 as bg

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def _tree(arity, depth, seed):
    """A complete tree whose frontier outgrows the cluster, relabelled, then a path from one leaf."""
    n, first = 1, [0]
    src, dst, level = [], [], [0]
    for _ in range(depth):
        nxt = []
        for u in level:
            for _ in range(arity):
                src.append(u)
                dst.append(n)
                nxt.append(n)
                n += 1
        level = nxt
    last = level[-1]
    for _ in range(50):
        src.append(last)
        dst.append(n)
        last = n
        n += 1
    perm = graphgen.permutation(n, seed=seed)
    return n, perm[np.array(src)].astype(np.int32), perm[np.array(dst)].astype(np.int32), int(perm[first[0]])


def _case(kind):
    if kind.startswith("tree"):
        return _tree(3, 10, 5) if kind == "tree4" else _tree(7, 6, 6)
    if kind == "grid":
        n, s, d = graphgen.grid(401, 127, 0.1, seed=4)
    elif kind == "er8":  # bounded degree up to 8: edges beyond it are left out
        n, s, d = graphgen.erdos_renyi(20011, 40000, seed=3)
        seen = np.zeros(n, int)
        keep = np.zeros(len(s), bool)
        for i, (a, b) in enumerate(zip(s, d)):
            if a != b and seen[a] < 8 and seen[b] < 8:
                keep[i] = True
                seen[a] += 1
                seen[b] += 1
        s, d = s[keep], d[keep]
    else:
        n = int(kind)
        s = np.arange(n - 1, dtype=np.int32)
        d = s + 1
    return n, s, d, int(s[0])


@pytest.mark.parametrize("kind", ["grid", "tree4", "tree8", "er8", "2", "31", "32", "33", "1000"])
@pytest.mark.parametrize("policy", [bg.BFS_POLICY_HEURISTIC, bg.BFS_POLICY_PUSH])
def test_small_rows_search(kind, policy):
    from paper_2607_17106_gb300 import build
    build.build()
    n, s, d, src = _case(kind)
    adj = oracle.build_adjacency(n, s, d)
    g = bg.Graph.build(n, s, d)
    assert g.info().deg_max <= 8
    srcs = np.array([src, int(d[-1])], np.int32)
    for gamma in (16.0, 1e-6):  # 1e-6: no level is read from the bitmap, the frontier alone ends the cluster's part
        got = {}
        for small in (bg.BFS_SMALL_AUTO, bg.BFS_SMALL_OFF):
            depth = torch.full((2, n), -9, dtype=torch.int32, device="cuda")
            parent = torch.full((2, n), -9, dtype=torch.int32, device="cuda")
            o = dict(batch=0, small_levels=small, policy=policy, gamma=gamma)
            g.run(srcs, depth, parent, bg.options(**o))
            g.sync()
            for j in range(2):
                ref, _ = oracle.bfs(adj, int(srcs[j]), with_parent=False)
                assert np.array_equal(depth[j].cpu().numpy(), ref)
                assert oracle.validate(adj, int(srcs[j]), ref, parent[j].cpu().numpy()) == 0
            only = torch.full((n,), -9, dtype=torch.int32, device="cuda")
            rec, lv = (bg.bfs_level_record * 2000)(), ctypes.c_int32(0)
            opt = bg.options(level_log_cap=2000, **o)
            opt.level_log, opt.levels_out = ctypes.cast(rec, ctypes.POINTER(bg.bfs_level_record)), ctypes.pointer(lv)
            g.run(srcs[:1], only, None, opt)  # depths alone
            g.sync()
            assert torch.equal(only, depth[0])
            got[small] = (lv.value, [(r.level, r.dir, r.f, r.e_f, r.m_u) for r in rec[: lv.value + 1]])
        assert got[bg.BFS_SMALL_AUTO] == got[bg.BFS_SMALL_OFF]
    with pytest.raises(bg.BfsError) as e:
        g.run(srcs[:1], only, None, bg.options(batch=0, max_levels=1, policy=policy))
        g.sync()
    assert e.value.status == bg.BFS_ERANGE
