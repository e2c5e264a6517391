"""Batched searches where the level code of the 64-lane kernel changes path.

Short-row push levels (maximum degree 1, 2, 4, 16) against the general ones
(17 and more), levels on both sides of the kept history (16), past it with
pull levels and with chunk units, batches of 1 lane short of full and of more
than one unit, vertex counts around a bitmap word, with and without parents.
Every lane's depths against the oracle, parents validated.
"""
import numpy as np
import pytest

import graphgen
import oracle
import paper_2607_17106_gb300 as bg

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def _ring_of_stars(stars, leaves):
    """Hubs on a path, each with leaves: long diameter and rows above the chunk size."""
    hubs = np.arange(stars, dtype=np.int32) * (leaves + 1)
    src = [hubs[:-1]] + [np.repeat(hubs, leaves).astype(np.int32)]
    dst = [hubs[1:]] + [(np.repeat(hubs, leaves) + np.tile(np.arange(1, leaves + 1), stars)).astype(np.int32)]
    return stars * (leaves + 1), np.concatenate(src), np.concatenate(dst)


def _case(kind):
    if kind == "pairs":
        n = 2001
        a = np.arange(0, n - 1, 2, dtype=np.int32)
        return n, a, a + 1
    if kind.startswith("path"):
        n = int(kind[4:])
        a = np.arange(n - 1, dtype=np.int32)
        return n, a, a + 1
    if kind == "grid":
        return graphgen.grid(211, 97, 0.1, seed=4)
    if kind.startswith("band"):  # vertex i joined to the next w: degree 2 w
        n, w = 3000, int(kind[4:])
        s = np.concatenate([np.arange(n - k, dtype=np.int32) for k in range(1, w + 1)])
        d = np.concatenate([np.arange(k, n, dtype=np.int32) for k in range(1, w + 1)])
        return n, s, d
    if kind == "stars":
        return _ring_of_stars(40, 90)
    return graphgen.rmat(13, 16, seed=5)


@pytest.mark.parametrize("kind", ["pairs", "path2", "path31", "path33", "path700", "grid", "band8", "band9", "stars", "rmat"])
@pytest.mark.parametrize("k", [2, 63, 64, 70])
def test_batch_levels(kind, k):
    from paper_2607_17106_gb300 import build
    build.build()
    n, s, d = _case(kind)
    adj = oracle.build_adjacency(n, s, d)
    g = bg.Graph.build(n, s, d)
    srcs = np.random.default_rng(k).integers(0, n, k).astype(np.int32)
    ref = [oracle.bfs(adj, int(v), with_parent=False)[0] for v in srcs]
    # push alone, the heuristic, and alternating forms (pull levels past the history, lists rebuilt); chunk 64: units;
    # pull alone, with serial scans that end inside a step of four
    for o in (dict(policy=bg.BFS_POLICY_PUSH), dict(), dict(schedule=[0, 2, 2, 0, 0], chunk=64),
              dict(policy=bg.BFS_POLICY_PULL, pull_serial=3), dict(policy=bg.BFS_POLICY_PULL, pull_serial=1)):
        for par in (True, False):
            depth = torch.full((k, n), -9, dtype=torch.int32, device="cuda")
            parent = torch.full((k, n), -9, dtype=torch.int32, device="cuda") if par else None
            g.run(srcs, depth, parent, bg.options(batch=1, **o))
            g.sync()
            got = depth.cpu().numpy()
            for j in range(k):
                assert np.array_equal(got[j], ref[j]), (o, j)
                if par and j % 9 == 0:
                    assert oracle.validate(adj, int(srcs[j]), ref[j], parent[j].cpu().numpy()) == 0


# Rows above MS_LONG_ROW_SMALL entries, scanned by a CTA in steps of 512: hubs
# joined to the same `width` vertices, their missing lanes complete in the
# first, the last or no step.
@pytest.mark.parametrize("width", [511, 512, 513, 1024, 4099, 9001])
@pytest.mark.parametrize("k", [1, 64, 96])
def test_long_rows(width, k):
    from paper_2607_17106_gb300 import build
    build.build()
    hubs = 300
    n = hubs + width + 40
    rng = np.random.default_rng(width + k)
    s = np.repeat(np.arange(hubs, dtype=np.int32), width)
    d = (hubs + np.tile(np.arange(width), hubs)).astype(np.int32)
    tail = np.arange(hubs + width, n, dtype=np.int32)  # a path into one end of the rows
    s, d = np.concatenate([s, tail[:-1], tail[-1:]]), np.concatenate([d, tail[1:], np.int32([n - 41])])
    adj = oracle.build_adjacency(n, s, d)
    g = bg.Graph.build(n, s, d)
    srcs = rng.integers(0, n, k).astype(np.int32)
    ref = {v: oracle.bfs(adj, v, with_parent=False)[0] for v in set(srcs.tolist())}
    for o in (dict(policy=bg.BFS_POLICY_PULL), dict()):
        for par in (True, False):
            depth = torch.full((k, n), -9, dtype=torch.int32, device="cuda")
            parent = torch.full((k, n), -9, dtype=torch.int32, device="cuda") if par else None
            g.run(srcs, depth, parent, bg.options(batch=1, **o))
            g.sync()
            got = depth.cpu().numpy()
            for j, v in enumerate(srcs.tolist()):
                assert np.array_equal(got[j], ref[v]), (o, j)
                if par and j % 9 == 0:
                    assert oracle.validate(adj, v, ref[v], parent[j].cpu().numpy()) == 0
    g.free()


# Rows a warp gives up once it has scanned MS_WARP_ENTRIES in a word, on graphs of
# more than two words a warp: what the warp found and what the CTA finds in the rest of the row
# must add up (depths, parents, levels past the history, the frontier's counts).
@pytest.mark.parametrize("width", [1024 + 32, 1024 + 33, 1700, 8192])
@pytest.mark.parametrize("k", [3, 64])
def test_rows_given_up(width, k):
    from paper_2607_17106_gb300 import build
    build.build()
    hubs, tail, n = 200, 40, 500_000
    rng = np.random.default_rng(width + k)
    s = np.repeat(np.arange(hubs, dtype=np.int32), width)
    d = (hubs + np.tile(np.arange(width), hubs)).astype(np.int32)
    path = np.arange(hubs + width, hubs + width + tail, dtype=np.int32)  # into the last entry of every hub's row
    s, d = np.concatenate([s, path]), np.concatenate([d, path[1:], np.int32([hubs + width - 1])])
    adj = oracle.build_adjacency(n, s, d)
    g = bg.Graph.build(n, s, d)
    srcs = np.concatenate([path[[0, 20, 39]], rng.integers(0, hubs + width + tail, k - 3)]).astype(np.int32)
    ref = {v: oracle.bfs(adj, v, with_parent=False)[0] for v in set(srcs.tolist())}
    for o in (dict(policy=bg.BFS_POLICY_PULL), dict(policy=bg.BFS_POLICY_PULL, pull_serial=1), dict()):
        for par in (True, False):
            depth = torch.full((k, n), -9, dtype=torch.int32, device="cuda")
            parent = torch.full((k, n), -9, dtype=torch.int32, device="cuda") if par else None
            g.run(srcs, depth, parent, bg.options(batch=1, **o))
            g.sync()
            got = depth.cpu().numpy()
            for j, v in enumerate(srcs.tolist()):
                assert np.array_equal(got[j], ref[v]), (o, j)
                if par and (j < 3 or j % 9 == 0):
                    assert oracle.validate(adj, v, ref[v], parent[j].cpu().numpy()) == 0
    g.free()
