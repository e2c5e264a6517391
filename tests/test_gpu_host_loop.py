"""The host-loop drive, one launch a level: its last launch finds the search
finished and says so while other CTAs are still reading the state.

Many short searches, each ending in such a launch, by every CTA size and with
ends of every kind: an empty frontier behind a push or a pull level, an isolated
source, the level limit.
"""
import ctypes

import numpy as np
import pytest

import graphgen
import oracle
import paper_2607_17106_gb300 as bg

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("threads", [256, 512, 1024])
@pytest.mark.parametrize("policy", [bg.BFS_POLICY_HEURISTIC, bg.BFS_POLICY_PULL])
def test_searches_that_end(threads, policy):
    from paper_2607_17106_gb300 import build
    build.build()
    n, s, d = graphgen.erdos_renyi(6007, 9000, seed=11)
    adj = oracle.build_adjacency(n, s, d)
    g = bg.Graph.build(n, s, d)
    rng = np.random.default_rng(3)
    deg = np.diff(adj.row_ptr)
    srcs = np.concatenate([rng.integers(0, n, 37), [int(np.argmin(deg)), int(s[0]), int(s[0])]]).astype(np.int32)
    ref = {int(v): oracle.bfs(adj, int(v), with_parent=False)[0] for v in srcs}
    opt = dict(batch=0, mode=bg.BFS_MODE_HOST_LOOP, block_threads=threads, policy=policy)
    for _ in range(4):
        depth = torch.full((len(srcs), n), -9, dtype=torch.int32, device="cuda")
        parent = torch.full((len(srcs), n), -9, dtype=torch.int32, device="cuda")
        g.run(srcs, depth, parent, bg.options(**opt))
        dh, ph = depth.cpu().numpy(), parent.cpu().numpy()
        for j, v in enumerate(srcs):
            assert np.array_equal(dh[j], ref[int(v)])
            assert oracle.validate(adj, int(v), dh[j], ph[j]) == 0
    lv = ctypes.c_int32(0)
    o = bg.options(**opt)
    o.levels_out = ctypes.pointer(lv)
    g.run(srcs[-1:], depth[0], None, o)
    assert lv.value == ref[int(srcs[-1])].max() + 1
    with pytest.raises(bg.BfsError) as e:
        g.run(srcs[-1:], depth[0], None, bg.options(max_levels=2, **opt))
    assert e.value.status == bg.BFS_ERANGE
