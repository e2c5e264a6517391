"""bfs_run_mixed keeps its workspace with the largest graph of a call.

Calls in a row that need more units, another chunk size, another largest graph,
or fewer of everything; a graph that is freed in between; an error in between;
and calls from several threads on streams of their own, of which only one finds
the workspace free.  Depths against the oracle.
"""
import threading

import numpy as np
import pytest

import graphgen
import oracle
import paper_2607_17106_gb300 as bg

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


class _Set:
    def __init__(self):
        from paper_2607_17106_gb300 import build
        build.build()
        self.adj, self.g = [], []
        for n, s, d in (graphgen.rmat(11, 16, seed=1), graphgen.erdos_renyi(5001, 20000, seed=2), graphgen.grid(90, 71, 0.1, seed=3)):
            self.adj.append(oracle.build_adjacency(n, s, d))
            self.g.append(bg.Graph.build(n, s, d))

    def call(self, goq, seed, **opt):
        rng = np.random.default_rng(seed)
        srcs = np.array([rng.integers(0, self.adj[q].n) for q in goq], np.int32)
        dep = [torch.full((self.adj[q].n,), -9, dtype=torch.int32, device="cuda") for q in goq]
        par = [torch.full((self.adj[q].n,), -9, dtype=torch.int32, device="cuda") for q in goq]
        bg.run_mixed(self.g, goq, srcs, dep, par, opt=bg.options(**opt) if opt else None)
        for i, q in enumerate(goq):
            ref, _ = oracle.bfs(self.adj[q], int(srcs[i]), with_parent=False)
            assert np.array_equal(dep[i].cpu().numpy(), ref), (i, q)
            assert oracle.validate(self.adj[q], int(srcs[i]), ref, par[i].cpu().numpy()) == 0


def test_calls_in_a_row():
    s = _Set()
    s.call([0, 1, 2, 0, 1], 1)
    s.call([2] * 3 + [0] * 70 + [1] * 130, 2)   # more units
    s.call([0, 0, 2], 3)                        # another largest graph
    s.call([0, 1, 2], 4, chunk=64)              # units of another size
    with pytest.raises(bg.BfsError) as e:       # a search that stops early leaves masks behind
        s.call([1, 2], 5, max_levels=3)
    assert e.value.status == bg.BFS_ERANGE
    s.call([1, 2, 2, 0], 6)
    s.g[2].free()
    n, a, b = graphgen.grid(60, 31, 0.0, seed=9)
    s.adj[2], s.g[2] = oracle.build_adjacency(n, a, b), bg.Graph.build(n, a, b)
    s.call([2, 1, 0, 2], 7)


def test_calls_from_threads():
    s = _Set()
    errors = []

    def work(t):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for i in range(4):
                    s.call([0, 1, 2, 1, 2][t % 2:], 100 * t + i)
                    torch.cuda.current_stream().synchronize()
        except BaseException as e:  # noqa: BLE001
            errors.append(e)

    threads = [threading.Thread(target=work, args=(t,)) for t in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors[0]
