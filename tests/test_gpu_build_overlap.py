"""A graph build waits for its own stream, not for work on others.

A kernel that only waits (0.3 s) runs on one stream while a graph is built on
another, with scratch that comes from the stream-ordered pool and scratch that
is too large for it, from device and from host edges.
"""
import numpy as np
import pytest

import paper_2607_17106_gb300 as bg

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [20000, 6000000])
@pytest.mark.parametrize("kind", ["symmetric", "directed", "host"])
def test_build_beside_another_stream(m, kind):
    from paper_2607_17106_gb300 import build
    build.build()
    n = 100003
    rng = np.random.default_rng(m)
    s, d = rng.integers(0, n, m).astype(np.int32), rng.integers(0, n, m).astype(np.int32)
    flags = bg.BFS_DEFAULT_FLAGS & ~bg.BFS_SYMMETRIZE if kind == "directed" else bg.BFS_DEFAULT_FLAGS
    src, dst = (s, d) if kind == "host" else (torch.from_numpy(s).cuda(), torch.from_numpy(d).cuda())
    busy, own = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda.synchronize()
    first = bg.Graph.build(n, src, dst, flags=flags, stream=own)  # loads the kernels
    torch.cuda.synchronize()
    done = torch.cuda.Event()
    with torch.cuda.stream(busy):
        torch.cuda._sleep(600_000_000)
        done.record()
    g = bg.Graph.build(n, src, dst, flags=flags, stream=own)
    still_busy = not done.query()
    torch.cuda.synchronize()
    assert still_busy
    assert all(np.array_equal(x, y) for x, y in zip(g.csr(), first.csr()))
