"""Connected components where the union-find kernel's paths change.

Chains of parents as long as the graph (natural-order and reversed paths, more
than one shortcut pass), rows around the lengths where a lane, a warp or the
whole grid hooks them, in a component that is not the largest one, and vertex
counts around a CTA's threads.  Labels are whole numbers and must equal the
oracle's.
"""
import numpy as np
import pytest

import graphgen
import oracle
import paper_2607_17106_gb300 as bg

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def _stars(lengths, giant):
    """A path of `giant` vertices, then for each length two stars of that many
    leaves whose centres are joined; ids shuffled."""
    src, dst, n = list(range(giant - 1)), list(range(1, giant)), giant
    for k in lengths:
        c0, c1 = n, n + 1
        leaves = np.arange(n + 2, n + 2 + 2 * k)
        src += [c0] + [c0] * k + [c1] * k
        dst += [c1] + list(leaves)
        n += 2 + 2 * k
    perm = graphgen.permutation(n, seed=11)
    return n, perm[np.array(src)].astype(np.int32), perm[np.array(dst)].astype(np.int32)


def _case(kind):
    if kind.startswith("path"):
        n = 200000
        a = np.arange(n - 1, dtype=np.int32)
        return (n, a, a + 1) if kind == "path" else (n, n - 1 - a, n - 2 - a)
    if kind == "rows":
        return _stars([1, 14, 15, 16, 17, 18, 19, 33, 4092, 4093, 4094, 4095, 4096, 9000], 60000)
    if kind == "rows-no-largest":  # no component stands out in the sample
        return _stars([5000, 4096, 4095, 4097], 2)
    if kind == "grid-natural":
        return graphgen.grid(700, 301, 0.1, seed=4, relabel=False)
    n = int(kind)
    s = np.arange(n - 1, dtype=np.int32)
    return n, s, np.full(n - 1, n - 1, np.int32)


@pytest.mark.parametrize("kind", ["path", "path-reversed", "rows", "rows-no-largest", "grid-natural", "2", "511", "512",
                                  "513", "1025"])
def test_components_forest_paths(kind):
    from paper_2607_17106_gb300 import build
    build.build()
    n, s, d = _case(kind)
    want = oracle.min_label(oracle.build_adjacency(n, s, d))
    g = bg.Graph.build(n, s, d)
    buf = torch.full((n + 1,), -7, dtype=torch.int32, device="cuda")
    for label in (buf[1:], buf[:n]):  # a 4-byte and a 16-byte boundary; the scratch is used twice
        g.components(label)
        assert np.array_equal(label.cpu().numpy(), want)
    assert g.components()[1] >= 1
