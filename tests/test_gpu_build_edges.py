"""The graph build where its sort, merge and row starts change.

Edge counts around a sorting tile (6144 keys) and several of them,
vertex counts on both sides of a change in the number of radix passes, every
combination of the flags that choose between the once-sorted symmetric build
and the general one, skewed and constant keys, and ids out of range that only
show in the raw list.  Rows must equal numpy's exactly.
"""
import numpy as np
import pytest

import paper_2607_17106_gb300 as bg

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

SYM, DEDUP, DROP, CSC = bg.BFS_SYMMETRIZE, bg.BFS_DEDUP, bg.BFS_DROP_SELF, bg.BFS_BUILD_CSC


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2607_17106_gb300 import build
    build.build()


def _rows(n, s, d, flags):
    s, d = s.astype(np.int64), d.astype(np.int64)
    if flags & SYM:
        s, d = np.concatenate([s, d]), np.concatenate([d, s])
    if flags & DROP:
        keep = s != d
        s, d = s[keep], d[keep]
    key = s * n + d
    key = np.unique(key) if flags & DEDUP else np.sort(key)
    s, d = key // n, key % n
    rp = np.searchsorted(s, np.arange(n + 1))
    t = np.sort(d * n + s)
    return rp, d, np.searchsorted(t // n, np.arange(n + 1)), t % n


def _check(n, s, d, flags, device):
    a, b = (torch.from_numpy(s).cuda(), torch.from_numpy(d).cuda()) if device else (s, d)
    g = bg.Graph.build(n, a, b, flags=flags)
    rp, col, cp, ccol = _rows(n, s, d, flags)
    for got, want in zip(g.csr() + g.csr(csc=True), (rp, col, cp, ccol)):
        assert np.array_equal(got, want)
    deg, din = np.diff(rp), np.diff(cp)
    i = g.info()
    assert (i.n, i.m, i.deg_max, i.n_isolated) == (n, len(col), deg.max(), int((din == 0).sum()))
    assert abs(i.deg_mean - deg.mean()) <= 1e-12 * max(1.0, deg.mean())
    g.free()


def _edges(kind, n, m, seed):
    rng = np.random.default_rng(seed)
    if kind == "uniform":
        return rng.integers(0, n, m).astype(np.int32), rng.integers(0, n, m).astype(np.int32)
    if kind == "skewed":  # a hub row, many repeats, self-loops
        s = (n * rng.random(m) ** 6).astype(np.int32)
        d = (n * rng.random(m) ** 3).astype(np.int32)
        d[::17] = s[::17]
        return s, d
    if kind == "constant":
        return np.full(m, n - 1, np.int32), np.full(m, 0, np.int32)
    return np.full(m, n // 2, np.int32), np.full(m, n // 2, np.int32)  # self-loops alone


@pytest.mark.parametrize("flags", [SYM | DEDUP | DROP | CSC, SYM | DEDUP | CSC, SYM | DROP, SYM, DEDUP | DROP | CSC,
                                   DEDUP, DROP | CSC, 0])
@pytest.mark.parametrize("kind", ["uniform", "skewed", "constant", "loops"])
def test_flags(flags, kind):
    _check(1537, *_edges(kind, 1537, 20011, 3), flags, device=True)


@pytest.mark.parametrize("m", [0, 1, 2, 31, 383, 384, 385, 6143, 6144, 6145, 12288, 49153, 65537, 131073])
@pytest.mark.parametrize("flags", [SYM | DEDUP | DROP | CSC, DEDUP | DROP | CSC])
def test_edge_counts(m, flags):
    _check(3001, *_edges("uniform", 3001, m, m), flags, device=m % 2 == 0)


# bits of an id: 1, 2, 9 and 10 (one and two passes by the lower part), 18 and 19, 20
@pytest.mark.parametrize("n", [1, 2, 3, 511, 512, 513, 262144, 262145, 700001])
@pytest.mark.parametrize("flags", [SYM | DEDUP | DROP | CSC, DEDUP | DROP | CSC])
def test_vertex_counts(n, flags):
    _check(n, *_edges("skewed", n, 30000, n), flags, device=True)


@pytest.mark.parametrize("bad", [5, 8, 1 << 20, -1])
@pytest.mark.parametrize("flags", [SYM | DEDUP | DROP | CSC, SYM, DEDUP])
def test_ids_out_of_range(bad, flags):
    for where in (0, 1):
        e = [np.zeros(9000, np.int32), np.ones(9000, np.int32)]
        e[where][8999] = bad
        with pytest.raises(bg.BfsError) as err:
            bg.Graph.build(5, e[0], e[1], flags=flags)
        assert err.value.status == bg.BFS_EINVAL


# Counting CTAs take 1, 2, .. 8 tiles, by the tiles of the sort over the CTAs
# there are: the second sort, of the keys kept, can have more chunks than the first.
@pytest.mark.parametrize("first,kept", [(2.0, 1.99), (2.0, 1.5), (3.01, 1.99), (3.01, 0.5)])
@pytest.mark.parametrize("flags", [SYM | DEDUP | DROP | CSC, DEDUP | DROP | CSC])
def test_second_sort_of_fewer_keys(first, kept, flags):
    ctas = 4 * torch.cuda.get_device_properties(0).multi_processor_count
    m, k = int(first * ctas * 6144) + 1, int(kept * ctas * 6144)
    s, d = _edges("uniform", 1 << 18, k, 11)
    r = np.arange(m) % k  # the rest repeats edges
    _check(1 << 18, s[r], d[r], flags, device=True)
