"""What the library does when a wait runs out or a runtime call fails.

No input makes the small levels' waits run out, the launch of their rows fail or
a copy fail, so the library is linked here with a copy of one file that gives a
wait up at the caller's limit (instead of a second at least), or whose first
launch or copy is refused by a fake of the runtime's call.
"""
import contextlib
import ctypes
import gc
import os
import subprocess

import numpy as np
import pytest

import graphgen
import oracle
import paper_2607_17106_gb300 as bg
from paper_2607_17106_gb300 import build

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

FAKE_LAUNCH = """
#include <cuda_runtime.h>
extern "C" { int fake_calls = 0; }
template <typename K, typename... A>
static cudaError_t fake_launch(const cudaLaunchConfig_t* c, K k, A... a) {
    return fake_calls++ == 0 ? cudaErrorLaunchOutOfResources : cudaLaunchKernelEx(c, k, a...);
}
#define cudaLaunchKernelEx fake_launch
"""
FAKE_COPY = """
#include <cuda_runtime.h>
extern "C" { int fake_calls = 0; }
static cudaError_t fake_copy(void* d, const void* s, size_t n, cudaMemcpyKind k, cudaStream_t st) {
    return fake_calls++ == 0 ? cudaErrorInvalidValue : cudaMemcpyAsync(d, s, n, k, st);
}
#define cudaMemcpyAsync fake_copy
"""


def _link(tmp, name, *flags):
    """The library with csrc/`name` compiled with `flags`."""
    build.build()
    src = os.path.join(build.CSRC, name)
    obj, lib = os.path.join(tmp, "variant.o"), os.path.join(tmp, "libbfsgb_variant.so")
    objs = [os.path.join(build.OUT_DIR, os.path.basename(s)[:-3] + ".o") for s in build.sources() if s != src]
    nvcc = build._nvcc()
    subprocess.run([nvcc, *build.ARCH, *build.NVCC_FLAGS, *flags, "-c", src, "-o", obj], check=True)
    subprocess.run([nvcc, *build.ARCH, "-shared", "-o", lib, obj, *objs], check=True)
    return lib


@contextlib.contextmanager
def _loaded(path):
    kept, bg._lib = bg._lib, None
    try:
        yield bg.load(path)
    finally:
        gc.collect()  # graphs are freed by the library that made them
        bg._lib = kept


def _search(g, n, src, **opt):
    depth = torch.full((n,), -9, dtype=torch.int32, device="cuda")
    parent = torch.full((n,), -9, dtype=torch.int32, device="cuda")
    g.run(np.array([src], np.int32), depth, parent, bg.options(batch=0, **opt))
    g.sync()
    return depth.cpu().numpy(), parent.cpu().numpy()


def _graph(kind):
    if kind == "grid":  # rows of 4
        return graphgen.grid(161, 127, 0.1, seed=4)
    n = 4000            # rows of 8: a ring with chords
    v = np.arange(n, dtype=np.int32)
    return n, np.concatenate([v, v, v]), np.concatenate([(v + 1) % n, (v + 17) % n, (v + 63) % n]).astype(np.int32)


def test_given_up_waits(tmp_path):
    # CTAs give up at their own times: some while others finish the level, hand
    # the search over or find it done.  The call reports it, or succeeds with the
    # right depths, and the next search on the same graph is right.
    lib = _link(str(tmp_path), "bfs_small.cu", "-DBFS_SMALL_WAIT_NS=0")
    with _loaded(lib):
        for kind in ("grid", "ring"):
            n, s, d = _graph(kind)
            adj = oracle.build_adjacency(n, s, d)
            g = bg.Graph.build(n, s, d)
            rng = np.random.default_rng(7)
            timeouts = {}
            for limit in (1, 200, 400, 600, 800, 1000, 1500, 2000, 4000, 1000000):
                timeouts[limit] = 0
                for src in rng.integers(0, n, 12):
                    ref, _ = oracle.bfs(adj, int(src), with_parent=False)
                    # gamma: with 1e-6 only the frontier's size ends the cluster's part
                    for gamma in (16.0, 1e-6):
                        try:
                            assert np.array_equal(_search(g, n, int(src), barrier_timeout_ns=limit, gamma=gamma)[0], ref)
                        except bg.BfsError as e:
                            assert e.status == bg.BFS_ETIMEOUT and f"exceeded {limit} ns" in str(e)
                            timeouts[limit] += 1
                depth, parent = _search(g, n, int(src))
                assert np.array_equal(depth, ref) and oracle.validate(adj, int(src), depth, parent) == 0
            g.free()
            assert timeouts[1] > 0


def test_rows_that_could_not_be_launched(tmp_path):
    fake = tmp_path / "fake.h"
    fake.write_text(FAKE_LAUNCH)
    lib = _link(str(tmp_path), "bfs_small.cu", "-include", str(fake))
    with _loaded(lib) as handle:
        launches = ctypes.c_int.in_dll(handle, "fake_calls")
        n, s, d = _graph("grid")
        adj = oracle.build_adjacency(n, s, d)
        g = bg.Graph.build(n, s, d)
        seen = []
        for src in (5, 700, 9000):
            ref, _ = oracle.bfs(adj, src, with_parent=False)
            depth, parent = _search(g, n, src)
            assert np.array_equal(depth, ref) and oracle.validate(adj, src, depth, parent) == 0
            seen.append(launches.value)
        g.free()
        # refused: the general kernel; then the rows and the search; then the search
        assert seen == [1, 3, 4]


def test_message_names_the_limit():
    # of the run that failed, also where bfs_sync reports it
    build.build()
    n, s, d = graphgen.rmat(14, 16, seed=1)
    g = bg.Graph.build(n, s, d)
    for k, opt in ((1, dict(batch=0)), (3, dict(batch=0)), (3, dict(batch=1))):
        depth = torch.empty((k, n), dtype=torch.int32, device="cuda")
        with pytest.raises(bg.BfsError) as e:
            g.run(s[:k], depth, None, bg.options(barrier_timeout_ns=7, **opt))
            g.sync()
        assert e.value.status == bg.BFS_ETIMEOUT and "exceeded 7 ns" in str(e.value)


def test_unit_count_that_failed(tmp_path):
    # a batch's chunk units are counted once per graph; a count that failed is
    # reported and not kept
    fake = tmp_path / "fake.h"
    fake.write_text(FAKE_COPY)
    lib = _link(str(tmp_path), "msbfs.cu", "-include", str(fake))
    with _loaded(lib):
        n, s, d = graphgen.rmat(13, 16, seed=1)
        adj = oracle.build_adjacency(n, s, d)
        g = bg.Graph.build(n, s, d)
        depth = torch.full((5, n), -9, dtype=torch.int32, device="cuda")
        run = lambda: bg.run_mixed([g], [0] * 5, s[:5], list(depth), opt=bg.options(chunk=64))  # noqa: E731
        with pytest.raises(bg.BfsError) as e:
            run()
        assert e.value.status == bg.BFS_ECUDA
        run()
        for j in range(5):
            assert np.array_equal(depth[j].cpu().numpy(), oracle.bfs(adj, int(s[j]), with_parent=False)[0])
        g.free()
