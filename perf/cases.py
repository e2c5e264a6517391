"""What a user of this library has it do, as cases that can be timed.

A case is a dict of plain values.  ``listed()`` gives the named ones,
``draw(rng)`` more of the same ranges; ``prepare`` makes the inputs of a case
on the GPU from a seed (graph, sources, output buffers, options), ``run`` is one
pass through the package's public calls, ``work`` the bytes and operations the
pass cannot do without, ``exact`` the same pass in 64 bits where the outputs
are computed numbers (the policy's training step).

Graphs are the families the repository generates (RMAT, Erdos-Renyi, the
relabelled grid with deleted edges), drawn here with torch so that inputs are
ready in a fraction of a second.  Sources are vertices with an edge, uniformly.

Searches and batches write the parent arrays too where ``parents`` is set.
What comes back of them is the depths: a vertex's parent is any of its
neighbours one level up, push levels let the first claim win, and two runs on
the same inputs name different, equally valid ones.
"""
import math

import numpy as np
import torch

import paper_2607_17106_gb300 as bg

DEV = "cuda"


def listed():
    return [
        # The smallest call there is: one search of the scale-14 graph, its
        # arrays in the L2 cache, the time all launch and level latency.
        dict(name="one-rmat14", op="search", kind="rmat", scale=14, ef=16, a=0.57, k=1, parents=True),
        # The headline: 64 searches of RMAT scale 22, one at a time, push and
        # pull levels, hubs of a hundred thousand neighbours.
        dict(name="search-rmat22", op="search", kind="rmat", scale=22, ef=16, a=0.57, k=64, parents=True),
        # The same on a graph without hubs: wide levels of short rows.
        dict(name="search-er22", op="search", kind="er", n=1 << 22, deg=16, directed=False, k=64, parents=True),
        # A long-diameter graph (road-like): thousands of levels of a few
        # thousand vertices each, one query.
        dict(name="search-grid4096", op="search", kind="grid", width=4096, height=4096, p_del=0.1, k=1, parents=True),
        # 64 sources at once on the largest graph of the configurations:
        # the throughput form, 8.6 GB of outputs.
        dict(name="batch-rmat24", op="batch", kind="rmat", scale=24, ef=16, a=0.57, rcm=False, k=64, parents=True),
        # A batch on a renumbered graph (Cuthill-McKee order, pull rows by
        # degree), depths alone: how a graph that is kept is searched.
        dict(name="batch-rmat22-rcm", op="batch", kind="rmat", scale=22, ef=16, a=0.57, rcm=True, k=64, parents=False),
        # A batch that fills half the lanes on a long-diameter graph of
        # ragged sides.
        dict(name="batch-grid2048", op="batch", kind="grid", width=2048, height=1531, p_del=0.1, rcm=False, k=32,
             parents=True),
        # A serving batch: 256 queries over graphs of scales 16 to 22, one call.
        dict(name="mixed-256", op="mixed", lo=16, hi=22, ef=16, a=0.57, queries=256, parents=True),
        # Components of a graph with hubs and many small components, and of
        # one with a long diameter.
        dict(name="components-rmat22", op="components", kind="rmat", scale=22, ef=16, a=0.57),
        dict(name="components-grid4096", op="components", kind="grid", width=4096, height=4096, p_del=0.1),
        # What every new graph costs first: 67 million edges on the device to
        # a symmetric, deduplicated CSR.
        dict(name="build-rmat22", op="build", kind="rmat", scale=22, ef=16, a=0.57),
        # One optimiser step of the direction policy on the training set's
        # 200,000 resampled levels.
        dict(name="train-200k", op="train", rows=200000, objective="regress"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_graph(rng, top):
    """A graph of up to about 2**top vertices (RMAT, ER) or as many grid cells."""
    kind = rng.choice(["rmat", "er", "grid"])
    if kind == "rmat":
        return dict(kind="rmat", scale=rng.randint(14, top), ef=rng.choice([8, 16, 32]) if top <= 22 else 16,
                    a=round(rng.uniform(0.45, 0.65), 3))
    if kind == "er":
        return dict(kind="er", n=_log_int(rng, 1 << 14, 1 << top), deg=rng.randint(6, 32), directed=rng.random() < 0.25)
    side = 1 << (top // 2 + 1)
    return dict(kind="grid", width=_log_int(rng, 200, side), height=_log_int(rng, 200, side),
                p_del=round(rng.uniform(0.0, 0.2), 3))


def draw(rng):
    op = rng.choice(["search", "search", "search", "batch", "batch", "mixed", "components", "build", "train"])
    if op == "search":
        c = dict(op=op, **_draw_graph(rng, 22), parents=rng.random() < 0.7)
        # a grid search takes thousands of levels: few sources
        c["k"] = rng.randint(1, 2) if c["kind"] == "grid" else _log_int(rng, 1, 64)
        return c
    if op == "batch":
        g = _draw_graph(rng, 22)
        rcm = g["kind"] == "rmat" and rng.random() < 0.3
        c = dict(op=op, **g, rcm=rcm, parents=rng.random() < 0.7)
        c["k"] = _log_int(rng, 2, 64 if c["kind"] == "grid" else 128)
        return c
    if op == "mixed":
        lo = rng.randint(12, 18)
        return dict(op=op, lo=lo, hi=rng.randint(lo + 1, 22), ef=16, a=round(rng.uniform(0.45, 0.65), 3),
                    queries=_log_int(rng, 16, 256), parents=rng.random() < 0.7)
    if op == "train":
        return dict(op=op, rows=_log_int(rng, 1000, 200000), objective=rng.choice(["regress", "ce"]))
    g = _draw_graph(rng, 22)
    if op == "components" and g["kind"] == "er":  # components are those of an undirected graph
        g["directed"] = False
    return dict(op=op, **g)


# ------------------------------------------------------------------- inputs
def _rmat(scale, ef, a, gen):
    """src, dst of ef << scale tuples: `scale` independent quadrant draws each
    (d = 0.05 and b = c = (1 - a - d) / 2: 0.57, 0.19, 0.19, 0.05 at a = 0.57)."""
    m = ef << scale
    b = (1.0 - a - 0.05) / 2
    src = torch.zeros(m, dtype=torch.int32, device=DEV)
    dst = torch.zeros(m, dtype=torch.int32, device=DEV)
    r = torch.empty(m, dtype=torch.float32, device=DEV)
    for _ in range(scale):
        r.uniform_(generator=gen)
        down = r >= a + b
        right = torch.where(down, r >= a + 2 * b, r >= a)
        src.mul_(2).add_(down)
        dst.mul_(2).add_(right)
    return 1 << scale, src, dst


def _er(n, deg, gen):
    m = max(1, n * deg // 2)
    return (n, torch.randint(n, (m,), generator=gen, device=DEV, dtype=torch.int32),
            torch.randint(n, (m,), generator=gen, device=DEV, dtype=torch.int32))


def _grid(width, height, p_del, gen):
    n = width * height
    perm = torch.randperm(n, generator=gen, device=DEV).to(torch.int32).view(height, width)
    right = torch.rand((height, width - 1), generator=gen, device=DEV) >= p_del
    down = torch.rand((height - 1, width), generator=gen, device=DEV) >= p_del
    src = torch.cat([perm[:, :-1][right], perm[:-1, :][down]])
    dst = torch.cat([perm[:, 1:][right], perm[1:, :][down]])
    return n, src, dst


def _edges(case, gen):
    if case["kind"] == "rmat":
        return _rmat(case["scale"], case["ef"], case["a"], gen)
    if case["kind"] == "er":
        return _er(case["n"], case["deg"], gen)
    return _grid(case["width"], case["height"], case["p_del"], gen)


def _flags(case):
    f = bg.BFS_DEFAULT_FLAGS
    if case.get("directed"):
        f &= ~bg.BFS_SYMMETRIZE
    if case.get("rcm"):
        f |= bg.BFS_REORDER_RCM | bg.BFS_PULL_HUBS_FIRST
    return f


def _sources(n, src, dst, k, gen):
    has = torch.zeros(n, dtype=torch.bool, device=DEV)
    keep = src != dst
    has[src[keep].long()] = True
    has[dst[keep].long()] = True
    cand = torch.nonzero(has).view(-1)
    pick = torch.randint(cand.numel(), (k,), generator=gen, device=DEV)
    return cand[pick].to(torch.int32).cpu().numpy()


def _policy_inputs(case, seed):
    """Weights as a fresh network has them (He), features with the spread of
    profiled levels, targets -log(T_c / T_min): at most 0, one of them 0."""
    rng = np.random.default_rng(seed)
    w = np.zeros(bg.BFS_MLP_NPARAM + bg.BFS_MLP_NNORM, np.float32)
    i, h, o = bg.BFS_MLP_IN, bg.BFS_MLP_HIDDEN, bg.BFS_MLP_OUT
    at = 0
    for rows, cols in ((h, i), (h, h), (o, h)):
        w[at:at + rows * cols] = rng.normal(0, math.sqrt(2.0 / cols), rows * cols)
        at += rows * cols + rows
    mean, std = rng.normal(0, 2, i).astype(np.float32), rng.uniform(0.5, 3, i).astype(np.float32)
    w[at:at + i], w[at + i:] = mean, 1.0 / std
    gen = torch.Generator(device=DEV).manual_seed(seed)
    X = torch.randn((case["rows"], i), generator=gen, device=DEV)
    X = (X * torch.from_numpy(std).to(DEV) + torch.from_numpy(mean).to(DEV)).contiguous()
    if case["objective"] == "ce":
        y = torch.randint(o, (case["rows"],), generator=gen, device=DEV, dtype=torch.int32)
    else:
        y = torch.rand((case["rows"], o), generator=gen, device=DEV).add_(1e-3).log_()
        y = (y - y.max(1, keepdim=True).values).contiguous()
    return w, X, y


LEARNING_RATE = 1e-3


def prepare(case, seed):
    op = case["op"]
    if op == "train":
        w, X, y = _policy_inputs(case, seed)
        return dict(op=op, policy=bg.Policy(w), X=X, y=y, rows=case["rows"], step=0, objective=case["objective"],
                    grad=torch.zeros(bg.BFS_MLP_NPARAM, device=DEV))
    gen = torch.Generator(device=DEV).manual_seed(seed)
    if op == "mixed":
        graphs, goq, srcs = [], [], []
        which = np.arange(case["queries"]) % (case["hi"] - case["lo"] + 1)  # as many queries on every graph
        for i, scale in enumerate(range(case["lo"], case["hi"] + 1)):
            n, s, d = _rmat(scale, case["ef"], case["a"], gen)
            graphs.append(bg.Graph.build(n, s, d))
            k = int((which == i).sum())
            goq += [i] * k
            srcs.append(_sources(n, s, d, k, gen))
            del s, d
        order = np.random.default_rng(case["queries"]).permutation(case["queries"])  # in no order
        goq, srcs = np.array(goq, np.int32)[order], np.concatenate(srcs)[order]
        sizes = [1 << (case["lo"] + int(i)) for i in goq]
        depth = torch.empty(sum(sizes), dtype=torch.int32, device=DEV)
        parent = torch.empty_like(depth) if case["parents"] else None
        return dict(op=op, graphs=graphs, goq=goq, srcs=srcs, depth=depth, depths=list(depth.split(sizes)),
                    parents=list(parent.split(sizes)) if parent is not None else None)
    n, s, d = _edges(case, gen)
    if op == "build":
        m = s.numel() * (1 if case.get("directed") else 2)
        return dict(op=op, n=n, src=s, dst=d, flags=_flags(case), csc=bool(case.get("directed")),
                    row_ptr=torch.empty(n + 1, dtype=torch.int32, device=DEV),
                    col=torch.full((m,), -1, dtype=torch.int32, device=DEV))  # room for a graph without repeats
    g = bg.Graph.build(n, s, d, flags=_flags(case))
    if op == "components":
        return dict(op=op, g=g, label=torch.empty(n, dtype=torch.int32, device=DEV))
    k = case["k"]
    srcs = _sources(n, s, d, k, gen)
    if case.get("rcm"):
        srcs = g.permutation()[srcs]
    depth = torch.empty((k, n), dtype=torch.int32, device=DEV)
    parent = torch.empty_like(depth) if case["parents"] else None
    return dict(op=op, g=g, srcs=srcs, depth=depth, parent=parent, opt=bg.options(batch=1 if op == "batch" else 0))


# --------------------------------------------------------------------- pass
def run(state):
    op = state["op"]
    if op in ("search", "batch"):
        state["g"].run(state["srcs"], state["depth"], state["parent"], state["opt"])
        return {"depth": state["depth"]}
    if op == "mixed":
        bg.run_mixed(state["graphs"], state["goq"], state["srcs"], state["depths"], state["parents"])
        return {"depth": state["depth"]}
    if op == "components":
        label, _ = state["g"].components(state["label"])
        return {"label": label}
    if op == "train":
        state["step"] += 1
        p = state["policy"]
        step = p.train_step_regress if state["objective"] == "regress" else p.train_step
        loss = step(state["X"], state["y"], state["rows"], LEARNING_RATE, state["step"], grad_out=state["grad"])
        return {"loss": loss, "grad": state["grad"]}
    # a new graph, read out into the caller's arrays, and freed (a graph
    # that is searched stays; a program that sweeps over graphs frees it)
    g = bg.Graph.build(state["n"], state["src"], state["dst"], flags=state["flags"])
    info = g.info()
    stream = torch.cuda.current_stream().cuda_stream
    if bg.load().bfs_graph_csr(g.handle, int(state["csc"]), state["row_ptr"].data_ptr(), state["col"].data_ptr(),
                               stream) != bg.BFS_OK:
        raise RuntimeError(bg.load().bfs_last_error().decode())
    out = {"row_ptr": state["row_ptr"], "col": state["col"], "m": int(info.m),
           "isolated": int(info.n_isolated), "deg_max": int(info.deg_max)}
    g.free()
    return out


# ---------------------------------------------------------------- the floor
def _size(case):
    """(vertices, directed entries before duplicates go) of the case's graph."""
    if case["kind"] == "rmat":
        return 1 << case["scale"], 2 * (case["ef"] << case["scale"])
    if case["kind"] == "er":
        m = max(1, case["n"] * case["deg"] // 2)
        return case["n"], m if case.get("directed") else 2 * m
    w, h = case["width"], case["height"]
    return w * h, int(2 * (1.0 - case["p_del"]) * (w * (h - 1) + h * (w - 1)))


def work(case):
    """Bytes: each input read once, each output written once.  Searches are
    counted as if one reading of the graph could serve all of a pass's."""
    op = case["op"]
    if op == "train":
        i, h, o = bg.BFS_MLP_IN, bg.BFS_MLP_HIDDEN, bg.BFS_MLP_OUT
        macs = i * h + h * h + h * o  # forward; the backward pass has twice as many, less the input gradient
        y = 4 if case["objective"] == "ce" else 4 * o
        return {"bytes": case["rows"] * (4 * i + y) + 4 * 5 * bg.BFS_MLP_NPARAM,
                "flops": 2.0 * case["rows"] * (3 * macs - i * h)}
    if op == "mixed":
        q = case["queries"] / (case["hi"] - case["lo"] + 1)
        total = 0.0
        for scale in range(case["lo"], case["hi"] + 1):
            n = 1 << scale
            total += q * n * (8 if case["parents"] else 4) + 4 * n + 8 * case["ef"] * n
        return {"bytes": total, "flops": 0}
    n, m = _size(case)
    graph = 4 * (n + 1) + 4 * m
    if op == "build":
        edges = m if case.get("directed") else m // 2
        return {"bytes": 8 * edges + graph, "flops": 0}
    if op == "components":
        return {"bytes": graph + 4 * n, "flops": 0}
    return {"bytes": graph + case["k"] * n * (8 if case["parents"] else 4), "flops": 0}


# ------------------------------------------------------------------ 64 bits
def exact(case, seed):
    """The training step's loss and gradient in 64 bits; depths, labels and
    CSR entries are whole numbers."""
    if case["op"] != "train":
        return None
    w, X, y = _policy_inputs(case, seed)
    i, h, o = bg.BFS_MLP_IN, bg.BFS_MLP_HIDDEN, bg.BFS_MLP_OUT
    t = torch.from_numpy(w).to(DEV).double()
    params, norm = t[:bg.BFS_MLP_NPARAM].clone().requires_grad_(True), t[bg.BFS_MLP_NPARAM:]
    shapes = ((h, i), (h,), (h, h), (h,), (o, h), (o,))
    parts = [p.view(s) for p, s in zip(params.split([math.prod(s) for s in shapes]), shapes)]
    x = (X.double() - norm[:i]) * norm[i:]
    z = torch.relu(torch.relu(x @ parts[0].T + parts[1]) @ parts[2].T + parts[3]) @ parts[4].T + parts[5]
    if case["objective"] == "ce":
        loss = torch.nn.functional.cross_entropy(z, y.long())
    else:
        loss = (z - y.double()).square().sum() / 2 / case["rows"]
    loss.backward()
    return {"loss": loss.detach(), "grad": params.grad}
