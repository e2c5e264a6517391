"""The policy's training step and forward pass at the row counts where the
kernels' tiles end: a warp's 32 rows, a CTA's 128, one pass of all resident
CTAs and a little more.  Gradient and loss against the oracle in FP64; the
tolerances are those the repository states for them (1e-4 of the largest
gradient entry, 1e-5 for logits), and a second run on the same inputs must
give the same bits, since no sum depends on the order CTAs finish in.
"""
import numpy as np
import pytest

import oracle
import paper_2607_17106_gb300 as bg

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def _inputs(rows):
    rng = np.random.default_rng(rows)
    w = rng.normal(0, 0.3, bg.BFS_MLP_NPARAM + bg.BFS_MLP_NNORM).astype(np.float32)
    w[bg.BFS_MLP_NPARAM + 10:] = rng.uniform(0.5, 2.0, 10)
    X = rng.normal(0, 1.5, (rows, 10)).astype(np.float32)
    return w, X, rng.integers(0, 3, rows).astype(np.int32), -rng.exponential(1.0, (rows, 3)).astype(np.float32)


@pytest.mark.parametrize("rows", [1, 31, 32, 33, 127, 128, 129, 2 * 152 * 128 - 1, 2 * 152 * 128 + 33])
@pytest.mark.parametrize("objective", ["ce", "regress"])
def test_training_step_tile_edges(rows, objective):
    from paper_2607_17106_gb300 import build
    build.build()
    w, X, y, t = _inputs(rows)
    pad = torch.full((rows * 10 + 1,), float("nan"), device="cuda")  # inputs off a 16-byte boundary
    pad[1:] = torch.from_numpy(X).cuda().view(-1)
    Xd = pad[1:]
    target = torch.from_numpy(y if objective == "ce" else t).cuda()
    P = w[:bg.BFS_MLP_NPARAM].astype(np.float64)
    Xn = (X.astype(np.float64) - w[-20:-10]) * w[-10:]  # the oracle takes normalised features
    if objective == "ce":
        ref_loss, ref = oracle.mlp_loss_grad(P, Xn, y)
    else:
        ref_loss, ref = oracle.mlp_regress_loss_grad(P, Xn, t.astype(np.float64))
    got = []
    for _ in range(2):
        p = bg.Policy(w)
        g = torch.empty(bg.BFS_MLP_NPARAM, device="cuda")
        step = p.train_step if objective == "ce" else p.train_step_regress
        loss = step(Xd, target, rows, 1e-3, 1, grad_out=g)
        got.append((loss, g.cpu().numpy(), p.weights()))
    assert got[0][0] == got[1][0] and all(np.array_equal(a, b) for a, b in zip(got[0][1:], got[1][1:]))
    assert abs(got[0][0] - ref_loss) <= 1e-5 * max(1.0, abs(ref_loss))
    assert np.max(np.abs(got[0][1] - ref)) <= 1e-4 * np.max(np.abs(ref))
    logits = torch.full((rows + 1, 3), 7.0, device="cuda")
    p = bg.Policy(w)
    p.forward(Xd, logits, rows)
    z = oracle.mlp_forward(P, Xn)
    assert np.max(np.abs(logits[:rows].cpu().numpy() - z)) <= 1e-5 * np.max(np.abs(z))
    assert (logits[rows] == 7.0).all()
