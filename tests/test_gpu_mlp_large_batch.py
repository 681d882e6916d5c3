"""Gradients of more rows than the fused training pass takes (32,768) go through the layer-by-layer products:
just below and just above that count, and a small batch on the same network afterwards.  Bars as
test_gpu_mlp.py's: 1e-3 on outputs, 1e-2 per gradient tensor, against the FP64 oracle with BF16 emulated."""
import numpy as np
import pytest

from oracle import mlp as M
from paper_1711_05075_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def split(flat, H):
    o, out = 0, {}
    for k, shape in (("W1", (H, 132)), ("b1", (H,)), ("W2", (H, H)), ("b2", (H,)), ("w3", (H,)), ("b3", (1,))):
        size = int(np.prod(shape))
        out[k] = np.asarray(flat[o:o + size], dtype=np.float64).reshape(shape)
        o += size
    return out


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a) - np.asarray(b)) / max(np.linalg.norm(b), 1e-30))


@pytest.mark.parametrize("H", [16, 48])
def test_both_sides_of_the_row_limit(H):
    import paper_1711_05075_gb300 as bc
    rng = np.random.default_rng(H)
    init = synth.mlp_init(H, H)
    X = np.zeros((32770, 144), np.float32)
    X[:, :132] = rng.uniform(-1, 1, (32770, 132))
    t = rng.normal(0, 1, 32770).astype(np.float32)
    Xd, td = torch.tensor(X, device="cuda"), torch.tensor(t, device="cuda")
    ctx = bc.Context(32, 6, synth.RADII_2)
    net = bc.MLP(ctx, H, init)
    p = split(init, H)
    for n in (100, 32768, 32769, 32770, 130):
        g, loss = net.grads(Xd[:n].contiguous(), td[:n].contiguous())
        lo, go = M.loss_and_grads(p, X[:n, :132].astype(np.float64), t[:n].astype(np.float64), bf=True)
        assert abs(float(loss.item()) - lo) <= 1e-4 * abs(lo)
        g = split(g.cpu().numpy(), H)
        for k in go:
            assert rel(g[k], go[k]) < 1e-2, (n, k, rel(g[k], go[k]))
    # a training step of either kind leaves weights that the fused forward pass reads
    for n in (32769, 64):
        net.train_step(Xd[:n].contiguous(), td[:n].contiguous(), 1e-2)
        yo, _ = M.forward(split(net.state()["params"], H), X[:200, :132].astype(np.float64), bf=True)
        assert rel(net.predict(Xd[:200].contiguous()).cpu().numpy(), yo) < 1e-3
    net.close()
    ctx.close()
