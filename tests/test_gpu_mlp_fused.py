"""The fused forward pass (hidden <= 256) against the FP64 oracle with BF16 rounding emulated, at hidden
sizes around its K blocks of 64 and row counts around its tiles of 128; and against the layer-by-layer
products, which the gradients of a wider network still take.  Bars as test_gpu_mlp.py's: 1e-3 on the
outputs (FP32 accumulation of BF16 products), 1e-2 per gradient tensor."""
import numpy as np
import pytest

from oracle import mlp as M
from paper_1711_05075_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def bc():
    if not torch.cuda.is_available():
        pytest.skip("CUDA device required")
    torch.cuda.set_device(0)
    import paper_1711_05075_gb300 as m
    return m


def split(flat, H):
    o, out = 0, {}
    for k, shape in (("W1", (H, 132)), ("b1", (H,)), ("W2", (H, H)), ("b2", (H,)), ("w3", (H,)), ("b3", (1,))):
        size = int(np.prod(shape))
        out[k] = np.asarray(flat[o:o + size], dtype=np.float64).reshape(shape)
        o += size
    return out


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a) - np.asarray(b)) / max(np.linalg.norm(b), 1e-30))


@pytest.mark.parametrize("H,n", [(16, 1), (48, 129), (64, 127), (80, 128), (112, 257), (128, 5), (192, 300), (240, 1000),
                                 (256, 4097), (272, 130)])
def test_forward_and_gradients(bc, H, n):
    rng = np.random.default_rng(H + n)
    init = synth.mlp_init(H, H)
    init[H * 132:H * 133] = rng.normal(0, 0.3, H)       # biases of both layers
    init[-(2 * H + 1):-(H + 1)] = rng.normal(0, 0.3, H)
    X = np.zeros((n, 144), np.float32)
    X[:, :132] = rng.uniform(-1, 1, (n, 132))
    t = rng.normal(0, 1, n).astype(np.float32)
    ctx = bc.Context(32, 6, synth.RADII_2)
    net = bc.MLP(ctx, H, init)
    Xd = torch.tensor(X, device="cuda")
    y = net.predict(Xd).cpu().numpy()
    # rows on a 4-byte boundary only
    off = torch.empty(n * 144 + 1, device="cuda")
    off[1:] = Xd.reshape(-1)
    y2 = torch.empty(n, device="cuda")
    bc.bc_mlp_predict(net.handle, off[1:], n, y2)
    p = split(init, H)
    yo, _ = M.forward(p, X[:, :132].astype(np.float64), bf=True)
    assert rel(y, yo) < 1e-3 and np.array_equal(y, y2.cpu().numpy())
    g, loss = net.grads(Xd, torch.tensor(t, device="cuda"))
    lo, go = M.loss_and_grads(p, X[:, :132].astype(np.float64), t.astype(np.float64), bf=True)
    assert abs(float(loss.item()) - lo) <= 1e-4 * abs(lo)
    g = split(g.cpu().numpy(), H)
    for k in go:
        assert rel(g[k], go[k]) < 1e-2, (k, rel(g[k], go[k]))
    # the weights change: the pass follows
    net.train_step(Xd, torch.tensor(t, device="cuda"), 1e-2)
    y3 = net.predict(Xd).cpu().numpy()
    yo3, _ = M.forward(split(net.state()["params"], H), X[:, :132].astype(np.float64), bf=True)
    assert rel(y3, yo3) < 1e-3
    st = net.state()
    st["params"] = init
    net.load_state(st)
    assert np.array_equal(net.predict(Xd).cpu().numpy(), y)
    net.close()
    ctx.close()


# A recorded forward pass follows the weights, and a recorded Adam step leaves them usable by later calls.
@pytest.mark.parametrize("H", [48, 256])
def test_recorded_passes_follow_the_weights(bc, H):
    n, s = 200, torch.cuda.Stream()
    rng = np.random.default_rng(H)
    with torch.cuda.stream(s):
        X = torch.zeros((n, 144), device="cuda")
        X[:, :132] = torch.tensor(rng.uniform(-1, 1, (n, 132)), device="cuda")
        t = torch.tensor(rng.normal(0, 1, n).astype(np.float32), device="cuda")
        y = torch.empty(n, device="cuda")
        ctx = bc.Context(32, 6, synth.RADII_2, stream=s)
        net = bc.MLP(ctx, H, synth.mlp_init(H, H))
        net.train_step(X, t, 1e-2)  # buffers exist, the forward pass has run
        net.predict(X)
    s.synchronize()
    forward, step = torch.cuda.CUDAGraph(), torch.cuda.CUDAGraph()
    with torch.cuda.graph(forward, stream=s):
        bc.bc_mlp_predict(net.handle, X, n, y)
    with torch.cuda.graph(step, stream=s):
        net.train_step(X, t, 1e-2)
    Xh = X[:, :132].double().cpu().numpy()
    for _ in range(2):
        with torch.cuda.stream(s):
            step.replay()
            forward.replay()
            eager = net.predict(X)
        s.synchronize()
        yo, _ = M.forward(split(net.state()["params"], H), Xh, bf=True)
        assert rel(y.cpu().numpy(), yo) < 1e-3 and torch.equal(y, eager)
    net.close()
    ctx.close()
