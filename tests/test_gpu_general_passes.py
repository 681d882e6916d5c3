"""The general passes -- k_spread, the tensor-core or radix z pass, k_fft_y, k_fft_x and three back-half
launches -- on shapes that reach across the period, which take them under the default tuning at N <= 128:
overlapped and ordinary launches, recorded graphs, repeated calls and switches to narrow shapes on one
context, against the FP64 oracle.  Bars as test_gpu_parity.py: rel-L2 1e-5 against the oracle, 1e-6 between
calls that differ only in the order of the spreading's float additions."""
import numpy as np
import pytest

import oracle as O
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


def across(seed, n=250):
    """A shape with knots on both sides of the period's edge."""
    A = synth.ellipsoid_shape(n, seed, synth.RADII_4, synth.PROBS_4, (0.6, 0.3, 0.4))
    A.xyz[0], A.xyz[1] = (-0.99, 0.1, 0.2), (0.99, -0.1, 0.1)
    return synth.Shape(A.xyz.astype(np.float32).astype(np.float64), A.level, A.radii)


def narrow(seed, n=200):
    B = synth.torus_shape(n, seed, synth.RADII_4, synth.PROBS_4)
    return synth.Shape(B.xyz.astype(np.float32).astype(np.float64), B.level, B.radii)


def rel(a, b):
    a, b = (np.asarray(x.double().cpu() if torch.is_tensor(x) else x) for x in (a, b))
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.fixture(scope="module")
def cases(bc):
    out = {}
    for N, W in ((32, 6), (96, 8), (128, 8)):
        A, B = across(3 + N), narrow(4 + N)
        q = synth.shoemake_quaternions(synth.SplitMix64(N), 2).astype(np.float32)
        out[N] = W, A, B, q, [O.band_limited_corr(A, B, q[r].astype(np.float64), N, 2.0) for r in range(2)]
    return out


@pytest.mark.parametrize("N", [32, 96, 128])
@pytest.mark.parametrize("zt", [1, 0])
def test_overlap_graphs_and_repeats(bc, cases, N, zt):
    W, A, B, q, refs = cases[N]
    ctx = bc.Context(N, W, synth.RADII_4)
    a, b = ctx.shape(A.xyz.astype(np.float32), A.level), ctx.shape(B.xyz.astype(np.float32), B.level)
    out = torch.empty((1, N, N, N), device="cuda")
    first = None
    for overlap in (1, 0):
        for graphs in (1, 0):
            ctx.set_tuning(z_transform=zt, persistent=0, overlap=overlap, graphs=graphs)
            for r in (0, 0, 0, 1, 1, 0):  # kernel by kernel, recorded, replayed; the rotation changes in between
                ctx.correlate(a, b, q[r:r + 1], out)
                ctx.sync()
                assert rel(out[0], refs[r]) <= 1e-5, (overlap, graphs, r, rel(out[0], refs[r]))
            first = out.clone() if first is None else first
            assert rel(out, first) <= 1e-6
    grids = ctx.correlate(a, b, q)  # A's spectrum through the cache, both rotations in one pass
    peak, _ = ctx.sweep(a, b, q)
    ctx.sync()
    for r in range(2):
        assert rel(grids[r], refs[r]) <= 1e-5
        assert abs(float(peak[r]) - refs[r].max()) <= 1e-5 * np.abs(refs[r]).max()
    ctx.close()


# the row-pair passes and the general ones share a context's workspaces: each has to leave them clear
def test_narrow_and_wide_in_turn(bc, cases):
    W, A, B, q, refs = cases[96]
    C = narrow(77)
    ref = O.band_limited_corr(C, B, q[0].astype(np.float64), 96, 2.0)
    ctx = bc.Context(96, W, synth.RADII_4)
    a, b, c = (ctx.shape(s.xyz.astype(np.float32), s.level) for s in (A, B, C))
    for _ in range(3):
        assert rel(ctx.correlate(a, b, q[:1])[0], refs[0]) <= 1e-5
        assert rel(ctx.correlate(c, b, q[:1])[0], ref) <= 1e-5
    # one wide shape in a batch of pairs: all of them take the general passes
    grids, _, _ = ctx.pairs([a, c], [b, b], np.concatenate([q[:1], q[:1]]), grids=True)
    ctx.sync()
    assert rel(grids[0], refs[0]) <= 1e-5 and rel(grids[1], ref) <= 1e-5
    ctx.close()
