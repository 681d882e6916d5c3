"""The default FP32 passes for shapes inside one period (row-pair spreading, z and y in
one launch, warp-private x lines, inverse planes) against the general passes of the same
context (z_transform 0: separate radix passes), over window widths, level counts, grids,
batches, shapes near the period and unaligned outputs; one case against the FP64 oracle.

Both sides are FP32 evaluations of the same sums (the same window and tables), each
within 1e-6 of the exact result at every W (test_gpu_parity.py: 2e-7 to 7e-7 where the
window's own error is smaller), so they differ by at most the sum, 2e-6."""
import numpy as np
import pytest

import oracle as O
from paper_1711_05075_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
TOL = 2e-6


@pytest.fixture(scope="module")
def bc():
    if not torch.cuda.is_available():
        pytest.skip("CUDA device required")
    torch.cuda.set_device(0)
    import paper_1711_05075_gb300 as m
    return m


def radii_of(L):
    return tuple(0.02 + 0.01 * i for i in range(L))


def knots(n, seed, L, semi=(0.5, 0.35, 0.25)):
    S = synth.ellipsoid_shape(n, seed, radii_of(L), (1.0,) * L, semi)
    return S.xyz.astype(np.float32), S.level


def rel(a, b):
    return float((a - b).double().norm() / b.double().norm())


# every window width and level count; odd and single knots; L = 1 and 3 with caps of either parity
@pytest.mark.parametrize("N,W,L,nA,nB,k", [
    (32, 2, 1, 40, 1, 1), (32, 3, 3, 33, 70, 3), (32, 10, 8, 500, 77, 2), (64, 4, 2, 100, 999, 1), (64, 9, 1, 300, 41, 5),
    (64, 5, 3, 1, 1, 1), (96, 7, 1, 222, 111, 2), (96, 8, 4, 4000, 31, 3), (96, 9, 3, 50, 1000, 1), (128, 6, 1, 700, 64, 2),
    (128, 10, 2, 65, 3000, 1), (128, 8, 8, 1500, 1501, 1)])
def test_matches_general_passes(bc, N, W, L, nA, nB, k):
    ctx = bc.Context(N, W, radii_of(L))
    q = synth.shoemake_quaternions(synth.SplitMix64(N + W), k).astype(np.float32)
    A, B = ctx.shape(*knots(nA, 3, L)), ctx.shape(*knots(nB, 4, L, (0.4, 0.2, 0.3)))
    got = ctx.correlate(A, B, q).clone()
    again = ctx.correlate(A, B, q).clone()       # boxes were left clear
    peak, arg = ctx.sweep(A, B, q, batch=2)
    gs = ctx.score(A, B, q, 0.02, 2.0).clone()
    ctx.set_tuning(z_transform=0)
    ref = ctx.correlate(A, B, q).clone()
    rs = ctx.score(A, B, q, 0.02, 2.0).clone()
    ctx.sync()
    assert rel(got, ref) <= TOL and rel(again, ref) <= TOL, (rel(got, ref), rel(again, ref))
    # the score's levels carry weights of both signs: its rounding is that of the unweighted sums
    # (a few units of TOL after the cancellation of R11's terms)
    assert rel(gs, rs) <= 4 * TOL, rel(gs, rs)
    flat = ref.reshape(k, -1)
    top = flat.max(dim=1).values
    scale = flat.abs().max(dim=1).values
    assert bool(((peak - top).abs() <= 1e-5 * scale).all())
    assert bool(((flat.gather(1, arg.long()[:, None])[:, 0] - top).abs() <= 1e-5 * scale).all())
    ctx.close()


# the widest shape the passes take, one just beyond (general passes), and one across the period
@pytest.mark.parametrize("N", [32, 96, 128])
@pytest.mark.parametrize("reach", [0.80, 0.93, 0.99, 1.2])
def test_wide_shapes(bc, N, reach):
    ctx = bc.Context(N, 8, radii_of(2))
    A, B = ctx.shape(*knots(400, 5, 2, (reach, 0.3, 0.7 * reach))), ctx.shape(*knots(50, 6, 2))
    q = synth.shoemake_quaternions(synth.SplitMix64(9), 2).astype(np.float32)
    got = ctx.correlate(A, B, q).clone()
    peak, _ = ctx.sweep(A, B, q)
    mixed, _ = ctx.sweep(B, A, q)
    m = bc.moments(ctx, A).clone()
    ctx.set_tuning(z_transform=0)
    ref = ctx.correlate(A, B, q).clone()
    ref2 = ctx.correlate(B, A, q).clone()
    mr = bc.moments(ctx, A).clone()
    ctx.sync()
    assert rel(got, ref) <= TOL, rel(got, ref)
    for p, r in ((peak, ref), (mixed, ref2)):
        top = r.reshape(2, -1).max(dim=1).values
        assert bool(((p - top).abs() <= 1e-5 * top.abs()).all())
    assert rel(m, mr) <= 1e-5
    ctx.close()


# ragged pairs whose boxes have different sizes and parities, and an output on a 4-byte boundary
def test_ragged_pairs_and_unaligned_output(bc):
    ctx = bc.Context(64, 9, radii_of(1))
    As = [ctx.shape(*knots(n, 10 + n, 1, (0.2 + 0.03 * i, 0.3, 0.1))) for i, n in enumerate((1, 30, 501, 90))]
    Bs = [ctx.shape(*knots(n, 50 + n, 1, (0.1, 0.15 + 0.05 * i, 0.3))) for i, n in enumerate((700, 2, 17, 64))]
    q = synth.shoemake_quaternions(synth.SplitMix64(2), 4).astype(np.float32)
    grids, peak, arg = ctx.pairs(As, Bs, q, grids=True)
    raw = torch.empty(64 ** 3 + 1, dtype=torch.float32, device="cuda")
    bc.bc_correlate(ctx.handle, As[2].handle, Bs[2].handle, q[2:3], 1, raw[1:], 1)
    ctx.set_tuning(z_transform=0)
    ref, rpeak, _ = ctx.pairs(As, Bs, q, grids=True)
    ctx.sync()
    for i in range(4):
        assert rel(grids[i], ref[i]) <= TOL, (i, rel(grids[i], ref[i]))
    assert rel(raw[1:], ref[2].reshape(-1)) <= TOL
    assert bool(((peak - rpeak).abs() <= 1e-5 * rpeak.abs()).all())
    ctx.close()


def test_oracle(bc):
    N, L = 64, 3
    xa, la = knots(300, 21, L)
    xb, lb = knots(80, 22, L, (0.2, 0.4, 0.1))
    q = synth.shoemake_quaternions(synth.SplitMix64(1), 1).astype(np.float32)
    ctx = bc.Context(N, 9, radii_of(L))
    got = ctx.correlate(ctx.shape(xa, la), ctx.shape(xb, lb), q)[0].double().cpu().numpy()
    ctx.sync()
    ref = O.band_limited_corr(synth.Shape(xa.astype(np.float64), la, radii_of(L)),
                              synth.Shape(xb.astype(np.float64), lb, radii_of(L)), q[0].astype(np.float64), N, 2.0)
    assert float(np.linalg.norm(got - ref) / np.linalg.norm(ref)) <= 1e-5
    ctx.close()
