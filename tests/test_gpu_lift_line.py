"""The lifted 4D NUFFT's passes for boxes narrower than the period (row-pair spreading, z and y in one
launch, warp-private x lines, r transforms with the collapse and the inverse x) against the direct 4D
NDFT of the same shapes (contraction "cuda", FP32), over grids, lifted axes, section counts beyond one
pass, single and odd knot counts.  Bar 1e-5, the method's FP32 target that test_gpu_lift.py holds both
forms to against the FP64 oracle."""
import numpy as np
import pytest

from paper_1711_05075_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
L, P, PR = 0.1, 2.0, 0.4


@pytest.fixture(scope="module")
def bc():
    if not torch.cuda.is_available():
        pytest.skip("CUDA device required")
    torch.cuda.set_device(0)
    import paper_1711_05075_gb300 as m
    return m


def knots(shape, seed, lo=0.01, hi=0.09):
    r = lo + (hi - lo) * synth.SplitMix64(seed).uniform(shape.xyz.shape[0])
    return np.concatenate([shape.xyz, r[:, None]], axis=1).astype(np.float32)


@pytest.mark.parametrize("N,Nr,nA,nB,slices", [
    (32, 16, 1, 1, (0.0,)), (32, 64, 33, 7, (0.0, 0.01, -0.02, 0.03, 0.05)), (64, 16, 200, 1, (0.0, 0.02)),
    (64, 64, 51, 300, (0.0,)), (96, 32, 77, 100, (0.0, 0.02, -0.01)), (96, 64, 20, 21, (0.04,)),
    (128, 16, 40, 30, tuple(0.005 * i for i in range(9))), (128, 32, 100, 101, (0.0, -0.03)), (128, 64, 15, 60, (0.0,))])
def test_matches_direct_form(bc, N, Nr, nA, nB, slices):
    A, B = knots(synth.ellipsoid_shape(nA, 3 + N), 5), knots(synth.torus_shape(nB, 4 + Nr), 6)
    A[:, :3] += np.float32(0.11)  # the two boxes start at different cells
    q = synth.shoemake_quaternions(synth.SplitMix64(N + Nr), 1)[0]
    lf, ld = bc.Lift(N, Nr, L, P, PR, contraction="nufft"), bc.Lift(N, Nr, L, P, PR, contraction="cuda")
    got, ref = lf.correlate(A, B, q, slices), ld.correlate(A, B, q, slices)
    again = lf.correlate(A, B, q, slices[:1])
    for s in range(len(slices)):
        d, r = (got[s] - ref[s]).double().norm(), ref[s].double().norm()
        # a section with little overlap is held to the largest section's size
        scale = max(float(r), 0.05 * max(float(x.double().norm()) for x in ref))
        assert float(d) <= 1e-5 * scale, (s, float(d / r))
    assert float((again[0] - got[0]).double().norm() / got[0].double().norm()) <= 2e-6
    lf.close()
    ld.close()


# radii that wrap along the lifted axis, or centres across the period, take the whole axis (the
# general passes) and then the narrow passes again on the same handle
def test_whole_axis_and_back(bc):
    N, Nr = 64, 32
    lf, ld = bc.Lift(N, Nr, L, P, PR, contraction="nufft"), bc.Lift(N, Nr, L, P, PR, contraction="cuda")
    q = synth.shoemake_quaternions(synth.SplitMix64(8), 1)[0]
    wide = knots(synth.ellipsoid_shape(60, 1, semi=(0.99, 0.2, 0.99)), 2)
    narrow, B = knots(synth.ellipsoid_shape(50, 3), 4), knots(synth.torus_shape(40, 5), 6)
    for A in (narrow, wide, narrow):
        got, ref = lf.correlate(A, B, q), ld.correlate(A, B, q)
        assert float((got - ref).double().norm() / ref.double().norm()) <= 1e-5
    lf.close()
    ld.close()
