"""Lifted shapes whose box takes a whole axis -- the lifted one alone, one spatial axis alone, all of them --
while the others stay narrow, in turn with narrow shapes on the same handle (the general passes and the line
passes share its workspace).  Against the direct 4D NDFT, bar 1e-5 as in test_gpu_lift_line.py."""
import numpy as np
import pytest

from paper_1711_05075_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
L, P, PR = 0.1, 2.0, 0.4


def knots(n, seed, ends=()):
    """Knots of a small ellipsoid, radii 0.03 to 0.07; per axis in `ends` two knots at the ends of its period."""
    x = synth.ellipsoid_shape(n, seed, semi=(0.3, 0.2, 0.25)).xyz
    k = np.concatenate([x, 0.03 + 0.04 * synth.SplitMix64(seed).uniform(n)[:, None]], axis=1).astype(np.float32)
    for i, a in enumerate(ends):
        k[2 * i, a], k[2 * i + 1, a] = (-0.99, 0.99) if a < 3 else (-0.195, 0.195)
    return k


@pytest.mark.parametrize("N,Nr", [(32, 16), (64, 32), (96, 16)])
@pytest.mark.parametrize("ends", [(3,), (0,), (1,), (2,), (0, 1, 2, 3)])
def test_one_whole_axis(N, Nr, ends):
    import paper_1711_05075_gb300 as bc
    lf, ld = bc.Lift(N, Nr, L, P, PR, contraction="nufft"), bc.Lift(N, Nr, L, P, PR, contraction="cuda")
    q = synth.shoemake_quaternions(synth.SplitMix64(8), 1)[0]
    small, whole, B = knots(50, 3), knots(60, 1, ends), knots(40, 5)
    for A, C in ((small, B), (whole, B), (small, whole), (small, B)):
        got, ref = lf.correlate(A, C, q), ld.correlate(A, C, q)
        assert float((got - ref).double().norm() / ref.double().norm()) <= 1e-5
    lf.close()
    ld.close()
