"""Lifted correlations of many sections: one call takes no longer than the r transforms of one pass and the
sections' own work would, and both forms of the passes agree with the direct 4D NDFT on either side of the
rule that chooses between them.  Bar 1e-5 as in test_gpu_lift_line.py."""
import time

import numpy as np
import pytest

from paper_1711_05075_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
L, P, PR = 0.1, 2.0, 0.4


def knots(shape, seed):
    r = 0.01 + 0.08 * synth.SplitMix64(seed).uniform(shape.xyz.shape[0])
    return torch.tensor(np.concatenate([shape.xyz, r[:, None]], axis=1), dtype=torch.float32, device="cuda")


def seconds(lf, A, B, q, slices):
    for _ in range(3):
        lf.correlate(A, B, q, slices)
    t = []
    for _ in range(9):
        t0 = time.perf_counter()
        lf.correlate(A, B, q, slices)  # the call synchronises
        t.append(time.perf_counter() - t0)
    return sorted(t)[4]


# Four sections and sixteen on the same shapes.  Sixteen sections add the inverse transforms and sums of
# twelve more (1.1 to 1.3 times the call of four by the general passes); with the r transforms repeated for
# every four sections the call was 2.3, 2.5 and 2.6 times as long.
@pytest.mark.parametrize("N,Nr,semi", [(32, 64, 0.5), (64, 64, 0.12), (96, 64, 0.12)])
def test_many_sections_do_not_repeat_the_call(N, Nr, semi):
    import paper_1711_05075_gb300 as bc
    A = knots(synth.ellipsoid_shape(300, 1, semi=(semi, 0.8 * semi, 0.6 * semi)), 3)
    B = knots(synth.ellipsoid_shape(300, 2, semi=(semi, 0.8 * semi, 0.6 * semi)), 4)
    q = synth.shoemake_quaternions(synth.SplitMix64(1), 1)[0]
    lf = bc.Lift(N, Nr, L, P, PR)
    few, many = (seconds(lf, A, B, q, tuple(0.004 * i for i in range(n))) for n in (4, 16))
    lf.close()
    assert many <= 1.9 * few, (few, many)


@pytest.mark.parametrize("N,Nr,ns", [(32, 16, 12), (32, 16, 13), (32, 32, 4), (32, 32, 5), (32, 64, 1), (64, 64, 4), (64, 64, 5)])
@pytest.mark.parametrize("semi", [0.5, 0.12])
def test_both_sides_of_the_rule_match_the_direct_form(N, Nr, ns, semi):
    import paper_1711_05075_gb300 as bc
    A = knots(synth.ellipsoid_shape(60, 5, semi=(semi, 0.7 * semi, 0.5 * semi)), 6)
    B = knots(synth.torus_shape(50, 7), 8)
    q = synth.shoemake_quaternions(synth.SplitMix64(N + Nr), 1)[0]
    slices = tuple(0.003 * i for i in range(ns))
    lf, ld = bc.Lift(N, Nr, L, P, PR, contraction="nufft"), bc.Lift(N, Nr, L, P, PR, contraction="cuda")
    got, ref = lf.correlate(A, B, q, slices), ld.correlate(A, B, q, slices)
    top = max(float(x.double().norm()) for x in ref)
    for s in range(ns):
        d, r = float((got[s] - ref[s]).double().norm()), float(ref[s].double().norm())
        assert d <= 1e-5 * max(r, 0.05 * top), (s, d / r)
    lf.close()
    ld.close()
