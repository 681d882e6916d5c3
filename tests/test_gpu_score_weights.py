"""Scores build only the form of the level weights that their passes read: every order of parameters, tuning
and shape size on one context gives what a context of its own gives."""
import numpy as np
import pytest

from paper_1711_05075_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def knots(semi, seed):
    A = synth.ellipsoid_shape(80, seed, synth.RADII_2, semi=semi)
    A.xyz[0], A.xyz[1] = (-semi[0], 0, 0), (semi[0], 0, 0)
    return A.xyz.astype(np.float32), A.level


@pytest.mark.parametrize("N", [32, 96])
def test_forms_follow_the_passes(N):
    import paper_1711_05075_gb300 as bc
    q = synth.shoemake_quaternions(synth.SplitMix64(3), 2).astype(np.float32)
    shapes = {"narrow": knots((0.4, 0.3, 0.2), 1), "wide": knots((0.99, 0.3, 0.2), 2)}
    b = knots((0.3, 0.2, 0.25), 3)

    def alone(shape, r0, lam, zt):
        ctx = bc.Context(N, 8, synth.RADII_2)
        ctx.set_tuning(z_transform=zt)
        out = ctx.score(ctx.shape(*shapes[shape]), ctx.shape(*b), q, r0, lam).clone()
        ctx.sync()
        ctx.close()
        return out

    ctx = bc.Context(N, 8, synth.RADII_2)
    S, B = {k: ctx.shape(*v) for k, v in shapes.items()}, ctx.shape(*b)
    for shape, r0, lam, zt in (("narrow", 0.02, 2.0, 1), ("wide", 0.02, 2.0, 1), ("narrow", 0.02, 2.0, 0), ("wide", 0.03, 2.0, 1),
                               ("narrow", 0.03, 2.0, 1), ("narrow", 0.03, 1.0, 1), ("narrow", 0.03, 1.0, 0), ("narrow", 0.02, 2.0, 1)):
        ctx.set_tuning(z_transform=zt)
        ref = alone(shape, r0, lam, zt)
        for _ in range(3):  # the second identical pass is recorded, the third replayed
            got = ctx.score(S[shape], B, q, r0, lam)
        peak, _ = ctx.score_sweep(S[shape], B, q, r0, lam)
        ctx.sync()
        scale = float(ref.double().norm())
        # same passes and weights; the spreading's float additions come in a run-dependent order
        assert float((got - ref).double().norm()) <= 2e-6 * scale, (shape, r0, lam, zt)
        top = ref.reshape(2, -1).max(dim=1).values
        assert bool(((peak - top).abs() <= 1e-5 * ref.abs().max()).all())
    ctx.close()
