"""A wait of the x pass that expires in one warp only: the block's other warps do not wait for it at a
barrier, the kernel ends, the expiry is reported, and later passes on the context are right."""
import numpy as np
import pytest

from paper_1711_05075_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [32, 128])
def test_one_warps_expired_wait_is_reported_and_the_block_ends(N):
    import paper_1711_05075_gb300 as bc
    ctx = bc.Context(N, 6, synth.RADII_2)
    A, B = synth.ellipsoid_shape(90, 3), synth.torus_shape(70, 4)
    sa, sb = ctx.shape(A.xyz.astype(np.float32), A.level), ctx.shape(B.xyz.astype(np.float32), B.level)
    q = synth.shoemake_quaternions(synth.SplitMix64(7), 3).astype(np.float32)
    before = ctx.correlate(sa, sb, q).clone()
    ctx.sync()
    assert ctx.selftest_wait() == 4 and "x pass" in bc.lib().bc_last_error().decode()
    ctx.sync()  # the error word was cleared
    after = ctx.correlate(sa, sb, q)
    ctx.sync()
    # the spreading's float additions come in a run-dependent order
    assert float((after - before).double().norm() / before.double().norm()) <= 1e-6
    ctx.close()
