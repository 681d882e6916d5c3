"""Single-configuration queries at many points (the column kernel) against the per-point kernel."""
import numpy as np
import pytest

from paper_1711_05075_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


# More points than one wave of the per-point kernel holds go to the column kernel
# (k_query_lines): the same points in one call against calls small enough for the
# per-point kernel.  Both are FP32 sums of the same terms from the same tables, each
# within 1e-6 of the exact value (the bars above), so they differ by at most 2e-6.
@pytest.mark.parametrize("N,mprime,npts", [(32, 1, 1300), (32, 7, 3001), (32, 14896, 1217), (64, 4096, 4097),
                                           (64, 125024, 2000), (128, 9000, 1500)])
def test_many_points_match_few(N, mprime, npts):
    import paper_1711_05075_gb300 as bc
    A, B = synth.ellipsoid_shape(200, 3), synth.torus_shape(150, 4)
    ctx = bc.Context(N, 6, A.radii)
    a, b = ctx.shape(A.xyz.astype(np.float32), A.level), ctx.shape(B.xyz.astype(np.float32), B.level)
    q = ctx.query(a, b, synth.shoemake_quaternions(synth.SplitMix64(5), 1)[0], mprime)
    t = torch.tensor(synth.SplitMix64(6).uniform(3 * npts).reshape(npts, 3) * 6 - 3, dtype=torch.float32, device="cuda")
    many = q.eval(t)
    few = torch.cat([q.eval(t[i:i + 500].contiguous()) for i in range(0, npts, 500)])
    ctx.sync()
    assert float((many - few).double().norm() / few.double().norm()) <= 2e-6
    ctx.close()
