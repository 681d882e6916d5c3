"""Creating a query: the modes and the records of the column kernel cost no more than the list of modes did."""
import time

import numpy as np
import pytest

from paper_1711_05075_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


# All 1,024,192 modes at N = 128: 14 ms on the GB300's host; with a comparison sort of the modes and a 21 MB
# list of places 88 ms (80 before there were records).  The oldest value is the bar.
def test_creation_of_a_query_of_all_modes():
    import paper_1711_05075_gb300 as bc
    A = synth.ellipsoid_shape(200, 3)
    ctx = bc.Context(128, 6, A.radii)
    a = ctx.shape(A.xyz.astype(np.float32), A.level)
    count, t = ((127 ** 3) + 1) // 2, []
    for _ in range(5):
        t0 = time.perf_counter()
        q = ctx.query(a, a, synth.IDENTITY_QUAT[0], count)
        t.append(time.perf_counter() - t0)
        q.close()
    ctx.close()
    assert sorted(t)[2] < 0.080, t
