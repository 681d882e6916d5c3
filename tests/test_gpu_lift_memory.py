"""A lifted handle takes the memory of the line passes' weight table only with the first call that reads it,
and a call for which there is no room is answered by the general passes."""
import numpy as np
import pytest

from paper_1711_05075_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
N, NR, L, P, PR = 96, 64, 0.1, 2.0, 0.4
TABLE = 8 * (N // 2) * (N // 2 + 1) * NR * (N // 2 + 1)  # 59 MB


def knots(shape, seed):
    r = 0.01 + 0.08 * synth.SplitMix64(seed).uniform(shape.xyz.shape[0])
    return torch.tensor(np.concatenate([shape.xyz, r[:, None]], axis=1), dtype=torch.float32, device="cuda")


def rel(a, b):
    return float((a - b).double().norm() / b.double().norm())


def free():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def test_weight_table_comes_with_the_first_call_that_reads_it_or_not_at_all():
    import paper_1711_05075_gb300 as bc
    q = synth.shoemake_quaternions(synth.SplitMix64(2), 1)[0]
    wide, narrow, B = (knots(s, i) for i, s in enumerate((synth.ellipsoid_shape(40, 1, semi=(0.99, 0.3, 0.2)),
                                                           synth.ellipsoid_shape(40, 2), synth.torus_shape(30, 3))))
    wide[0, 0], wide[1, 0] = -0.99, 0.99  # the box takes the whole x axis: the general passes
    ld = bc.Lift(N, NR, L, P, PR, contraction="cuda")
    ref = {k: ld.correlate(s, B, q).clone() for k, s in (("wide", wide), ("narrow", narrow))}
    ld.close()
    bc.Lift(N, NR, L, P, PR, contraction="nufft").close()  # modules and pools of the library
    before = free()
    lf = bc.Lift(N, NR, L, P, PR, contraction="nufft")
    assert before - free() < TABLE // 2
    assert rel(lf.correlate(wide, B, q), ref["wide"]) <= 1e-5  # the workspace exists from here on
    torch.cuda.empty_cache()
    out = torch.empty((1, N, N, N), device="cuda")
    sl = np.zeros(1, np.float32)
    hog = torch.empty(free() - TABLE // 2, dtype=torch.uint8, device="cuda")  # room for half of the table
    assert free() < TABLE
    bc.bc_lift_correlate(lf.handle, narrow, len(narrow), B, len(B), q.astype(np.float32), sl, 1, out, 1)
    assert rel(out, ref["narrow"]) <= 1e-5
    del hog
    torch.cuda.empty_cache()
    before = free()
    assert rel(lf.correlate(narrow, B, q), ref["narrow"]) <= 1e-5
    assert before - free() >= TABLE
    assert rel(lf.correlate(narrow, B, q), ref["narrow"]) <= 1e-5
    lf.close()
