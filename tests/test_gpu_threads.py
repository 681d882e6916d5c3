"""Contexts used from two threads at once, with shapes of different sizes: a pass whose shared memory
depends on the shapes must not fail because a call in the other thread needed less of it."""
import threading

import numpy as np
import pytest

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


def run_threads(bodies):
    errors, start = [], threading.Barrier(len(bodies))

    def guarded(body):
        try:
            start.wait()
            body()
        except Exception as e:  # reported by the test below
            errors.append(repr(e))

    ts = [threading.Thread(target=guarded, args=(b,)) for b in bodies]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not errors, errors[:2]


def rel(a, b):
    return float((a - b).double().norm() / b.double().norm())


# launched kernel by kernel, so that every call sets its kernels up anew
def test_correlations_of_wide_and_narrow_shapes(bc):
    N, jobs = 64, []
    for i, (reach, L) in enumerate(((0.85, 4), (0.5, 4), (0.85, 4), (0.6, 4), (0.99, 8), (0.99, 1))):  # the last two across the period
        radii = tuple(0.02 + 0.01 * k for k in range(L))
        A = synth.ellipsoid_shape(30, 3 + i, radii, (1.0,) * L, (reach, 0.7 * reach, 0.8 * reach))
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            ctx = bc.Context(N, 8, radii, stream=stream)
            ctx.set_tuning(graphs=0)
            a = ctx.shape(A.xyz.astype(np.float32), A.level)
            out = torch.empty((1, N, N, N), device="cuda")
            q = synth.shoemake_quaternions(synth.SplitMix64(i), 1).astype(np.float32)
            ctx.correlate(a, a, q, out)
            ctx.sync()
        jobs.append((ctx, a, q, out, out.clone()))
    torch.cuda.synchronize()

    def body(ctx, a, q, out, ref):
        def go():
            for _ in range(300):
                for _ in range(10):
                    ctx.correlate(a, a, q, out)
                ctx.sync()
        return go

    run_threads([body(*j) for j in jobs])
    for ctx, a, q, out, ref in jobs:
        assert rel(out, ref) <= 1e-6  # the spreading's float additions come in a run-dependent order
        ctx.close()


def test_queries_and_lifted_calls_of_different_sizes(bc):
    jobs = []
    for N, m in ((128, 300000), (128, 100000)):
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            A = synth.ellipsoid_shape(60, N)
            ctx = bc.Context(N, 6, A.radii, stream=stream)
            a = ctx.shape(A.xyz.astype(np.float32), A.level)
            q = ctx.query(a, a, synth.IDENTITY_QUAT[0], m)
            t = torch.rand((2000, 3), device="cuda")
            g = torch.empty(2000, device="cuda")
            bc.bc_query_eval(q.handle, t, 2000, g, 1)
            ctx.sync()
        jobs.append((ctx, q, t, g, g.clone()))
    lifts = []
    for hi, semi in ((0.09, 0.8), (0.02, 0.5)):
        A = synth.ellipsoid_shape(60, 9, semi=(semi, 0.5, 0.4))
        r = 0.01 + (hi - 0.01) * synth.SplitMix64(2).uniform(60)
        stream = torch.cuda.Stream()
        k = torch.tensor(np.concatenate([A.xyz, r[:, None]], axis=1), dtype=torch.float32, device="cuda")
        lf = bc.Lift(96, 32, 0.1, 2.0, 0.4, stream=stream)
        lifts.append((lf, k, lf.correlate(k, k, synth.IDENTITY_QUAT[0]).clone()))
    torch.cuda.synchronize()

    def query(ctx, q, t, g, ref):
        def go():
            for _ in range(1500):
                bc.bc_query_eval(q.handle, t, 2000, g, 1)
            ctx.sync()
        return go

    def lift(lf, k, ref):
        def go():
            for _ in range(60):
                out = lf.correlate(k, k, synth.IDENTITY_QUAT[0])
            assert rel(out, ref) <= 1e-5
        return go

    run_threads([query(*j) for j in jobs] + [lift(*l) for l in lifts])
    for ctx, q, t, g, ref in jobs:
        assert torch.equal(g, ref)
        ctx.close()
    for lf, _, _ in lifts:
        lf.close()
