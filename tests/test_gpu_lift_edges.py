"""Lifted correlations of knots on the edges of the fine grid's cells, where the first cell of a stencil turns on
the last bit of the knot's coordinate: the box search and the spreading of the 4D NUFFT have to agree on it.
Against the direct 4D NDFT, bar 1e-5 as in test_gpu_lift_line.py."""
import numpy as np
import pytest

from paper_1711_05075_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
L, P, PR = 0.1, 2.0, 0.4


def edge_knots(n, N, Nr, seed, span):
    """n knots whose coordinates are whole numbers of cells (rounded to float32), corners of the box among them."""
    g = np.random.default_rng(seed)
    k = g.integers(-span, span + 1, (n, 3))
    k[:2] = [[-span] * 3, [span] * 3]
    r = g.integers(1, max(2, int(0.24 * 2 * Nr)), n)
    return np.concatenate([k * (P / (2 * N)), (r * (PR / (2 * Nr)))[:, None]], axis=1).astype(np.float32)


QUATS = {"identity": (1, 0, 0, 0), "quarter turn": (0.5 ** 0.5, 0, 0, 0.5 ** 0.5), "third turn": (0.5, 0.5, 0.5, 0.5),
         "general": synth.shoemake_quaternions(synth.SplitMix64(5), 1)[0]}


@pytest.mark.parametrize("N,Nr", [(64, 32), (96, 16), (96, 32)])
@pytest.mark.parametrize("turn", list(QUATS))
def test_knots_on_cell_edges(N, Nr, turn):
    import paper_1711_05075_gb300 as bc
    A, B = edge_knots(300, N, Nr, 1, N // 4), edge_knots(200, N, Nr, 2, N // 3)
    lf, ld = bc.Lift(N, Nr, L, P, PR, contraction="nufft"), bc.Lift(N, Nr, L, P, PR, contraction="cuda")
    got, ref = lf.correlate(A, B, QUATS[turn]), ld.correlate(A, B, QUATS[turn])
    assert float((got - ref).double().norm() / ref.double().norm()) <= 1e-5
    lf.close()
    ld.close()
