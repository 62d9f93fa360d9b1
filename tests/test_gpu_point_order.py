"""A value of H depends on its point and loop alone: the same points in another order, alone, and
among others give the same bits (MTS_MIXED chooses a form by the point's distance)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from paper_2503_18479_gb300 import workloads as W  # noqa: E402
from paper_2503_18479_gb300.simulator import Simulator  # noqa: E402


def _basis(loops, pts, precision):
    off, vx, vy, vz = W.loops_to_arrays(loops)
    N, om = len(loops), np.array([4e8])
    px, py, pz = (np.ascontiguousarray(pts[:, i]) for i in range(3))
    st = W.Structure(off, vx, vy, vz, px, py, pz, np.full(N, .1), om, W.drive_uniform_field(loops, om), np.zeros(0, np.int64))
    return Simulator(W.Workload("order", [st], np.full((1, N), 1e-10), 1e-3), precision).export_basis()[0].cpu().numpy().reshape(-1, N)


@pytest.mark.parametrize("precision", ["mixed", "bf16", "fp64"])
def test_point_order(precision):
    rng = np.random.default_rng(0)
    loops = W.square_array(1, 1, seg_per_side=4) + [W.circular_loop(.034, 33)]
    # all around the distance where the form changes (three times that of the furthest vertex)
    pts = rng.standard_normal((1000, 3))
    pts *= (rng.uniform(.07, .15, 1000) / np.linalg.norm(pts, axis=1))[:, None]
    H = _basis(loops, pts, precision)
    order = rng.permutation(len(pts))
    assert np.array_equal(_basis(loops, pts[order], precision), H[order])
    for i in range(0, 1000, 111):
        assert np.array_equal(_basis(loops, pts[i:i + 1], precision)[0], H[i])
