"""Rows of H at the loss points (MTS_MIXED): FP64 sums rounded once, for loops of fewer, as many and
more sides than the four threads that share one, more loops than a CTA takes at once, repeated
loss points and a second structure. Reference: the FP64 oracle; bound per value: one FP32 rounding
(2^-24 = 6e-8), and 1e-12 of the largest for values that cancel."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from paper_2503_18479_gb300 import workloads as W  # noqa: E402
from paper_2503_18479_gb300.simulator import Simulator  # noqa: E402


def _triangle(cx):
    return np.array([cx, cx + .04, cx + .01]), np.array([0., .01, .05]), np.zeros(3)


@pytest.mark.parametrize("loops", [
    lambda: [_triangle(0.)],
    lambda: W.square_array(3, 1, seg_per_side=16),
    lambda: [W.circular_loop(.025, 63, .055 * i) for i in range(7)],
    lambda: W.square_array(13, 5, seg_per_side=2),
], ids=["triangle", "squares", "circles", "65"])
def test_loss_rows(loops):
    rng = np.random.default_rng(3)
    sts, refs = [], []
    for lp in (loops(), W.square_array(2, 2, seg_per_side=4)):
        off, vx, vy, vz = W.loops_to_arrays(lp)
        N, om, P = len(lp), np.array([4e8]), 140
        pts = [rng.uniform(-.2, .2, P), rng.uniform(-.2, .2, P), rng.uniform(.01, .05, P)]
        li = np.array([0, 139, 77, 77, 5], np.int64)
        sts.append(W.Structure(off, vx, vy, vz, *pts, np.full(N, .1), om, W.drive_uniform_field(lp, om), li))
        refs.append(np.asarray(oracle.basis(off, vx, vy, vz, *pts, 1e-3)).reshape(P, N)[li])
    nports, nloss = sum(s.n_ports for s in sts), 10
    sim = Simulator(W.Workload("rows", sts, np.full((1, nports), 1e-10), 1e-3, target=np.zeros(nloss)), "mixed")
    H = sim.export_basis()[0].cpu().numpy()
    o = 0
    for s, ref in zip(sts, refs):
        got = H[o:o + s.n_points * s.n_ports].reshape(s.n_points, s.n_ports)[s.loss_idx]
        assert np.all(np.abs(got - ref) <= 2.0 ** -24 * np.abs(ref) + 1e-12 * np.abs(ref).max())
        o += s.n_points * s.n_ports
