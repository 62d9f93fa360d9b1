"""Where MTS_MIXED takes its rows at the loss points from FP64 sums: up to 64 points of a structure, or
as many as its loops have sides (one rounding from the oracle); beyond that they are the rows that
the field has anyway, to the bit. Each structure of a batch counts for itself."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from paper_2503_18479_gb300 import workloads as W  # noqa: E402
from paper_2503_18479_gb300.simulator import Simulator  # noqa: E402


def _basis(parts):
    sts = []
    for loops, pts, idx in parts:
        off, vx, vy, vz = W.loops_to_arrays(loops)
        om = np.array([4e8])
        sts.append(W.Structure(off, vx, vy, vz, *pts, np.full(len(loops), .1), om,
                               W.drive_uniform_field(loops, om), idx))
    nports, nloss = sum(s.n_ports for s in sts), sum(len(s.loss_idx) for s in sts)
    wl = W.Workload("rows", sts, np.full((1, nports), 1e-10), 1e-3, target=np.zeros(nloss) if nloss else None)
    H, out, o = Simulator(wl, "mixed").export_basis()[0].cpu().numpy(), [], 0
    for s in sts:
        out.append(H[o:o + s.n_points * s.n_ports].reshape(s.n_points, s.n_ports))
        o += s.n_points * s.n_ports
    return out


def test_fp64_rows_up_to_the_sides():
    rng = np.random.default_rng(4)
    shapes = [W.square_array(4, 4, seg_per_side=4), W.square_array(4, 5, seg_per_side=1),
              [W.circular_loop(.025, 63, .055 * i) for i in range(3)], W.square_array(30, 9, seg_per_side=1)]
    sides = [64, 80, 189, 1080]
    parts = []
    for loops, n in zip(shapes, sides):
        P = n + 60
        pts = [rng.uniform(-.2, .4, P), rng.uniform(-.2, .4, P), rng.uniform(.01, .05, P)]
        parts.append((loops, pts, rng.permutation(P)[:n + 1]))  # one more than the sides
    most = [(l, p, i[:-1]) for l, p, i in parts]
    none = [(l, p, i[:0]) for l, p, i in parts]
    for plain, many, exact, (loops, pts, idx) in zip(_basis(none), _basis(parts), _basis(most), most):
        assert np.array_equal(many, plain)
        off, vx, vy, vz = W.loops_to_arrays(loops)
        ref = np.asarray(oracle.basis(off, vx, vy, vz, *pts, 1e-3)).reshape(plain.shape)
        d = np.abs(exact - ref)[idx]
        assert (d <= 2.0 ** -24 * np.abs(ref[idx]) + 1e-12 * np.abs(ref).max()).all()
