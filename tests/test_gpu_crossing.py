"""M of loops in two planes whose sides cross at a distance, closest inside both sides: M12 itself
against the oracle, which sums over segments. Bound: the stated 1e-10 of MTS_FP64 (M is built in
FP64 for every precision)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from paper_2503_18479_gb300 import workloads as W  # noqa: E402
from paper_2503_18479_gb300.simulator import Simulator  # noqa: E402


def _square(side, angle, z, cuts):
    """Square loop turned by `angle`, each side cut at the fractions `cuts`."""
    c, s, h = np.cos(angle), np.sin(angle), side / 2
    q = np.array([[c * x - s * y, s * x + c * y, z] for x, y in ((-h, -h), (h, -h), (h, h), (-h, h))])
    v = np.concatenate([q[i] + np.asarray(cuts)[:, None] * (q[(i + 1) % 4] - q[i]) for i in range(4)])
    return v[:, 0].copy(), v[:, 1].copy(), v[:, 2].copy()


CUTS = {"2": np.arange(2) / 2, "16": np.arange(16) / 16, "64": np.arange(64) / 64,
        "uneven": np.concatenate([np.arange(12) / 64, np.arange(2, 11) / 10 - .01])}


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("cuts", list(CUTS))
@pytest.mark.parametrize("side", [.05, .2])
def test_crossing_sides(side, cuts, precision):
    for angle in (10, 30, 45):
        for gap in (.001, .002, .005):
            loops = [_square(side, .2, 0, CUTS[cuts]), _square(.98 * side, .2 + np.radians(angle), gap, CUTS["16"])]
            off, vx, vy, vz = W.loops_to_arrays(loops)
            om, pts = np.array([4e8]), [np.zeros(1), np.zeros(1), np.full(1, .02)]
            st = W.Structure(off, vx, vy, vz, *pts, np.full(2, .1), om, W.drive_uniform_field(loops, om), np.zeros(0, np.int64))
            M = Simulator(W.Workload("cross", [st], np.full((1, 2), 1e-10), 1e-3), precision).export_basis()[1].cpu().numpy()
            status, ref = oracle.inductance(off, vx, vy, vz, 1e-3, None)
            assert status == 0
            # (the reference evaluates [1, 0] with the roles of the loops exchanged, on other panels)
            assert np.abs(M.reshape(2, 2)[0] / ref[0] - 1).max() <= 1e-10, (angle, gap)
