"""H and M on whole straight sides against the oracle, which sums over segments: loops whose
segments merge (any rotation, any first vertex, uneven and long subdivisions, repeated
vertices), and oblique pairs too close for the panels of one side (a vertex touching the inside
of another loop's side). Bounds: the stated 1e-10 of MTS_FP64 and 1e-6 of MTS_MIXED."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from paper_2503_18479_gb300 import workloads as W  # noqa: E402
from paper_2503_18479_gb300.simulator import Simulator  # noqa: E402


def _polygon(corners, segs, roll=0):
    """Closed polygon whose side q is cut at the fractions segs[q] (int: evenly)."""
    out = []
    for q, c in enumerate(corners):
        d = np.asarray(corners[(q + 1) % len(corners)]) - c
        cut = np.arange(segs[q]) / segs[q] if np.isscalar(segs[q]) else np.asarray(segs[q])
        out += [c + f * d for f in cut]
    v = np.roll(np.array(out), -roll, axis=0)
    return v[:, 0].copy(), v[:, 1].copy(), v[:, 2].copy()


def _square(cx, cy, side, angle, z=0.0):
    c, s, h = np.cos(angle), np.sin(angle), side / 2
    return [np.array([cx + c * x - s * y, cy + s * x + c * y, z])
            for x, y in ((-h, -h), (h, -h), (h, h), (-h, h))]


def _touching():
    a = _square(0.0, 0.0, 0.05, 0.0)
    mid = np.array([0.025, 0.0125, 0.0])  # a vertex inside the right side when it has 4 segments
    b = [mid, mid + [0.04, -0.02, 0.0], mid + [0.045, 0.03, 0.0]]
    return [_polygon(a, [4] * 4), _polygon(b, [3, 5, 2])]


CASES = {
    "axis": lambda: W.square_array(3, 2, seg_per_side=16),
    "rolled": lambda: [_polygon(_square(0, 0, .05, 0), [16] * 4, roll=5), _polygon(_square(.055, 0, .05, 0), [16] * 4, roll=63)],
    "rotated": lambda: [_polygon(_square(0, 0, .05, .3), [16] * 4, 3), _polygon(_square(.06, .01, .05, .9), [7] * 4)],
    "uneven": lambda: [_polygon(_square(0, 0, .05, .0), [[0, .1, .7], 1, [0, .5, .5, .9], 70], 2), _polygon(_square(.06, 0, .05, 0), [150, 1, 64, 65])],
    "near": lambda: [_polygon(_square(0, 0, .05, 0), [16] * 4), _polygon(_square(.0253 + .05 * 2 ** -.5, 0, .05, np.pi / 4), [16] * 4)],
    "touching": _touching,
    "many": lambda: [W.circular_loop(.025, 40), _polygon(_square(.06, 0, .05, .2), [16] * 4), W.circular_loop(.02, 17, -.06, 0)],
}


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-10), ("mixed", 1e-6)])
@pytest.mark.parametrize("name", list(CASES))
def test_sides_against_segments(name, precision, tol):
    loops = CASES[name]()
    off, vx, vy, vz = W.loops_to_arrays(loops)
    rng = np.random.default_rng(1)
    pts = [rng.uniform(-.1, .1, 300), rng.uniform(-.1, .1, 300), rng.uniform(.0005, .05, 300)]
    pts[0][200:], pts[1][200:] = 50 * pts[0][200:], 50 * pts[1][200:]  # far points
    N, om = len(loops), np.array([4e8])
    st = W.Structure(off, vx, vy, vz, *pts, np.full(N, .1), om, W.drive_uniform_field(loops, om), np.zeros(0, np.int64))
    sim = Simulator(W.Workload("sides", [st], np.full((1, N), 1e-10), 1e-3), precision)
    H, M = (x.cpu().numpy() for x in sim.export_basis())
    Ho = oracle.basis(off, vx, vy, vz, *pts, 1e-3)
    status, Mo = oracle.inductance(off, vx, vy, vz, 1e-3, None)
    assert status == 0
    assert np.linalg.norm(M.reshape(N, N) - Mo) <= 1e-10 * np.linalg.norm(Mo)
    H, Ho = H.reshape(300, N), np.asarray(Ho).reshape(300, N)
    for sl in (slice(0, 200), slice(200, 300)):
        assert np.linalg.norm(H[sl] - Ho[sl]) <= tol * np.linalg.norm(Ho[sl])
