"""H at points inside the wire, where the field of the segment beside the point is scaled and that
of its neighbours on the same straight side is not: around the middle of a segment, a joint of two
segments, a corner and on the axis, for sides of one, few and many segments, some shorter than the
wire's radius. Reference: the oracle, segment by segment. Bounds: the stated 1e-10 of MTS_FP64;
1e-6 of the largest value for the FP32 basis of the others."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from paper_2503_18479_gb300 import workloads as W  # noqa: E402
from paper_2503_18479_gb300.simulator import Simulator  # noqa: E402

RW = 1e-3


def _square(segs, angle):
    c, s, h = np.cos(angle), np.sin(angle), .025
    q = np.array([[c * x - s * y, s * x + c * y, 0.] for x, y in ((-h, -h), (h, -h), (h, h), (-h, h))])
    v = np.concatenate([q[i] + (np.arange(segs) / segs)[:, None] * (q[(i + 1) % 4] - q[i]) for i in range(4)])
    return v[:, 0].copy(), v[:, 1].copy(), v[:, 2].copy()


def _points(loop, rng):
    """Points at 0 .. 1.2 wire radii around vertices and segment middles, and on the axis."""
    v = np.stack(loop, 1)
    base = np.concatenate([v, (v + np.roll(v, -1, 0)) / 2])
    base = np.concatenate([base, base + 1e-5 * rng.standard_normal(base.shape)])
    base = base[rng.permutation(len(base))[:150]]
    u = rng.standard_normal((len(base), 3))
    u *= (RW * rng.choice([.2, .5, .9, .999, 1.001, 1.2], len(base)) / np.linalg.norm(u, axis=1))[:, None]
    flat = u.copy()
    flat[:, 2] = 0
    return np.concatenate([base + u, base + flat, v[::max(1, len(v) // 8)]])


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-10), ("mixed", 1e-6), ("bf16", 1e-6)])
@pytest.mark.parametrize("segs", [1, 2, 16, 64])
@pytest.mark.parametrize("angle", [0., .3])
def test_inside_wire(segs, angle, precision, tol):
    rng = np.random.default_rng(int(segs + 10 * angle))
    loops = [_square(segs, angle), W.circular_loop(.01, 40, .1, 0.)]
    pts = np.concatenate([_points(l, rng) for l in loops])
    P, om = len(pts), np.array([4e8])
    off, vx, vy, vz = W.loops_to_arrays(loops)
    comp = rng.integers(0, 3, P).astype(np.int8)
    px, py, pz = (np.ascontiguousarray(pts[:, i]) for i in range(3))
    loss = np.arange(0, P, 7, dtype=np.int64)  # their rows have a kernel of their own
    st = W.Structure(off, vx, vy, vz, px, py, pz, np.full(2, .1), om, W.drive_uniform_field(loops, om), loss, pcomp=comp)
    wl = W.Workload("wire", [st], np.full((1, 2), 1e-10), RW, target=np.zeros(len(loss)))
    H = Simulator(wl, precision).export_basis()[0].cpu().numpy().reshape(P, 2)
    ref = np.asarray(oracle.basis(off, vx, vy, vz, px, py, pz, RW, comp=comp)).reshape(P, 2)
    assert np.abs(H - ref).max() <= tol * np.abs(ref).max()
