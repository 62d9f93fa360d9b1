"""Panels of the blocked solve at the edges of its sizes: the last panel partly filled, a thread's
one or two rows just used up, CTAs too small for the panel in registers, trailing chunks of up
to 32, 64 and 128 columns. Reference: A I = V in FP64 with the exported M; bound: the stated 1e-6
of MTS_MIXED."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from paper_2503_18479_gb300 import workloads as W  # noqa: E402
from paper_2503_18479_gb300.simulator import Simulator  # noqa: E402


@pytest.mark.parametrize("nx,ny,threads", [
    (13, 5, 0), (73, 1, 0), (16, 5, 0), (97, 1, 0), (127, 1, 0), (16, 8, 0), (16, 8, 256), (16, 8, 512),
    (43, 3, 0), (17, 15, 0), (16, 16, 0), (257, 1, 0), (16, 16, 128), (23, 15, 128), (23, 15, 256),
    (27, 19, 0), (31, 33, 0), (32, 32, 0),
])
def test_currents(nx, ny, threads):
    N = nx * ny
    rng = np.random.default_rng(N)
    loops = W.square_array(nx, ny, seg_per_side=1)
    off, vx, vy, vz = W.loops_to_arrays(loops)
    om = 2 * np.pi * np.array([60e6, 66e6])
    pts = [rng.uniform(-0.3, 0.3, 3), rng.uniform(-0.3, 0.3, 3), rng.uniform(0.02, 0.04, 3)]
    V = W.drive_uniform_field(loops, om)
    st = W.Structure(off, vx, vy, vz, *pts, np.full(N, 0.1), om, V, np.zeros(0, np.int64))
    C = rng.uniform(20e-12, 200e-12, size=(2, N))
    sim = Simulator(W.Workload("sizes", [st], C, 1e-3), "mixed")
    sim.tuning = dict(sim.tuning, large_threads=threads)
    I = sim.forward(torch.from_numpy(C), want_I=True, want_loss=False)["I"].cpu().numpy().reshape(2, 2, N)
    M = sim.export_basis()[1].cpu().numpy().reshape(N, N)
    for b in range(2):
        for f in range(2):
            A = 1j * om[f] * M + np.diag(0.1 + 1 / (1j * om[f] * C[b]))
            ref = np.linalg.solve(A, np.asarray(V).reshape(2, N)[f])
            assert np.linalg.norm(I[b, f] - ref) <= 1e-6 * np.linalg.norm(ref)
