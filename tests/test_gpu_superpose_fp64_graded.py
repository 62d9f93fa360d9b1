"""FP64 superposition of graded data at sizes that take the tensor-core form: ports that are nearly
open beside a driven one, points right above them, so that large values of H meet small currents.
Reference: the product of the exported basis and the returned currents in extended precision. Bound
per value: that of a plain FP64 sum, (N + 4) 2^-52 sum |H_k I_k|."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from paper_2503_18479_gb300 import workloads as W  # noqa: E402
from paper_2503_18479_gb300.simulator import Simulator  # noqa: E402


@pytest.mark.parametrize("nx,ny,F,P,n_cfg,grade", [
    (8, 8, 1, 1100, 48, 1.0),      # an ordinary array
    (8, 8, 1, 1100, 48, 1e4),
    (8, 8, 2, 1029, 25, 1e9),
    (9, 7, 1, 1100, 49, 1e14),     # odd rows
    (5, 1, 1, 9001, 33, 1e9),
    (13, 5, 1, 1700, 33, 1e9),     # 65 ports: a second chunk of one
    (12, 11, 1, 901, 40, 1e12),    # three chunks
])
def test_graded(nx, ny, F, P, n_cfg, grade):
    rng = np.random.default_rng(7)
    N = nx * ny
    loops = W.square_array(nx, ny, seg_per_side=1)
    off, vx, vy, vz = W.loops_to_arrays(loops)
    om = 2 * np.pi * np.linspace(60e6, 68e6, F)
    R = .1 * grade ** rng.uniform(0, 1, N)
    R[0] = .1
    V = np.zeros((F, N), complex)
    V[:, 0] = 1 + .3j  # one port is driven
    at = rng.integers(0, N, P)  # points around the wires of every loop
    pts = np.stack([np.array([vx, vy, vz])[:, off[at] + rng.integers(0, 4, P)]])[0].T + rng.normal(0, .004, (P, 3))
    pts[:, 2] = np.abs(pts[:, 2]) + .002
    px, py, pz = (np.ascontiguousarray(pts[:, i]) for i in range(3))
    st = W.Structure(off, vx, vy, vz, px, py, pz, R, om, V, np.zeros(0, np.int64))
    C = rng.uniform(20e-12, 200e-12, size=(n_cfg, N))
    sim = Simulator(W.Workload("graded", [st], C, 1e-3), "fp64")
    out = sim.forward(torch.from_numpy(C), want_I=True, want_loss=False)
    H = sim.export_basis()[0].cpu().numpy().reshape(P, N)
    I = out["I"].cpu().numpy().reshape(n_cfg * F, N)
    B = out["B"].cpu().numpy().reshape(n_cfg * F, P)
    assert np.isfinite(I).all()
    for part in (np.real, np.imag):
        i = part(I)
        ref = sum(np.multiply.outer(i[:, k].astype(np.longdouble), H[:, k]) for k in range(N))
        assert (np.abs(part(B) - ref) <= (N + 4) * 2.0 ** -52 * (np.abs(i) @ np.abs(H).T)).all()
