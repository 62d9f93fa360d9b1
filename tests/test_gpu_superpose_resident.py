"""Superposition with the column tile resident in shared memory: port counts around the edges of
K chunks and of a tail chunk packed as one tile (at most 16 columns), the largest that stays
resident and the first that does not, with column tiles that change inside a CTA and partial
tiles on both sides. Reference: H I of the exported basis and the returned currents in FP64;
bound: the stated 1e-6 of MTS_MIXED on B, 1e-2 of MTS_BF16."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from paper_2503_18479_gb300 import workloads as W  # noqa: E402
from paper_2503_18479_gb300.simulator import Simulator  # noqa: E402


@pytest.mark.parametrize("precision,tol", [("mixed", 1e-6), ("bf16", 1e-2)])
@pytest.mark.parametrize("nx,ny,P,n_cfg", [
    (8, 8, 2563, 130),     # one chunk
    (13, 5, 130, 12801),   # 65: a tail of one column; two point tiles per column tile
    (10, 8, 2563, 130),    # 80: the widest packed tail
    (9, 9, 2563, 130),     # 81: the first that is not packed
    (16, 8, 2563, 130),    # 128: no tail
    (13, 10, 2563, 130),   # 130: two chunks and a packed tail
    (16, 12, 2563, 130),   # 192: the largest resident one in three pieces
    (15, 13, 2563, 130),   # 195: four chunks, streamed
    (32, 18, 131, 70),     # 576: nine tiles in one piece
])
def test_resident(nx, ny, P, n_cfg, precision, tol):
    rng = np.random.default_rng(nx * ny)
    loops = W.square_array(nx, ny, seg_per_side=1)
    off, vx, vy, vz = W.loops_to_arrays(loops)
    om = 2 * np.pi * np.array([63.6e6])
    pts = [rng.uniform(-0.3, 0.3, P), rng.uniform(-0.3, 0.3, P), rng.uniform(0.02, 0.04, P)]
    st = W.Structure(off, vx, vy, vz, *pts, np.full(nx * ny, 0.1), om, W.drive_uniform_field(loops, om),
                     np.zeros(0, np.int64))
    C = rng.uniform(20e-12, 200e-12, size=(n_cfg, nx * ny))
    sim = Simulator(W.Workload("resident", [st], C, 1e-3), precision)
    out = sim.forward(torch.from_numpy(C), want_I=True, want_loss=False,
                      B_out=torch.full((n_cfg, P), float("nan"), dtype=torch.complex64, device="cuda"))
    H = sim.export_basis()[0].reshape(P, nx * ny)
    I = out["I"].reshape(n_cfg, nx * ny)
    ref = torch.complex(I.real @ H.T, I.imag @ H.T)
    assert torch.linalg.norm(out["B"] - ref) <= tol * torch.linalg.norm(ref)
