"""SIMT superposition (few systems a structure): port counts at the edges of its K chunks and
vector forms, numbers of systems at the edges of its 4, 8 and 16, point counts beyond one unit of
tiles. Reference: H I of the exported basis and the returned currents in FP64; bound: the stated
1e-6 of MTS_MIXED on B."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from paper_2503_18479_gb300 import workloads as W  # noqa: E402
from paper_2503_18479_gb300.simulator import Simulator  # noqa: E402


@pytest.mark.parametrize("nx,ny,F,P,n_cfg", [
    (1, 1, 3, 130, 1), (4, 1, 4, 129, 1), (3, 2, 5, 513, 1), (4, 3, 8, 700, 1), (8, 8, 9, 515, 1),
    (17, 4, 16, 515, 1), (9, 8, 3, 1100, 5), (16, 8, 1, 515, 1), (16, 8, 16, 640, 1), (16, 9, 11, 200, 3),
])
def test_simt(nx, ny, F, P, n_cfg):
    N = nx * ny
    rng = np.random.default_rng(N + F)
    loops = W.square_array(nx, ny, seg_per_side=1)
    off, vx, vy, vz = W.loops_to_arrays(loops)
    om = 2 * np.pi * np.linspace(60e6, 68e6, F)
    pts = [rng.uniform(-0.3, 0.3, P), rng.uniform(-0.3, 0.3, P), rng.uniform(0.02, 0.04, P)]
    st = W.Structure(off, vx, vy, vz, *pts, np.full(N, 0.1), om, W.drive_uniform_field(loops, om),
                     np.zeros(0, np.int64))
    C = rng.uniform(20e-12, 200e-12, size=(n_cfg, N))
    sim = Simulator(W.Workload("simt", [st], C, 1e-3), "mixed")
    sim.tuning = dict(sim.tuning, simt_max_sys=1000)
    out = sim.forward(torch.from_numpy(C), want_I=True, want_loss=False,
                      B_out=torch.full((n_cfg, F * P), float("nan"), dtype=torch.complex64, device="cuda"))
    H = sim.export_basis()[0].reshape(P, N)
    I = out["I"].reshape(n_cfg * F, N)
    ref = torch.complex(I.real @ H.T, I.imag @ H.T).reshape(n_cfg, F * P)
    assert torch.linalg.norm(out["B"] - ref) <= 1e-6 * torch.linalg.norm(ref)
