"""Superpositions whose tensor-core products share an accumulator give the same bits on every call:
the FP64 digit form, and the resident column tile with its two widths of product (2 and 3 K chunks,
a packed last chunk or not, one column tile and several). Against the FP64 product of basis and
currents: 1e-6 for MTS_MIXED and 1e-12 for MTS_FP64."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from paper_2503_18479_gb300 import workloads as W  # noqa: E402
from paper_2503_18479_gb300.simulator import Simulator  # noqa: E402


@pytest.mark.parametrize("nx,ny,P,n_cfg,precision", [
    (8, 8, 9000, 320, "fp64"),
    (13, 11, 4000, 100, "fp64"),
    (13, 5, 12000, 500, "mixed"),   # 65 ports: one full chunk, one packed
    (13, 10, 12000, 500, "mixed"),  # 130: two full, one packed
    (15, 10, 12000, 60, "mixed"),   # 150: three full
    (12, 16, 9000, 500, "mixed"),   # 192: three full
    (13, 8, 12000, 500, "mixed"),   # 104: two full
    (20, 10, 12000, 500, "bf16"),
])
def test_repeated_calls(nx, ny, P, n_cfg, precision):
    rng = np.random.default_rng(1)
    loops = W.square_array(nx, ny, seg_per_side=1)
    off, vx, vy, vz = W.loops_to_arrays(loops)
    N, om = nx * ny, np.array([4e8])
    pts = [rng.uniform(-.3, .3, P), rng.uniform(-.3, .3, P), rng.uniform(.02, .04, P)]
    st = W.Structure(off, vx, vy, vz, *pts, np.full(N, .1), om, W.drive_uniform_field(loops, om), np.zeros(0, np.int64))
    C = rng.uniform(20e-12, 200e-12, (n_cfg, N))
    sim = Simulator(W.Workload("order", [st], C, 1e-3), precision)
    Cg = torch.from_numpy(C).cuda()
    out = sim.forward(Cg, want_I=True, want_loss=False)
    first, I = out["B"].clone(), out["I"].cpu().numpy().reshape(n_cfg, N)
    H = sim.export_basis()[0].cpu().numpy().reshape(P, N)
    ref = I.real @ H.T + 1j * (I.imag @ H.T)
    tol = {"fp64": 1e-12, "mixed": 1e-6, "bf16": 1e-2}[precision]
    assert np.linalg.norm(first.cpu().numpy().reshape(n_cfg, P) - ref) <= tol * np.linalg.norm(ref)
    for _ in range(60):
        assert torch.equal(sim.forward(Cg, want_loss=False)["B"], first)
