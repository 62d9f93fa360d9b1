"""Rows of the field that the tensor-core superposition writes: partial column tiles, one and
several structures, one and several frequencies, odd point counts, and the running-sum
epilogue (more than 256 ports). Reference: H I of the exported basis and the returned currents
in FP64; bound: the stated 1e-6 of MTS_MIXED on B."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from paper_2503_18479_gb300 import workloads as W  # noqa: E402
from paper_2503_18479_gb300.simulator import Simulator  # noqa: E402


def _structure(nx, ny, F, P, rng):
    loops = W.square_array(nx, ny, seg_per_side=1)
    off, vx, vy, vz = W.loops_to_arrays(loops)
    om = 2 * np.pi * np.linspace(60e6, 68e6, F)
    pts = [rng.uniform(-0.2, 0.2, P), rng.uniform(-0.2, 0.2, P), rng.uniform(0.02, 0.04, P)]
    return W.Structure(off, vx, vy, vz, *pts, np.full(nx * ny, 0.1), om,
                       W.drive_uniform_field(loops, om), np.zeros(0, np.int64))


@pytest.mark.parametrize("shapes,n_cfg", [
    ([(3, 2, 3, 131)], 43),                   # 129 systems: two full column tiles and one row
    ([(3, 2, 1, 128)], 64),                   # exactly one column tile
    ([(2, 1, 1, 257), (3, 3, 1, 40)], 65),    # two structures, one frequency: stride sumFP
    ([(2, 1, 5, 130), (8, 9, 2, 129), (1, 1, 64, 3)], 27),  # rows wrap inside and across tiles
    ([(18, 16, 2, 131)], 33),                 # running sum, one structure
    ([(18, 16, 3, 70), (2, 2, 2, 9)], 23),    # running sum, several structures
])
def test_rows(shapes, n_cfg):
    rng = np.random.default_rng(5)
    ss = [_structure(*sh, rng) for sh in shapes]
    C = rng.uniform(20e-12, 200e-12, size=(n_cfg, sum(s.n_ports for s in ss)))
    sim = Simulator(W.Workload("rows", ss, C, 1e-3), "mixed")
    sim.tuning = dict(sim.tuning, simt_max_sys=-1)
    out = sim.forward(torch.from_numpy(C), want_I=True, want_loss=False,
                      B_out=torch.full((n_cfg, sim.sumFP), float("nan"), dtype=torch.complex64, device="cuda"))
    H, _ = sim.export_basis()
    H, I, B = H.cpu().numpy(), out["I"].cpu().numpy(), out["B"].cpu().numpy()
    ho = io = bo = 0
    for s in ss:
        N, P, F = s.n_ports, s.n_points, s.n_freq
        Hs = H[ho:ho + P * N].reshape(P, N)
        Is = I[:, io:io + F * N].reshape(n_cfg, F, N)
        ref = np.einsum("pk,bfk->bfp", Hs, Is)
        got = B[:, bo:bo + F * P].reshape(n_cfg, F, P)
        assert np.linalg.norm(got - ref) <= 1e-6 * np.linalg.norm(ref)
        ho, io, bo = ho + P * N, io + F * N, bo + F * P
