"""FP64 superposition at sizes that take the tensor-core form (digit products, one structure):
odd port, point and system counts, several K chunks, infinities and NaN, and results at the
bottom of the FP64 range. Reference: the FP64 product of the exported basis and the returned
currents. Bound per value, for two sums of N products each and the dropped digits: (N + 4) 2^-52
sum |H_k I_k| + N 2^-58 max|H| max|I| over 64-port chunks, plus the subnormal spacing."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from paper_2503_18479_gb300 import workloads as W  # noqa: E402
from paper_2503_18479_gb300.simulator import Simulator  # noqa: E402


def _sim(nx, ny, F, P, n_cfg, scale=1.0, bad=False, seed=3):
    rng = np.random.default_rng(seed)
    loops = W.square_array(nx, ny, seg_per_side=1)
    off, vx, vy, vz = W.loops_to_arrays(loops)
    om = 2 * np.pi * np.linspace(60e6, 68e6, F)
    pts = [rng.uniform(-0.2, 0.2, P), rng.uniform(-0.2, 0.2, P), rng.uniform(0.02, 0.04, P)]
    st = W.Structure(off, vx, vy, vz, *pts, np.full(nx * ny, 0.1), om,
                     scale * W.drive_uniform_field(loops, om), np.zeros(0, np.int64))
    C = rng.uniform(20e-12, 200e-12, size=(n_cfg, nx * ny))
    if bad:
        C[n_cfg // 2, 0] = np.nan
    return Simulator(W.Workload("fp64", [st], C, 1e-3), "fp64"), C


@pytest.mark.parametrize("nx,ny,F,P,n_cfg,scale,bad", [
    (5, 1, 1, 9001, 33, 1.0, False),
    (16, 1, 3, 2999, 41, 1.0, False),
    (9, 7, 1, 1153, 65, 1.0, False),    # odd rows: 8-byte loads
    (8, 8, 2, 1024, 48, 1.0, False),
    (8, 8, 1, 1281, 31, 1.0, True),     # a NaN configuration
    (8, 8, 1, 1281, 31, 1e-298, False), # subnormal fields
    (13, 5, 1, 1700, 33, 1.0, False),   # 65 ports: second chunk of one
    (12, 11, 1, 901, 40, 1.0, True),    # three chunks
])
def test_fp64_tensor_superposition(nx, ny, F, P, n_cfg, scale, bad):
    sim, C = _sim(nx, ny, F, P, n_cfg, scale, bad)
    N = nx * ny
    out = sim.forward(torch.from_numpy(C), want_I=True, want_loss=False,
                      B_out=torch.full((n_cfg, F * P), float("nan"), dtype=torch.complex128, device="cuda"))
    H = sim.export_basis()[0].cpu().numpy().reshape(P, N)
    I = out["I"].cpu().numpy().reshape(n_cfg * F, N)
    B = out["B"].cpu().numpy().reshape(n_cfg * F, P)
    ref = I.real @ H.T + 1j * (I.imag @ H.T)
    nan = np.isnan(I).any(axis=1)
    assert nan.sum() == (F if bad else 0)
    assert np.isnan(B[nan]).all() and np.isfinite(B[~nan]).all()
    top = sum(np.abs(H[:, k:k + 64]).max(1)[None] * np.abs(I[:, k:k + 64]).max(1)[:, None] for k in range(0, N, 64))
    for part in (np.real, np.imag):
        bound = (N + 4) * 2.0 ** -52 * (np.abs(part(I)) @ np.abs(H).T) + N * 2.0 ** -58 * top + N * 2.0 ** -1073
        assert (np.abs(part(B) - part(ref)) <= bound)[~nan].all()
