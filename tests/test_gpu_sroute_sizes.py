"""Scattering route at the edges of the eight-lane row sums and of the sweeps' 32-row slots: port
counts around multiples of 8 and 32 up to the limit of 96, several external ports, and loss
points beyond one staged chunk. Reference: the FP64 oracle; bound: 1e-6 (MTS_MIXED) and 1e-10
(MTS_FP64)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from helpers import rel  # noqa: E402
from paper_2503_18479_gb300.sroute import SRoute  # noqa: E402


@pytest.mark.parametrize("prec,tol", [("mixed", 1e-6), ("fp64", 1e-10)])
@pytest.mark.parametrize("n0,n1,L", [(1, 1, 3), (7, 2, 17), (8, 1, 64), (31, 1, 65), (32, 3, 33), (33, 1, 40),
                                     (63, 1, 130), (64, 2, 64), (65, 1, 65), (96, 1, 193), (95, 2, 97)])
def test_sizes(n0, n1, L, prec, tol):
    rng = np.random.default_rng(100 * n0 + n1)
    P, n, n_cfg, F = 200, n0 + n1, 3, 2

    def cn(*shape):
        return rng.standard_normal(shape) + 1j * rng.standard_normal(shape)

    S0, sc = cn(F, n0, n0) * (0.5 / np.sqrt(n0)), cn(F, n, n) * (0.2 / np.sqrt(n))
    field = cn(F, P, n0) * 1e-6
    pos = [(i, i) for i in range(n0)] + [(0, n0)] + ([(0, n0 - 1), (n0 - 1, n0 // 2)] if n0 > 6 else [])
    rows, cols = (np.array(x, np.int32) for x in zip(*pos))
    svar = rng.uniform(-0.8, 0.8, (n_cfg, F, len(pos))) + 1j * rng.uniform(-0.8, 0.8, (n_cfg, F, len(pos)))
    li = np.sort(rng.choice(P, size=L, replace=False)).astype(np.int64)
    t = np.abs(rng.standard_normal((F, n1, L))) * 1e-6
    sr = SRoute(S0, field, rows, cols, n1, sc_const=sc, loss_idx=li, target=t, precision=prec)
    out = sr.forward(torch.from_numpy(svar), want_B=True, want_W=True)
    g = sr.backward(out, grad_loss=torch.ones(n_cfg, dtype=torch.float64, device="cuda"))
    assert sr.status(out["tape"], n_cfg) == (0, 0)
    ref = oracle.sroute_pipeline(S0, field, sc, rows, cols, svar, li, t)
    for k in ("W", "B", "loss"):
        assert rel(out[k].cpu().numpy(), ref[k]) < tol, k
    assert rel(g.cpu().numpy(), oracle.sroute_gradient(S0, field, sc, rows, cols, svar, li, t)) < tol
