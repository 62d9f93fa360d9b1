"""Autograd entry points: a gradient of the loss alone runs no field adjoint (its launches are
those of the direct backward call), and equals the direct call bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from paper_2503_18479_gb300 import native as nv  # noqa: E402
from paper_2503_18479_gb300 import workloads as W  # noqa: E402
from paper_2503_18479_gb300.simulator import Simulator  # noqa: E402
from paper_2503_18479_gb300.sroute import SRoute  # noqa: E402


def _launches(fn):
    n0 = nv.mts_launch_count()
    out = fn()
    return nv.mts_launch_count() - n0, out


def test_loss_gradient_skips_the_field():
    wl = W.array_8x8(n_cfg=20, grid=9, planes=(0.02,))
    sim = Simulator(wl, "mixed")
    C = torch.from_numpy(wl.C).cuda().requires_grad_(True)
    B, loss = sim(C)
    n_auto, _ = _launches(lambda: loss.sum().backward())
    out = sim.forward(C.detach())
    n_direct, g = _launches(lambda: sim.backward(out["ev"], out["tape"], grad_loss=torch.ones_like(out["loss"])))
    assert n_auto == n_direct
    assert torch.equal(C.grad, g)


def test_sroute_loss_gradient_skips_the_field():
    sw = W.sroute_array(2, 2, n_cfg=5, grid=6, planes=(0.02,))
    sr = SRoute(sw.S0, sw.field, sw.rows, sw.cols, sw.n1, sc_const=sw.sc_const, loss_idx=sw.loss_idx,
                target=sw.target)
    rng = np.random.default_rng(0)
    sv = torch.from_numpy(0.5 * np.exp(1j * rng.uniform(-3, 3, (5, 1, 4)))).cuda().requires_grad_(True)
    B, loss = sr(sv)
    n_auto, _ = _launches(lambda: loss.sum().backward())
    out = sr.forward(sv.detach())
    n_direct, g = _launches(lambda: sr.backward(out, grad_loss=torch.ones_like(out["loss"])))
    assert n_auto == n_direct
    assert torch.equal(sv.grad, g)
