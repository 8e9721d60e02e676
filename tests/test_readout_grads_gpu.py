"""The read-out's gradients in a type of their own (single-precision
directions) are tensors of their own: one that is kept holds no other's
memory, starts where any tensor starts, and takes part in differentiable
operations in place."""
import pytest

import paper_2006_14927_gb300 as P
import workloads
from paper_2006_14927_gb300.autograd import telescope_readout
from parity import FP32, context, host_tracks

pytestmark = pytest.mark.gpu


def test_direction_gradients_share_nothing():
    import torch
    sc = workloads.adjoint_300gev(n=5001)
    ctx, tr = context(sc), host_tracks(sc, FP32)
    dev = P.device_tracks(tr, FP32, t_ref=sc["t_ref"])
    dirs = [dev[k].requires_grad_() for k in ("ux", "uy", "uz")]
    atm = sc["atm"]
    params = torch.tensor(atm["a"] + atm["b"] + atm["c"], dtype=torch.float64)
    D, T = telescope_readout(ctx, dev, params, atm, 3, FP32)
    grads = torch.autograd.grad(D.sum() + T.sum(), dirs)
    scale = torch.ones(5001, device="cuda", requires_grad=True)
    for g in grads:
        assert g.dtype == torch.float32 and float(g.abs().max()) > 0
        assert g.untyped_storage().nbytes() == 4 * 5001 and g.data_ptr() % 16 == 0
        g.mul_(scale)
