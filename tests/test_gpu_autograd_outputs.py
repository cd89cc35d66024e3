"""autograd.closure where the loss uses one of its two outputs: the other's gradient arrives as
None, the result is that of explicit zeros."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("used", ["coefficients", "moments", "both", "neither"])
def test_unused_outputs(used, prec):
    """The same kernels on the same numbers, so equal: a None stands for zeros."""
    from paper_2606_15622_gb300 import api, autograd
    rng = np.random.default_rng(1)
    counts = np.array([(3, 40, 61, 90)[c % 4] for c in range(200)])
    off = torch.from_numpy(np.concatenate([[0], np.cumsum(counts)]).astype(np.int64)).cuda()
    dtype = torch.float64 if prec == "fp64" else torch.float32
    v = torch.from_numpy(rng.standard_normal((3, int(off[-1])))).to(dtype).cuda().requires_grad_()
    tau = torch.linspace(0.5, 2.0, 200, dtype=torch.float64, device="cuda")
    p = api.default_params(min_particles=8)
    gY = torch.from_numpy(rng.standard_normal((200, 9))).cuda()
    gM = torch.from_numpy(rng.standard_normal((200, 30))).cuda()
    m, y, fl = autograd.closure(v, off, tau, prec=prec, params=p)
    if used == "neither":
        loss = 0.0 * y.sum()
        gY = torch.zeros_like(gY)
    else:
        loss = sum(x for x, on in (((gY * y).sum(), used != "moments"), ((gM * m).sum(), used != "coefficients")) if on)
    loss.backward()
    gY = gY if used != "moments" else torch.zeros_like(gY)
    gM = gM if used in ("moments", "both") else torch.zeros_like(gM)
    _, gv = api.fp_closure_backward(v.detach(), off, tau, m.detach(), y.detach(), fl, gY, grad_moments_in=gM, params=p,
                                    want_grad_moments=False)
    assert torch.equal(v.grad, gv)
    assert used == "neither" or (gv != 0).any()
