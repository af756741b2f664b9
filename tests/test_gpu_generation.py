"""A backward pass after another call on the same problem took the problem's tables: the gradient
is that of the forward pass's parameters, bit for bit."""
import numpy as np
import pytest

from paper_1801_10277_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("between", ["render", "hess", "fit", "elbo_grad"])
@pytest.mark.parametrize("prec", [0, 1])
def test_backward_after_another_call(prec, between):
    import torch
    from paper_1801_10277_gb300 import autograd
    from paper_1801_10277_gb300 import celeste as cel
    prob = synth.config(0)
    other = prob.theta.copy()
    other[:, 0:2] += 0.7
    other[:, synth.I_SCALE] *= 1.3
    P = cel.Problem(prob)
    want = P.elbo_grad(prob.theta, precision=prec)[2]
    theta = torch.from_numpy(prob.theta).cuda().requires_grad_(True)
    total = autograd.elbo(theta, P, prec)
    if between == "fit":
        P.fit(other, precision=prec, max_iter=1, max_sweeps=1, refine_fp64=0)
    elif between in ("hess", "elbo_grad"):
        getattr(P, between)(other, precision=1 - prec)
    else:
        getattr(P, between)(other)
    total.backward()
    np.testing.assert_array_equal(theta.grad.cpu().numpy(), want)
    P.close()
