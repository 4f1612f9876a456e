"""Constant gradients on a table of one column, with programs without constants
(which run through the evaluator) among the others."""
import numpy as np
import pytest

from paper_2110_11226_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_rows", [1, 130, 1027, 4096])
def test_gradient_of_one_column(n_rows):
    """Sums of positive terms of at most six roundings each: no cancellation."""
    import torch

    from paper_2110_11226_gb300 import gp
    O = synth.OP
    x, add, mul, absn = (O["var"], 0, 0.0), (O["add"], 0, 0.0), (O["mul"], 0, 0.0), (O["abs"], 0, 0.0)
    c = (O["const"], 0, 0.75)
    progs = [[x], [mul, x, x], [add, absn, x, absn, x], [c], [mul, c, x], [add, c, mul, x, x]]
    rng = np.random.default_rng(n_rows)
    X = torch.from_numpy(rng.uniform(1.0, 2.0, (1, n_rows)).astype(np.float32)).cuda()
    y = torch.zeros(n_rows, device="cuda")
    nodes, off = synth.pack(progs)
    grad, fit = gp.gp_const_grad(gp.nodes_to_device(nodes), torch.from_numpy(off).cuda(), X, y, None, "mse")
    d = X[0].double()
    one = torch.ones_like(d)
    vals = [d, d * d, 2 * d, 0.75 * one, 0.75 * d, 0.75 + d * d]
    parts = [None, None, None, one, d, one]  # d value / d constant
    want = torch.zeros(len(progs), 16, dtype=torch.float64)
    for i, (v, p) in enumerate(zip(vals, parts)):
        if p is not None:
            want[i, 0] = (2 * v * p).mean()
    np.testing.assert_allclose(fit.cpu().numpy(), [float((v * v).mean()) for v in vals], rtol=2e-6)
    np.testing.assert_allclose(grad.cpu().numpy(), want.numpy(), rtol=2e-6, atol=0)
