"""Weighted squared errors at the ends of the float range are the same wherever
the row lies: in a whole sub-tile, in the ragged last one, and in the plain
evaluator."""
import numpy as np
import pytest

from paper_2110_11226_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("metric", ["mse", "rmse"])
@pytest.mark.parametrize("n_rows", [256, 1027, 5003])
def test_square_past_the_float_range(metric, n_rows):
    import torch

    from paper_2110_11226_gb300 import gp
    # ordinary values, and a column with one row far out, as it is and times a
    # constant (the gradient's own kernel)
    x1 = (synth.OP["var"], 1, 0.0)
    nodes, off = synth.pack([[(synth.OP["var"], 0, 0.0)], [x1],
                             [(synth.OP["mul"], 0, 0.0), (synth.OP["const"], 0, 1.0), x1]])
    pn, po = gp.nodes_to_device(nodes), torch.from_numpy(off).cuda()
    rng = np.random.default_rng(n_rows)
    X0 = rng.uniform(1.0, 2.0, (2, n_rows)).astype(np.float32)
    w0 = rng.uniform(0.5, 1.5, n_rows).astype(np.float32)
    y = torch.zeros(n_rows, device="cuda")
    # the square overflows: NaN under a zero weight, else infinite; it does not: finite
    for error, weight in ((1e25, 0.0), (-1e25, 0.0), (1e20, 1e-10), (-3e19, 1e-30), (1e19, 1e-30), (1e19, 0.0)):
        over = error * error > float(np.finfo(np.float32).max)
        for row in (0, 5, n_rows // 2, n_rows - 1):
            X, w = X0.copy(), w0.copy()
            X[1, row], w[row] = error, weight
            dX, dw = torch.from_numpy(X).cuda(), torch.from_numpy(w).cuda()
            got = [gp.gp_evaluate_plain(pn, po, dX, y, dw, metric)]
            got += [gp.gp_evaluate_ex(pn, po, dX, y, dw, metric, opts=gp.EvalOpts(rows_per_thread=r)) for r in (4, 8)]
            got.append(gp.gp_const_grad(pn, po, dX, y, dw, metric)[1])
            for g in got:
                g = g.cpu().numpy()
                assert np.isfinite(g[0])
                if over:
                    assert np.all(np.isnan(g[1:]) if weight == 0.0 else np.isposinf(g[1:])), (error, weight, row, g)
                else:  # at most 256 FP32 additions in a row, of one sign
                    want = np.sum(w.astype(np.float64) * X[1].astype(np.float64) ** 2) / np.sum(w.astype(np.float64))
                    want = np.sqrt(want) if metric == "rmse" else want
                    np.testing.assert_allclose(g[1:], want, rtol=256 * 2.0 ** -24)
