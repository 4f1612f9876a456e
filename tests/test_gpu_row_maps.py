"""How a lane's rows are laid out (consecutive, 16-byte loads; or every 32nd
row, 4-byte loads, in ragged sub-tiles and unaligned columns) must not show
in any prediction, and in a fitness only as a summation order."""
import numpy as np
import pytest

import oracle
from paper_2110_11226_gb300 import synth

pytestmark = pytest.mark.gpu

IEEE = ("add", "sub", "mul", "div", "sqrt", "abs", "neg", "inv")


@pytest.mark.parametrize("n_feat", [1, 2, 5])
@pytest.mark.parametrize("n_rows", [1, 31, 32, 33, 127, 128, 255, 256, 257, 260, 2047, 2048, 2052, 4099])
@pytest.mark.parametrize("offset", [0, 1])
def test_predictions_and_fitness(n_feat, n_rows, offset):
    import torch

    from paper_2110_11226_gb300 import gp
    nodes, off = synth.ramped_half_and_half(40, 2, 6, IEEE, n_feat, seed=7)
    rng = np.random.default_rng(n_rows)
    X = rng.uniform(-4, 4, size=(n_feat, n_rows)).astype(np.float32)
    y = rng.uniform(-1, 1, size=n_rows).astype(np.float32)
    w = rng.uniform(0.5, 2.0, size=n_rows).astype(np.float32)
    ref = oracle.predict32(nodes, off, X)
    pn, po = gp.nodes_to_device(nodes), torch.from_numpy(off).cuda()

    def at(a):  # the array `offset` floats past an aligned address
        buf = torch.empty(a.size + offset, device="cuda")
        v = buf[offset:]
        v.copy_(torch.from_numpy(a.ravel()))
        return v.view(a.shape)
    dX, dy, dw = at(X), at(y), at(w)
    for rpt in (4, 8):
        out = torch.full((40 * n_rows + offset,), 7.0, device="cuda")[offset:].view(40, n_rows)
        gp.gp_predict_ex(pn, po, dX, gp.make_opts(rows_per_thread=rpt), out=out)
        np.testing.assert_array_equal(out.cpu().numpy(), ref)
    # weighted MAE of the very predictions: a lane adds at most 16 terms
    # before the compensated sum, 13 more adds combine lanes and warps, and
    # the product and difference round once each: (16 + 13 + 2) 2^-24 < 2e-6
    with np.errstate(all="ignore"):
        e = np.abs(ref.astype(np.float64) - y)
        want = (e * w).sum(1) / w.astype(np.float64).sum()
    for rpt in (4, 8, 16):
        got = gp.gp_evaluate_ex(pn, po, dX, dy, dw, "mae", gp.make_opts(rows_per_thread=rpt)).cpu().numpy()
        fin = np.isfinite(want) & (want < 1e37)
        assert fin.any()
        np.testing.assert_allclose(got[fin], want[fin], rtol=2e-6)
