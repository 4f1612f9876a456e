"""tan, sq, cube, max and min in the fast loop of the extended class: on edge
arguments they give the bits of the C++ functions that the pre-pass folds
constants with (NaN where those do), at 4 and 8 rows per lane, with columns in
registers and columns read from memory."""
import numpy as np
import pytest

from paper_2110_11226_gb300 import synth

pytestmark = pytest.mark.gpu

EDGE = np.array([0.0, 1e-40, 2.0 ** -61, 2.0 ** -60, 1e-8, 0.001, 0.5, np.pi / 4, 1.0, np.pi / 2, 1.5707964,
                 np.pi, 3.25, 4.712389, 100.0, 1e4, 65535.0, 65536.0, 7e4, 1e19, 2.0 ** 64, 3e38, np.inf],
                np.float64)
EDGE = np.concatenate([EDGE, -EDGE, [np.nan]]).astype(np.float32)


@pytest.mark.parametrize("n_feat", [2, 5])
@pytest.mark.parametrize("rpt", [4, 8])
def test_loop_matches_the_folded_value(n_feat, rpt):
    import torch

    from paper_2110_11226_gb300 import gp
    O, V, C = synth.OP, synth.OP["var"], synth.OP["const"]
    n = len(EDGE)
    a, b = (g.ravel() for g in np.meshgrid(EDGE, EDGE, indexing="ij"))
    X = np.zeros((n_feat, n * n), np.float32)
    X[0], X[n_feat - 1] = a, b
    unary, binary = ("tan", "sq", "cube"), ("max", "min")
    progs = [[(O[f], 0, 0.0), (V, 0, 0.0)] for f in unary]
    progs += [[(O[f], 0, 0.0), (V, 0, 0.0), (V, n_feat - 1, 0.0)] for f in binary]
    folded = [[(O[f], 0, 0.0), (C, 0, float(c))] for f in unary for c in EDGE]
    folded += [[(O[f], 0, 0.0), (C, 0, float(p)), (C, 0, float(q))] for f in binary for p, q in zip(a, b)]
    nodes, off = synth.pack(progs + folded)
    pred = gp.gp_predict_ex(gp.nodes_to_device(nodes), torch.from_numpy(off).cuda(), torch.from_numpy(X).cuda(),
                            gp.make_opts(rows_per_thread=rpt)).cpu().numpy()
    got, want = pred[:len(progs)], pred[len(progs):, 0]
    want = np.concatenate([np.repeat(want[:3 * n].reshape(3, n), n, axis=1), want[3 * n:].reshape(2, n * n)])
    nan = np.isnan(want)
    np.testing.assert_array_equal(np.isnan(got), nan)
    np.testing.assert_array_equal(got[~nan].view(np.uint32), want[~nan].view(np.uint32))
