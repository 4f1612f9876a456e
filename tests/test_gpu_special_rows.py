"""A few special values (NaN, infinities, zeros) among ordinary ones: the ordinary
rows keep the bits that they have without them, the special ones get the value
that the pre-pass folds, at 4 and 8 rows per lane, in the common and the
extended class, with columns in registers and columns read from memory."""
import numpy as np
import pytest

from paper_2110_11226_gb300 import synth

pytestmark = pytest.mark.gpu

SPECIAL = np.array([np.nan, np.inf, -np.inf, 0.0, -0.0], np.float32)
UNARY = ("sqrt", "log", "exp", "sin", "cos", "tan", "abs", "neg", "inv", "sq", "cube", "tanh")


@pytest.mark.parametrize("which", [[0], [1, 2], [3, 4], [0, 1, 2, 3, 4]], ids=["nan", "inf", "zero", "all"])
@pytest.mark.parametrize("n_feat", [2, 5])
@pytest.mark.parametrize("rpt", [4, 8])
def test_special_rows_among_ordinary_ones(rpt, n_feat, which):
    import torch

    from paper_2110_11226_gb300 import gp
    O, V, C = synth.OP, synth.OP["var"], synth.OP["const"]
    rng = np.random.default_rng(n_feat)
    n = 3000
    clean = (rng.uniform(0.1, 50.0, (n_feat, n)) * rng.choice([-1.0, 1.0], (n_feat, n))).astype(np.float32)
    X = clean.copy()
    at = rng.random((n_feat, n)) < 0.01
    X[at] = rng.choice(SPECIAL[which], at.sum())
    a, b = 0, n_feat - 1
    progs = [[(O[f], 0, 0.0), (V, a, 0.0)] for f in UNARY]
    progs += [[(O[f], 0, 0.0), (V, a, 0.0), (V, b, 0.0)] for f in ("div", "add", "mul", "max", "min")]
    progs += [[(O["div"], 0, 0.0), (C, 0, 1.5), (V, a, 0.0)], [(O["div"], 0, 0.0), (V, a, 0.0), (C, 0, -1.5)]]
    # a stack operand, and a word after the special one
    progs += [[(O["div"], 0, 0.0), (O["neg"], 0, 0.0), (V, a, 0.0), (O["neg"], 0, 0.0), (V, b, 0.0)],
              [(O["sin"], 0, 0.0), (O["neg"], 0, 0.0), (V, a, 0.0)]]

    def predict(progs, X):
        nodes, off = synth.pack(progs)
        return gp.gp_predict_ex(gp.nodes_to_device(nodes), torch.from_numpy(off).cuda(), torch.from_numpy(X).cuda(),
                                gp.make_opts(rows_per_thread=rpt)).cpu().numpy()

    got, base = predict(progs, X), predict(progs, clean)
    rows = np.flatnonzero(at[a] | at[b])
    assert len(rows) > 20
    # the programs with the columns' values in their place are constants
    def fold(p, r):
        return [(C, 0, float(X[f, r])) if op == V else (op, f, c) for op, f, c in p]
    want = predict([fold(p, r) for p in progs for r in rows], np.ones((1, 1), np.float32))[:, 0].reshape(len(progs), -1)
    plain = np.setdiff1d(np.arange(n), rows)
    np.testing.assert_array_equal(got[:, plain].view(np.uint32), base[:, plain].view(np.uint32))
    special = got[:, rows]
    nan = np.isnan(want)
    np.testing.assert_array_equal(np.isnan(special), nan)
    np.testing.assert_array_equal(special[~nan].view(np.uint32), want[~nan].view(np.uint32))
