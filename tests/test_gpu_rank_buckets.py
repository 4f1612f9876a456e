"""The rank fitness by buckets: sizes at the edges of its bucket counts and
tiles, and values that a sample of the predictions misjudges or that fill
buckets with ties."""
import numpy as np
import pytest

import oracle
from paper_2110_11226_gb300 import synth

pytestmark = pytest.mark.gpu

CAP, AIM, OVERSAMPLE, MOST = 6144, 2048, 16, 2048  # gp_rank.cu's bucket sizes


def _sampled(n):
    """the rows that the splitters are drawn from (all, for one bucket)"""
    if n <= CAP:
        return np.arange(n)
    s = 1
    while s < -(-n // AIM) * OVERSAMPLE:
        s *= 2
    return (2 * np.arange(s, dtype=np.int64) + 1) * n // (2 * s)


def _columns(n, rng):
    u = rng.standard_normal(n).astype(np.float32)
    cols = [u, np.arange(n, dtype=np.float32), rng.integers(-3, 4, n).astype(np.float32),
            rng.integers(0, 5000, n).astype(np.float32), (np.exp(u) ** 8).astype(np.float32)]
    tight = (1.0 + 1e-5 * rng.random(n)).astype(np.float32)
    tight[n // 2] = 1e30
    hidden = rng.random(n).astype(np.float32) + 1.0   # above every splitter
    hidden[_sampled(n)] = rng.random(len(_sampled(n))).astype(np.float32) * 1e-3
    zeros = np.where(rng.random(n) < 0.5, 0.0, u).astype(np.float32)
    zeros[::3] *= -1.0                                 # -0 and +0 tie
    return np.stack(cols + [tight, hidden, zeros])


@pytest.mark.parametrize("n", [1, 2, 3, 511, CAP - 1, CAP, CAP + 1, 8191, 8192, 8193, 3 * 8192 + 5,
                               200_003, MOST * AIM, MOST * AIM + 1])
def test_rank_fitness(n):
    """Equal to the definition on the device's own values within the rounding
    of the FP32 result (2^-24) and of two FP64 evaluations (n 2^-53)."""
    import torch

    from paper_2110_11226_gb300 import gp
    rng = np.random.default_rng(n)
    X = _columns(n, rng)
    if n > 3_000_000:
        X = X[[0, 2, 6]]
    y = np.round(rng.standard_normal(n), 3).astype(np.float32)
    V = synth.OP["var"]
    progs = [[(V, f, 0.0)] for f in range(len(X))] + [[(synth.OP["const"], 0, 1.5)]]
    nodes, off = synth.pack(progs)
    pn, po = gp.nodes_to_device(nodes), torch.from_numpy(off).cuda()
    dX, dy = torch.from_numpy(X).cuda(), torch.from_numpy(y).cuda()
    got = gp.gp_evaluate(pn, po, dX, dy, None, "spearman").cpu().numpy()
    again = gp.gp_evaluate(pn, po, dX, dy, None, "spearman").cpu().numpy()
    np.testing.assert_array_equal(got.view(np.uint32), again.view(np.uint32))
    want = np.array([oracle.spearman_of(c.astype(np.float64), y.astype(np.float64)) for c in X] + [0.0])
    np.testing.assert_allclose(got, want, rtol=1e-6, atol=1e-9)
    X[0, n // 2] = np.nan
    got = gp.gp_evaluate(pn, po, torch.from_numpy(X).cuda(), dy, None, "spearman").cpu().numpy()
    assert np.isnan(got[0]) and not np.isnan(got[1:]).any()
