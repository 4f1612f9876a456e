"""The device pre-pass at the edges of its 32-node chunks and of its row sums.

Its program scan works on 32 nodes at a time with counts carried from chunk
to chunk, so programs of 1, 31, 32, 33, ... 255 nodes, and constant-only
subtrees that lie across a chunk's edge, are where it can go wrong.  The
total weight is summed by up to 512 blocks of at least 1024 rows.
"""
import numpy as np
import pytest

import oracle
from paper_2110_11226_gb300 import synth

pytestmark = pytest.mark.gpu

VAR, CONST, ADD, SUB, MUL, DIV, ABS, NEG = 1, 0, 2, 3, 4, 5, 12, 13


def _sized(rng, n, binary):
    """a random valid prefix list of exactly n nodes over IEEE operators; its
    left operands are terminals or short constant-only subtrees"""
    if n == 1:
        return [(VAR, int(rng.integers(2)), 0.0)] if rng.random() < 0.7 else [(CONST, 0, float(rng.uniform(1, 2)))]
    if n == 2 or not binary or rng.random() < 0.3:
        return [(int(rng.choice([ABS, NEG])), 0, 0.0)] + _sized(rng, n - 1, binary)
    k = int(min(n - 2, rng.choice([1, 1, 2, 4, 7])))
    if rng.random() < 0.5:  # constant-only: a chain of one-operand functions over a constant
        left = [(NEG, 0, 0.0)] * (k - 1) + [(CONST, 0, float(rng.uniform(1, 2)))]
    else:
        left = _sized(rng, k, False)
    return [(int(rng.choice([ADD, SUB, MUL, DIV])), 0, 0.0)] + left + _sized(rng, n - 1 - k, binary)


@pytest.mark.parametrize("length", [1, 2, 31, 32, 33, 63, 64, 65, 127, 128, 129, 224, 225, 254, 255])
def test_programs_at_chunk_edges(length):
    import torch

    from paper_2110_11226_gb300 import gp
    rng = np.random.default_rng(length)
    progs = [_sized(rng, length, b) for b in (True, False) for _ in range(9)]
    assert all(len(p) == length for p in progs)
    # a valid program, one node short, one too many, a bad code in front
    progs += [progs[0][1:], progs[0] + [(VAR, 0, 0.0)], [(40, 0, 0.0)] + progs[0][1:]]
    nodes, off = synth.pack(progs)
    X = rng.uniform(-2, 2, size=(2, 300)).astype(np.float32)
    pn, po = gp.nodes_to_device(nodes), torch.from_numpy(off).cuda()
    dX = torch.from_numpy(X).cuda()
    st = torch.zeros(len(progs), dtype=torch.int32, device="cuda")
    gp.gp_evaluate_ex(pn, po, dX, dX[0].contiguous(), out_status=st)
    _, want_st, _ = gp.gp_validate_host(nodes, off, 2)
    np.testing.assert_array_equal(st.cpu().numpy(), want_st)
    ok = want_st == 0
    assert ok[:18].all()
    got = gp.gp_predict(pn, po, dX).cpu().numpy()
    assert np.isnan(got[~ok]).all()
    good = [p for p, v in zip(progs, ok) if v]
    np.testing.assert_array_equal(got[ok], oracle.predict32(*synth.pack(good), X))
    gp.gp_last_device_status()


@pytest.mark.parametrize("n_rows", [1, 255, 1023, 1024, 1025, 524_287, 524_288, 524_289, 1_500_001])
def test_total_weight(n_rows):
    """x0 = 1 against y = 0 under weights w: MSE and MAE are sum w / sum w.
    The numerator is summed in FP32 -- 8 or 16 terms in a lane, then
    compensated, 5 + 8 adds across the block -- so it is off by at most
    (16 + 13) 2^-24 < 2e-6 relative; a total that missed or doubled a row
    would be off by 1 / n or by its weight."""
    import torch

    from paper_2110_11226_gb300 import gp
    nodes, off = synth.pack([[(VAR, 0, 0.0)]])
    g = torch.Generator(device="cuda").manual_seed(n_rows)
    w = torch.rand(n_rows, generator=g, device="cuda") + 0.5
    w[-1] = 0.25 * n_rows + 1.0  # the last row carries a fifth of the total
    one, zero = torch.ones(1, n_rows, device="cuda"), torch.zeros(n_rows, device="cuda")
    pn, po = gp.nodes_to_device(nodes), torch.from_numpy(off).cuda()
    for metric in ("mse", "mae"):
        f = float(gp.gp_evaluate(pn, po, one, zero, w, metric)[0])
        assert abs(f - 1.0) <= 2e-6, (metric, f)
        f = float(gp.gp_evaluate(pn, po, one, zero, None, metric)[0])
        assert f == 1.0
    # y = x0 up to sign and scale: the correlation is 1
    x = torch.randn(1, n_rows, generator=g, device="cuda")
    if n_rows > 1:
        r = float(gp.gp_evaluate(pn, po, x, (-2.0 * x[0]).contiguous(), w, "pearson")[0])
        assert abs(r - 1.0) <= 1e-5


@pytest.mark.parametrize("length", [1, 2, 31, 32, 33, 64, 65, 128, 129, 254, 255])
def test_mutation_at_chunk_edges(length):
    """The mutation step scans its lists 32 nodes at a time too: parents and
    donors of exactly `length` nodes, every kind, bit for bit."""
    import torch

    from paper_2110_11226_gb300 import gp
    rng = np.random.default_rng(1000 + length)
    progs = [_sized(rng, length, b) for b in (True, False) for _ in range(20)]
    nodes, off = synth.pack(progs)
    parents = rng.integers(0, 40, 2 * 300).astype(np.int32)
    for kind in ("crossover", "subtree", "hoist", "point"):
        probs = dict(p_crossover=0.0, p_subtree=0.0, p_hoist=0.0, p_point=0.0, p_replace=0.3)
        probs["p_" + kind] = 1.0
        out, oo, k = gp.gp_mutate(gp.nodes_to_device(nodes), torch.from_numpy(off).cuda(), 2,
                                  torch.from_numpy(parents).cuda(), gp.make_mut_params(**probs), seed=length)
        wn, wo, wk = oracle.mutate(nodes, off, 2, parents, seed=length, **probs)
        np.testing.assert_array_equal(oo.cpu().numpy(), wo)
        np.testing.assert_array_equal(k.cpu().numpy(), wk)
        assert gp.nodes_from_device(out[:int(wo[-1])]).tobytes() == wn.tobytes()


@pytest.mark.parametrize("k", [1, 3, 4, 5, 8, 21])
def test_tournament_sizes(k):
    """Draws come four at a time: sizes around multiples of four."""
    import torch

    from paper_2110_11226_gb300 import gp
    fit = np.random.default_rng(k).standard_normal(77).astype(np.float32)
    fit[5] = np.nan
    for greater in (False, True):
        got = gp.gp_tournament_ex(torch.from_numpy(fit).cuda(), 129, k, 9, greater_is_better=greater)
        np.testing.assert_array_equal(got.cpu().numpy(),
                                      oracle.tournament(fit, 129, k, 9, greater_is_better=greater))
