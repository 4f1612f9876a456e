"""Calls that follow one another without a synchronisation share the library's
workspace and overlap at their edges: every result must be that of the call
on its own, whatever ran before, with inputs rewritten between calls and in a
captured graph."""
import numpy as np
import pytest

from paper_2110_11226_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_feat", [2, 6])
def test_back_to_back_calls(n_feat):
    import torch

    from paper_2110_11226_gb300 import gp
    sets = (synth.FULL_SET, synth.EXTENDED_SET, synth.PAPER_SET, synth.FULL_SET)
    pops = []
    for i, funcs in enumerate(sets):
        # every class: a few programs with deep compiled stacks among the others
        nodes, off = synth.ramped_half_and_half(150 + 90 * i, 2, 8, funcs, n_feat, seed=i)
        deep = [(2, 0, 0.0)] * 11 + [(12, 0, 0.0), (1, 0, 0.0)] * 12
        nodes, off = synth.pack(synth.unpack(nodes, off) + [deep] * (i + 1))
        pops.append((gp.nodes_to_device(nodes), torch.from_numpy(off).cuda()))
    g = torch.Generator(device="cuda").manual_seed(5)
    n = 5003
    Xs = [torch.randn(n_feat, n, generator=g, device="cuda") for _ in range(3)]
    ys = [torch.randn(n, generator=g, device="cuda") for _ in range(3)]
    X, y = Xs[0].clone(), ys[0].clone()
    metrics = ("mse", "pearson", "mae")
    want = {}
    for p in range(len(pops)):
        for d in range(3):
            torch.cuda.synchronize()
            want[p, d] = gp.gp_evaluate(*pops[p], Xs[d], ys[d], None, metrics[d]).cpu()
    rng = np.random.default_rng(1)
    calls, got = [], []
    for _ in range(60):  # nothing waits in here
        p, d = int(rng.integers(len(pops))), int(rng.integers(3))
        X.copy_(Xs[d])
        y.copy_(ys[d])
        calls.append((p, d))
        got.append(gp.gp_evaluate(*pops[p], X, y, None, metrics[d]))
    for key, f in zip(calls, got):
        assert torch.equal(f.cpu().nan_to_num(-1.0), want[key].nan_to_num(-1.0)), key
    # the same chain captured and replayed, the inputs rewritten inside it
    ws = torch.empty(max(gp.gp_workspace_size(o.numel() - 1, n, n_feat) for _, o in pops), dtype=torch.uint8,
                     device="cuda")
    out = [torch.empty(o.numel() - 1, device="cuda") for _, o in pops]
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        for p in range(len(pops)):
            X.copy_(Xs[p % 3])
            y.copy_(ys[p % 3])
            gp.gp_evaluate_ex(*pops[p], X, y, None, metrics[p % 3], out=out[p], ws=ws)
    for _ in range(3):
        graph.replay()
    torch.cuda.synchronize()
    for p in range(len(pops)):
        assert torch.equal(out[p].cpu().nan_to_num(-1.0), want[p, p % 3].nan_to_num(-1.0)), p
