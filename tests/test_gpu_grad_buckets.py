"""The constant gradient at the edges of its buckets (what a program's stack and
constants need of shared memory), where the packed stack, tangents and sums of a
warp are largest, with marked divisions by and of columns among them."""
import numpy as np
import pytest

from paper_2110_11226_gb300 import synth

pytestmark = pytest.mark.gpu


def _program(depth, n_consts, n_feat, X, theta):
    """a sum of depth leaves, all of them on the stack at once, that hold the
    constants in turn; (prefix nodes, its value for theta, in 64 bits)"""
    O = synth.OP
    leaves = [([(O["var"], i % n_feat, 0.0)], X[i % n_feat]) for i in range(depth)]
    if depth > 1:  # (a plain column would be an operand, not a stack value)
        leaves = [([(O["abs"], 0, 0.0)] + p, v) for p, v in leaves]
    for k in range(n_consts):
        i, f, c = k % depth, (k + 1) % n_feat, (O["const"], 0, float(theta[k]))
        x = (O["var"], f, 0.0)
        p, v = leaves[i]
        form = k % 4
        if form == 0:    # x / (c e) * x
            p, v = [(O["mul"], 0, 0.0), (O["div"], 0, 0.0), x, (O["mul"], 0, 0.0), c] + p + [x], \
                X[f] / (theta[k] * v) * X[f]
        elif form == 1:  # (e / c) / x
            p, v = [(O["div"], 0, 0.0), (O["div"], 0, 0.0)] + p + [c, x], v / theta[k] / X[f]
        elif form == 2:  # c / e + x
            p, v = [(O["add"], 0, 0.0), (O["div"], 0, 0.0), c] + p + [x], theta[k] / v + X[f]
        else:            # x (e + c)
            p, v = [(O["mul"], 0, 0.0), x, (O["add"], 0, 0.0)] + p + [c], X[f] * (v + theta[k])
        leaves[i] = p, v
    nodes = [(O["add"], 0, 0.0)] * (depth - 1)
    for p, _ in leaves:
        nodes = nodes + p
    return nodes, sum(v for _, v in leaves)


@pytest.mark.parametrize("n_rows", [1, 1027, 3072])
@pytest.mark.parametrize("n_feat", [2, 5])
def test_gradient_at_the_bucket_edges(n_feat, n_rows):
    import torch

    from paper_2110_11226_gb300 import gp
    # 4 (depth - 1) + 5 constants around 51, 70 and 108 units, deep stacks, none
    shapes = [(1, 1), (1, 10), (5, 7), (4, 8), (8, 4), (8, 5), (1, 14), (1, 15), (6, 10), (6, 11), (8, 8),
              (8, 9), (3, 16), (8, 16), (8, 0), (9, 1), (12, 16), (20, 16), (2, 2), (2, 14), (16, 4)]
    rng = np.random.default_rng(n_feat)
    X = torch.from_numpy(rng.uniform(1.0, 2.0, (n_feat, n_rows)).astype(np.float32)).cuda()
    y = torch.zeros(n_rows, device="cuda")
    progs, want, fits = [], torch.zeros(len(shapes), 16, dtype=torch.float64), []
    for i, (depth, n_consts) in enumerate(shapes):
        # (the prefix order of the constants is not the order of theta)
        theta = torch.from_numpy(rng.uniform(0.5, 1.5, n_consts).astype(np.float32)).double().cuda()
        theta.requires_grad_(True)
        p, v = _program(depth, n_consts, n_feat, X.double(), theta)
        progs.append(p)
        fit = (v * v).mean()
        fits.append(fit.item())
        if n_consts:
            (g,) = torch.autograd.grad(fit, theta)
            order = [int(np.argmin([abs(t - c) for t in theta.tolist()])) for op, _, c in p if op == synth.OP["const"]]
            assert sorted(order) == list(range(n_consts))
            want[i, :n_consts] = g.cpu()[order]
    nodes, off = synth.pack(progs)
    grad, fit = gp.gp_const_grad(gp.nodes_to_device(nodes), torch.from_numpy(off).cuda(), X, y, None, "mse")
    # two of them need more than the 20 values that a program's own stack may hold
    binary = {synth.OP[f] for f in ("add", "mul", "div")}
    deepest = [max(np.cumsum([0 if op == synth.OP["abs"] else -1 if op in binary else 1 for op, _, _ in p[::-1]]))
               for p in progs]
    for i, d in enumerate(deepest):
        if d > 20:
            fits[i] = want[i] = np.nan
    assert sum(d > 20 for d in deepest) == 2
    # every term is positive up to the sign that a constant's gradient has as a
    # whole: no cancellation, at most some 60 roundings in a row
    np.testing.assert_allclose(fit.cpu().numpy(), fits, rtol=1e-5)
    np.testing.assert_allclose(grad.cpu().numpy(), want.numpy(), rtol=1e-5, atol=0)


def test_back_to_back_gradients():
    """Gradients, evaluations and Adam steps with nothing waiting between them,
    and captured, equal each call alone."""
    import torch

    from paper_2110_11226_gb300 import gp
    g = torch.Generator(device="cuda").manual_seed(3)
    n, n_feat = 4099, 5
    X = torch.randn(n_feat, n, generator=g, device="cuda")
    y = torch.randn(n, generator=g, device="cuda")
    w = torch.rand(n, generator=g, device="cuda") + 0.5
    pops = []
    for i in range(3):
        nodes, off = synth.ramped_half_and_half(100 + 150 * i, 2, 7, synth.FULL_SET, n_feat, seed=i, max_consts=16)
        pops.append((gp.nodes_to_device(nodes), torch.from_numpy(off).cuda()))
    want = []
    for nodes, off in pops:
        for ww in (None, w):
            torch.cuda.synchronize()
            grad, fit = gp.gp_const_grad(nodes, off, X, y, ww, "mse")
            torch.cuda.synchronize()
            want.append((grad.cpu(), fit.cpu(), gp.gp_evaluate(nodes, off, X, y, ww, "mse").cpu()))

    def run(out):
        for nodes, off in pops:
            for ww in (None, w):
                grad, fit = gp.gp_const_grad(nodes, off, X, y, ww, "mse")
                out.append((grad, fit, gp.gp_evaluate(nodes, off, X, y, ww, "mse")))

    got = []
    for _ in range(4):
        run(got)
    graph, captured = torch.cuda.CUDAGraph(), []
    with torch.cuda.graph(graph):
        run(captured)
    for _ in range(3):
        graph.replay()
    torch.cuda.synchronize()
    for i, tensors in enumerate(got + captured):
        for a, b in zip(tensors, want[i % len(want)]):
            assert torch.equal(a.cpu().nan_to_num(-1.0), b.nan_to_num(-1.0)), i
