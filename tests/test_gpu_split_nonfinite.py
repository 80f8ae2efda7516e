"""FP32 networks with operands that are not finite, through planes, several k-blocks and splits: every result
that IEEE arithmetic makes infinite or NaN is so (the class does not depend on the order of a sum far from
overflow), the others are those of the finite rows, and no wait of the pipeline runs out however many results
have to be formed again (an infinite row of the output gradient makes every weight gradient of the last two
layers infinite)."""
import types

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def df():
    import __graft_entry__ as g
    g.build()
    import paper_2508_18969_gb300 as m
    return m


def _net(widths, seed):
    rng = np.random.default_rng(seed)
    W = [(rng.uniform(-1, 1, (o, i)) * np.sqrt(6.0 / (i + o))).astype(np.float32) for i, o in zip(widths[:-1], widths[1:])]
    b = [rng.uniform(-0.1, 0.1, o).astype(np.float32) for o in widths[1:]]
    k, m = widths[0], widths[-1]
    return types.SimpleNamespace(widths=list(widths), W=W, b=b, lam=0.1, dt=0.0, n_layers=len(W), in_mean=np.zeros(k),
                                 in_std=np.ones(k), out_mean=np.zeros(m), out_std=np.ones(m))


def _gelu(z):
    c, a = 0.7978845608028654, 0.044715
    t = torch.tanh(c * (z + a * z ** 3))
    return 0.5 * z * (1 + t), 0.5 * (1 + t) + 0.5 * z * (1 - t * t) * c * (1 + 3 * a * z * z)


def _same_class(got, want, tol):
    assert torch.equal(torch.isnan(got), torch.isnan(want))
    assert torch.equal(torch.isposinf(got), torch.isposinf(want)) and torch.equal(torch.isneginf(got), torch.isneginf(want))
    f = torch.isfinite(want)
    if f.any():
        assert (got[f].double() - want[f].double()).abs().max() <= tol * want[f].double().abs().max()


@pytest.mark.parametrize("widths,rows", [((33, 130, 70, 6), 300), ((34, 300, 257, 40), 5000)])
def test_forward(df, widths, rows):
    net = _net(widths, 1)
    net.W[0][:, 0] = np.abs(net.W[0][:, 0])                 # +inf in input 0: every hidden value +inf
    net.W[1][:, :] = np.abs(net.W[1])
    net.W[2][0], net.W[2][1] = np.abs(net.W[2][0]), -np.abs(net.W[2][1])
    net.W[2][2], net.W[2][2, 5] = np.abs(net.W[2][2]), 0.0
    x = np.random.default_rng(2).normal(size=(rows, widths[0])).astype(np.float32)
    clean = x.copy()
    bad = [3, 129, rows // 2, rows - 1]
    x[bad[0], 0] = np.inf
    x[bad[1], 0] = np.nan
    x[bad[2], 7] = -np.inf
    x[bad[3], 0], x[bad[3], 7] = np.inf, -np.inf
    pn = df.PropNet(net, precision=df.DF_FP32, batch_cells=4096)
    dev = lambda a: torch.tensor(a, device="cuda")
    for h in (pn.mlp_forward(dev(x)), pn.mlp_forward_train(dev(x))):
        z = dev(x[bad]).double()
        for l, (W, b) in enumerate(zip(net.W, net.b)):
            z = z @ dev(W).double().T + dev(b).double()
            z = _gelu(z)[0] if l < 2 else z
        _same_class(h[bad], z, 0.0)
        assert torch.isposinf(h[bad[0], 0]) and torch.isneginf(h[bad[0], 1]) and torch.isnan(h[bad[0], 2])
        others = np.setdiff1d(np.arange(rows), bad)
        assert torch.equal(h[others], pn.mlp_forward(dev(clean))[others])
    pn.close()


@pytest.mark.parametrize("widths,rows", [((11, 65, 33, 9), 129), ((11, 257, 96, 9), 5003),
                                         ((32, 1600, 800, 400, 30), 262145)])
def test_infinite_gradient(df, widths, rows):
    net = _net(widths, 3)
    gen = torch.Generator(device="cuda").manual_seed(rows)
    x = torch.randn(rows, widths[0], device="cuda", generator=gen)
    dO = torch.randn(rows, widths[-1], device="cuda", generator=gen) / rows
    dO[rows // 3, 1] = float("inf")
    pn = df.PropNet(net, precision=df.DF_FP32, batch_cells=128)
    pn.mlp_forward_train(x)
    dX = pn.mlp_backward(dO)
    assert pn.step_summary()[0] != df._lib.DF_ERR_TIMEOUT
    H, G, W = [x], [], [torch.tensor(w, device="cuda") for w in net.W]
    for w, b in zip(W[:-1], net.b[:-1]):
        h, g = (t.float() for t in _gelu((H[-1] @ w.T + torch.tensor(b, device="cuda")).double()))
        H.append(h)
        G.append(g)
    dZ = dO
    for l in range(len(W) - 1, -1, -1):
        gW, gb = pn.params(l, df._lib.DF_PARAM_GRADS, widths=widths)
        _same_class(gW, dZ.T @ H[l], 1e-3)
        _same_class(gb, dZ.sum(0), 1e-3)
        dZ = dZ @ W[l]
        if l:
            dZ = dZ * G[l - 1]
    _same_class(dX, dZ, 1e-3)
    assert not torch.isfinite(pn.params(len(W) - 1, df._lib.DF_PARAM_GRADS, widths=widths)[0][1]).any()
    pn.close()
