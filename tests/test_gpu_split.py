"""FP32 networks on the tensor cores (three BF16 planes per operand) at the edges of their tiles.

Bound per layer, from the arithmetic: the products left out and the planes' rounding stay below
2^-22 |a||w|, the tensor core truncates at most 24 additions per k-block of 64 (below 2^-22 of the
block's absolute sum in all, since the first 20 add terms 2^-8 of the last four), and the k-blocks are
added in FP32: (8 + K / 64) 2^-23 (|H| |W|^T + |b|). GELU has slopes below 1.13 and is evaluated to
2^-21 of |z|; errors of a layer's inputs pass through |W|.
"""
import types

import numpy as np
import pytest

from oracle import network as onw

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def df():
    import torch
    import __graft_entry__ as g
    g.build()
    import paper_2508_18969_gb300 as m
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return m


def _net(widths, seed):
    rng = np.random.default_rng(seed)
    W, b = [], []
    for i, o in zip(widths[:-1], widths[1:]):
        lim = np.sqrt(6.0 / (i + o))
        W.append(rng.uniform(-lim, lim, (o, i)).astype(np.float32).astype(np.float64))
        b.append(rng.uniform(-0.1, 0.1, o).astype(np.float32).astype(np.float64))
    k, m = widths[0], widths[-1]
    return types.SimpleNamespace(widths=list(widths), W=W, b=b, lam=0.1, dt=0.0, n_layers=len(W),
                                 in_mean=np.zeros(k), in_std=np.ones(k), out_mean=np.zeros(m),
                                 out_std=np.ones(m))


def _bound(net, x):
    H, E = x, np.zeros_like(x)
    for l, (W, b) in enumerate(zip(net.W, net.b)):
        K = W.shape[1]
        s = np.abs(H) @ np.abs(W).T + np.abs(b)
        z = H @ W.T + b
        E = E @ np.abs(W).T + (8 + K / 64) * 2.0 ** -23 * s
        if l + 1 < len(net.W):
            E = 1.13 * E + 2.0 ** -21 * np.abs(z)
            z = onw.gelu_tanh(z)
        H = z
    return H, E


@pytest.mark.parametrize("widths,rows", [
    ((3, 1), 1), ((3, 31), 127), ((18, 32, 33), 128), ((33, 64, 65, 63), 129), ((34, 65, 1), 255),
    ((32, 257, 96, 5), 257), ((11, 256, 128, 64, 9), 4097), ((32, 640, 129, 40), 20011),
    ((32, 1600, 800, 400, 30), 19969),
])
def test_matches_fp64(df, widths, rows):
    import torch
    net = _net(widths, 5 + rows)
    x = np.random.default_rng(rows).normal(size=(rows, widths[0])).astype(np.float32)
    pn = df.PropNet(net, precision=df.DF_FP32, batch_cells=max(128, min(rows, 8192)))
    got = pn.mlp_forward(torch.tensor(x, device="cuda")).cpu().numpy().astype(np.float64)
    want, tol = _bound(net, x.astype(np.float64))
    assert np.all(np.abs(got - want) <= tol), np.max(np.abs(got - want) / tol)
    pn.close()


def test_values_beyond_bf16_and_not_finite(df):
    """A linear layer passes infinities with the weights' signs, NaN as NaN, and FP32 values that
    would round to a BF16 infinity; other rows of the tile are not touched."""
    import torch
    net = _net((6, 70), 3)
    x = np.random.default_rng(4).normal(size=(200, 6)).astype(np.float32)
    clean = x.copy()
    x[3, 1] = np.inf
    x[64, 2] = -np.inf
    x[65, 0], x[65, 1] = np.inf, np.nan
    x[199, 5] = np.finfo(np.float32).max
    pn = df.PropNet(net, precision=df.DF_FP32, batch_cells=256)
    got = pn.mlp_forward(torch.tensor(x, device="cuda")).cpu().numpy()
    base = pn.mlp_forward(torch.tensor(clean, device="cuda")).cpu().numpy()
    W = net.W[0]
    assert np.array_equal(got[3], np.sign(W[:, 1]) * np.inf)
    assert np.array_equal(got[64], -np.sign(W[:, 2]) * np.inf)
    assert np.isnan(got[65]).all()
    big = np.abs(x[199].astype(np.float64)) @ np.abs(W).T
    want = x[199].astype(np.float64) @ W.T
    fits = np.abs(want) < np.finfo(np.float32).max
    assert fits.any() and np.all(np.abs(got[199].astype(np.float64) - want)[fits] <= 2.0 ** -19 * big[fits])
    others = np.setdiff1d(np.arange(200), [3, 64, 65, 199])
    assert np.array_equal(got[others], base[others])
    pn.close()
