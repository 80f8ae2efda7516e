"""Backward pass at the edges of its tiles: odd and ragged widths and batches, operands read along their
columns, column sums, one Adam launch over padded layers.

Bounds by running error analysis against FP64: every stored operand (weights, inputs, activations, GELU'
values, gradients) carries a relative rounding u, sums at most u of their absolute terms, and the hidden
errors pass through |W| and the slopes of GELU (below 1.13) and GELU' (below 1.2, with GELU' itself below
1.13). u = 2^-8 for BF16 (storage 2^-9, hardware tanh 2^-11); 2^-16 for FP32 (three exact planes; FP32 sums
of up to 65 k-blocks and split-K partials: (8 + 65) 2^-23)."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


def _gelu(z):
    c = np.sqrt(2.0 / np.pi)
    t = np.tanh(c * (z + 0.044715 * z ** 3))
    return 0.5 * z * (1 + t), 0.5 * (1 + t) + 0.5 * z * (1 - t * t) * c * (1 + 3 * 0.044715 * z * z)


def _reference(net, x, dO, u):
    """(dX, [dW], [db]) in FP64 and elementwise bounds."""
    a = np.abs
    H, E, hs, gs = x, u * a(x), [], []
    L = len(net.W)
    for l, (W, b) in enumerate(zip(net.W, net.b)):
        hs.append((H, E))
        Z = H @ W.T + b
        EZ = (E @ a(W).T) * (1 + u) + 3 * u * (a(H) @ a(W).T + a(b))
        if l + 1 < L:
            H, G = _gelu(Z)
            E = 1.13 * EZ + u * a(H) + u * a(Z)
            gs.append((G, 1.2 * EZ + u * (1 + a(G))))
    D, ED, dW, db = dO, u * a(dO), [None] * L, [None] * L
    for l in range(L - 1, -1, -1):
        (Hi, EHi), W = hs[l], net.W[l]
        dW[l] = (D.T @ Hi, ED.T @ a(Hi) + a(D).T @ EHi + ED.T @ EHi + 3 * u * (a(D).T @ a(Hi)))
        db[l] = (D.sum(0), ED.sum(0) + 3 * u * a(D).sum(0))
        S, ES = D @ W, ED @ a(W) * (1 + u) + 3 * u * (a(D) @ a(W))
        if l:
            G, EG = gs[l - 1]
            ED = ES * (a(G) + EG) + (a(D) @ a(W)) * EG
            D = S * G
            ED = ED + u * a(D)
    return (S, ES), dW, db


@pytest.mark.parametrize("prec,u", [("DF_FP32", 2.0 ** -16), ("DF_BF16", 2.0 ** -8)])
@pytest.mark.parametrize("n,hidden,rows", [(9, (33, 65), 1), (9, (31, 129, 40), 127), (9, (256, 128, 64), 129),
                                           (31, (257, 96), 4097), (32, (130, 34), 1000)])
def test_gradients_within_error_analysis(prec, u, n, hidden, rows):
    import torch
    import __graft_entry__ as g
    g.build()
    import paper_2508_18969_gb300 as df
    widths = [n + 2, *hidden, n]
    mech = synth.mechanism.make_mechanism(n, 1, 3)
    net = synth.network.make_network(widths, n, seed=rows)
    st = df.State(mech, net, precision=getattr(df, prec), batch_cells=max(128, rows))
    rng = np.random.default_rng(rows + n)
    x = rng.normal(size=(rows, n + 2)).astype(np.float32)
    dO = (rng.normal(size=(rows, n)) / rows).astype(np.float32)
    st.mlp_forward_train(torch.tensor(x, device="cuda"))
    dX = st.mlp_backward(torch.tensor(dO, device="cuda"))
    (wantX, EX), dW, db = _reference(net, x.astype(np.float64), dO.astype(np.float64), u)
    host = lambda t: t.cpu().numpy().astype(np.float64)
    assert np.all(np.abs(host(dX) - wantX) <= EX + 1e-30)
    for l in range(len(widths) - 1):
        W, b = st.params(l, df._lib.DF_PARAM_GRADS, widths=widths)
        assert np.all(np.abs(host(W) - dW[l][0]) <= dW[l][1] + 1e-30), l
        assert np.all(np.abs(host(b) - db[l][0]) <= db[l][1] + 1e-30), l
    before = [[host(t) for t in st.params(l, widths=widths)] for l in range(len(widths) - 1)]
    grads = [[host(t) for t in st.params(l, df._lib.DF_PARAM_GRADS, widths=widths)] for l in range(len(widths) - 1)]
    st.adam_step(lr=1e-3, eps=1e-8)
    for l, (w, gr) in enumerate(zip(before, grads)):   # first step: p - lr g / (|g| + eps), in FP32
        for p0, gg, p1 in zip(w, gr, st.params(l, widths=widths)):
            want = p0 - 1e-3 * gg / (np.abs(gg) + 1e-8)
            assert np.all(np.abs(host(p1) - want) <= 1e-3 * 1e-4 + 2.0 ** -23 * np.abs(p0)), l
    st.close()
