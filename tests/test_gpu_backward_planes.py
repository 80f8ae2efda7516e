"""FP32 gradients at batches and widths so small that losing a third BF16 plane would show. Bounds per GEMM as in
test_gpu_split.py: (8 + k-blocks + splits) 2^-23 of the absolute terms; GELU to 2^-21 of |z| and GELU' (values
below 1.13, slopes below 1.2) to 2^-20 of 1 + |z|. Those are worst cases; in the 2-norm, where errors of single
terms are independent, FP32 arithmetic leaves 2^-22 to 2^-21 of a weight gradient, and operands of two planes
(off by up to 2^-18 each) 2^-18: the line lies at 2^-20, and the same products with two planes per operand,
formed on the host, are above it."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


def _gelu(z):
    c = np.sqrt(2.0 / np.pi)
    t = np.tanh(c * (z + 0.044715 * z ** 3))
    return 0.5 * z * (1 + t), 0.5 * (1 + t) + 0.5 * z * (1 - t * t) * c * (1 + 3 * 0.044715 * z * z)


def _two_planes(a):
    def bf16(v):
        u = v.astype(np.float32).view(np.uint32).astype(np.uint64)
        return ((u + 0x7FFF + ((u >> 16) & 1)) & 0xFFFF0000).astype(np.uint32).view(np.float32).astype(np.float64)
    h = bf16(a)
    return h + bf16(a - h)


@pytest.mark.parametrize("n,hidden,rows", [(9, (33, 65), 1), (9, (31, 64, 40), 3), (30, (96, 33), 2)])
def test_gradients(n, hidden, rows):
    import torch
    import __graft_entry__ as g
    g.build()
    import paper_2508_18969_gb300 as df
    widths = [n + 2, *hidden, n]
    net = synth.network.make_network(widths, n, seed=rows)
    st = df.State(synth.mechanism.make_mechanism(n, 1, 3), net, batch_cells=128)
    rng = np.random.default_rng(rows + n)
    x = rng.normal(size=(rows, n + 2)).astype(np.float32).astype(np.float64)
    dO = rng.normal(size=(rows, n)).astype(np.float32).astype(np.float64)
    dev = lambda a: torch.tensor(a, device="cuda", dtype=torch.float32)
    host = lambda t: t.cpu().numpy().astype(np.float64)
    st.mlp_forward_train(dev(x))
    dX = host(st.mlp_backward(dev(dO)))
    grads = [[host(t) for t in st.params(l, df._lib.DF_PARAM_GRADS, widths=widths)] for l in range(len(widths) - 1)]
    st.close()
    a, L = np.abs, len(net.W)
    gemm = lambda k: (8 + (k + 63) // 64 + 1) * 2.0 ** -23   # (one split: fewer than eight k-blocks)
    H, E, hs, gs = x, np.zeros_like(x), [], []
    for l, (W, b) in enumerate(zip(net.W, net.b)):
        hs.append((H, E))
        Z = H @ W.T + b
        EZ = E @ a(W).T + gemm(W.shape[1]) * ((a(H) + E) @ a(W).T + a(b))
        if l + 1 < L:
            H, G = _gelu(Z)
            E = 1.13 * EZ + 2.0 ** -21 * a(Z)
            gs.append((G, 1.2 * EZ + 2.0 ** -20 * (1 + a(Z))))
    D, ED = dO, np.zeros_like(dO)
    for l in range(L - 1, -1, -1):
        (Hi, EHi), W = hs[l], net.W[l]
        want = D.T @ Hi
        tol = ED.T @ (a(Hi) + EHi) + a(D).T @ EHi + gemm(rows) * (a(D).T @ a(Hi))
        assert np.all(a(grads[l][0] - want) <= tol + 1e-37), (l, np.max(a(grads[l][0] - want) / (tol + 1e-37)))
        off = lambda got: np.linalg.norm(got - want) / np.linalg.norm(want)
        assert off(grads[l][0]) <= 2.0 ** -20 < off(_two_planes(D).T @ _two_planes(Hi)), l
        assert np.all(a(grads[l][1] - D.sum(0)) <= ED.sum(0) + gemm(rows) * a(D).sum(0) + 1e-37), l
        S, ES = D @ W, ED @ a(W) + gemm(W.shape[0]) * ((a(D) + ED) @ a(W))
        if l:
            G, EG = gs[l - 1]
            ED = (ES * (a(G) + EG) + a(S) * EG) + 2.0 ** -23 * a(S * G)
            D = S * G
    assert np.all(a(dX - S) <= ES + 1e-37)
