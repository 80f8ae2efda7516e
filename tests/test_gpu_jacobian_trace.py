"""Jacobian of the step with positive mass fractions below FP32's normal range (1.2e-38) and below the point
where a double-float pair loses its low part (1e-31): their Box-Cox root Y^lambda is 2e-4 to 0.3, so they
count like any other species. Against the formulas in FP64 with the oracle's network.

Bound: the network and its tangents are FP32 (2e-6 of their absolute terms), an error e of the base
Y^lambda + lambda du (lambda du ~ 0.35 to FP32: e <= 4e-7) moves base^(m - 1) by (m - 1) e / base, m <= 64,
base >= 0.2: below 1e-3 of the absolute terms in all."""
import numpy as np
import pytest

import synth
from oracle import network as onw

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [10, 64])
@pytest.mark.parametrize("n", [5, 18])
def test_trace_species(m, n):
    import torch
    import __graft_entry__ as g
    g.build()
    import paper_2508_18969_gb300 as df
    lam = 1.0 / m
    mech = synth.mechanism.make_mechanism(n, 1, 3)
    net = synth.network.make_network([n + 2, 32, n], n, seed=4, lam=lam)
    net.in_mean[2:], net.in_std[2:] = -0.5 * m, 0.25 * m
    net.out_mean[:], net.out_std[:] = 0.35 * m, 0.05 * m
    rng = np.random.default_rng(n)
    N = 64
    Y = rng.dirichlet(np.full(n, 1.0), N).T
    Y[0] = np.array([1e-31, 1e-35, 1e-38, 1e-40])[np.arange(N) % 4]
    Y[-1, ::5] = 0.0
    Y = np.ascontiguousarray(Y / Y.sum(0))
    T, p = rng.uniform(900.0, 2500.0, N), rng.uniform(6e6, 1.5e7, N)
    st = df.State(mech, net, T_react=0.0, batch_cells=128)
    status = torch.empty(N, dtype=torch.int32, device="cuda")   # (large changes: some T' leave the bracket)
    st.chem_step(*(torch.tensor(a, device="cuda") for a in (T, p, Y)), status=status)
    ok = status.cpu().numpy() == 0
    J, dT = (t.cpu().numpy().astype(np.float64) for t in st.chem_jacobian(*(torch.tensor(a, device="cuda") for a in (T, p, Y))))
    st.close()
    x = onw.normalise_inputs(net, T, p, Y)
    O, (z0, _) = onw.mlp_forward(net, x, return_pre=True)
    G = onw.gelu_tanh_grad(z0)
    # dv_t/dx and the network's tangents [N, n, n + 1] with their absolute sums
    bc = np.maximum(Y, 1e-12) ** (lam - 1.0)
    sc = np.concatenate([np.full((1, N), 1.0 / net.in_std[0]), bc / net.in_std[2:, None]]).T
    cols = [0] + list(range(2, n + 2))
    def tangents(f):
        return np.einsum("ko,no,oc,nc->nkc", f(net.W[1]), f(G), f(net.W[0][:, cols]), sc)
    own = np.zeros((N, n, n + 1))
    own[:, np.arange(n), 1 + np.arange(n)] = bc.T
    ju = net.out_std[:, None] * tangents(lambda a: a) + own
    ja = net.out_std[:, None] * tangents(np.abs) + own
    base = (np.where(Y > 0, Y, 0.0) ** lam + lam * (net.out_std[:, None] * O.T + net.out_mean[:, None])).T
    assert base.min() > 0.2
    zl = base ** (m - 1)
    S = (zl * base).sum(1)[:, None, None]
    Yp = (zl * base)[:, :, None] / S
    def columns(u):
        return zl[:, :, None] * u / S, Yp * np.einsum("nk,nkc->nc", zl, u)[:, None, :] / S
    a, b = columns(ju)
    aa, ba = columns(ja)
    eye = np.zeros((n, n + 1))
    eye[np.arange(n), 1 + np.arange(n)] = 1.0
    err = np.abs(J - (a - b - eye))
    tol = 1e-3 * (aa + ba) + 2.0 ** -23 * eye + 1e-37
    assert ok.sum() >= 4 and np.array_equal(np.isfinite(dT).all(1), ok)
    assert np.all(err[ok] <= tol[ok]), np.max((err / tol)[ok], axis=(0, 2))
