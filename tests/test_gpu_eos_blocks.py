"""The equation-of-state kernels in small blocks (launches that one wave of them holds) against the large
blocks of a big launch, on the same cells. Both run the same double-float operations, whose errors stay
below 1e-10 of the terms; the increment's FP32 power is good to 1e-6 of the increment, which the
renormalisation spreads over a cell's species."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu
BIG = 120001


@pytest.mark.parametrize("name", ["layer1d-30sp-1m", "small-fp32-4k"])
@pytest.mark.parametrize("n", [1, 63, 65, 4097, 40001])
def test_small_blocks_match_large(name, n):
    import torch
    import __graft_entry__ as g
    g.build()
    import paper_2508_18969_gb300 as df
    mech, net, T, p, Y = synth.configs.build(name, n_cells=4096)
    rep = lambda a, m: torch.tensor(np.ascontiguousarray(np.tile(a, m // 4096 + 1)[..., :m]), device="cuda")
    st = df.State(mech, net, batch_cells=BIG)
    out = []
    for m in (n, BIG):
        Tm, pm, Ym = rep(T, m), rep(p, m), rep(Y, m)
        h0, Z, x, s = st.eos_pre(Tm, pm, Ym)
        O = torch.sin(torch.arange(m * mech.n, device="cuda", dtype=torch.float32)).reshape(m, mech.n)
        Y0 = Ym.clone()
        s2 = st.eos_post(O, h0, Tm, pm, Ym)
        out.append([t[..., :n] for t in (h0, Z, s, s2, Tm, Ym, Y0)] + [x[:n]])
    (h0, Z, s, s2, T1, Y1, Y0, x), (H0, ZZ, S, S2, TT, YY, _, X) = out
    assert torch.equal(s, S) and torch.equal(s2, S2)
    torch.testing.assert_close(Z, ZZ, rtol=1e-10, atol=0)
    torch.testing.assert_close(h0, H0, rtol=1e-10, atol=1e-10 * float(H0.abs().max()))
    torch.testing.assert_close(x, X, rtol=1e-6, atol=2e-6)
    torch.testing.assert_close(T1, TT, rtol=1e-8, atol=0)
    inc = (YY - Y0).abs()
    assert torch.all((Y1 - YY).abs() <= 1e-6 * (inc + inc.sum(0, keepdim=True)) + 1e-13 * YY)
    st.close()
