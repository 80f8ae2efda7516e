"""A cell's results do not depend on how many cells its launch holds, bit for bit, in any precision: short
launches take smaller equation-of-state blocks, other network tiles and the one-launch compaction. (The host
step, which cuts the cells into chunks, promises the device step's results.)"""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["DF_FP32", "DF_BF16", "DF_FP8_E4M3"])
@pytest.mark.parametrize("n,hidden", [(9, (256, 128, 64)), (17, (100, 60)), (31, (1600, 800, 96))])
def test_same_bits(prec, n, hidden):
    import __graft_entry__ as g
    g.build()
    import paper_2508_18969_gb300 as df
    N = 120_011
    mech = synth.mechanism.make_mechanism(n, 1, 3)
    net = synth.network.make_network([n + 2, *hidden, n], n, seed=2)
    T, p, Y = synth.fields.training_states(mech, N, 11)[:3]
    st = df.State(mech, net, precision=getattr(df, prec), T_react=600.0, batch_cells=N)
    Td, pd, Yd = (torch.tensor(a, device="cuda") for a in (T, p, Y))
    h0, Z, x, _ = st.eos_pre(Td, pd, Yd)
    O = st.mlp_forward(x)
    for m in (1, 130, 3001, 20011):
        assert torch.equal(O[:m], st.mlp_forward(x[:m].contiguous())), m
    m = 5001
    Tm, pm, Ym = Td[:m].clone(), pd[:m].clone(), Yd[:, :m].clone()
    for a, b in zip(st.eos_pre(Tm, pm, Ym), (h0, Z, x)):
        assert torch.equal(a, b[:m])
    st.eos_post(O[:m].contiguous(), h0[:m].contiguous(), Tm, pm, Ym)
    Tb, Yb = Td.clone(), Yd.clone()
    st.eos_post(O, h0, Tb, pd, Yb)
    assert torch.equal(Tm, Tb[:m]) and torch.equal(Ym, Yb[:, :m])
    st.chem_step(Td, pd, Yd)
    for chunk in (4001, 40_009):
        Th, ph, Yh = (torch.tensor(a).pin_memory() for a in (T, p, Y))
        st.chem_step_host(Th, ph, Yh, chunk_cells=chunk)
        torch.cuda.synchronize()
        assert torch.equal(Th, Td.cpu()) and torch.equal(Yh, Yd.cpu()), chunk
    st.close()
