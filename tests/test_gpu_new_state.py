"""A state or network that was just created (or has just grown its training buffers) used at once on a
non-blocking stream, which nothing orders behind the legacy stream: all set-up work has to be complete when
the call that does it returns. Compared bit for bit with the same call once the device is idle."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def df():
    import __graft_entry__ as g
    g.build()
    import paper_2508_18969_gb300 as m
    return m


@pytest.mark.parametrize("prec", ["DF_FP32", "DF_BF16", "DF_FP8_E4M3"])
def test_first_call_on_a_non_blocking_stream(df, prec):
    mech = synth.mechanism.make_mechanism(9, 1, 3)
    net = synth.network.make_network([11, 2048, 2048, 1024, 9], 9, seed=1)
    x = torch.randn(333, 11, device="cuda")
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    for _ in range(3):
        st = df.State(mech, net, precision=getattr(df, prec), batch_cells=65536)
        with torch.cuda.stream(side):
            first = st.mlp_forward(x)
        torch.cuda.synchronize()
        assert torch.equal(first, st.mlp_forward(x))
        torch.cuda.synchronize()
        st.close()


@pytest.mark.parametrize("prec", ["DF_FP32", "DF_BF16"])
def test_first_training_call_on_a_non_blocking_stream(df, prec):
    mech = synth.mechanism.make_mechanism(9, 1, 3)
    net = synth.network.make_network([11, 64, 4096, 9], 9, seed=1)
    x, dO = torch.randn(20011, 11, device="cuda"), torch.randn(20011, 9, device="cuda")
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    st = df.State(mech, net, precision=getattr(df, prec), batch_cells=128)
    st.mlp_forward_train(x[:1])          # masters and moments; the batch buffers grow below
    out = []
    for _ in range(2):
        torch.cuda.synchronize()
        with torch.cuda.stream(side):
            out.append([st.mlp_forward_train(x), st.mlp_backward(dO)])
        torch.cuda.synchronize()
        out[-1] += [t for l in range(3) for t in st.params(l, df._lib.DF_PARAM_GRADS, widths=net.widths)]
        torch.cuda.synchronize()
    for a, b in zip(*out):
        assert torch.equal(a, b)
    st.close()
