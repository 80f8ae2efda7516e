"""Short launches of a low-precision network take a narrower pair tile where its waves cost less. The tile
does not enter an element's sum (the same products in the same order), so the outputs are the same bits as
those of the same rows in a long launch."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["DF_BF16", "DF_FP8_E4M3"])
def test_short_launches_give_the_same_bits(prec):
    import torch
    import __graft_entry__ as g
    g.build()
    import paper_2508_18969_gb300 as df
    mech, net, _, _, _ = synth.configs.build("layer1d-30sp-1m", n_cells=64)
    st = df.State(mech, net, precision=getattr(df, prec), batch_cells=40064)
    x = torch.tensor(np.random.default_rng(7).normal(size=(40011, net.widths[0])).astype(np.float32), device="cuda")
    want = st.mlp_forward(x)
    for n in (1, 255, 257, 1500, 3001, 6000, 9500, 12001):
        assert torch.equal(st.mlp_forward(x[:n]), want[:n]), n
    st.close()
