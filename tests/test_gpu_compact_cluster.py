"""The reacting-cell list of one cluster of blocks (16,385 to 32,768 cells): exact at the edges of a block's
range and of the rule, and with blocks that have no cell or no reacting cell. Exact."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [16385, 20479, 24577, 28673, 32767, 32768, 32769])
@pytest.mark.parametrize("cold", [False, True])
def test_cluster_list_is_exact(n, cold):
    import torch
    import __graft_entry__ as g
    g.build()
    import paper_2508_18969_gb300 as df
    import synth
    mech, net, _, _, _ = synth.configs.build("small-fp32-4k", n_cells=64)
    T = np.random.default_rng(n).uniform(100.0, 1200.0, n)
    if cold:
        T[4096:n - 3] = 300.0
    st = df.State(mech, net, T_react=600.0, batch_cells=128)
    idx, cnt = st.active_compact(torch.tensor(T, device="cuda"))
    want = np.nonzero(T > 600.0)[0]
    assert int(cnt.item()) == want.size
    assert np.array_equal(idx[:want.size].cpu().numpy(), want)
    st.close()
