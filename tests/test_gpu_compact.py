"""The reacting-cell list at the edges of its launch rule: one block up to 16,384 cells (four or sixteen
cells a thread), two launches beyond, a third (the scan of chunk counts) beyond 2048 chunks. Exact."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 31, 4095, 4097, 16384, 16385, 20480, 2048 * 4096, 2048 * 4096 + 1])
def test_list_is_exact(n):
    import torch
    import __graft_entry__ as g
    g.build()
    import paper_2508_18969_gb300 as df
    import synth
    mech, net, _, _, _ = synth.configs.build("small-fp32-4k", n_cells=64)
    rng = np.random.default_rng(n)
    T = rng.uniform(100.0, 1200.0, n)
    T[rng.integers(0, n, 5)] = [np.nan, np.inf, -np.inf, 600.0, np.nextafter(600.0, 601.0)]
    st = df.State(mech, net, T_react=600.0, batch_cells=128)
    idx, cnt = st.active_compact(torch.tensor(T, device="cuda"))
    want = np.nonzero(T > 600.0)[0]
    assert int(cnt.item()) == want.size
    assert np.array_equal(idx[:want.size].cpu().numpy(), want)
    st.close()
