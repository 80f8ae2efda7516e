"""The equation-of-state kernels at the edges of their species loops (pairs of species, four-wide tables, both
size classes): an odd and an even count, the largest of each class. Properties within 1e-10 of the oracle's
terms (1e-9 for c_p, as in the parity tests). The Jacobian against central differences of the oracle's step:
their truncation is O(1e-8) relative, FP32 tangents carry 2e-6 of the output spread."""
import numpy as np
import pytest

import synth
from oracle import pr_eos as ope
from oracle import step as ostep
from oracle.thermo import species_h_molar

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [5, 15, 16, 17, 31, 32])
def test_properties_and_jacobian(n):
    import torch
    import __graft_entry__ as g
    g.build()
    import paper_2508_18969_gb300 as df
    mech = synth.mechanism.make_mechanism(n, 1, 11)
    net = synth.network.make_network([n + 2, 64, 32, n], n, seed=n)
    T, p, Y = synth.fields.training_states(mech, 193, 5)[:3]
    dev = lambda a: torch.tensor(np.ascontiguousarray(a), device="cuda")
    host = lambda t: t.cpu().numpy().astype(np.float64)
    st = df.State(mech, net, T_react=0.0, batch_cells=256)
    rho, h, cp, Z = (host(t) for t in st.real_fluid_props(dev(T), dev(p), dev(Y)))
    o = ope.state(mech, T, p, Y)
    scale = np.sum(np.abs(Y * species_h_molar(mech.nasa, T) / mech.W[:, None]), axis=0) + np.abs(o["h_dep"] / o["W_mix"])
    np.testing.assert_allclose(Z, o["Z"], rtol=1e-10)
    np.testing.assert_allclose(rho, o["rho"], rtol=1e-10)
    np.testing.assert_allclose(cp, o["cp"], rtol=1e-9)
    assert np.max(np.abs(h - o["h"]) / scale) <= 1e-10
    k = 24
    J, dTn = (host(t) for t in st.chem_jacobian(dev(T[:k]), dev(p[:k]), dev(Y[:, :k])))
    Jf, dTf = ostep.chem_step_jacobian_fd(mech, net, T[:k], p[:k], Y[:, :k], dY_rel=1e-4, dY_min=1e-4)
    mask, tm = np.isfinite(Jf), np.isfinite(dTf)
    assert np.abs(J - Jf)[mask].max() <= 2e-6 + 1e-4 * np.abs(Jf[mask]).max()
    assert (np.abs(dTn - dTf)[tm] / (np.abs(dTf[tm]) + 1.0)).max() <= 1e-4
    st.close()
