"""Real-fluid properties where the cubic is delicate: on either side of a saturation line (which of two roots
has the least Gibbs energy), near the critical points and next to merging roots, and in the dilute limit,
with trace species down to 1e-60; the compressibility that the reaction step starts from, and the derivatives
of T' of a step that changes nothing.

Bounds. The mixing sums are good to 2^-42 of their terms, so the cubic's value at a root is off by at most
2^-41 of its terms' absolute sum S, the root by that over |f'(Z)|, and c_p, whose departure part goes with
1 / f'(Z), by f''(Z) / f'(Z) of the root's error, on top of 2^-40 of its terms. Near the saturation line the
roots' Gibbs energies differ by about |dp / p|, which FP64 resolves for p >= 1 kPa."""
import numpy as np
import pytest

import synth
from oracle import pr_eos as o
from oracle.thermo import species_h_molar

pytestmark = pytest.mark.gpu
TRACE = [0.0, 1e-30, 1e-38, 1e-45, 1e-60]
MECH = synth.mechanism.make_mechanism(9, 1, 3)


def _composition(rng, i):
    if i % 2:
        y = rng.dirichlet(np.full(MECH.n, 0.5))
        y[rng.integers(MECH.n)] = TRACE[i % 5]
        return y / y.sum()
    y = np.full(MECH.n, TRACE[(i // 2) % 5])
    y[rng.integers(MECH.n)] = 1.0
    return y


def _cubic(t, q, y):
    """(A, B, (c2, c1, c0)) at temperature t, pressures q and composition y."""
    q = np.atleast_1d(np.asarray(q, dtype=np.float64))
    X = np.repeat(o.mole_fractions(MECH.W, y[:, None])[0], len(q), 1)
    a, _, _, b = o.mixture_params(MECH, X, np.full(len(q), t))
    A, B = a * q / (o.R * t) ** 2, b * q / (o.R * t)
    return A, B, o.cubic_coefficients(A, B)


def _bisect(f, lo, hi):
    flo = f(lo)
    for _ in range(60):
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if f(mid) * flo > 0 else (lo, mid)
    return lo


def _crossing(y, t, value, lo):
    """First pressure above lo at which value(A, B, coefficients) changes sign, or None."""
    qs = np.logspace(np.log10(lo), 7.5, 200)
    v = value(*_cubic(t, qs, y))
    j = np.flatnonzero(v[:-1] * v[1:] < 0)
    return _bisect(lambda q: value(*_cubic(t, q, y))[0], qs[j[0]], qs[j[0] + 1]) if len(j) else None


def _gibbs_gap(A, B, c):
    r = o.cubic_real_roots(*c)
    three = np.isfinite(r[2]) & (r[0] > B)
    with np.errstate(all="ignore"):
        return np.where(three, o.gibbs_departure(r[0], A, B) - o.gibbs_departure(r[2], A, B), np.nan)


def _discriminant(A, B, c):
    P, Q = c[1] - c[0] ** 2 / 3, 2 * c[0] ** 3 / 27 - c[0] * c[1] / 3 + c[2]
    return (Q / 2) ** 2 + (P / 3) ** 3


def _states(kind):
    rng = np.random.default_rng({"saturation": 3, "critical": 4, "dilute": 5}[kind])
    out, i = [], 0
    while len(out) < 360:
        y, i = _composition(rng, i), i + 1
        Tpc = float((y / MECH.W * MECH.Tc).sum() / (y / MECH.W).sum())
        if kind == "saturation":
            t = Tpc * rng.uniform(0.35, 0.95)
            q = _crossing(y, t, _gibbs_gap, 1e3)
            out += [(t, q * (1 + s * e), y) for e in (1e-2, 1e-3, 1e-4) for s in (-1, 1)] if q else []
        elif kind == "critical" and i % 3:
            t = Tpc * rng.uniform(0.6, 0.98)
            q = _crossing(y, t, _discriminant, 1e3)
            out += [(t, q * (1 + s * e), y) for e in (1e-2, 1e-4, 1e-6) for s in (-1, 1)] if q else []
        elif kind == "critical":
            k, y = i % MECH.n, np.full(MECH.n, TRACE[i % 5])
            y[k] = 1.0
            e = 10.0 ** -rng.integers(1, 6)
            out += [(MECH.Tc[k] * (1 + a * e), MECH.pc[k] * (1 + b * e), y) for a in (-1, 1) for b in (-1, 1)]
        else:
            out.append((rng.uniform(250.0, 3000.0), 10 ** rng.uniform(-6.0, -2.0), y))
    T, p, Y = zip(*out)
    return np.array(T), np.array(p), np.ascontiguousarray(np.array(Y).T)


@pytest.mark.parametrize("kind", ["saturation", "critical", "dilute"])
def test_properties(kind):
    import torch
    import __graft_entry__ as g
    g.build()
    import paper_2508_18969_gb300 as df
    T, p, Y = _states(kind)
    net = synth.network.make_network([11, 32, 9], 9, seed=1)
    st = df.State(MECH, net, T_react=0.0, batch_cells=128)
    rho, h, cp, Z = (t.cpu().numpy() for t in st.real_fluid_props(*(torch.tensor(a, device="cuda") for a in (T, p, Y))))
    st.close()
    s = o.state(MECH, T, p, Y)
    A, B, Zo = s["A"], s["B"], s["Z"]
    if kind == "dilute":   # Z = 1 + B - A + O(p^2), the square below 1e-18
        assert np.max(np.abs(Z - (1.0 + (B - A)))) <= 2.0 ** -50
    terms = Zo ** 3 + (1 + B) * Zo ** 2 + (A + 3 * B ** 2 + 2 * B) * Zo + A * B + B ** 2 + B ** 3
    slope = np.abs(3 * Zo ** 2 - 2 * (1 - B) * Zo + A - 3 * B ** 2 - 2 * B)
    dZ = 2.0 ** -41 * terms / slope
    assert np.max(np.abs(Z - Zo) / (dZ + 2.0 ** -50 * Zo)) <= 1.0
    np.testing.assert_array_less(np.abs(rho / s["rho"] - 1), dZ / Zo + 2.0 ** -41)
    # dh/dZ at fixed T, p: R T + (T a' - a) / (2 sqrt2 b) d ln(ratio)/dZ
    pull = np.abs(T * s["da"] - s["a_m"]) / (2 * o.SQ2 * s["b_m"])
    dL = np.abs(1 / (Zo + (1 + o.SQ2) * B) - 1 / (Zo + (1 - o.SQ2) * B))
    h_abs = np.abs(s["h_ig"]) + np.abs(s["h_dep"] / s["W_mix"]) + pull * np.abs(o.log_ratio(Zo, B)) / s["W_mix"]
    h_abs += np.sum(np.abs(Y * species_h_molar(MECH.nasa, T)) / MECH.W[:, None], axis=0)
    assert np.max(np.abs(h - s["h"]) / ((o.R * T + pull * dL) / s["W_mix"] * dZ + 2.0 ** -40 * h_abs)) <= 1.0
    curve = np.abs(6 * Zo - 2 * (1 - B)) + 2 * (1 + B)
    dep = np.abs(s["cp"]) + o.R / s["W_mix"] * 10
    assert np.max(np.abs(cp - s["cp"]) / (dep * (2.0 ** -39 + 2 * curve * dZ / slope + 2 * dZ / (Zo - B)))) <= 1.0


def test_step_and_jacobian_next_to_saturation():
    """eos_pre's root is the one of least Gibbs energy: the other phase's Z is a factor off. With a network that
    changes nothing (du = 0), h(T', p, Y) = h(T, p, Y) and h, homogeneous of degree 1 in Y, give dT'/dT = 1 and
    dT'/dY_j = h / c_p; double-float errors of the root, by its slope, and of h's cancelling terms stay far
    below the bound, which a state of the other phase misses by its heat of evaporation."""
    import torch
    import __graft_entry__ as g
    g.build()
    import paper_2508_18969_gb300 as df
    T, p, Y = _states("saturation")
    net = synth.network.make_network([11, 32, 9], 9, seed=1)
    for W, b in zip(net.W, net.b):
        W[:], b[:] = 0, 0
    net.out_mean[:] = 0
    dev = [torch.tensor(a, device="cuda") for a in (T, p, Y)]
    s = o.state(MECH, T, p, Y)
    st = df.State(MECH, net, T_react=0.0, batch_cells=512)
    _, Z, _, status = (t.cpu().numpy() for t in st.eos_pre(*dev))
    assert not status.any()
    np.testing.assert_allclose(Z, s["Z"], rtol=1e-6)
    _, dT = (t.cpu().numpy() for t in st.chem_jacobian(*dev))
    st.close()
    np.testing.assert_allclose(dT[:, 0], 1.0, rtol=1e-6)
    scale = np.sum(np.abs(Y * species_h_molar(MECH.nasa, T)) / MECH.W[:, None], axis=0) + np.abs(s["h_dep"] / s["W_mix"])
    j = Y.argmax(0)   # (Box-Cox slopes are floored for trace species)
    off = np.abs(dT[np.arange(len(T)), 1 + j] - s["h"] / s["cp"]) * np.abs(s["cp"]) / scale
    assert off.max() <= 1e-6, off.max()


@pytest.mark.parametrize("kind", ["critical", "dilute"])
def test_jacobian_of_the_unchanged_cell(kind):
    """dT'/dT = 1 and dT'/dY_j = h / c_p (above) where c_p is ill conditioned: its bound of test_properties at both
    ends of the step, and its change over the error of T', 2^-40 of h's terms over c_p."""
    import torch
    import __graft_entry__ as g
    g.build()
    import paper_2508_18969_gb300 as df
    T, p, Y = _states(kind)
    net = synth.network.make_network([11, 32, 9], 9, seed=1)
    for W, b in zip(net.W, net.b):
        W[:], b[:] = 0, 0
    net.out_mean[:] = 0
    st = df.State(MECH, net, T_react=0.0, batch_cells=512)
    J, dT = (t.cpu().numpy() for t in st.chem_jacobian(*(torch.tensor(a, device="cuda") for a in (T, p, Y))))
    st.close()
    s = o.state(MECH, T, p, Y)
    A, B, Z, cp = s["A"], s["B"], s["Z"], np.abs(s["cp"])
    terms = Z ** 3 + (1 + B) * Z ** 2 + (A + 3 * B ** 2 + 2 * B) * Z + A * B + B ** 2 + B ** 3
    slope = np.abs(3 * Z ** 2 - 2 * (1 - B) * Z + A - 3 * B ** 2 - 2 * B)
    dZ = 2.0 ** -41 * terms / slope
    scale = np.sum(np.abs(Y * species_h_molar(MECH.nasa, T)) / MECH.W[:, None], axis=0) + np.abs(s["h_dep"] / s["W_mix"])
    bend = np.abs(o.state(MECH, T * (1 + 1e-7), p, Y)["cp"] - o.state(MECH, T * (1 - 1e-7), p, Y)["cp"]) / (2e-7 * T)
    rel = 2.0 ** -39 + 2 * (np.abs(6 * Z - 2 * (1 - B)) + 2 * (1 + B)) * dZ / slope + 2 * dZ / (Z - B)
    rel = 2 * rel * (1 + 10 * o.R / s["W_mix"] / cp) + 2.0 ** -40 * scale / cp * bend / cp
    assert np.all(np.abs(dT[:, 0] - 1) <= rel), np.max(np.abs(dT[:, 0] - 1) / rel)
    j = Y.argmax(0)
    off = np.abs(dT[np.arange(len(T)), 1 + j] - s["h"] / s["cp"])
    assert np.all(off <= (2.0 ** -39 + rel) * scale / cp), np.max(off / ((2.0 ** -39 + rel) * scale / cp))
