"""Workloads for timing the library through its Python binding, with inputs made on the GPU from a
seed and an FP64 evaluation of the same quantities in plain torch.

The sizes are those of the repository's named workloads (synth/configs.py, bench.py) and of its
tests: the 9-species network 11-256-128-64-9 on 4096 cells, the 30-species network
32-1600-800-400-30 up to 2^20 cells per batch, property networks of hidden widths 2048-1024-512
and 1024-512-256, sparse systems of 64^3 to 100^3 cells in block rows of 512, and odd sizes in
between (a rank's part of a decomposed mesh is never a round number).

A case is a dict of plain values:
  kind    what is called: "step" (State.chem_step), "net" (State.mlp_forward), "grad"
          (State.mlp_forward_train + mlp_backward), "train" (State.train_step), "jac"
          (State.chem_jacobian), "prop" (PropNet.infer), "eos" (State.real_fluid_props), "solver"
          (Solver.fv_laplacian + convert + gauss_seidel + residual)
  n       cells, rows or states;  net: network size, "small" (9 species) or "large" (30 species),
          for "prop" "density" or "transport";  prec: "fp32", "bf16" or "fp8";  field: which states
"""
from __future__ import annotations

import functools
import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_2508_18969_gb300 as df

R = 8.31446261815324
SQ2 = math.sqrt(2.0)
NETS = {
    "small": (9, (11, 256, 128, 64, 9)),
    "large": (30, (32, 1600, 800, 400, 30)),
    "density": (30, (32, 1024, 512, 256, 1)),
    "transport": (30, (32, 2048, 1024, 512, 4)),
}
PREC = {"fp32": df.DF_FP32, "bf16": df.DF_BF16, "fp8": df.DF_FP8_E4M3}
LAM = 0.1
F64 = torch.float64


def listed():
    return [
        # one step of a small flame on the default (FP32) precision: the smallest call, latency
        {"name": "step_small_fp32_4k", "kind": "step", "net": "small", "prec": "fp32",
         "field": "uniform", "n": 4096},
        # a rank's share of a decomposed mesh: an odd number of cells, well below one full batch
        {"name": "step_bf16_20k", "kind": "step", "net": "large", "prec": "bf16",
         "field": "layer", "n": 20011},
        # the headline step: a 2^20-cell mixing layer, every cell through the network
        {"name": "step_bf16_1m", "kind": "step", "net": "large", "prec": "bf16",
         "field": "layer", "n": 1 << 20},
        # a partly reacting field (30 % hot cells) in FP8: compaction, several batches, the largest
        # field
        {"name": "step_fp8_react_4m", "kind": "step", "net": "large", "prec": "fp8",
         "field": "reacting", "n": 4000037},
        # the network alone at the default precision, an ordinary batch of rows
        {"name": "net_fp32_131k", "kind": "net", "net": "large", "prec": "fp32", "n": 131072},
        # the network on a few thousand rows (ragged last tile), as a caller's own model has it
        {"name": "net_bf16_3k", "kind": "net", "net": "large", "prec": "bf16", "n": 3001},
        # one Adam step of the training recipe (bench.py --mode train: 65,536 states)
        {"name": "train_bf16_64k", "kind": "train", "net": "large", "prec": "bf16", "n": 65536},
        # forward and backward of the differentiable network op in FP32, an odd batch
        {"name": "grad_fp32_10k", "kind": "grad", "net": "large", "prec": "fp32", "n": 10007},
        # Jacobians of the step (implicit coupling, sensitivities) of a block of cells
        {"name": "jac_bf16_20k", "kind": "jac", "net": "large", "prec": "bf16",
         "field": "training", "n": 20000},
        # temperature and transport properties from the property network
        {"name": "prop_bf16_200k", "kind": "prop", "net": "transport", "prec": "bf16", "n": 200003},
        # density, enthalpy, heat capacity and Z of a field: what a flow solver asks each step
        {"name": "eos_props_260k", "kind": "eos", "net": "large", "prec": "fp32",
         "field": "layer", "n": 262144},
        # one transport-equation solve: assembly, conversion, two Gauss-Seidel sweeps, residual
        {"name": "solver_1m", "kind": "solver", "nx": 101, "ny": 99, "nz": 100, "part": 512, "n": 999900},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "net", "net", "grad", "train", "jac", "prop", "eos", "solver"])
    if kind == "solver":
        d = [_log_int(rng, 20, 95) for _ in range(3)]
        return {"kind": kind, "nx": d[0], "ny": d[1], "nz": d[2], "part": rng.choice([256, 512, 1024]),
                "n": d[0] * d[1] * d[2]}
    c = {"kind": kind, "net": rng.choice(["small", "large", "large"])}
    c["prec"] = rng.choice({"step": ["fp32", "bf16", "fp8"], "net": ["fp32", "bf16", "fp8"],
                            "grad": ["fp32", "bf16"], "train": ["fp32", "bf16"],
                            "jac": ["fp32", "bf16"], "prop": ["fp32", "bf16"], "eos": ["fp32"]}[kind])
    if kind == "prop":
        c["net"] = rng.choice(["density", "transport"])
    if kind in ("step", "jac", "eos"):
        c["field"] = rng.choice(["uniform", "layer", "training"] + (["reacting"] if kind == "step" else []))
    top = {"step": 900000, "net": 500000, "grad": 60000, "train": 65000, "jac": 20000,
           "prop": 200000, "eos": 300000}[kind]
    if c["prec"] == "fp32" and kind != "eos":
        top //= 6
    c["n"] = _log_int(rng, 300, top)
    return c


# ---------------------------------------------------------------- mechanism, networks, fields

@functools.lru_cache(maxsize=None)
def _mech(n):
    """A C/H/O mechanism of the recipe of synth/mechanism.py (its own draws)."""
    rng = np.random.default_rng(20250818 + n)
    pool = [(x, y, z) for x in range(3) for y in range(5) for z in range(3) if x + y + z]
    fixed = [(0, 0, 2), (1, 4, 0), (0, 2, 1), (1, 0, 2)]   # O2, CH4, H2O, CO2
    rest = [c for c in pool if c not in fixed]
    comp = np.array(fixed + [rest[i] for i in rng.permutation(len(rest))[: n - 4]], dtype=np.float64)
    k = np.triu(rng.uniform(0.0, 0.1, (n, n)).astype(np.float32).astype(np.float64), 1)
    nasa = np.zeros((n, 7))
    nasa[:, 0] = rng.uniform(3.5, 6.0, n)
    nasa[:, 1] = rng.uniform(0.0, 2.0e-3, n)
    nasa[:, 2] = rng.uniform(-4.0e-8, 4.0e-8, n)
    nasa[:, 3] = rng.uniform(-4.0e-12, 4.0e-12, n)
    nasa[:, 4] = rng.uniform(-4.0e-16, 4.0e-16, n)
    nasa[:, 5] = rng.uniform(-20000.0, 30000.0, n)
    nasa[:4, 5] = (-1000.0, -10000.0, -30000.0, -48000.0)
    nasa[:, 6] = rng.uniform(-5.0, 12.0, n)
    return SimpleNamespace(n=n, W=comp @ np.array([12.011, 1.008, 15.999]) * 1e-3,
                           Tc=rng.uniform(100.0, 800.0, n), pc=rng.uniform(2.0e6, 10.0e6, n),
                           omega=rng.uniform(0.0, 0.4, n), kij=k + k.T, nasa=nasa)


@functools.lru_cache(maxsize=None)
def _net(name):
    """Xavier-uniform weights and small biases, exact in binary32; Z-score constants as
    synth/network.py states them (a property network reads h in place of T)."""
    n, widths = NETS[name]
    rng = np.random.default_rng(20250820 + sum(widths))
    W, b = [], []
    for i, o in zip(widths[:-1], widths[1:]):
        lim = math.sqrt(6.0 / (i + o))
        W.append(rng.uniform(-lim, lim, (o, i)).astype(np.float32).astype(np.float64))
        b.append(rng.uniform(-0.05, 0.05, o).astype(np.float32).astype(np.float64))
    prop = name in ("density", "transport")
    first = (0.0, 2.0e6) if prop else (1500.0, 1000.0)
    m = widths[-1]
    return SimpleNamespace(widths=list(widths), W=W, b=b, lam=LAM, dt=1e-7,
                           in_mean=np.r_[first[0], 12.5e6, np.full(n, -4.0)],
                           in_std=np.r_[first[1], 5.0e6, np.full(n, 3.0)],
                           out_mean=np.zeros(m), out_std=np.full(m, 1.0 if prop else 1e-3))


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _uniform(g, n, lo=0.0, hi=1.0):
    return torch.rand(n, generator=g, device="cuda", dtype=F64) * (hi - lo) + lo


def _fields(mech, field, N, g):
    """(T, p, Y) of synth/fields.py's recipes: states along a mixing-and-burning line of O2 and
    CH4, minor species log-uniform."""
    n, W = mech.n, mech.W
    burn = lambda z: torch.exp(-(((z - 0.2) / 0.1) ** 2))
    p = torch.full((N,), 10.0e6, device="cuda", dtype=F64)
    T = None
    if field == "uniform":
        zf, c = _uniform(g, N), _uniform(g, N)
        T, p = _uniform(g, N, 100.0, 3500.0), _uniform(g, N, 5.0e6, 20.0e6)
    elif field == "reacting":
        hot = _uniform(g, N) < 0.3
        zf = torch.where(hot, _uniform(g, N, 0.07, 0.33), _uniform(g, N))
        c = torch.where(hot, burn(zf), torch.zeros_like(zf))
    else:
        if field == "layer":
            x = -1.0 + (torch.arange(N, device="cuda", dtype=F64) + 0.5) * (2.0 / N)
        else:
            x, p = _uniform(g, N, -1.0, 1.0), _uniform(g, N, 5.0e6, 20.0e6)
        zf = 0.5 * (1.0 + torch.tanh(x / 0.1))
        c = burn(zf)
    if T is None:
        mix = 100.0 * (1.0 - zf) + 150.0 * zf
        T = mix + c * (3500.0 - mix)
    Y = torch.zeros(n, N, device="cuda", dtype=F64)
    s = 2.0 * W[0] / W[1]
    m = c * torch.minimum(zf, (1.0 - zf) / s)
    Y[0], Y[1] = 1.0 - zf - s * m, zf - m
    Y[2], Y[3] = m * (2.0 * W[2] / W[1]), m * (W[3] / W[1])
    Y[4:] = 10.0 ** (torch.rand(n - 4, N, generator=g, device="cuda", dtype=F64) * 5.0 - 8.0)
    Y.clamp_(min=0.0)
    Y /= Y.sum(0, keepdim=True)
    return T, p, Y


def _rows(widths, N, g):
    """Normalised network inputs, O(1) values."""
    return torch.randn(N, widths[0], generator=g, device="cuda", dtype=torch.float32).clamp_(-2.5, 2.5)


def _target(Y, g):
    """States a little later: the Box-Cox coordinates moved by O(1e-3)."""
    u = Y ** LAM + LAM * 1e-3 * torch.randn(Y.shape, generator=g, device="cuda", dtype=F64)
    Yt = u.clamp_(min=0.0) ** (1.0 / LAM)
    return Yt / Yt.sum(0, keepdim=True)


def _mesh(case, seed):
    """The mesh recipe of synth/mesh.py: a hexahedral grid with extra diagonal faces, numbered at
    random, faces in LDU order. Returns host (owner, neighbour) int32 and the face scale."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    n = nx * ny * nz
    g = _gen(seed)
    i = torch.arange(n, device="cuda").reshape(nz, ny, nx)
    pairs = [(i[:, :, :-1], i[:, :, 1:], 1.0), (i[:, :-1], i[:, 1:], 1.0), (i[:-1], i[1:], 1.0)]
    for a, b in ((i[:, :-1, :-1], i[:, 1:, 1:]), (i[:-1, :, :-1], i[1:, :, 1:]), (i[:-1, :-1], i[1:, 1:])):
        keep = torch.rand(a.shape, generator=g, device="cuda") < 0.15
        pairs.append((a[keep], b[keep], 0.3))
    a = torch.cat([q[0].reshape(-1) for q in pairs])
    b = torch.cat([q[1].reshape(-1) for q in pairs])
    w = torch.cat([torch.full((q[0].numel(),), q[2], device="cuda", dtype=F64) for q in pairs])
    new = torch.randperm(n, generator=g, device="cuda")
    a, b = new[a], new[b]
    own, nei = torch.minimum(a, b), torch.maximum(a, b)
    order = torch.argsort(own * n + nei)
    to = lambda t: t[order].to(torch.int32).cpu().numpy()
    return to(own), to(nei), w[order].cpu().numpy()


# ---------------------------------------------------------------- prepare and run

def _inputs(case, seed):
    """The inputs of a case on the GPU (host arrays for the mesh)."""
    kind, g = case["kind"], _gen(seed)
    if kind == "solver":
        own, nei, w = _mesh(case, seed)
        n = case["n"]
        new, pp = df.mesh_decompose(n, own, nei, max(1, n // case["part"]))
        own, nei, old, _ = df.mesh_renumber(n, own, nei, new)
        w = torch.from_numpy(w[old]).cuda()
        rn = lambda k: torch.randn(k, generator=g, device="cuda", dtype=F64)
        return dict(own=own, nei=nei, pp=pp, g=w * torch.exp(0.5 * rn(own.size)),
                    s=0.5 * torch.exp(0.3 * rn(n)), b=rn(n), x0=0.1 * rn(n))
    n, widths = NETS[case["net"]]
    if kind in ("net", "grad"):
        d = dict(x=_rows(widths, case["n"], g))
        if kind == "grad":
            d["dO"] = torch.randn(case["n"], widths[-1], generator=g, device="cuda",
                                  dtype=torch.float32) / case["n"]
        return d
    T, p, Y = _fields(_mech(n), case.get("field", "training"), case["n"], g)
    d = dict(T=T, p=p, Y=Y)
    if kind == "train":
        d["Yt"] = _target(Y, g)
    elif kind == "prop":
        d["h"] = 2.0e6 * torch.randn(case["n"], generator=g, device="cuda", dtype=F64)
    return d


def prepare(case, seed):
    kind, s = case["kind"], _inputs(case, seed)
    s["kind"] = kind
    if kind == "solver":
        s["S"] = df.Solver(case["n"], s.pop("own"), s.pop("nei"), s.pop("pp"))
        s["x"] = torch.empty_like(s["x0"])
        return s
    net = _net(case["net"])
    prec = PREC[case["prec"]]
    s["widths"] = net.widths
    if kind == "prop":
        s["st"] = df.PropNet(net, precision=prec)
        return s
    # a state's batch: the library's default for field steps, the caller's batch otherwise
    batch = 0 if kind == "step" else min(1 << 20, max(case["n"], 128))
    s["st"] = df.State(_mech(NETS[case["net"]][0]), net, precision=prec, batch_cells=batch,
                       T_react=600.0 if case.get("field") == "reacting" else 0.0)
    if kind == "step":
        s["T1"], s["Y1"] = torch.empty_like(s["T"]), torch.empty_like(s["Y"])
        s["status"] = torch.empty(case["n"], dtype=torch.int32, device="cuda")
    return s


def run(s):
    kind = s["kind"]
    if kind == "step":
        # the flow solver hands over its fields, the step works on them in place
        s["T1"].copy_(s["T"])
        s["Y1"].copy_(s["Y"])
        s["st"].chem_step(s["T1"], s["p"], s["Y1"], status=s["status"])
        return s["T1"], s["Y1"], s["status"]
    if kind == "net":
        return s["st"].mlp_forward(s["x"])
    if kind == "grad":
        st = s["st"]
        O = st.mlp_forward_train(s["x"])
        dX = st.mlp_backward(s["dO"])
        return O, dX, _grads(s)
    if kind == "train":
        loss = s["st"].train_step(s["T"], s["p"], s["Y"], s["Yt"], lr=1e-4)
        return loss, _grads(s)
    if kind == "jac":
        return s["st"].chem_jacobian(s["T"], s["p"], s["Y"])
    if kind == "prop":
        return s["st"].infer(s["h"], s["p"], s["Y"])
    if kind == "eos":
        return s["st"].real_fluid_props(s["T"], s["p"], s["Y"])
    S = s["S"]
    lo, dg, up = S.fv_laplacian(s["g"], s["s"])
    S.convert(lo, dg, up)
    s["x"].copy_(s["x0"])
    S.gauss_seidel(s["b"], s["x"], 2)
    return dg, s["x"], S.residual(s["b"], s["x"])


def _grads(s):
    return [s["st"].params(l, df._lib.DF_PARAM_GRADS, widths=s["widths"]) for l in range(len(s["widths"]) - 1)]


def work(case):
    kind, N = case["kind"], case["n"]
    if kind == "solver":
        nx, ny, nz = case["nx"], case["ny"], case["nz"]
        f = (nx - 1) * ny * nz + nx * (ny - 1) * nz + nx * ny * (nz - 1)
        f += 0.15 * ((nx - 1) * (ny - 1) * nz + (nx - 1) * ny * (nz - 1) + nx * (ny - 1) * (nz - 1))
        # assembly, conversion, two sweeps, residual: each matrix value, column and vector once
        return {"bytes": 16 * f + 24 * N + 16 * f + 16 * N + 3 * (20 * f + 32 * N),
                "flops": 2 * f + 3 * (4 * f + 2 * N)}
    n, widths = NETS[case["net"]]
    mac = sum(i * o for i, o in zip(widths[:-1], widths[1:]))
    par = 4 * mac
    eos = 2 * n * (n - 1) + 30 * n + 150   # one real-fluid state
    if kind == "net":
        return {"bytes": 4 * N * (widths[0] + widths[-1]) + par, "flops": 2 * mac * N}
    if kind == "grad":
        return {"bytes": 4 * N * (2 * widths[0] + 2 * widths[-1]) + 2 * par, "flops": 6 * mac * N}
    if kind == "train":   # weights, moments and gradients once, no input gradient
        return {"bytes": 16 * N * (n + 1) + 7 * par,
                "flops": (6 * mac - 2 * widths[0] * widths[1]) * N + eos * N}
    if kind == "prop":
        return {"bytes": 8 * N * (n + 2 + widths[-1]) + par, "flops": 2 * mac * N}
    if kind == "eos":
        return {"bytes": 8 * N * (n + 2 + 4), "flops": eos * N}
    if kind == "jac":
        return {"bytes": N * (8 * (n + 2) + 4 * n * (n + 1) + 8 * (n + 1)),
                "flops": (2 * mac + (n + 1) * 2 * (mac - widths[0] * widths[1])) * N + 6 * eos * N}
    a = 0.3 if case["field"] == "reacting" else 1.0
    return {"bytes": 8 * N + a * N * 16 * (n + 1) + 4 * N, "flops": a * N * (2 * mac + 3 * eos)}


# ---------------------------------------------------------------- the same in FP64

def _gelu(z):
    t = torch.tanh(0.7978845608028654 * (z + 0.044715 * z ** 3))
    return 0.5 * z * (1.0 + t)


def _dgelu(z):
    c = 0.7978845608028654
    t = torch.tanh(c * (z + 0.044715 * z ** 3))
    return 0.5 * (1.0 + t) + 0.5 * z * (1.0 - t * t) * c * (1.0 + 3 * 0.044715 * z * z)


def _dev(net):
    t = lambda a: torch.from_numpy(np.asarray(a)).cuda()
    return [t(w) for w in net.W], [t(b) for b in net.b]


def _mlp(W, b, x, chunk=65536):
    out = []
    for x0 in x.split(chunk):
        for l in range(len(W)):
            x0 = torch.addmm(b[l], x0, W[l].T)
            if l + 1 < len(W):
                x0 = _gelu(x0)
        out.append(x0)
    return torch.cat(out)


def _norm_in(net, first, p, Y):
    t = lambda a: torch.from_numpy(np.asarray(a)).cuda()
    x = torch.cat([first[None], p[None], (Y.clamp(min=0.0) ** LAM - 1.0) / LAM])
    return ((x - t(net.in_mean)[:, None]) / t(net.in_std)[:, None]).T.contiguous()


def _composition(mech, Y):
    """Composition sums of the Peng-Robinson mixture and of the ideal-gas enthalpy."""
    t = lambda a: torch.from_numpy(np.asarray(a)).cuda()[:, None]
    inv = (Y / t(mech.W)).sum(0)
    X = Y / t(mech.W) / inv
    sac = np.sqrt(0.45724 * R ** 2 * mech.Tc ** 2 / mech.pc)
    kap = 0.37464 + 1.54226 * mech.omega - 0.26992 * mech.omega ** 2
    K = torch.from_numpy(1.0 - mech.kij).cuda()
    u, v = X * t(sac * (1.0 + kap)), X * t(sac * kap / np.sqrt(mech.Tc))
    Ku, Kv = K @ u, K @ v
    c = mech.nasa[:, [5, 0, 1, 2, 3, 4]] * R / np.array([1.0, 1.0, 2.0, 3.0, 4.0, 5.0])
    e = [(Y * t(c[:, j] / mech.W)).sum(0) for j in range(6)]
    return dict(inv=inv, b=(X * t(0.07780 * R * mech.Tc / mech.pc)).sum(0), e=e,
                A0=(u * Ku).sum(0), A1=(u * Kv).sum(0), A2=(v * Kv).sum(0))


def _root(A, B):
    """The real root above B of least departure Gibbs energy."""
    c2, c1, c0 = B - 1.0, A - 3 * B * B - 2 * B, B * B + B ** 3 - A * B
    P = c1 - c2 * c2 / 3.0
    Q = 2.0 * c2 ** 3 / 27.0 - c2 * c1 / 3.0 + c0
    disc = (Q / 2) ** 2 + (P / 3) ** 3
    w = -Q / 2 - torch.where(Q >= 0, 1.0, -1.0) * torch.sqrt(disc.clamp(min=0.0))
    u = torch.sign(w) * w.abs() ** (1.0 / 3.0)
    one = torch.where(u != 0, u - P / (3.0 * u), torch.zeros_like(u))
    m = 2.0 * torch.sqrt((-P / 3.0).clamp(min=1e-300))
    phi = torch.arccos((3.0 * Q / (P * m)).clamp(-1.0, 1.0))
    best, gb = torch.full_like(A, math.nan), torch.full_like(A, math.inf)
    for k in range(3):
        three = m * torch.cos(phi / 3.0 - 2.0 * math.pi * k / 3.0)
        Z = torch.where(disc > 0, one, three) - c2 / 3.0
        for _ in range(8):
            f, fp = ((Z + c2) * Z + c1) * Z + c0, (3.0 * Z + 2.0 * c2) * Z + c1
            Zn = Z - f / torch.where(fp == 0, torch.ones_like(fp), fp)
            less = (((Zn + c2) * Zn + c1) * Zn + c0).abs() < f.abs()
            Z = torch.where(less, Zn, Z)
        g = Z - 1.0 - torch.log(Z - B) - A / (2 * SQ2 * B) * torch.log((Z + (1 + SQ2) * B) / (Z + (1 - SQ2) * B))
        ok = (Z > B) & ((disc <= 0) | (k == 0)) & (g < gb - 1e-12)
        best, gb = torch.where(ok, Z, best), torch.where(ok, g, gb)
    return best


def _state(m, T, p):
    """(h, Z) at (T, p) of the composition m, differentiable (the root through one Newton step
    of the cubic from its detached value)."""
    am = m["A0"] - 2.0 * m["A1"] * torch.sqrt(T) + m["A2"] * T
    da = m["A2"] - m["A1"] / torch.sqrt(T)
    A, B = am * p / (R * T) ** 2, m["b"] * p / (R * T)
    with torch.no_grad():
        Z0 = _root(A, B)
        slope = 3 * Z0 * Z0 - 2 * (1 - B) * Z0 + A - 3 * B * B - 2 * B
    Z = Z0 - (((Z0 + B - 1.0) * Z0 + A - 3 * B * B - 2 * B) * Z0 + B * B + B ** 3 - A * B) / slope
    L = torch.log((Z + (1 + SQ2) * B) / (Z + (1 - SQ2) * B))
    hd = R * T * (Z - 1.0) + (T * da - am) / (2 * SQ2 * m["b"]) * L
    h = hd * m["inv"]
    for j in range(6):
        h = h + m["e"][j] * T ** j
    return h, Z


def _h_cp(m, T, p):
    with torch.enable_grad():
        Tg = T.detach().clone().requires_grad_(True)
        h, Z = _state(m, Tg, p)
        cp, = torch.autograd.grad(h.sum(), Tg)
    return h.detach(), cp, Z.detach()


def _solve_T(m, p, h0, T):
    lo, hi = torch.full_like(T, 50.0), torch.full_like(T, 5000.0)
    T = T.clamp(50.0, 5000.0)
    for _ in range(80):
        h, cp, _ = _h_cp(m, T, p)
        f = h - h0
        hi, lo = torch.where(f >= 0, T, hi), torch.where(f < 0, T, lo)
        Tn = T - f / cp
        small = (Tn - T).abs() <= 1e-13 * T
        Tn = torch.where(small | ((Tn > lo) & (Tn < hi)), Tn, 0.5 * (lo + hi))
        T = Tn
        if bool(small.all()):
            break
    return T


def _new_Y(net, Y, O):
    sd = torch.from_numpy(net.out_std).cuda()[:, None]
    u = (Y.clamp(min=0.0) ** LAM + LAM * sd * O.T).clamp(min=0.0)
    z = u ** (1.0 / LAM)
    return z / z.sum(0), u


def exact(case, seed):
    s, kind = _inputs(case, seed), case["kind"]
    if kind == "solver":
        return _exact_solver(s, case["n"])
    net = _net(case["net"])
    mech = _mech(NETS[case["net"]][0])
    W, b = _dev(net)
    if kind == "net":
        return _mlp(W, b, s["x"].double())
    if kind == "prop":
        return _mlp(W, b, _norm_in(net, s["h"], s["p"], s["Y"])).T.contiguous()
    if kind == "grad":
        return _exact_grad(W, b, s["x"].double(), lambda O: s["dO"].double(), True)
    T, p, Y = s["T"], s["p"], s["Y"]
    if kind == "train":
        sd = torch.from_numpy(net.out_std).cuda()
        Oh = ((s["Yt"] ** LAM - Y ** LAM) / LAM).T / sd
        B = Y.shape[1]
        O, _, gr = _exact_grad(W, b, _norm_in(net, T, p, Y), lambda O: 2.0 * (O - Oh) / B, False)
        return ((O - Oh) ** 2).sum().reshape(1) / B, gr
    if kind == "eos":
        m = _composition(mech, Y)
        h, cp, Z = _h_cp(m, T, p)
        return p / (m["inv"] * Z * R * T), h, cp, Z
    if kind == "jac":
        return _exact_jac(mech, net, W, b, T, p, Y)
    live = T > (600.0 if case["field"] == "reacting" else 0.0)
    Tl, pl, Yl = T[live], p[live], Y[:, live]
    h0, _ = _state(_composition(mech, Yl), Tl, pl)
    Yn, _ = _new_Y(net, Yl, _mlp(W, b, _norm_in(net, Tl, pl, Yl)))
    T, Y = T.clone(), Y.clone()
    T[live] = _solve_T(_composition(mech, Yn), pl, h0, Tl)
    Y[:, live] = Yn
    return T, Y, None


def _exact_grad(W, b, x, dO_of, want_dx, chunk=32768):
    """(O, dx or None, [(dW, db)]) of the network with output gradient dO_of(O)."""
    O = _mlp(W, b, x)
    dO = dO_of(O)
    gr = [(torch.zeros_like(w), torch.zeros_like(v)) for w, v in zip(W, b)]
    dxs = []
    for x0, d in zip(x.split(chunk), dO.split(chunk)):
        H, Zs = [x0], []
        for l in range(len(W)):
            Zs.append(torch.addmm(b[l], H[-1], W[l].T))
            H.append(_gelu(Zs[-1]))
        for l in reversed(range(len(W))):
            gr[l][0].addmm_(d.T, H[l])
            gr[l][1].add_(d.sum(0))
            d = d @ W[l]
            if l:
                d = d * _dgelu(Zs[l - 1])
        dxs.append(d)
    return O, torch.cat(dxs) if want_dx else None, gr


def _exact_jac(mech, net, W, b, T, p, Y, chunk=2500):
    n, N = Y.shape
    isd = 1.0 / torch.from_numpy(net.in_std).cuda()
    osd = torch.from_numpy(net.out_std).cuda()
    Js, dTs = [], []
    for c0 in range(0, N, chunk):
        Tc, pc, Yc = T[c0:c0 + chunk], p[c0:c0 + chunk], Y[:, c0:c0 + chunk].contiguous()
        M = Tc.shape[0]
        bcp = Yc.clamp(min=1e-12) ** (LAM - 1.0)                       # [n, M]
        x = _norm_in(net, Tc, pc, Yc)
        t = torch.zeros(M, n + 1, n + 2, device="cuda", dtype=F64)      # dx/dv
        t[:, 0, 0] = isd[0]
        k = torch.arange(n, device="cuda")
        t[:, 1 + k, 2 + k] = bcp.T * isd[2:]
        for l in range(len(W)):
            z = torch.addmm(b[l], x, W[l].T)
            t = t @ W[l].T
            if l + 1 < len(W):
                t, x = t * _dgelu(z)[:, None, :], _gelu(z)
        Yn, u = _new_Y(net, Yc, z)
        S = (u ** (1.0 / LAM)).sum(0)
        ju = t * osd                                                    # d(BC coordinate)/dv [M, n+1, n]
        ju[:, 1 + k, k] += bcp.T
        jz = torch.where(u > 0, u ** (1.0 / LAM - 1.0), torch.zeros_like(u)).T[:, None, :] * ju
        jy = (jz - Yn.T[:, None, :] * jz.sum(2, keepdim=True)) / S[:, None, None]
        J = jy.clone()
        J[:, 1 + k, k] -= 1.0
        Js.append(J.transpose(1, 2).contiguous())

        def grad_h(Tx, Yx):
            with torch.enable_grad():
                Tg, Yg = Tx.clone().requires_grad_(True), Yx.clone().requires_grad_(True)
                h, _ = _state(_composition(mech, Yg), Tg, pc)
                gT, gY = torch.autograd.grad(h.sum(), (Tg, Yg))
            return h.detach(), gT, gY
        h0, gT0, gY0 = grad_h(Tc, Yc)
        T1 = _solve_T(_composition(mech, Yn), pc, h0, Tc)
        _, cp1, gY1 = grad_h(T1, Yn)
        dh = torch.cat([gT0[:, None], gY0.T], 1)
        dTs.append((dh - (jy @ gY1.T[:, :, None])[:, :, 0]) / cp1[:, None])
    return torch.cat(Js), torch.cat(dTs)


def _exact_solver(s, n):
    own, nei = (torch.from_numpy(np.asarray(a)).cuda().long() for a in (s["own"], s["nei"]))
    g, b = s["g"], s["b"]
    diag = s["s"].clone().index_add_(0, own, g).index_add_(0, nei, g)
    pp = torch.from_numpy(np.asarray(s["pp"])).cuda()
    part = torch.searchsorted(pp, torch.arange(n, device="cuda"), right=True)
    row, col, val = torch.cat([own, nei]), torch.cat([nei, own]), torch.cat([-g, -g])
    low = (part[row] == part[col]) & (col < row)
    mat = lambda k: torch.sparse_coo_tensor(torch.stack([row[k], col[k]]), val[k], (n, n)).to_sparse_csr()
    Lo, Up = mat(low), mat(~low)
    x = s["x0"].clone()
    for _ in range(2):
        rhs = b - (Up @ x[:, None])[:, 0]
        z = rhs / diag
        while True:   # forward substitution by levels: exact once nothing moves any more
            zn = (rhs - (Lo @ z[:, None])[:, 0]) / diag
            if bool((zn == z).all()):
                break
            z = zn
        x = z
    r = b - diag * x - ((Lo @ x[:, None]) + (Up @ x[:, None]))[:, 0]
    return diag, x, r
