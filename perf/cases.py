"""Performance cases of the library: what its users have it do, through its public entry points.

Families: cell bounds (every precision, mode, activation and the rounding-error inflation), point
evaluation, the proposer's training gradient and its inference, and whole extractions.  Networks are
the committed fits (``synth/data``: 3 -> 64 x 2 -> 1, 3 -> 256 x 5 -> 1, 3 -> 512 x 8 -> 1) or
unfitted MLPs of the widths, depths and activations the library's tests use.  A seed turns a
committed network into another one of the same work: the domain cube is mapped onto itself by one
of its 48 symmetries, and the iso-values move by a few percent of their spacing.
"""
from __future__ import annotations

import math
from pathlib import Path

import numpy as np
import torch

import paper_2402_13861_gb300 as isx

DATA = Path(__file__).resolve().parents[1] / "synth" / "data"
FITTED = {"small": (64, 2), "scientific": (256, 5), "large": (512, 8)}     # hidden width, hidden layers
F64 = torch.float64
ACTIVE_PER_AREA, TRIS_PER_AREA = 16, 16    # output capacity per iso-value and grid face


# ---- the cases -----------------------------------------------------------------------------------
def listed():
    return [
        # a handful of boxes on the smallest network, as a caller that refines a few nodes at a time asks
        dict(name="bound_bf16_few", family="bound", net="small", prec="bf16", mode="clt", inflate=False, n=9,
             boxes="boxes", lo=1, hi=10),
        # the level loop's dominant call: one chunk of a fine level of the 256-wide scientific network, UP
        dict(name="bound_bf16_scientific", family="bound", net="scientific", prec="bf16", mode="clt", inflate=False,
             n=262144, boxes="cubes", lo=6, hi=9),
        # rigorous bounds (rounding errors enclosed), all octree scales
        dict(name="bound_bf16_inflated", family="bound", net="relu", w=128, H=4, prec="bf16", mode="sound",
             inflate=True, n=20011, boxes="cubes", lo=3, hi=9),
        # sound bounds of the 512-wide, 8-layer network
        dict(name="bound_bf16_large", family="bound", net="large", prec="bf16", mode="sound", inflate=False, n=12007,
             boxes="cubes", lo=6, hi=9),
        # float32 bounds, the precision of a caller that checks or does not trust bf16
        dict(name="bound_fp32_scientific", family="bound", net="scientific", prec="fp32", mode="clt", inflate=False,
             n=20003, boxes="cubes", lo=5, hi=9),
        # an ELU network of the signed-distance workload's shape, anisotropic boxes (every symbol is alive)
        dict(name="bound_fp32_elu", family="bound", net="elu", w=128, H=4, prec="fp32", mode="clt", inflate=False,
             n=5003, boxes="boxes", lo=1, hi=10),
        # the reduced range-analysis baseline
        dict(name="bound_rafixed", family="bound", net="scientific", prec="fp32", mode="rafixed", inflate=False,
             n=131075, boxes="cubes", lo=6, hi=9),
        # corner values of the 512-wide network (float32, the default evaluation precision)
        dict(name="eval_fp32_large", family="eval", net="large", prec="fp32", n=300007),
        # corner values of the scientific network on the tensor cores
        dict(name="eval_bf16_scientific", family="eval", net="scientific", prec="bf16", n=2100003),
        # one training batch of the proposer, at the size its training uses
        dict(name="proposer_grad", family="proposer", op="grad", n=8192),
        # interactive extraction of the small network at 64^3: launches and host round trips count
        dict(name="extract_small", family="extract", net="small", level=6, n_iso=1, mode="clt", k=3.0, prec="fp32",
             eval_prec="fp32", kd_tree=False, stop=-1),
        # the headline: 512^3, eight iso-values, UP with k = 3
        dict(name="extract_scientific", family="extract", net="scientific", level=9, n_iso=8, mode="clt", k=3.0,
             prec="bf16", eval_prec="bf16", kd_tree=False, stop=-1),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(max(lo, hi))))))


def draw(rng):
    family = rng.choice(["bound"] * 7 + ["eval"] * 3 + ["proposer"] * 2 + ["extract"] * 3)
    if family == "bound":
        c = dict(family="bound", prec=rng.choice(["bf16", "bf16", "fp32"]))
        c["net"] = rng.choice(["small", "scientific", "scientific", "large", "relu", "relu", "elu", "sine"])
        if c["net"] not in FITTED:
            c["w"] = rng.choice([64, 128, 256, 512]) if c["prec"] == "bf16" else 16 * rng.randint(1, 32)
            c["H"] = rng.randint(1, 8)
        if c["net"] in ("elu", "sine"):
            c["mode"] = "clt"
        else:
            c["mode"] = rng.choice(["clt", "clt", "sound", "sound", "raua"] + (["rafixed"] if c["prec"] == "fp32" else []))
        c["inflate"] = c["mode"] in ("sound", "rafixed") and rng.random() < 0.4
        c["boxes"] = rng.choice(["cubes", "cubes", "boxes"])
        c["lo"] = rng.randint(1, 7)
        c["hi"] = rng.randint(c["lo"], 10)
        w, H = _shape(c)
        dense = _bound_flops(w, H, 1.0, c["mode"])                       # every symbol alive
        c["n"] = _log_int(rng, 1, min(300000, (1.5e14 if c["prec"] == "bf16" else 1e13) / dense))
        return c
    if family == "eval":
        c = dict(family="eval", prec=rng.choice(["fp32", "bf16"]))
        if c["prec"] == "bf16":
            c["net"] = rng.choice(["scientific", "scientific", "relu", "sine", "elu"])
        else:
            c["net"] = rng.choice(["small", "scientific", "large", "large", "relu", "sine", "elu"])
        if c["net"] not in FITTED:
            c["w"] = rng.choice([128, 256]) if c["prec"] == "bf16" else 16 * rng.randint(1, 32)
            c["H"] = rng.randint(2, 8)
        w, H = _shape(c)
        c["n"] = _log_int(rng, 1, min(1 << 23, 3e12 / _eval_flops(w, H)))
        return c
    if family == "proposer":
        op = rng.choice(["grad", "predict"])
        return dict(family="proposer", op=op, n=_log_int(rng, 32, 65536 if op == "grad" else 1 << 21))
    c = dict(family="extract", net=rng.choice(["small", "scientific", "scientific", "large"]))
    c["prec"] = rng.choice(["fp32", "bf16"]) if c["net"] == "small" else "bf16"
    c["eval_prec"] = "bf16" if c["net"] == "scientific" else "fp32"
    c["level"] = rng.randint(3, {"small": 6, "scientific": 8, "large": 7}[c["net"]])
    c["n_iso"] = rng.randint(1, 8) if c["net"] == "scientific" else 1
    c["mode"] = "sound" if c["net"] == "large" else rng.choice(["clt", "clt", "sound"])
    c["k"] = rng.choice([2.0, 3.0, 4.0])
    c["kd_tree"] = rng.random() < 0.15
    c["stop"] = rng.choice([-1, -1, max(1, c["level"] - 2)])
    return c


# ---- networks ------------------------------------------------------------------------------------
def _shape(case):
    return FITTED[case["net"]] if case["net"] in FITTED else (case["w"], case["H"])


def _act(case):
    return case["net"] if case["net"] in ("elu", "sine") else "relu"


def _layers(case, seed):
    """(W, b) float32 pairs and iso-values."""
    r = np.random.default_rng([seed, 17])
    if case["net"] in FITTED:
        with np.load(DATA / f"{case['net']}.npz") as z:
            layers = [(z[f"W{l}"], z[f"b{l}"]) for l in range(int(z["n_layers"]))]
            isos = z["isos"].astype(np.float64)
        # a symmetry of the cube [-1, 1]^3: axes permuted, some of them mirrored
        W0 = layers[0][0][:, r.permutation(3)] * r.choice([-1.0, 1.0], size=3).astype(np.float32)
        layers[0] = (np.ascontiguousarray(W0), layers[0][1])
        step = isos[1] - isos[0] if len(isos) > 1 else 0.1 * abs(isos[0])
        return layers, isos + 0.05 * step * r.uniform(-1.0, 1.0, size=len(isos))
    w, H = case["w"], case["H"]
    dims = [3] + [w] * H + [1]
    layers = []
    for l, (fi, fo) in enumerate(zip(dims[:-1], dims[1:])):
        if case["net"] == "sine":                   # SIREN initialisation, omega_0 = 30 folded in
            lim = 1.0 / fi if l == 0 else math.sqrt(6.0 / fi) / 30.0
            s = 30.0 if l < H else 1.0
            W, b = s * r.uniform(-lim, lim, size=(fo, fi)), s * r.uniform(-1.0, 1.0, size=fo) / math.sqrt(fi)
        else:                                       # He initialisation, small biases as after a fit
            W, b = r.normal(0.0, math.sqrt(2.0 / fi), size=(fo, fi)), r.normal(0.0, 0.1, size=fo)
        layers.append((W.astype(np.float32), b.astype(np.float32)))
    return layers, np.zeros(1)


def _boxes(case, seed):
    """n boxes inside [-1, 1]^3: octree cubes of levels lo .. hi, or boxes with log-uniform half-widths
    2^-hi .. 2^-lo per axis."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    n = case["n"]
    if case["boxes"] == "cubes":
        level = torch.randint(case["lo"], case["hi"] + 1, (n, 1), generator=g, device="cuda")
        cells = torch.exp2(level.to(F64))
        ijk = torch.floor(torch.rand((n, 3), generator=g, device="cuda", dtype=F64) * cells)
        lo = -1.0 + 2.0 * ijk / cells
        hi = lo + 2.0 / cells
    else:
        e = torch.rand((n, 3), generator=g, device="cuda", dtype=F64)
        h = torch.exp2(-(case["lo"] + (case["hi"] - case["lo"]) * e))
        c = (torch.rand((n, 3), generator=g, device="cuda", dtype=F64) * 2.0 - 1.0) * (1.0 - h)
        lo, hi = c - h, c + h
    return lo.float().contiguous(), hi.float().contiguous()


def _proposer_inputs(case, seed):
    with np.load(DATA / "proposer.npz") as z:
        params, mean, std = z["params"].astype(np.float32), z["mean"].astype(np.float32), z["std"].astype(np.float32)
    r = np.random.default_rng([seed, 23])
    params = params * (1.0 + 0.02 * r.standard_normal(params.shape)).astype(np.float32)
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    x = torch.randn((case["n"], 8), generator=g, device="cuda")
    feat = torch.tensor(mean, device="cuda") + torch.tensor(std, device="cuda") * x
    label = (torch.rand(case["n"], generator=g, device="cuda") < 0.3).float()
    return params, mean, std, feat.contiguous(), label


# ---- prepare / run ---------------------------------------------------------------------------------
def prepare(case, seed):
    s = dict(case=case)
    if case["family"] == "proposer":
        params, mean, std, s["feat"], s["label"] = _proposer_inputs(case, seed)
        s["proposer"] = isx.Proposer(params, mean, std)
        return s
    layers, isos = _layers(case, seed)
    s["net"] = isx.Inr(layers, act=_act(case))
    if case["family"] == "bound":
        s["lo"], s["hi"] = _boxes(case, seed)
    elif case["family"] == "eval":
        g = torch.Generator(device="cuda")
        g.manual_seed(seed)
        s["xyz"] = torch.rand((case["n"], 3), generator=g, device="cuda") * 2.0 - 1.0
    else:
        s["isos"] = [float(c) for c in isos[:case["n_iso"]]]
        # the caller's output buffers, sized as it sizes them: active cells and triangles grow with the
        # surfaces' area; cleared, so that what lies past the counts is the same for everybody
        area = case["n_iso"] * 4 ** case["level"]
        na, nt = min(8 ** case["level"], ACTIVE_PER_AREA * area + 65536), TRIS_PER_AREA * area + 65536
        i32 = dict(dtype=torch.int32, device="cuda")
        s["buffers"] = dict(code=torch.zeros(na, **i32), mask=torch.zeros(na, **i32), active_cap=na,
                            vert=torch.zeros((nt, 3, 3), device="cuda"),
                            edge=torch.zeros((nt, 3), dtype=torch.int64, device="cuda"),
                            iso=torch.zeros(nt, **i32), cell=torch.zeros(nt, **i32), tri_cap=nt)
    return s


def run(state):
    c = state["case"]
    if c["family"] == "bound":
        return state["net"].bound_cells(state["lo"], state["hi"], mode=c["mode"], prec=c["prec"], inflate=c["inflate"])
    if c["family"] == "eval":
        return state["net"].eval_points(state["xyz"], prec=c["prec"])
    if c["family"] == "proposer":
        if c["op"] == "grad":
            return state["proposer"].grad(state["feat"], state["label"])
        return state["proposer"].predict(state["feat"])
    buf = state["buffers"]
    out = state["net"].extract(c["level"], state["isos"], mode=c["mode"], k=c["k"], prec=c["prec"],
                               eval_prec=c["eval_prec"], kd_tree=c["kd_tree"], bound_stop_level=c["stop"],
                               active_cap=buf["active_cap"], tri_cap=buf["tri_cap"], buffers=buf)
    return {**{k: buf[k] for k in ("code", "mask", "vert", "edge", "iso", "cell")},
            **{k: np.array(out[k]) for k in ("n_active", "n_tris", "n_points", "cells_bounded", "cells_kept",
                                             "cells_visited")}}


# ---- work ------------------------------------------------------------------------------------------
def _symbol_share(case):
    """Share of a layer's neurons whose activation creates a noise symbol (a ReLU away from its kink
    creates none): measured for the committed networks on fine cells, more than half of them on coarse
    boxes, all of them for smooth activations and where rounding errors are carried in symbols."""
    if _act(case) != "relu" or case["inflate"]:
        return 1.0
    if case["net"] in FITTED and case["boxes"] == "cubes" and case["lo"] >= 5:
        return 0.018 if case["net"] == "large" else 0.07
    return 0.6


def _bound_flops(w, H, share, mode):
    """Of one cell: the centre and three input rows, and every symbol's row, through the hidden layers."""
    rows = 5.0 * (H - 1) if mode == "rafixed" else 4.0 * (H - 1) + share * w * (H - 1) * (H - 2) / 2.0
    return 2.0 * w * w * rows + 2.0 * w * (16.0 + share * w * max(0, H - 1))


def _eval_flops(w, H):
    return 2.0 * (4.0 * w + (H - 1.0) * w * w)


def work(case):
    if case["family"] == "proposer":
        macs = 8 * 64 + 2 * 64 * 64 + 64
        grad = case["op"] == "grad"
        return {"bytes": 36.0 * case["n"] + 4.0 * 8961 * (2 if grad else 1),
                "flops": 2.0 * case["n"] * macs * (3 if grad else 1)}
    w, H = _shape(case)
    weights = 4.0 * (4 * w + (H - 1) * w * (w + 1) + w + 1)
    if case["family"] == "bound":
        return {"bytes": 32.0 * case["n"] + weights, "flops": case["n"] * _bound_flops(w, H, _symbol_share(case), case["mode"])}
    if case["family"] == "eval":
        return {"bytes": 16.0 * case["n"] + weights, "flops": case["n"] * _eval_flops(w, H)}
    # bounded cells and active cells per iso-value, both close to multiples of the surfaces' area
    area = case["n_iso"] * 4.0 ** (case["level"] if case["stop"] < 0 else case["stop"])
    cells = 4.0 * 4.0 * area
    fine = case["n_iso"] * 4.0 ** case["level"]
    return {"bytes": 68.0 * 4.0 * fine + weights,
            "flops": cells * _bound_flops(w, H, 0.03, case["mode"]) + 4.0 * fine * _eval_flops(w, H)}


# ---- 64-bit values ---------------------------------------------------------------------------------
def _relu_sound(c, r):
    l, u = c - r, c + r
    cross = (l < 0) & (u > 0)
    alpha = torch.where(cross, u / (u - l).clamp_min(1e-300), (l >= 0).to(F64))
    beta = torch.where(cross, -0.5 * alpha * l, torch.zeros_like(l))
    return alpha, alpha * c + beta, beta


def _least_squares(act, mu, sg):
    """alpha, alpha mu + beta and gamma of the least-squares line of the activation under N(mu, sg^2)."""
    s2 = sg * sg
    if act == "sine":
        a = torch.exp(-0.5 * s2)
        alpha, centre = a * torch.cos(mu), a * torch.sin(mu)
        g2 = 0.5 * (1.0 - torch.exp(-2.0 * s2) * torch.cos(2.0 * mu)) - centre ** 2 - alpha ** 2 * s2
        return alpha, centre, torch.sqrt(g2.clamp_min(0.0))
    safe = sg.clamp_min(1e-300)
    t = mu / safe
    Phi, Q = 0.5 * torch.erfc(-t / math.sqrt(2.0)), 0.5 * torch.erfc(t / math.sqrt(2.0))
    gauss = torch.exp(-0.5 * t * t)
    phi = gauss / math.sqrt(2.0 * math.pi)
    if act == "relu":
        centre = mu * Phi + sg * phi
        g2 = Phi * Q * (t * t + 1.0) + (Q - Phi) * t * phi - phi * phi
        return Phi, centre, torch.where(t.abs() < 40.0, sg * torch.sqrt(g2.clamp_min(0.0)), torch.zeros_like(sg))

    def lognormal(k):                               # E[e^{kX}; X <= 0]
        y = (t + k * sg) / math.sqrt(2.0)
        return torch.where(y >= 0, 0.5 * torch.special.erfcx(y.clamp_min(0.0)) * gauss,
                           0.5 * torch.erfc(y) * torch.exp(torch.where(y >= 0, torch.zeros_like(mu), k * mu + 0.5 * k * k * s2)))

    b1, b2 = lognormal(1.0), lognormal(2.0)
    alpha = Phi + b1
    centre = mu * Phi + sg * phi + b1 - Q
    g2 = (mu * mu + s2) * Phi + mu * sg * phi + b2 - 2.0 * b1 + Q - centre ** 2 - alpha ** 2 * s2
    return alpha, centre, torch.sqrt(g2.clamp_min(0.0))


def _exact_bound(layers, act, lo, hi, mode, share):
    W = [torch.tensor(w, device="cuda", dtype=F64) for w, _ in layers]
    b = [torch.tensor(v, device="cuda", dtype=F64) for _, v in layers]
    H, w, n = len(layers) - 1, layers[0][0].shape[0], lo.shape[0]
    clt = mode == "clt"
    centre, spread = torch.empty(n, device="cuda", dtype=F64), torch.empty(n, device="cuda", dtype=F64)
    m = int(max(8, min(8192, 1.5e8 / (w * (4 + share * w * H)))))
    for a in range(0, n, m):
        x, h = 0.5 * (lo[a:a + m].to(F64) + hi[a:a + m].to(F64)), 0.5 * (hi[a:a + m].to(F64) - lo[a:a + m].to(F64))
        if clt:
            h = h / math.sqrt(3.0)
        c = x @ W[0].T + b[0]
        I = h[:, :, None] * W[0].T[None]
        G, owner = torch.zeros((0, w), device="cuda", dtype=F64), torch.zeros(0, device="cuda", dtype=torch.int64)
        priv = torch.zeros_like(c)
        for j in range(1, H + 1):
            f = (lambda v: v * v) if clt else torch.abs
            r = f(I).sum(1)
            r.index_add_(0, owner, f(G))
            r = torch.sqrt(r) if clt else r + priv
            alpha, act_c, gamma = _least_squares(act, c, r) if clt else _relu_sound(c, r)
            if j == H:
                break
            I = (I * alpha[:, None]) @ W[j].T
            if mode == "rafixed":
                priv = (alpha * priv + gamma) @ W[j].abs().T
            else:
                cell, nrn = torch.nonzero(gamma > (1e-7 * r if clt else 0.0), as_tuple=True)
                G = torch.cat([(G * alpha[owner]) @ W[j].T, gamma[cell, nrn, None] * W[j].T[nrn]])
                owner = torch.cat([owner, cell])
            c = act_c @ W[j].T + b[j]
        v, wo = alpha * W[H][0], W[H][0]
        yi, yg, yn = (I * v[:, None]).sum(-1), (G * v[owner]).sum(-1), gamma * wo
        if mode in ("clt", "raua"):
            s = (yi ** 2).sum(1).index_add_(0, owner, yg ** 2) + (yn ** 2).sum(1)
            s = torch.sqrt(s / 3.0 if mode == "raua" else s)
        else:
            s = yi.abs().sum(1).index_add_(0, owner, yg.abs()) + yn.abs().sum(1) + (alpha * priv) @ wo.abs()
        centre[a:a + m], spread[a:a + m] = act_c @ wo + b[H][0], s
    return centre, spread


def exact(case, seed):
    if case["family"] == "proposer":
        params, mean, std, feat, label = _proposer_inputs(case, seed)
        p = torch.tensor(params, device="cuda", dtype=F64, requires_grad=True)
        a = (feat.to(F64) - torch.tensor(mean, device="cuda", dtype=F64)) / torch.tensor(std, device="cuda", dtype=F64)
        o = 0
        for fi, fo in ((8, 64), (64, 64), (64, 64), (64, 1)):
            a = a @ p[o:o + fi * fo].view(fo, fi).T + p[o + fi * fo:o + fi * fo + fo]
            o += fi * fo + fo
            a = torch.relu(a) if fo > 1 else a[:, 0]
        if case["op"] == "predict":
            return a.detach()
        loss = torch.nn.functional.binary_cross_entropy_with_logits(a, label.to(F64))
        loss.backward()
        return p.grad, loss.detach().reshape(1)
    if case["family"] == "extract":                 # cell lists and meshes: compared value by value
        return None
    w, H = _shape(case)
    layers, _ = _layers(case, seed)
    if case["family"] == "eval":
        x = torch.Generator(device="cuda")
        x.manual_seed(seed)
        x = torch.rand((case["n"], 3), generator=x, device="cuda") * 2.0 - 1.0
        f = {"relu": torch.relu, "elu": torch.nn.functional.elu, "sine": torch.sin}[_act(case)]
        W = [(torch.tensor(u, device="cuda", dtype=F64), torch.tensor(v, device="cuda", dtype=F64)) for u, v in layers]
        out = torch.empty(case["n"], device="cuda", dtype=F64)
        for a in range(0, case["n"], 1 << 18):
            y = x[a:a + (1 << 18)].to(F64)
            for l, (u, v) in enumerate(W):
                y = y @ u.T + v
                if l < H:
                    y = f(y)
            out[a:a + (1 << 18)] = y[:, 0]
        return out
    share = _symbol_share(case)
    # the inflated interval has no single right value; float64 over 12 TFLOP takes too long
    if case["inflate"] or case["n"] * _bound_flops(w, H, share, case["mode"]) > 1.2e13:
        return None
    lo, hi = _boxes(case, seed)
    return _exact_bound(layers, _act(case), lo, hi, case["mode"], share)
