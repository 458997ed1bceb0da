"""Timed cases of the chemistry-step library: the calls a reacting-flow solver makes, at its sizes.

Every case is one pass through the public entry points of `paper_2402_18858_gb300.chem` on seeded
synthetic cells (fresh-gas / burnt-gas mixing lines with a radical pool and random temperatures).
The sizes run from a small patch of cells, where launches and the latency of single cells count, to
the million-cell blocks of one GPU; the mechanisms are the three of `workload.py` (9, 30 and 53
species) and the networks the two committed checkpoints and the one-network-per-species form.

    listed()             the standing cases
    draw(rng)            one more case of the same ranges
    prepare(case, seed)  handles, inputs and output buffers on the GPU
    run(state)           one pass; returns its outputs
    work(case)           bytes and flops one pass cannot do without
    exact(case, seed)    the same outputs in 64 bits by plain torch (None where there are none)
"""
import functools
import math
import os
import struct
import tempfile

import numpy as np
import torch

from paper_2402_18858_gb300 import chem, workload as wl

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
MODELS = os.path.join(ROOT, "paper_2402_18858_gb300", "models")
MECH_SEED = {"h2_9": 0, "c_30": 1, "c_53": 5}
FLOW_DT = {"h2_9": 1e-6, "c_30": 5e-6, "c_53": 1e-5}        # flow step of each mechanism's workload (s)
CKPT = {"c_30": "ann_c30_seed1.ckpt", "c_53": "ann_c53_seed5.ckpt"}
HIDDEN = {"c_30": (1600, 800, 400), "c_53": (2000, 1000, 504), "h2_9": (256, 128)}
# FP64 operations of one direct integration per cell: the mean counts of right-hand sides,
# Jacobians, factorisations and solves over the workload times their operations
DI_FLOPS = {"h2_9": 1.24e5, "c_30": 6.12e6, "c_53": 1.85e7}
R_GAS, P_STD = 8.314462618, 101325.0
DEV = "cuda"


def listed():
    return [
        # a refined patch or the last cells of a load-balanced block: one cell's latency decides
        {"name": "di-30sp-patch", "op": "di", "kind": "c_30", "cells": 150},
        # the small hydrogen workload: short kernels, few unknowns
        {"name": "di-9sp-4k", "op": "di", "kind": "h2_9", "cells": 4096},
        # direct integration of a block of cells, the reference path of every flow step
        {"name": "di-30sp-12k", "op": "di", "kind": "c_30", "cells": 12345},
        # the large mechanism, where the Newton matrix does not fit the lanes of a warp
        {"name": "di-53sp-3k", "op": "di", "kind": "c_53", "cells": 3001},
        # production and heat release rates of a field (diagnostics, explicit sub-steps)
        {"name": "rates-30sp-200k", "op": "rates", "kind": "c_30", "cells": 200_000},
        # property update after every chemistry step: c_p, h, viscosity and conductivity in FP64
        {"name": "thermo-30sp-1m", "op": "thermo", "kind": "c_30", "cells": 1_000_000, "from_h": False, "mixed": False},
        # temperature from the transported enthalpy and properties with FP32 transport sums
        {"name": "thermo-53sp-from-h", "op": "thermo", "kind": "c_53", "cells": 120_007, "from_h": True, "mixed": True},
        # filtered reaction source of the turbulence-chemistry closure
        {"name": "pasr-30sp-1m", "op": "pasr", "kind": "c_30", "cells": 1_000_000},
        # the network alone, on two uneven inference chunks
        {"name": "forward-30sp-400k", "op": "forward", "kind": "c_30", "cells": 400_001, "per_species": False},
        # the learned chemistry step with its checks and the fallback, on a large block
        {"name": "learned-30sp-400k", "op": "learned", "kind": "c_30", "cells": 400_003, "indexed": False},
        # the same on a small list of cells, where the launches count
        {"name": "learned-53sp-2k", "op": "learned", "kind": "c_53", "cells": 2048, "indexed": True},
        # one optimisation step of a new network's training
        {"name": "train-30sp-16k", "op": "train", "kind": "c_30", "cells": 16_384},
    ]


def _log_size(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["di", "di", "di", "rates", "thermo", "thermo", "pasr", "forward", "learned", "train"])
    case = {"op": op}
    if op == "di":
        case["kind"] = rng.choice(["h2_9", "c_30", "c_53"])
        case["cells"] = _log_size(rng, 64, {"h2_9": 60_000, "c_30": 12_000, "c_53": 3_000}[case["kind"]])
    elif op in ("rates", "pasr"):
        case["kind"] = rng.choice(["h2_9", "c_30", "c_53"])
        case["cells"] = _log_size(rng, 1_000, 200_000 if op == "rates" else 900_000)
    elif op == "thermo":
        case["kind"] = rng.choice(["h2_9", "c_30", "c_53"])
        case["cells"] = _log_size(rng, 1_000, 400_000 if case["kind"] == "c_53" else 1_000_000)
        case["from_h"] = rng.random() < 0.5
        case["mixed"] = rng.random() < 0.5
    elif op == "forward":
        case["kind"] = rng.choice(["h2_9", "c_30", "c_53"])
        case["per_species"] = case["kind"] == "h2_9"
        case["cells"] = _log_size(rng, 500, 300_000)
    elif op == "learned":
        case["kind"] = rng.choice(["c_30", "c_53"])
        case["cells"] = _log_size(rng, 500, 300_000)
        case["indexed"] = rng.random() < 0.5
    else:
        case["kind"] = "c_30"
        case["cells"] = 8 * _log_size(rng, 128, 4_096)
    return case


# ------------------------------------------------------------------------------------------
# inputs
# ------------------------------------------------------------------------------------------
@functools.lru_cache(maxsize=None)
def _mechanism(kind):
    return wl.make_mechanism(kind, MECH_SEED[kind])


@functools.lru_cache(maxsize=None)
def _endpoints(kind):
    """Mass fractions of the fresh mixture and its products over equivalence ratios in [0.6, 1]."""
    m = _mechanism(kind)
    nu, nb = wl.unburnt_and_burnt_moles(m, np.linspace(0.6, 1.0, 4096))
    major = (nu.sum(axis=1) > 0) | (nb.sum(axis=1) > 0)
    return wl.moles_to_mass_fractions(m, nu), wl.moles_to_mass_fractions(m, nb), major


def _load(kind):
    folder = os.path.join(tempfile.gettempdir(), f"chem_mech_{os.getuid()}")
    return chem.chem_load_mech(wl.mechanism_file(kind, MECH_SEED[kind], folder))


def _states(kind, n, seed):
    """T [n], p [n], Y [K, n]: the distribution of workload.make_states, drawn on the GPU."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    u = lambda *shape: torch.rand(*shape, dtype=torch.float64, device=DEV, generator=g)  # noqa: E731
    Yu, Yb, major = (torch.as_tensor(a, device=DEV) for a in _endpoints(kind))
    K = Yu.shape[0]
    pick = (u(n) * Yu.shape[1]).long().clamp_(max=Yu.shape[1] - 1)
    xi = u(n)
    T = 300.0 + 2200.0 * u(n)
    pool = xi * 10.0 ** (4.0 * u(K, n) - 7.0) + 10.0 ** (3.0 * u(K, n) - 12.0)
    Y = torch.where(major[:, None], Yu[:, pick] * (1.0 - xi) + Yb[:, pick] * xi, pool)
    Y *= torch.exp(0.05 * torch.randn(K, n, dtype=torch.float64, device=DEV, generator=g))
    Y /= Y.sum(dim=0)
    return T, torch.full_like(T, wl.P_ATM), Y.contiguous()


def _network(gm, case):
    if case.get("per_species"):
        return chem.chem_ann_create_per_species(gm, list(HIDDEN[case["kind"]]), seed=3)
    if case["op"] == "train":
        return chem.chem_ann_create(gm, list(HIDDEN[case["kind"]]), seed=3)
    return chem.chem_ann_load(gm, os.path.join(MODELS, CKPT[case["kind"]]))


def _features(ann, T, p, Y, **kw):
    X = torch.empty((T.numel(), 64), dtype=torch.bfloat16, device=DEV)
    chem.chem_ann_features(ann, T, p, Y, X, **kw)
    return X


def prepare(case, seed):
    op, kind, n = case["op"], case["kind"], case["cells"]
    gm = _load(kind)
    T, p, Y = _states(kind, n, seed)
    s = {"op": op, "gm": gm, "dt": FLOW_DT[kind], "p": p, "T0": T, "Y0": Y}
    if op in ("di", "learned"):
        s.update(T=T.clone(), Y=Y.clone(), status=torch.empty(n, dtype=torch.int32, device=DEV))
    if op == "di":
        s["ws"] = torch.empty(chem.chem_workspace_bytes(gm, n), dtype=torch.uint8, device=DEV)
    elif op == "rates":
        s.update(wdot=torch.empty_like(Y), hrr=torch.empty_like(T))
    elif op == "thermo":
        s["out"] = [torch.empty_like(T) for _ in range(4)]
        s["mixed"] = case["mixed"]
        if case["from_h"]:
            # the transported enthalpy belongs to a temperature near the last known one
            s["h_in"] = _nasa(_mechanism(kind), T, Y)[1]
            g = torch.Generator(device=DEV).manual_seed(seed + 1)
            s["T_guess"] = T + 60.0 * (torch.rand(n, dtype=torch.float64, device=DEV, generator=g) - 0.5)
            s["T_new"] = torch.empty_like(T)
    elif op == "pasr":
        g = torch.Generator(device=DEV).manual_seed(seed + 1)
        s["Y1"] = Y * (1.0 + 1e-3 * torch.randn(Y.shape, dtype=torch.float64, device=DEV, generator=g))
        lu = lambda lo, hi: torch.exp(math.log(lo) + (math.log(hi) - math.log(lo))  # noqa: E731
                                      * torch.rand(n, dtype=torch.float64, device=DEV, generator=g))
        s.update(rho=lu(0.12, 1.2), k=lu(1e-3, 10.0), eps=lu(1.0, 1e6), nu=lu(1.5e-5, 4e-4))
        s["k"][torch.rand(n, device=DEV, generator=g) < 0.05] = 0.0
        s.update(omega=torch.empty_like(Y), kappa=torch.empty_like(T))
    else:
        s["ann"] = ann = _network(gm, case)
        if op == "train":
            _prepare_training(s, n)
        else:
            s["ws"] = torch.empty(chem.chem_ann_workspace_bytes(ann, n), dtype=torch.uint8, device=DEV)
        if op == "forward":
            if case["per_species"]:
                chem.chem_ann_fit_norm(ann, T, p, Y, Y * 1.01)
            s["X"] = _features(ann, T, p, Y)
            s["U"] = torch.empty((n, ann.n_out_pad), dtype=torch.float32, device=DEV)
        if op == "learned" and case["indexed"]:
            g = torch.Generator(device=DEV).manual_seed(seed + 1)
            s["idx"] = torch.randperm(n, device=DEV, generator=g).int()[: max(1, (3 * n) // 4)].contiguous()
    torch.cuda.synchronize()
    return s


def _prepare_training(s, n):
    """Features and targets of n samples: the states and their direct integration over dt."""
    ann, T, p, Y0 = s["ann"], s["T0"], s["p"], s["Y0"]
    T1, Y1 = T.clone(), Y0.clone()
    status = torch.empty(n, dtype=torch.int32, device=DEV)
    ws = torch.empty(chem.chem_workspace_bytes(s["gm"], n), dtype=torch.uint8, device=DEV)
    chem.chem_step_di(s["gm"], s["dt"], T1, p, Y1, status, workspace=ws, rtol=1e-6, atol_Y=1e-12)
    chem.chem_ann_fit_norm(ann, T, p, Y0, Y1)
    s["bcty"] = torch.empty((n, ann.n_out), dtype=torch.float32, device=DEV)
    s["X"] = _features(ann, T, p, Y0, bcty=s["bcty"])
    s["Ut"] = torch.empty((n, ann.n_out_pad), dtype=torch.float32, device=DEV)
    chem.chem_ann_targets(ann, Y0, Y1, s["Ut"])
    s["loss"] = torch.zeros(4, dtype=torch.float32, device=DEV)


# ------------------------------------------------------------------------------------------
# one pass
# ------------------------------------------------------------------------------------------
def run(s):
    op, gm = s["op"], s["gm"]
    if op == "di":
        s["T"].copy_(s["T0"])
        s["Y"].copy_(s["Y0"])
        chem.chem_step_di(gm, s["dt"], s["T"], s["p"], s["Y"], s["status"], workspace=s["ws"])
        return {"T": s["T"], "Y": s["Y"], "status": s["status"]}
    if op == "rates":
        chem.chem_rates(gm, s["T0"], s["p"], s["Y0"], s["wdot"], s["hrr"])
        return {"wdot": s["wdot"], "hrr": s["hrr"]}
    if op == "thermo":
        cp, h, mu, kappa = s["out"]
        out = {"cp": cp, "h": h, "mu": mu, "kappa": kappa}
        if "h_in" in s:
            chem.thermo_props(gm, s["T_guess"], s["Y0"], cp, h, mu, kappa, h_in=s["h_in"], T_out=s["T_new"],
                              mixed_precision=s["mixed"])
            out["T"] = s["T_new"]
        else:
            chem.thermo_props(gm, s["T0"], s["Y0"], cp, h, mu, kappa, mixed_precision=s["mixed"])
        return out
    if op == "pasr":
        chem.chem_pasr_source(gm, s["dt"], s["rho"], s["Y0"], s["Y1"], s["k"], s["eps"], s["nu"], s["omega"],
                              s["kappa"])
        return {"omega": s["omega"], "kappa": s["kappa"]}
    if op == "forward":
        chem.chem_ann_forward(s["ann"], s["X"], s["U"], s["ws"])
        return {"U": s["U"]}
    if op == "learned":
        s["T"].copy_(s["T0"])
        s["Y"].copy_(s["Y0"])
        idx = s.get("idx")
        # the fallback's tolerances are those the learned step is served with
        chem.chem_step_ann(gm, s["ann"], s["dt"], s["T"], s["p"], s["Y"], s["status"], s["ws"], idx=idx, di_rtol=1e-5,
                           di_atol_Y=1e-10)
        return {"T": s["T"], "Y": s["Y"], "status": s["status"] if idx is None else s["status"][: idx.numel()]}
    chem.chem_ann_train_step(s["ann"], s["X"], s["Ut"], s["bcty"], loss_out=s["loss"])
    return {"grad": chem.chem_ann_get_params(s["ann"], 1), "loss": s["loss"]}


def _network_weights(case):
    """Multiply-adds of one row through the network (the checkpoints' padded input and output)."""
    h, K = HIDDEN[case["kind"]], _mechanism(case["kind"]).n_species
    out = 1 if case.get("per_species") else (32 if K <= 32 else 64)
    dims = (64,) + h + (out,)
    return (K if case.get("per_species") else 1) * sum(a * b for a, b in zip(dims, dims[1:])), K, out


def work(case):
    op, n = case["op"], case["cells"]
    m = _mechanism(case["kind"])
    K, I = m.n_species, m.n_reactions
    state = 8.0 * (K + 2) * n                 # T, p, Y
    if op == "di":
        return {"bytes": 2 * state, "flops": DI_FLOPS[case["kind"]] * n}
    if op == "rates":
        return {"bytes": state + 8.0 * (K + 1) * n, "flops": n * (30.0 * I + 40.0 * K)}
    if op == "thermo":
        # inputs T, Y (and h); outputs c_p, h, mu, kappa (and T); Wilke's sum over species pairs
        return {"bytes": 8.0 * (K + 1 + 4 + 2 * case["from_h"]) * n, "flops": n * (6.0 * K * K + 80.0 * K)}
    if op == "pasr":
        return {"bytes": 8.0 * (3 * K + 5) * n, "flops": 4.0 * K * n}
    macs, _, out = _network_weights(case)
    if op == "forward":
        n_out = 32 if K <= 32 else 64
        return {"bytes": 128.0 * n + 4.0 * n_out * n + 2.0 * macs, "flops": 2.0 * macs * n}
    if op == "learned":
        cells = max(1, (3 * n) // 4) if case["indexed"] else n
        return {"bytes": 8.0 * (2 * K + 3) * cells + 4.0 * cells + 2.0 * macs, "flops": 2.0 * macs * cells}
    # inputs, targets and raw features; weights, gradients and Adam's moments read and written
    return {"bytes": (128.0 + 4.0 * 32 + 4.0 * K) * n + 28.0 * macs, "flops": 6.0 * macs * n}


# ------------------------------------------------------------------------------------------
# the same results in 64 bits by plain torch
# ------------------------------------------------------------------------------------------
def exact(case, seed):
    op = case["op"]
    if op in ("di", "learned"):
        # a stiff integration to full accuracy takes minutes in plain torch; the learned step
        # decides per cell between a BF16 network and that integration
        return None
    s = prepare(case, seed)
    m = _mechanism(case["kind"])
    if op == "rates":
        return _exact_rates(m, s["T0"], s["p"], s["Y0"])
    if op == "thermo":
        return _exact_thermo(m, s, case["from_h"])
    if op == "pasr":
        return _exact_pasr(s)
    if op == "forward" and not case["per_species"]:
        layers = _read_checkpoint(os.path.join(MODELS, CKPT[case["kind"]]))
    else:
        layers = _unflatten(chem.chem_ann_get_params(s["ann"], 0), s["ann"])
    if op == "forward":
        return {"U": _exact_forward(layers, s["X"].double(), s["U"].shape[1])}
    return _exact_training(layers, s)


def _t(a):
    return torch.as_tensor(np.asarray(a, dtype=np.float64), device=DEV)


def _nasa(m, T, Y=None):
    """Mixture c_p and h per kg (with Y), or per species c_p/R, h/RT and s/R [K, n]."""
    lo, hi, invW = _t(m.nasa_low), _t(m.nasa_high), 1.0 / _t(m.W)
    cp, h, e = [], [], []
    lnT = torch.log(T)
    for k in range(m.n_species):
        a = torch.where(T >= m.T_mid, hi[k][:, None], lo[k][:, None])
        cp.append(a[0] + T * (a[1] + T * (a[2] + T * (a[3] + T * a[4]))))
        h.append(a[0] + T * (a[1] / 2 + T * (a[2] / 3 + T * (a[3] / 4 + T * a[4] / 5))) + a[5] / T)
        if Y is None:
            e.append(a[0] * lnT + T * (a[1] + T * (a[2] / 2 + T * (a[3] / 3 + T * a[4] / 4))) + a[6])
    cp, h = torch.stack(cp), torch.stack(h)
    if Y is None:
        return cp, h, torch.stack(e)
    yw = Y * invW[:, None]
    return R_GAS * (yw * cp).sum(dim=0), R_GAS * T * (yw * h).sum(dim=0)


def _exact_rates(m, T, p, Y):
    rho = p / (R_GAS * T * (Y / _t(m.W)[:, None]).sum(dim=0))
    C = rho * Y / _t(m.W)[:, None]
    _, h, s = _nasa(m, T)
    g, lnT, RT = h - s, torch.log(T), R_GAS * T
    wdot = torch.zeros_like(Y)
    for r in m.reactions:
        k = r.A * torch.exp(r.b * lnT - r.Ea / RT)
        M = None
        if r.kind >= 1:
            M = C.sum(dim=0)
            for sp, a in r.eff.items():
                M = M + (a - 1.0) * C[sp]
        if r.kind == 2:
            pr = r.low[0] * torch.exp(r.low[1] * lnT - r.low[2] / RT) * M / k
            a, T3, T1 = r.troe[:3]
            fc = (1 - a) * torch.exp(-T / T3) + a * torch.exp(-T / T1)
            if len(r.troe) > 3:
                fc = fc + torch.exp(-r.troe[3] / T)
            lf, lp = torch.log10(fc), torch.log10(pr)
            x = lp - 0.4 - 0.67 * lf
            f1 = x / (0.75 - 1.27 * lf - 0.14 * x)
            k = k * pr / (1 + pr) * 10.0 ** (lf / (1 + f1 * f1))
        dg = g[r.products].sum(dim=0) - g[r.reactants].sum(dim=0)
        dnu = len(r.products) - len(r.reactants)
        q = k * (C[r.reactants].prod(dim=0) - torch.exp(dg) * (RT / P_STD) ** dnu * C[r.products].prod(dim=0))
        if r.kind == 1:
            q = q * M
        for sp in r.reactants:
            wdot[sp] -= q
        for sp in r.products:
            wdot[sp] += q
    return {"wdot": wdot, "hrr": -(h * RT * wdot).sum(dim=0)}


def _exact_thermo(m, s, from_h):
    Y = s["Y0"]
    T = s["T_guess"].clone() if from_h else s["T0"]
    if from_h:
        for _ in range(50):
            cp, h = _nasa(m, T, Y)
            T = (T - (h - s["h_in"]) / cp).clamp(200.0, 6000.0)
    cp, h = _nasa(m, T, Y)
    W, L = _t(m.W), torch.log(T)
    X = Y / W[:, None]
    X = X / X.sum(dim=0)
    poly = lambda c: c[:, 0:1] + L * (c[:, 1:2] + L * (c[:, 2:3] + L * c[:, 3:4]))  # noqa: E731
    mu, lam = torch.exp(poly(_t(m.mu_fit))), torch.exp(poly(_t(m.lam_fit)))
    mix = torch.zeros_like(T)
    for k in range(m.n_species):
        ratio = torch.sqrt(mu[k] / mu) * ((W / W[k]) ** 0.25)[:, None]
        phi = (1.0 + ratio) ** 2 / torch.sqrt(8.0 * (1.0 + W[k] / W))[:, None]
        mix += X[k] * mu[k] / (X * phi).sum(dim=0)
    out = {"cp": cp, "h": h, "mu": mix, "kappa": 0.5 * ((X * lam).sum(dim=0) + 1.0 / (X / lam).sum(dim=0))}
    if from_h:
        out["T"] = T
    return out


def _exact_pasr(s, y_min=1e-10, r_min=1e-9):
    Y0, Y1, dt = s["Y0"], s["Y1"], s["dt"]
    d = Y1 - Y0
    formed = (Y1 >= y_min) & (d > r_min * Y1)
    tau_c = torch.where(formed, dt * Y1 / d, torch.zeros_like(d)).max(dim=0).values
    tau_m = torch.where(s["k"] > 0, torch.sqrt(torch.sqrt(s["nu"] / s["eps"]) * s["k"] / s["eps"]),
                        torch.zeros_like(tau_c))
    tot = tau_c + tau_m
    kappa = torch.where(tot > 0, tau_c / tot, torch.ones_like(tot))
    return {"omega": kappa * s["rho"] * d / dt, "kappa": kappa}


def _read_checkpoint(path):
    """Layers [(W, b)] of a committed network, by its file format."""
    with open(path, "rb") as f:
        f.read(8)
        _, L, _, n_norm, flags = struct.unpack("<5i", f.read(20))
        dims = struct.unpack(f"<{L + 1}i", f.read(4 * (L + 1)))
        take = lambda n: np.frombuffer(f.read(4 * n), dtype="<f4")  # noqa: E731
        take(n_norm)
        layers = []
        for a, b in zip(dims, dims[1:]):
            layers.append((_t(take(a * b)).view(b, a), _t(take(b))))
            if flags & 1:
                take(2 * (a * b + b))
    return layers


def _unflatten(flat, ann):
    """Layers [(W, b)] from the flat parameters; per-species networks stacked, [K, out, in], [K, out]."""
    lead, at, layers = ((ann.groups,) if ann.groups > 1 else ()), 0, []
    for a, b in zip(ann.dims, ann.dims[1:]):
        nw, nb = ann.groups * a * b, ann.groups * b
        layers.append((_t(flat[at:at + nw]).view(*lead, b, a), _t(flat[at + nw:at + nw + nb]).view(*lead, b)))
        at += nw + nb
    return layers


def _gelu(z):
    return 0.5 * z * (1.0 + torch.erf(z * math.sqrt(0.5)))


def _exact_forward(layers, X, n_out, rows=16_384):
    """Rows of X [n, 64] through one network or, with stacked weights, one network per species."""
    outs = []
    for x in X.split(rows):
        stacked = layers[0][0].dim() == 3
        nets = range(layers[0][0].shape[0]) if stacked else [None]
        cols = []
        for g in nets:
            a = x
            for i, (W, b) in enumerate(layers):
                W, b = (W, b) if g is None else (W[g], b[g])
                a = a @ W.T + b
                if i < len(layers) - 1:
                    a = _gelu(a)
            cols.append(a)
        u = cols[0] if len(cols) == 1 else torch.cat(cols, dim=1)
        outs.append(torch.nn.functional.pad(u, (0, n_out - u.shape[1])))
    return torch.cat(outs)


def _exact_training(layers, s, w_data=1.0, w_mass=0.1, lam=0.1):
    """Loss (data and mass terms) and its gradient at the given weights."""
    K, n_in, norm = s["ann"].n_out, s["ann"].n_in, chem.chem_ann_get_norm(s["ann"])
    mean, sd = _t(norm[4 * n_in:4 * n_in + K]), _t(norm[4 * n_in + K:])
    params = [t.clone().requires_grad_(True) for layer in layers for t in layer]
    a = s["X"].double()
    for i in range(0, len(params), 2):
        a = a @ params[i].T + params[i + 1]
        if i < len(params) - 2:
            a = _gelu(a)
    u = a[:, :K]
    data = ((u - s["Ut"][:, :K].double()) ** 2).mean()
    t = (lam * (s["bcty"].double() + u * sd + mean) + 1.0).clamp(min=0.0)
    mass = ((t ** 10).sum(dim=1) - 1.0).abs().mean()
    total = w_data * data + w_mass * mass
    total.backward()
    loss = torch.stack([total, data, mass, torch.zeros_like(total)]).detach()
    return {"grad": torch.cat([q.grad.flatten() for q in params]), "loss": loss}
