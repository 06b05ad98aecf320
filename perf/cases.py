"""Performance cases of the layer refinement library.

Each case is one thing that a program which quantizes a model with this
library does, called through the public Python binding: refining a layer
(from a handful of rows to the widest projection of a decoder block), with the
Hessian prepared on the way or on the propagation-corrected target, refitting
and scoring a host quantizer's state, accumulating a calibration Hessian, and
writing a refined layer back.  The layer sizes, group sizes, bit widths and
iteration counts are those of ``synth/layers.py``, the tests and the
benchmark, and ranges around them.

Inputs follow the recipe of ``synth/layers.py`` (low-rank correlated
activations with a few outlier channels, weights with outliers, a
round-to-nearest host state), drawn on the GPU from the seed alone.
"""
import math

import torch

from paper_2609_38599_gb300 import jarq

DEV = "cuda"
RIDGE, EPS, TAU = 1e-4, 1.1920929e-07, 1e-5


# ---------------------------------------------------------------- the cases

def _refine(name, din, dout, g, bits, K, early_stop):
    return {"name": name, "kind": "refine", "din": din, "dout": dout, "g": g, "bits": bits,
            "K": K, "early_stop": early_stop}


def listed():
    return [
        # the smallest layer a program refines (unit-sized projection, g = 64):
        # launches and latency
        _refine("refine_tiny", 256, 256, 64, 3, 5, False),
        # a small projection of odd size: ragged row tile, odd group count,
        # default stopping
        _refine("refine_ragged", 1344, 1000, 64, 4, 3, True),
        # the benchmark's attention projection with its full iteration budget
        _refine("refine_attn_k10", 4096, 4096, 128, 3, 10, False),
        # the same projection at group size 64 (64 scales a row), the paper's
        # default budget and early stop
        _refine("refine_attn_g64", 4096, 4096, 64, 3, 3, True),
        # the widest input (86 groups a row), 4-bit
        _refine("refine_down", 11008, 4096, 128, 4, 3, True),
        # the most output rows
        _refine("refine_gate", 4096, 14336, 128, 3, 3, True),
        # the first layer on a new calibration Hessian: prepare, refine, release
        {"name": "prepare_refine", "kind": "prepare", "din": 4096, "dout": 4096, "g": 128,
         "bits": 3, "K": 3, "early_stop": True},
        # a layer after quantized predecessors: propagation-corrected target
        {"name": "refine_mu", "kind": "mu", "din": 4096, "dout": 4096, "g": 128, "bits": 3,
         "K": 3, "early_stop": True, "mu": 0.5},
        # a host state scored and its scales refitted, codes kept
        {"name": "fit_and_score", "kind": "fit", "din": 4096, "dout": 4096, "g": 128, "bits": 4},
        # calibration one sequence at a time
        {"name": "hessian_sequences", "kind": "hessian", "din": 4096, "tokens": 2048,
         "batches": 4},
        # calibration of the widest input in large batches
        {"name": "hessian_wide", "kind": "hessian", "din": 11008, "tokens": 32768, "batches": 1},
        # a refined layer cast and packed for serving
        {"name": "writeback", "kind": "writeback", "din": 4096, "dout": 11008, "g": 128,
         "bits": 3, "dtype": "float16"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["refine"] * 6 + ["prepare", "mu", "fit", "hessian", "hessian", "writeback"])
    if kind == "hessian":
        din = 8 * _log_int(rng, 8, 11008 // 8)
        return {"kind": kind, "din": din, "tokens": _log_int(rng, 100, 32768),
                "batches": rng.choice([1, 2, 3])}
    g = rng.choice([64, 128, 128])
    G = _log_int(rng, 2, min(11008 // g, 128) if kind in ("refine", "writeback") else 4096 // g)
    din = g * G
    bits = rng.choice([2, 3, 3, 4, 4, 8])
    K = rng.choice([1, 2, 3, 3, 5, 10])
    dout = _log_int(rng, 33, 14336)
    if kind == "writeback":
        return {"kind": kind, "din": din, "dout": dout, "g": g, "bits": bits,
                "dtype": rng.choice(["float16", "bfloat16", "float32"])}
    if kind == "fit":
        return {"kind": kind, "din": din, "dout": dout, "g": g, "bits": bits}
    # no dearer than the largest listed refinement
    top = 3 * 4096 * 11008 ** 2
    dout = max(33, min(dout, top // (K * din * din)))
    case = {"kind": kind, "din": din, "dout": dout, "g": g, "bits": bits, "K": K,
            "early_stop": rng.random() < 0.6}
    if kind == "mu":
        case["mu"] = round(rng.uniform(0.1, 0.9), 2)
    return case


# ---------------------------------------------------------------- inputs

def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _randn(gen, *shape):
    return torch.randn(*shape, generator=gen, device=DEV)


def _activation_law(gen, din):
    """(L, sqrt(D), col): x = (L u + sqrt(D) e) * col, u and e standard normal."""
    rank = max(1, min(64, din // 16))
    L = _randn(gen, din, rank)
    D = torch.rand(din, generator=gen, device=DEV) * 0.95 + 0.05
    col = torch.ones(din, device=DEV)
    n_out = max(1, min(32, din // 256))
    col[torch.randperm(din, generator=gen, device=DEV)[:n_out]] = 30.0
    return L, D.sqrt(), col


def _activations(gen, law, n):
    L, sd, col = law
    return (_randn(gen, n, L.shape[1]) @ L.T + _randn(gen, n, L.shape[0]) * sd) * col


def _hessian(gen, din):
    n = max(2048, din)
    X = _activations(gen, _activation_law(gen, din), n)
    H = X.T @ X / n
    H.diagonal().add_(0.01 * H.diagonal().mean())
    return H


def _layer(gen, dout, din, g, bits):
    """Weights and their round-to-nearest host state."""
    W = _randn(gen, dout, din) * 0.015
    W = torch.where(torch.rand(dout, din, generator=gen, device=DEV) < 0.001, W * 10.0, W)
    qmax = (1 << bits) - 1
    Wg = W.view(dout, din // g, g)
    lo, hi = Wg.amin(2), Wg.amax(2)
    S = (hi - lo) / qmax
    Z = torch.clamp(torch.round(-lo / S), 0, qmax)
    Q = torch.clamp(torch.round(Wg / S[..., None]) + Z[..., None], 0, qmax)
    return W, S, Q.reshape(dout, din).to(torch.uint8), Z.to(torch.int32)


def _mu_grams(gen, din):
    """H = X~^T X~ / n + nu2 I, K = X~^T X / n, XX = X^T X / n for drifted inputs."""
    n = max(2048, din)
    Xq = _activations(gen, _activation_law(gen, din), n).half().float()
    Xf = (Xq + 0.05 * Xq.std(0) * (0.5 * _randn(gen, n, din) +
                                   (Xq / Xq.std(0)).roll(1, 1))).half().float()
    H, K, XX = Xq.T @ Xq / n, Xq.T @ Xf / n, Xf.T @ Xf / n
    nu2 = 0.01 * float(H.diagonal().mean())
    H.diagonal().add_(nu2)
    return H, K, XX, nu2


def prepare(case, seed):
    gen = _gen(seed)
    kind, din = case["kind"], case["din"]
    st = {"case": case}
    if kind == "hessian":
        law = _activation_law(gen, din)
        law = (law[0] * (2.0 / math.sqrt(law[0].shape[1])), law[1], law[2])
        st["X"] = [_activations(gen, law, case["tokens"]).half() for _ in range(case["batches"])]
        return st
    g, bits = case["g"], case["bits"]
    st["W"], st["S"], st["Q"], st["Z"] = _layer(gen, case["dout"], din, g, bits)
    if kind == "writeback":
        # a refined layer: a few of its signed scales are negative
        neg = torch.rand(st["S"].shape, generator=gen, device=DEV) < 0.03
        st["S"] = torch.where(neg, -st["S"], st["S"])
        return st
    if kind == "mu":
        st["H"], st["K"], st["XX"], st["nu2"] = _mu_grams(gen, din)
    else:
        st["H"] = _hessian(gen, din)
    if kind != "prepare":
        # a program prepares a Hessian once and refines all its layers on it
        st["hess"] = jarq.prepare(st["H"], g)
    return st


# ---------------------------------------------------------------- one pass

def _stats(S, Q, r):
    return {"S": S, "Q": Q, "L_host": r.L_host, "L_final": r.L_final, "iters": r.iters,
            "accepted": r.accepted, "ridge_hits": r.ridge_hits, "row_status": r.row_status}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "hessian":
        H = None
        for X in state["X"]:
            H = jarq.accumulate_hessian(X, H)
        return H
    W, Z, bits, g = state["W"], state["Z"], case["bits"], case["g"]
    # the host state stays with the program; the library refines copies in place
    S, Q = state["S"].clone(), state["Q"].clone()
    if kind == "writeback":
        Z = Z.clone()
        jarq.canonicalize(S, Q, Z, g, bits)
        return {"S": S, "Q": Q, "Z": Z, "W": jarq.dequantize(S, Q, Z, g, bits, case["dtype"]),
                "packed": jarq.pack_codes(Q, bits)}
    if kind == "fit":
        F0 = jarq.objective(state["hess"], W, S, Q, Z, bits)
        F_before, F_after = jarq.fit_scales(state["hess"], W, S, Q, Z, bits, "joint")
        return {"F0": F0, "S": S, "F_before": F_before, "F_after": F_after}
    opt = {"max_iters": case["K"], "early_stop": int(case["early_stop"])}
    if kind == "mu":
        r = jarq.refine_mu(state["hess"], W, S, Q, Z, bits, state["K"], state["XX"], case["mu"],
                           state["nu2"], **opt)
    elif kind == "prepare":
        hess = jarq.prepare(state["H"], g)
        r = jarq.refine(hess, W, S, Q, Z, bits, **opt)
        hess.close()
    else:
        r = jarq.refine(state["hess"], W, S, Q, Z, bits, **opt)
    return _stats(S, Q, r)


# ---------------------------------------------------------------- what a pass cannot do without

def work(case):
    kind, d = case["kind"], case["din"]
    if kind == "hessian":
        n = case["tokens"] * case["batches"]
        return {"bytes": 2 * n * d + 4 * d * d, "flops": n * d * (d + 1)}
    p, g, bits = case["dout"], case["g"], case["bits"]
    G = d // g
    if kind == "writeback":
        out = {"float32": 4, "float16": 2, "bfloat16": 2}[case["dtype"]]
        return {"bytes": p * d * (2 + out) + 4 * p * ((d * bits + 31) // 32) + 16 * p * G,
                "flops": p * d}
    gram = p * g * g * G * (G + 1)      # c_i^T H_ih c_h for h <= i
    layer = 4 * p * d + p * d + 8 * p * G + 4 * d * d
    if kind == "fit":
        return {"bytes": layer + 4 * p * G + 24 * p,
                "flops": 4 * p * d * d + gram + p * G ** 3 // 3}
    K = case["K"]
    # target projection, then per iteration the Gram matrices, the solve, the
    # sweep's products and its back substitutions; the Gram matrices once more
    # for the final objective
    flops = 2 * p * d * d + (K + 1) * gram + K * (2 * p * d * d + p * d * g + p * G ** 3 // 3)
    if kind == "mu":
        flops += 4 * p * d * d
        layer += 8 * d * d
    if kind == "prepare":
        flops += d * g * g + d * d * g
    return {"bytes": layer + p * d + 4 * p * G + 32 * p, "flops": flops}


def tolerance(case):
    kind = case["kind"]
    if kind == "writeback":
        return "exact"          # whole numbers, and one correct rounding of an exact product
    if kind == "hessian":
        # float32 sums of exact fp16 products: 1.9e-6 and 5.3e-6 off 64 bits
        return {"rel": 8e-6, "max": 2.5e-5}
    if kind == "fit":
        # a float32 residual product for the score (1.1e-7, 3.5e-7), float32 scales
        return {"rel": 5e-7, "max": 2e-6}
    # a proposal decided the other way at a near-tie moves its row's codes and
    # scales from there on: against 64 bits up to 0.2 % of the rows of a layer
    # part, the scales are off by 1.3e-3 (one value by 0.26) and the objectives by 3.8e-3
    return {"rel": 1.5e-2, "max": 0.9, "differ": 8e-3}


# ---------------------------------------------------------------- 64-bit values

def _grams(C, H, G, g):
    """Gram[j, i, h] = c_i^T H_ih c_h for every row."""
    p = C.shape[0]
    out = torch.empty(p, G, G, dtype=torch.float64, device=DEV)
    for h in range(G):
        HC = C[:, h * g:(h + 1) * g] @ H[h * g:(h + 1) * g]
        out[:, :, h] = (HC * C).view(p, G, g).sum(2)
    return out


def _objective(wHw, rhs, Gram, S):
    return wHw - 2 * (S * rhs).sum(1) + (S * (Gram @ S[..., None])[..., 0]).sum(1)


def _solve(Gram, rhs):
    """Joint scales in 64 bits, rounded once to float32; with the ridge where it is needed."""
    Gram = 0.5 * (Gram + Gram.mT)
    Lc, info = torch.linalg.cholesky_ex(Gram)
    ridge = info > 0
    if bool(ridge.any()):
        eye = torch.eye(Gram.shape[1], dtype=Gram.dtype, device=DEV)
        Gram = torch.where(ridge[:, None, None], Gram + RIDGE * eye, Gram)
        Lc, info = torch.linalg.cholesky_ex(Gram)
    S = torch.cholesky_solve(rhs[..., None], Lc)[..., 0]
    return S.float().double(), ridge


def _sweep(P, H, R, S, C, Z, live_rows, qmax, G, g):
    """One Gauss-Seidel sweep of bounded Babai proposals; returns the accepted count."""
    acc = torch.zeros(P.shape[0], dtype=torch.int32, device=DEV)
    Sx = S.repeat_interleave(g, 1)
    for i in range(G):
        si = slice(i * g, (i + 1) * g)
        s, z, Ri = S[:, i:i + 1], Z[:, i:i + 1], R[i]
        Hr = P[:, si] - (Sx * C) @ H[:, si]
        live = live_rows & (s[:, 0].abs() > EPS)
        y = torch.linalg.solve_triangular(Ri.mT, Hr.T, upper=False).T / torch.where(
            live[:, None], s, torch.ones_like(s))
        # relative to the current codes: x_l = q_l + (y_l - sum_{h>l} R_lh delta_h) / R_ll
        q = C[:, si] + z
        u, delta = y.T.contiguous(), torch.zeros(g, P.shape[0], dtype=torch.float64, device=DEV)
        qT = q.T.contiguous()
        for l in range(g - 1, -1, -1):
            dl = torch.clamp(torch.round(qT[l] + u[l] / Ri[l, l]), 0, qmax) - qT[l]
            delta[l] = dl
            if l:
                u[:l].addr_(Ri[:l, l], dl, alpha=-1)
        Rd = Ri @ delta
        dF = (s[:, 0] ** 2) * ((Rd - 2 * y.T) * Rd).sum(0)
        ok = live & torch.isfinite(dF) & (dF < 0)
        C[:, si] += torch.where(ok[:, None], delta.T, torch.zeros_like(q))
        acc += ok.int()
    return acc


def _exact_refine(case, st):
    p, d, g, bits, K = (case[k] for k in ("dout", "din", "g", "bits", "K"))
    G, qmax = d // g, (1 << case["bits"]) - 1
    H = st["H"].double()
    H = 0.5 * (H + H.T)
    W, S, Z = st["W"].double(), st["S"].double(), st["Z"].double()
    C = st["Q"].double() - Z.repeat_interleave(g, 1)
    P = W @ H
    wHw = (W * P).sum(1)
    if case["kind"] == "mu":
        mu, nu2 = case["mu"], st["nu2"]
        KW = W @ st["K"].double().T
        ww = (W * W).sum(1)
        wHw = ((1 - mu) ** 2 * (W * (W @ st["XX"].double().T)).sum(1)
               + 2 * mu * (1 - mu) * (W * KW).sum(1) + mu ** 2 * (wHw - nu2 * ww) + nu2 * ww)
        P = mu * P + (1 - mu) * (KW + nu2 * W)
    R = [torch.linalg.cholesky(H[i * g:(i + 1) * g, i * g:(i + 1) * g]).mT.contiguous()
         for i in range(G)]
    rows = lambda v: torch.full((p,), v, dtype=torch.int32, device=DEV)  # noqa: E731
    active = torch.ones(p, dtype=torch.bool, device=DEV)
    iters, accepted, ridge_hits = rows(0), rows(0), rows(0)
    Gram = _grams(C, H, G, g)
    rhs = (P * C).view(p, G, g).sum(2)
    L_host = _objective(wHw, rhs, Gram, S)
    L_prev = L_host
    for k in range(1, K + 1):
        if k > 1:
            Gram = _grams(C, H, G, g)
            rhs = (P * C).view(p, G, g).sum(2)
        S_new, ridge = _solve(Gram, rhs)
        S = torch.where(active[:, None], S_new, S)
        ridge_hits += (ridge & active).int()
        iters = torch.where(active, torch.full_like(iters, k), iters)
        L = _objective(wHw, rhs, Gram, S)
        if case["early_stop"] and k >= 2:
            dec = L_prev - L
            active = active & ~((dec / L_prev.abs().clamp_min(EPS) <= TAU) | (dec.abs() <= TAU))
        L_prev = L
        accepted += _sweep(P, H, R, S, C, Z, active, qmax, G, g)
    L_final = _objective(wHw, (P * C).view(p, G, g).sum(2), _grams(C, H, G, g), S)
    Q = (C + Z.repeat_interleave(g, 1)).to(torch.uint8)
    if p * d * K > 2e7:
        # so many decisions that some fall at a near-tie: either side of it is
        # right, and how far the rows then part says nothing about the sums
        S = L_final = None
    return {"S": S, "Q": Q, "L_host": L_host, "L_final": L_final, "iters": iters,
            "accepted": accepted, "ridge_hits": ridge_hits, "row_status": rows(0)}


def exact(case, seed):
    kind, d = case["kind"], case["din"]
    st = prepare(case, seed)
    if kind == "hessian":
        return sum(X.double().T @ X.double() for X in st["X"])
    g, bits = case["g"], case["bits"]
    G = d // g
    if kind == "writeback":
        S, Q, Z = st["S"], st["Q"].int(), st["Z"]
        neg = S < 0
        negx = neg.repeat_interleave(g, 1)
        qmax = (1 << bits) - 1
        S, Z, Q = S.abs(), torch.where(neg, qmax - Z, Z), torch.where(negx, qmax - Q, Q)
        What = S.double().repeat_interleave(g, 1) * (Q - Z.repeat_interleave(g, 1))
        return {"S": S.double(), "Q": None, "Z": None, "W": What, "packed": None}
    if kind == "fit":
        H = st["H"].double()
        H = 0.5 * (H + H.T)
        W, S, Z = st["W"].double(), st["S"].double(), st["Z"].double()
        C = st["Q"].double() - Z.repeat_interleave(g, 1)
        P = W @ H
        wHw, rhs = (W * P).sum(1), (P * C).view(-1, G, g).sum(2)
        Gram = _grams(C, H, G, g)
        F = _objective(wHw, rhs, Gram, S)
        S_new, _ = _solve(Gram, rhs)
        return {"F0": F, "S": S_new, "F_before": F, "F_after": _objective(wHw, rhs, Gram, S_new)}
    return _exact_refine(case, st)
