"""Cases for timing the library through its public entry points.

A SOAP case is one optimizer step in the steady state of a run: the factors hold the mean of the
gradients' outer products, the bases their eigenbases, the moments their stationary values, and
each pass takes the next of a few gradients (a training loop never steps twice on one gradient).
Gradients follow the package's synthetic workloads: G = c (A + 0.3 N), A = U diag(s) V^T with
s_i ~ i^-1.5 and ||s|| = 1, N i.i.d. N(0, 1/cols), weights N(0, 0.02^2).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2607_20548_gb300 import soap as S

DEV = "cuda:0"


# ---- the cases ---------------------------------------------------------------------------

def listed():
    """shapes: "count*rows*cols*sides" tokens, sides L, R or LR (the preconditioned ones)."""
    return [
        # one 256 x 512 weight, both sides: the smallest workload, bound by launches and latency
        {"name": "soap_256x512", "kind": "soap", "shapes": "1*256*512*LR", "kl": 0, "every": 1, "grads": 8},
        # a dense transformer block of hidden 2048 and FFN 8192 (attention, gate/up, down)
        {"name": "soap_dense_block", "kind": "soap", "shapes": "4*2048*2048*LR,2*2048*8192*LR,1*8192*2048*LR", "kl": 0,
         "every": 1, "grads": 2},
        # one fine-grained MoE layer: 64 experts (gate, up, down) and the router, one batched step
        {"name": "soap_moe_layer", "kind": "soap", "shapes": "128*2048*768*LR,64*768*2048*LR,1*2048*64*LR", "kl": 0,
         "every": 1, "grads": 2},
        # an embedding or LM head: the vocabulary side carries no preconditioner
        {"name": "soap_lm_head", "kind": "soap", "shapes": "1*2048*32768*L", "kl": 0, "every": 1, "grads": 2},
        # the KL-Shampoo factor form on eight experts (a rank's share of a layer)
        {"name": "soap_kl_experts", "kind": "soap", "shapes": "8*2048*768*LR", "kl": 1, "every": 1, "grads": 4},
        # the four attention matrices with the basis refreshed every tenth step
        {"name": "soap_attention_f10", "kind": "soap", "shapes": "4*2048*2048*LR", "kl": 0, "every": 10, "grads": 4},
        # ragged vocabulary-like sides that no TMA copy can read: the CUDA-core path
        {"name": "soap_ragged", "kind": "soap", "shapes": "2*512*1001*L,1*257*768*R", "kl": 0, "every": 1, "grads": 8},
        # resume: every state piece set from a checkpoint, one step, every piece read back
        {"name": "resume_768x2048", "kind": "resume", "shapes": "1*768*2048*LR", "kl": 0, "every": 1, "grads": 1},
        # the stand-alone QR refresh on the largest factor and on a batch of hidden-sized ones
        {"name": "qr_8192", "kind": "qr", "n": 8192, "batch": 1, "static": False},
        {"name": "qr_2048x16", "kind": "qr", "n": 2048, "batch": 16, "static": False},
        # the stand-alone fp32-accurate product at a rotation's size, ragged, accumulating into C
        {"name": "gemm_2052x770x2044", "kind": "gemm", "M": 2052, "N": 770, "K": 2044, "batch": 4, "beta": 0.5},
        # Muon on the dense block's matrices
        {"name": "muon_dense_block", "kind": "muon", "shapes": "4*2048*2048*LR,2*2048*8192*LR,1*8192*2048*LR", "steps": 16},
    ]


def _size(rng, lo, hi, unit):
    """A multiple of `unit` in [lo, hi], spread over the logarithm."""
    return max(lo, min(hi, unit * round(math.exp(rng.uniform(math.log(lo), math.log(hi))) / unit)))


def draw(rng):
    kind = rng.choice(["soap", "soap", "soap", "resume", "qr", "qr", "gemm", "muon"])
    if kind in ("soap", "resume"):
        toks, cost = [], 0.0
        for _ in range(1 if kind == "resume" else rng.randint(1, 3)):
            r = _size(rng, 64, 3072, 4)
            # the longer side at most four times the shorter: what a few gradients' factors fill
            c = _size(rng, max(64, r // 4), min(3072, 4 * r), 4)
            sides = rng.choice(["LR", "LR", "LR", "L", "R"])
            if sides == "L" and rng.random() < 0.3:
                c += 1  # a ragged identity side
            if sides == "R" and rng.random() < 0.3:
                r += 1
            one = (r + c) ** 3
            k = 1 if kind == "resume" else max(1, min(_size(rng, 1, 64, 1), int((1.5e12 - cost) / one)))
            if cost + k * one > 2e12:
                continue
            cost += k * one
            toks.append("%d*%d*%d*%s" % (k, r, c, sides))
        return {"kind": kind, "shapes": ",".join(toks), "kl": rng.choice([0, 0, 1]), "every": rng.choice([1, 1, 1, 10]),
                "grads": 1 if kind == "resume" else 8}
    if kind == "qr":
        n = _size(rng, 36, 4096, 4)
        if n <= 512 and rng.random() < 0.5:
            return {"kind": "qr", "n": n, "batch": rng.randint(1, 2), "static": True}
        return {"kind": "qr", "n": n, "batch": max(1, min(_size(rng, 1, 128, 1), int(2e11 / n ** 3))), "static": False}
    if kind == "gemm":
        M, N, K = _size(rng, 16, 4096, 1), _size(rng, 16, 4096, 1), _size(rng, 16, 4096, 4)
        return {"kind": "gemm", "M": M, "N": N, "K": K, "batch": max(1, min(_size(rng, 1, 64, 1), int(2e11 / (M * N * K)))),
                "beta": rng.choice([0.0, 0.5, 1.0])}
    r, c = _size(rng, 64, 4096, 8), _size(rng, 64, 4096, 8)
    k = max(1, min(_size(rng, 1, 64, 1), int(1e11 / (r * c * min(r, c)))))
    return {"kind": "muon", "shapes": "%d*%d*%d*LR" % (k, r, c), "steps": rng.choice([5, 16])}


def _groups(case):
    """[(count, rows, cols, left, right)]"""
    out = []
    for tok in case["shapes"].split(","):
        k, r, c, sides = tok.split("*")
        out.append((int(k), int(r), int(c), "L" in sides, "R" in sides))
    return out


# ---- inputs ------------------------------------------------------------------------------

def _gen(seed, *more):
    h = seed & 0x7FFFFFFF
    for m in more:
        h = (h * 1000003 + m + 12345) & 0x7FFFFFFFFFFF
    return torch.Generator(device=DEV).manual_seed(h)


def _orth(n, k, g):
    """k orthonormal columns of length n: a cosine basis with its rows and columns shuffled and
    their signs drawn."""
    rows = torch.randperm(n, generator=g, device=DEV).double()
    cols = torch.randperm(n, generator=g, device=DEV)[:k].double()
    q = torch.cos((rows[:, None] + 0.5) * (cols[None, :] * (math.pi / n))).mul_(math.sqrt(2.0 / n))
    q[:, cols == 0] = math.sqrt(1.0 / n)
    sr = torch.randint(0, 2, (n, 1), generator=g, device=DEV).double().mul_(2).sub_(1)
    sc = torch.randint(0, 2, (1, k), generator=g, device=DEV).double().mul_(2).sub_(1)
    return (q * sr * sc).float()


def _group_inputs(gi, count, m, n, left, right, seed, ngrads, beta1):
    """One shape group: weights, gradients and the steady state, [count, ., .] tensors."""
    g = _gen(seed, gi)
    k = min(m, n)
    sv = torch.arange(1, k + 1, dtype=torch.float64, device=DEV).pow(-1.5)
    sv = (sv / sv.norm()).float()
    # many matrices of one shape (experts): uneven scales, log-uniform in [1e-2, 1]
    c = torch.exp(torch.rand(count, generator=g, device=DEV) * math.log(1e-2)) if count > 4 else torch.ones(count, device=DEV)
    noise = 0.3 / math.sqrt(n)
    d = {"W": torch.randn(count, m, n, generator=g, device=DEV).mul_(0.02), "c": c}
    A = torch.empty(count, m, n, device=DEV)
    V = torch.empty(count, m, n, device=DEV)
    if left:
        d["QL"] = torch.empty(count, m, m, device=DEV)
    if right:
        d["QR"] = torch.empty(count, n, n, device=DEV)
    for b in range(count):
        U = _orth(m, m if left else k, g)
        X = _orth(n, n if right else k, g)
        A[b] = c[b] * ((U[:, :k] * sv) @ X[:, :k].T)
        # the second moment of the rotated gradient
        if left and right:
            rot = torch.zeros(m, n, device=DEV)
            rot.diagonal().copy_(sv)
        elif left:
            rot = torch.zeros(m, n, device=DEV)
            rot[:k] = sv[:, None] * X[:, :k].T
        else:
            rot = torch.zeros(m, n, device=DEV)
            rot[:, :k] = U[:, :k] * sv
        V[b] = c[b] * c[b] * (rot * rot + noise * noise)
        if left:
            d["QL"][b] = U
        if right:
            d["QR"][b] = X
    c3 = c.view(-1, 1, 1)
    if left:
        d["L"] = torch.matmul(A, A.transpose(1, 2))
        d["L"].diagonal(dim1=1, dim2=2).add_((0.09 * c * c)[:, None])
    if right:
        d["R"] = torch.matmul(A.transpose(1, 2), A)
        d["R"].diagonal(dim1=1, dim2=2).add_((0.09 * m / n * c * c)[:, None])
    d["V"] = V
    draw_noise = lambda s: torch.randn(count, m, n, generator=g, device=DEV).mul_(s).mul_(c3)  # noqa: E731
    d["M"] = A + draw_noise(noise * math.sqrt((1 - beta1) / (1 + beta1)))
    d["G"] = [A + draw_noise(noise) for _ in range(ngrads)]
    return d


PIECES = (("M", S.STATE_MHAT), ("V", S.STATE_V), ("L", S.STATE_L), ("R", S.STATE_R), ("QL", S.STATE_QL), ("QR", S.STATE_QR))


def _hparams(case):
    return S.default_hparams(kl=case["kl"], eig_every=case["every"])


def _soap_inputs(case, seed):
    b1 = float(_hparams(case).beta1)
    return [_group_inputs(gi, k, m, n, left, right, seed, case["grads"], b1)
            for gi, (k, m, n, left, right) in enumerate(_groups(case))]


def _qr_input(case, seed, dtype=torch.float32):
    """P = F Q as the refresh meets it: Q the eigenbasis of the mean factor, F that factor after
    one more gradient."""
    n = case["n"]
    out = []
    for b in range(case["batch"]):
        g = _gen(seed, 7, b)
        sv = torch.arange(1, n + 1, dtype=torch.float64, device=DEV).pow(-1.5)
        sv = (sv / sv.norm()).float()
        U = _orth(n, n, g)
        G = (U * sv) @ torch.randn(n, n, generator=g, device=DEV).mul_(1.0 / math.sqrt(n))
        G += torch.randn(n, n, generator=g, device=DEV).mul_(0.3 / math.sqrt(n))
        F = 0.95 * ((U * (sv * sv + 0.09)) @ U.T) + 0.05 * (G @ G.T)
        out.append(F @ U)
    return torch.stack(out)


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("soap", "resume"):
        data = _soap_inputs(case, seed)
        shapes, pieces = [], []
        for (k, m, n, left, right), d in zip(_groups(case), data):
            for b in range(k):
                shapes.append((m, n, left, right))
                pieces.append({p: d[p][b] for p, _ in PIECES if p in d})
        opt = S.SoapOptimizer(shapes, _hparams(case), device=0)
        st = {"kind": kind, "opt": opt, "W": [d["W"] for d in data], "i": 0,
              "params": [w for d in data for w in d["W"].unbind(0)],
              "grads": [[w for d in data for w in d["G"][j].unbind(0)] for j in range(case["grads"])]}
        if kind == "resume":
            st["saved"] = pieces
            st["W0"] = [d["W"].clone() for d in data]
            return st
        for i, p in enumerate(pieces):
            for name, which in PIECES:
                if name in p:
                    opt.state_set(i, which, p[name])
        opt.t = 1000
        torch.cuda.synchronize()
        return st
    if kind == "qr":
        return {"kind": kind, "P": _qr_input(case, seed), "static": case["static"], "tol": float(S.default_hparams().qr_tol)}
    if kind == "gemm":
        g = _gen(seed, 3)
        M, N, K, b = case["M"], case["N"], case["K"], case["batch"]
        return {"kind": kind, "beta": case["beta"], "A": torch.randn(b, M, K, generator=g, device=DEV),
                "B": torch.randn(b, N, K, generator=g, device=DEV).mul_(1.0 / math.sqrt(K)),
                "C0": torch.randn(b, M, N, generator=g, device=DEV)}
    assert kind == "muon", kind
    W, G, M = [], [], []
    for gi, (k, m, n, _, _) in enumerate(_groups(case)):
        g = _gen(seed, gi, 5)
        A = torch.randn(k, m, n, generator=g, device=DEV).mul_(1.0 / math.sqrt(m * n))
        W.append(torch.randn(k, m, n, generator=g, device=DEV).mul_(0.02))
        G.append(A + torch.randn(k, m, n, generator=g, device=DEV).mul_(0.3 / math.sqrt(n * m)))
        M.append(A + torch.randn(k, m, n, generator=g, device=DEV).mul_(0.07 / math.sqrt(n * m)))
    opt = S.MuonOptimizer([(m, n) for k, m, n, _, _ in _groups(case) for _ in range(k)], ns_steps=case["steps"], device=0)
    for i, x in enumerate(x for grp in M for x in grp.unbind(0)):
        opt.state_set(i, x)
    torch.cuda.synchronize()
    return {"kind": kind, "opt": opt, "W": W, "params": [x for grp in W for x in grp.unbind(0)],
            "grads": [x for grp in G for x in grp.unbind(0)]}


def run(st):
    kind = st["kind"]
    if kind == "soap":
        g = st["grads"][st["i"] % len(st["grads"])]
        st["i"] += 1
        st["opt"].step(st["params"], g)
        return st["W"]
    if kind == "resume":
        opt = st["opt"]
        for w, w0 in zip(st["W"], st["W0"]):
            w.copy_(w0)
        opt.t = 1000
        for i, p in enumerate(st["saved"]):
            for name, which in PIECES:
                if name in p:
                    opt.state_set(i, which, p[name])
        opt.step(st["params"], st["grads"][0])
        return {"W": st["W"], "state": [{name: opt.state_get(i, which) for name, which in PIECES if name in p}
                                        for i, p in enumerate(st["saved"])]}
    if kind == "qr":
        Q, skip = (S.soap_qr_static if st["static"] else S.soap_qr)(st["P"], st["tol"])
        return {"Q": Q, "skip": skip}
    if kind == "gemm":
        if st["beta"] == 0.0:
            return S.soap_gemm_tf32x4(st["A"], st["B"])
        return S.soap_gemm_tf32x4(st["A"], st["B"], beta=st["beta"], C=st["C0"].clone())
    st["opt"].step(st["params"], st["grads"])
    return st["W"]


# ---- what a pass cannot do without -------------------------------------------------------

def work(case):
    kind = case["kind"]
    if kind in ("soap", "resume"):
        by = fl = 0.0
        ref = 1.0 / case["every"]
        for k, m, n, left, right in _groups(case):
            b = 4.0 * 7 * m * n  # W, M, v read and written, G read
            f = 10.0 * m * n
            for on, a, o in ((left, m, n), (right, n, m)):
                if not on:
                    continue
                b += 4.0 * (a * a + (1 + ref) * a * a)        # the factor's half in and out; the basis in, and out on a refresh
                f += a * a * o                                # the factor's EMA, a symmetric product
                f += ref * (2.0 + 8.0 / 3.0) * a ** 3         # power step, QR with explicit Q
                f += 3 * 2.0 * a * a * o                      # gradient and moment into the basis, the update out
                if case["kl"] and left and right:
                    f += 2.0 * a ** 3 + 2.0 * a * a * o
            by += k * b
            fl += k * f
        return {"bytes": by, "flops": fl}
    if kind == "qr":
        n, b = case["n"], case["batch"]
        return {"bytes": 8.0 * b * n * n, "flops": 8.0 / 3.0 * b * float(n) ** 3}
    if kind == "gemm":
        M, N, K, b = case["M"], case["N"], case["K"], case["batch"]
        return {"bytes": 4.0 * b * (M * K + N * K + M * N * (2 if case["beta"] else 1)), "flops": 2.0 * b * M * N * K}
    by = fl = 0.0
    for k, m, n, _, _ in _groups(case):
        r, c = min(m, n), max(m, n)
        by += k * 4.0 * 5 * m * n  # W and M read and written, G read
        fl += k * case["steps"] * (1.0 * r * r * c + 1.0 * r ** 3 + 2.0 * r * r * c)  # X X^T and A A^T are symmetric
    return {"bytes": by, "flops": fl}


# ---- the same in 64 bits -----------------------------------------------------------------

def _q64(P):
    Q, R = torch.linalg.qr(P)
    return Q * torch.where(torch.diagonal(R, dim1=-2, dim2=-1) < 0, -1.0, 1.0).to(P.dtype).unsqueeze(-2)


def _step64(d, G, m, n, hp, refresh):
    """One step of a shape group in 64 bits (the steady state has no zero columns)."""
    f = lambda x: float(np.float32(x))  # noqa: E731  (the library takes its hyper-parameters in 32 bits)
    b, b1, b2, eps, lr, wd = (f(x) for x in (hp.factor_beta, hp.beta1, hp.beta2, hp.eps, hp.lr, hp.weight_decay))
    x = {k: v.double() for k, v in d.items() if k in ("W", "M", "V", "L", "R", "QL", "QR")}
    G = G.double()
    T = lambda a: a.transpose(1, 2)  # noqa: E731
    left, right = "QL" in x, "QR" in x
    Y, X, aL, aR = G, T(G), 1 - b, 1 - b
    if hp.kl and left and right:
        lam = lambda F, Q: (Q * (F @ Q)).sum(1).clamp_min(0)  # noqa: E731
        lamL, lamR = lam(x["L"], x["QL"]), lam(x["R"], x["QR"])
        Y = (G @ x["QR"]) * ((1 - b) / (n * (lamR + eps))).sqrt()[:, None, :]
        X = (T(G) @ x["QL"]) * ((1 - b) / (m * (lamL + eps))).sqrt()[:, None, :]
        aL = aR = 1.0
    elif hp.kl:
        aL, aR = (1 - b) / (n * (1 + eps)), (1 - b) / (m * (1 + eps))
    x["M"] = b1 * x["M"] + (1 - b1) * G
    g, mo = G, x["M"]
    if left:
        x["L"] = b * x["L"] + aL * (Y @ T(Y))
        if refresh:
            x["QL"] = _q64(x["L"] @ x["QL"])
        g, mo = T(x["QL"]) @ g, T(x["QL"]) @ mo
    if right:
        x["R"] = b * x["R"] + aR * (X @ T(X))
        if refresh:
            x["QR"] = _q64(x["R"] @ x["QR"])
        g, mo = g @ x["QR"], mo @ x["QR"]
    x["V"] = b2 * x["V"] + (1 - b2) * g * g
    u = mo / (x["V"].sqrt() + eps)
    if left:
        u = x["QL"] @ u
    if right:
        u = u @ T(x["QR"])
    x["W"] = (1 - lr * wd) * x["W"] - lr * u
    return x


def exact(case, seed):
    kind = case["kind"]
    if kind in ("soap", "resume"):
        refresh = 1001 % case["every"] == 0
        if work(case)["flops"] > 1.5e12:
            return None
        hp = _hparams(case)
        out = []
        for (k, m, n, _, _), d in zip(_groups(case), _soap_inputs(case, seed)):
            G = d.pop("G")[0]
            per = max(1, int(3e8 / (m * n + m * m + n * n)))
            parts = [_step64({p: v[i:i + per] for p, v in d.items()}, G[i:i + per], m, n, hp, refresh) for i in range(0, k, per)]
            out.append({p: torch.cat([q[p] for q in parts]) for p in parts[0]})
        if kind == "soap":
            return [o["W"] for o in out]
        return {"W": [o["W"] for o in out],
                "state": [{p: o[p][b] for p, _ in PIECES if p in o} for o in out for b in range(o["W"].shape[0])]}
    if kind == "qr":
        if work(case)["flops"] > 1.5e12:
            return None
        Q = torch.cat([_q64(p.double().unsqueeze(0)) for p in _qr_input(case, seed)])
        return {"Q": Q, "skip": None}
    if kind == "gemm":
        st = prepare(case, seed)
        out = torch.matmul(st["A"].double(), st["B"].double().transpose(1, 2))
        return out + case["beta"] * st["C0"].double() if case["beta"] else out
    return None  # Newton-Schulz in bf16 has no value in 64 bits that its rounding follows
