"""What the performance of this library is measured on: the calls that its users make, over the
range of sizes that they make them with.

Every case is one call (or one short sequence of calls) of the public Python entry points on
inputs resident on the GPU, except the scikit-learn style front end, which works on host arrays.
Signals follow the problem statement y = A x + noise with a planted sparse x.

    listed()            the cases
    draw(rng)           one more case of the same ranges
    prepare(case, seed) inputs, the handle and the prepared dictionary (what a program keeps)
    run(state)          one pass, and its outputs
    work(case)          bytes and operations one pass cannot do without
    exact(case, seed)   the outputs in 64 bits (plain torch), None where there is no such value
"""
from __future__ import annotations

import math

import torch

from paper_2407_06434_gb300 import omp, orthogonal_mp

DEV = "cuda"
TRAIN_STEPS = 4       # minibatches of one training pass
EXACT_FLOPS = 6e12    # the 64-bit solve of a larger case would take too long


def _solve(name, M, N, B, S, prec, **kw):
    return {"name": name, "kind": "solve", "M": M, "N": N, "B": B, "S": S, "s_min": S, "prec": prec,
            "coherent": False, "sigma": 1e-3, "eps": 0.0, **kw}


def listed():
    return [
        # A small dictionary and a handful of signals (the smoke test's problem): the shortest
        # call, all latency and launches.
        _solve("small_fp32", 64, 256, 16, 8, "fp32"),
        # One target over a large dictionary, as OrthogonalMatchingPursuit.fit(X, y) has it:
        # coding a signal as it arrives.
        _solve("one_signal_bf16", 1024, 8192, 1, 32, "bf16"),
        # Sparse coding of 16 x 16 image patches over a 4 x overcomplete dictionary.
        _solve("patches_bf16", 256, 1024, 5000, 32, "bf16"),
        # The default precision on the benchmark's batch: ordinary batched coding.
        _solve("batch_bf16", 1024, 8192, 4096, 32, "bf16"),
        # The largest dictionary, coherent atoms and the 8-bit correlation.
        _solve("coherent_fp8", 4096, 32768, 4096, 64, "fp8", coherent=True, sigma=1e-2, unit_coef=True),
        # Signals of very different sparsity stopped at a residual norm: the batch thins out.
        _solve("uneven_bf16", 2048, 16384, 8192, 128, "bf16", s_min=4, sigma=1e-6, eps=1e-3),
        # Plain single precision throughout (no quantised correlation), a ragged batch.
        _solve("plain_fp32", 1024, 8192, 1000, 32, "fp32"),
        # Few long atoms (face recognition): the solve in Gram space.
        {"name": "gram_face", "kind": "gram", "M": 8064, "N": 1207, "B": 1200, "S": 30, "s_min": 30,
         "prec": "bf16", "coherent": False, "sigma": 1e-3, "eps": 0.0},
        # Dictionary learning: the atoms have just been updated, so the dictionary is prepared
        # again and a minibatch is coded with it.
        {"name": "new_dictionary_bf16", "kind": "recode", "M": 1024, "N": 8192, "B": 1024, "S": 16,
         "s_min": 16, "prec": "bf16", "coherent": False, "sigma": 1e-3, "eps": 0.0},
        # The learned proposal: network inference, the restricted iteration and the fallback.
        {"name": "learned_bf16", "kind": "learned", "M": 1024, "N": 8192, "B": 4096, "S": 48, "s_min": 48,
         "prec": "bf16", "coherent": False, "sigma": 1e-3, "eps": 0.0, "hidden": 1024, "topk": 256},
        # Training the proposal: a few minibatches forward, backward and AdamW, then the weights.
        {"name": "train_proposal", "kind": "train", "M": 1024, "N": 8192, "B": 4096, "S": 48, "s_min": 48,
         "prec": "bf16", "coherent": False, "sigma": 1e-3, "eps": 0.0, "hidden": 1024, "topk": 256},
        # The scikit-learn style function on host arrays, from the numpy dictionary to the dense
        # coefficients: nothing is kept between calls.
        {"name": "sklearn_host", "kind": "estimator", "M": 512, "N": 2048, "B": 300, "S": 24, "s_min": 24,
         "prec": "bf16", "coherent": False, "sigma": 1e-3, "eps": 0.0},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _cost(c):
    """Rough seconds of a pass: the correlations, the gathered atom rows, the training GEMMs."""
    M, N, B, S = c["M"], c["N"], c["B"], c["S"]
    rate = {"fp32": 4e13, "bf16": 6e14, "fp8": 7e14}[c["prec"]]
    t = 2.0 * M * N * B * S / rate + 2.0 * B * S * (S + 20) * M / 8e12 + 20e-6 * S
    if c["kind"] in ("recode", "estimator"):
        t += 2.0 * M * N * N / 4e13
    if c["kind"] == "gram":
        t = 2.0 * M * N * B / 2e13 + 2.0 * B * S * S * N / 8e12
    if c["kind"] == "train":
        t = TRAIN_STEPS * 12.0 * B * N * c["hidden"] / 2e14
    return t


def draw(rng):
    while True:
        kind = rng.choice(["solve", "solve", "solve", "solve", "gram", "recode", "learned", "train", "estimator"])
        M = _log(rng, 48, 4096)
        N = min(32768, max(128, int(M * rng.uniform(1.5, 10))))
        B = _log(rng, 1, 8192)
        S = _log(rng, 4, min(128, M // 6 + 4))
        c = {"kind": kind, "M": M, "N": N, "B": B, "S": S, "s_min": S,
             "prec": rng.choice(["fp32", "bf16", "bf16", "fp8"]), "coherent": False, "sigma": 1e-3, "eps": 0.0}
        if kind == "solve":
            c["coherent"] = rng.random() < 0.25
            if rng.random() < 0.3:
                c.update(s_min=max(1, S // 8), eps=1e-3, sigma=1e-6)
        elif kind == "gram":
            c.update(M=_log(rng, 128, 8192), N=_log(rng, 128, 4096), S=_log(rng, 4, 48))
            c["S"] = c["s_min"] = min(c["S"], c["M"] // 6)
        elif kind == "recode":
            c.update(prec=rng.choice(["bf16", "fp8"]), S=min(S, 32))
            c["s_min"] = c["S"]
        elif kind in ("learned", "train"):
            c.update(M=_log(rng, 128, 1024), prec="bf16", hidden=rng.choice([256, 512, 1024]))
            c.update(N=64 * max(8, int(c["M"] * rng.uniform(3, 8) / 64)), S=min(48, c["M"] // 8))
            c.update(s_min=c["S"], topk=rng.choice([64, 128, 256]), B=max(64, B // 64 * 64) if kind == "train" else max(64, B))
            c["B"] = min(c["B"], 4096)
        else:
            c.update(M=_log(rng, 48, 1024), prec=rng.choice(["fp32", "bf16"]), B=_log(rng, 1, 1000))
            c.update(N=int(c["M"] * rng.uniform(1.5, 6)), S=_log(rng, 4, min(32, c["M"] // 6)))
            c["s_min"] = c["S"]
        c["coherent"] = c["coherent"] and c["N"] % 2 == 0
        if _cost(c) <= 0.04 and c["S"] <= min(c["M"], c["N"]):
            return c


# ------------------------------------------------------------------------------------- inputs
def _gen(seed, stream):
    g = torch.Generator(device=DEV)
    g.manual_seed(1000003 * int(seed) + stream)
    return g


def _dictionary(c, seed):
    """(N, M) atom rows of unit norm; A is its transpose (column-major)."""
    N, M = c["N"], c["M"]
    g = _gen(seed, 0)
    G = torch.randn((N, M), generator=g, device=DEV)
    if c["coherent"]:  # pairs of atoms that share a direction (inner product about 0.3)
        mate = torch.randperm(N, generator=g, device=DEV) % (N // 2)
        H = torch.randn((N // 2, M), generator=g, device=DEV)
        G = math.sqrt(0.7) * G + math.sqrt(0.3) * H[mate]
    G /= torch.linalg.vector_norm(G, dim=1, keepdim=True)
    return G.contiguous()


def _signals(c, At, seed, B=None):
    """Y (B, M) = planted signals plus noise, and the planted supports (B, S) int32, -1 padded."""
    N, M, S = c["N"], c["M"], c["S"]
    B = B or c["B"]
    g = _gen(seed, 1)
    sup = torch.empty((B, S), dtype=torch.int64, device=DEV)
    for lo in range(0, B, 1024):
        hi = min(B, lo + 1024)
        sup[lo:hi] = torch.rand((hi - lo, N), generator=g, device=DEV).topk(S, dim=1).indices
    if c.get("unit_coef"):
        coef = torch.rand((B, S), generator=g, device=DEV) * 0.5 + 0.5
        coef *= torch.randint(0, 2, (B, S), generator=g, device=DEV) * 2 - 1
    else:
        coef = torch.randn((B, S), generator=g, device=DEV)
    if c["s_min"] < S:
        n = torch.randint(c["s_min"], S + 1, (B, 1), generator=g, device=DEV)
        off = torch.arange(S, device=DEV)[None, :] >= n
        coef[off] = 0.0
        sup_out = torch.where(off, -1, sup).to(torch.int32)
    else:
        sup_out = sup.to(torch.int32)
    Y = torch.randn((B, M), generator=g, device=DEV) * c["sigma"]
    for j in range(S):
        Y += coef[:, j, None] * At[sup[:, j]]
    return Y.contiguous(), sup_out.contiguous()


def _weights(c, seed):
    """Initial parameters of the proposal network: small random layers, an output bias at the prior
    logit of an atom being in the support, and a skip term that spans a few logits."""
    N, H, S = c["N"], c["hidden"], c["S"]
    g = _gen(seed, 2)
    W1 = (torch.rand((H, N), generator=g, device=DEV) * 2 - 1) / (8 * math.sqrt(N))
    W2 = (torch.rand((N, H), generator=g, device=DEV) * 2 - 1) / (8 * math.sqrt(H))
    b1 = torch.zeros(H, device=DEV)
    b2 = torch.full((N,), math.log(S / (N - S)), device=DEV)
    beta = torch.full((1,), 4.0 * math.sqrt(c["M"]), device=DEV)
    return W1, b1, W2, b2, beta


def prepare(case, seed):
    c = case
    At = _dictionary(c, seed)
    if c["kind"] == "estimator":
        Y, _ = _signals(c, At, seed)
        return {"case": c, "X": At.t().cpu().numpy().copy(), "y": Y.t().cpu().numpy().copy()}
    st = {"case": c, "A": At.t()}
    st["Y"], sup = _signals(c, At, seed)
    st["solver"] = omp.OmpSolver(c["M"], c["N"], max_batch=c["B"], max_iters=c["S"], precision=c["prec"])
    if c["kind"] != "recode":
        omp.omp_prepare_dictionary(st["solver"].h, st["A"])
    if c["kind"] in ("learned", "train"):
        st["prop"] = omp.Proposal(st["solver"].h, hidden=c["hidden"], topk=c["topk"], train_batch=max(64, c["B"] // 64 * 64),
                                  pos_weight=(c["N"] - c["S"]) / c["S"])
        st["prop"].set_weights(*_weights(c, seed))
        if c["kind"] == "train":  # minibatches of their own, labelled with the planted supports
            more = [_signals(c, At, int(seed) + 7919 * (i + 1)) for i in range(TRAIN_STEPS - 1)]
            st["batches"] = [(st["Y"], sup)] + more
        else:  # the residual-drop thresholds, from a solve of other signals of the same kind
            Yc, _ = _signals(c, At, int(seed) + 7919, B=min(c["B"], 2048))
            X = torch.empty((Yc.shape[0], c["S"]), device=DEV)
            lab = torch.empty((Yc.shape[0], c["S"]), dtype=torch.int32, device=DEV)
            drops = torch.empty((Yc.shape[0], c["S"]), device=DEV)
            omp.omp_solve_batch_trace(st["solver"].h, st["A"], Yc, c["S"], 0.0, X, lab, drops)
            st["prop"].calibrate(drops, 1e-3)
    torch.cuda.synchronize()
    return st


# --------------------------------------------------------------------------------------- runs
def run(state):
    c = state["case"]
    if c["kind"] == "estimator":
        return orthogonal_mp(state["X"], state["y"], n_nonzero_coefs=c["S"], precision=c["prec"], return_n_iter=True)
    s, A, Y, B, S = state["solver"], state["A"], state["Y"], c["B"], c["S"]
    if c["kind"] == "solve":
        return s.solve(A, Y, S, c["eps"], diagnostics=True)
    if c["kind"] == "gram":
        return s.solve_gram(A, Y, S, c["eps"], diagnostics=True)
    if c["kind"] == "recode":
        omp.omp_prepare_dictionary(s.h, A)
        return s.solve(A, Y, S, c["eps"], diagnostics=True)
    if c["kind"] == "learned":
        X = torch.empty((B, S), device=DEV)
        sup = torch.empty((B, S), dtype=torch.int32, device=DEV)
        n_iter = torch.empty(B, dtype=torch.int32, device=DEV)
        resid = torch.empty(B, device=DEV)
        fallback = torch.empty(B, dtype=torch.int32, device=DEV)
        omp.omp_solve_batch_learned(s.h, state["prop"], A, Y, S, c["eps"], X, sup, n_iter, resid, fallback)
        return X, sup, n_iter, resid, fallback
    p, N, H = state["prop"], c["N"], c["hidden"]
    loss = torch.empty(TRAIN_STEPS, device=DEV)
    for i, (Yi, labels) in enumerate(state["batches"]):
        p.train_step(A, Yi, labels, loss[i:i + 1])
    W = [torch.empty(n, device=DEV) for n in ((H, N), H, (N, H), N, 1)]
    p.get_weights(*W)
    return [loss] + W


# --------------------------------------------------------------------------------------- work
def work(case):
    c = case
    M, N, B, S = c["M"], c["N"], c["B"], c["S"]
    out = B * S * 8 + B * 12
    if c["kind"] == "train":
        H = c["hidden"]
        params = 2 * N * H + N + H + 1
        # forward and backward GEMMs; the signals and labels, weights and both moments read and
        # written per step
        return {"bytes": TRAIN_STEPS * (B * (M + S) * 4 + M * N * 4 + params * 24) + params * 4,
                "flops": TRAIN_STEPS * (2 * B * N * M + 10 * B * N * H)}
    steps = S if c["s_min"] == S else (S + c["s_min"]) // 2  # steps a signal takes
    tri = 2 * B * steps * steps * M // 2     # the residual update's gathered rows, 2 per element
    b = 4 * M * N + 4 * B * M + out
    f = 2 * M * N * B * steps + tri
    if c["kind"] == "gram":                  # one correlation, then Gram rows
        f = 2 * M * N * B + B * steps * steps * N
        b += 4 * N * N
    elif c["kind"] == "recode":              # the Gram matrix, half of it (it is symmetric)
        f += M * N * N
        b += 4 * N * N
    elif c["kind"] == "estimator":
        f += M * N * N
        b = 4 * M * N + 4 * B * M + 4 * N * B
    elif c["kind"] == "learned":             # features, network, the candidates' correlations
        H, K = c["hidden"], c["topk"]
        f = 2 * B * N * M + 4 * B * N * H + 2 * B * K * M + B * steps * steps * K + tri
        b += 4 * 2 * N * H
    return {"bytes": int(b), "flops": int(f)}


# -------------------------------------------------------------------------------------- exact
def _omp64(At, Y, S, eps):
    """Alg. 1 in FP64: greedy picks of the largest |<r, a>| / ||a||, an orthonormal basis of the
    support by Gram-Schmidt (twice), coefficients by back-substitution. (X, support, ||r||)"""
    At, Y = At.double(), Y.double()
    B, M = Y.shape
    inv = 1.0 / torch.linalg.vector_norm(At, dim=1)
    ynorm = torch.linalg.vector_norm(Y, dim=1)
    r = Y.clone()
    Q = torch.zeros((B, S, M), dtype=torch.float64, device=At.device)
    Rm = torch.eye(S, dtype=torch.float64, device=At.device).repeat(B, 1, 1)
    beta = torch.zeros((B, S), dtype=torch.float64, device=At.device)
    sup = torch.full((B, S), -1, dtype=torch.int64, device=At.device)
    live = ynorm > 0
    for k in range(S):
        n = torch.empty(B, dtype=torch.int64, device=At.device)
        for lo in range(0, B, 1024):
            n[lo:lo + 1024] = ((r[lo:lo + 1024] @ At.t()).abs_() * inv).argmax(dim=1)
        v = At[n]
        for _ in range(2):
            if k:
                h = torch.einsum("bkm,bm->bk", Q[:, :k], v)
                v = v - torch.einsum("bk,bkm->bm", h, Q[:, :k])
                Rm[:, :k, k] += h
        d = torch.linalg.vector_norm(v, dim=1)
        q = torch.where(live[:, None], v / d[:, None], torch.zeros_like(v))
        Q[:, k] = q
        Rm[:, k, k] = torch.where(live, d, torch.ones_like(d))
        Rm[:, :k, k] = torch.where(live[:, None], Rm[:, :k, k], torch.zeros_like(Rm[:, :k, k]))
        b = torch.einsum("bm,bm->b", q, r)
        beta[:, k] = b
        r = r - b[:, None] * q
        sup[:, k] = torch.where(live, n, sup[:, k])
        live = live & (torch.linalg.vector_norm(r, dim=1) > eps * ynorm)
    X = torch.linalg.solve_triangular(Rm, beta[:, :, None], upper=True)[:, :, 0]
    return X, sup, torch.linalg.vector_norm(r, dim=1)


def _exact_train(c, seed):
    """TRAIN_STEPS AdamW steps of the proposal network in FP64 (lr 1e-3, betas 0.9 and 0.999)."""
    At = _dictionary(c, seed)
    batches = [_signals(c, At, seed)] + [_signals(c, At, int(seed) + 7919 * (i + 1)) for i in range(TRAIN_STEPS - 1)]
    At = At.double()
    At = At / torch.linalg.vector_norm(At, dim=1, keepdim=True)
    P = [p.double().requires_grad_(True) for p in _weights(c, seed)]
    m, v = [torch.zeros_like(p) for p in P], [torch.zeros_like(p) for p in P]
    pw = torch.tensor((c["N"] - c["S"]) / c["S"], dtype=torch.float64, device=DEV)
    losses = []
    for t, (Y, labels) in enumerate(batches, 1):
        x = (Y.double() @ At.t()) / torch.linalg.vector_norm(Y.double(), dim=1, keepdim=True)
        y = torch.zeros_like(x)
        y.scatter_(1, labels.long().clamp(min=0), (labels >= 0).double())
        W1, b1, W2, b2, beta = P
        o = torch.nn.functional.gelu(x @ W1.t() + b1) @ W2.t() + b2 + beta * x.abs()
        loss = torch.nn.functional.binary_cross_entropy_with_logits(o, y, pos_weight=pw)
        grads = torch.autograd.grad(loss, P)
        losses.append(loss.detach())
        with torch.no_grad():
            for p, g, mi, vi in zip(P, grads, m, v):
                mi.mul_(0.9).add_(g, alpha=0.1)
                vi.mul_(0.999).addcmul_(g, g, value=0.001)
                p -= 1e-3 * (mi / (1 - 0.9 ** t)) / ((vi / (1 - 0.999 ** t)).sqrt() + 1e-8)
    return [torch.stack(losses)] + [p.detach() for p in P]


def exact(case, seed):
    c = case
    if c["kind"] == "learned":
        return None
    if c["kind"] == "train":
        return _exact_train(c, seed) if TRAIN_STEPS * 12.0 * c["B"] * c["N"] * c["hidden"] <= EXACT_FLOPS else None
    if 2.0 * c["M"] * c["N"] * c["B"] * c["S"] > EXACT_FLOPS or 8.0 * c["B"] * c["S"] * c["M"] > 2e10:
        return None
    At = _dictionary(c, seed)
    Y, _ = _signals(c, At, seed)
    X, sup, rn = _omp64(At, Y, c["S"], c["eps"])
    if c["kind"] == "estimator":
        coef = torch.zeros((c["B"], c["N"]), dtype=torch.float64, device=DEV)
        coef.scatter_(1, sup.clamp(min=0), torch.where(sup >= 0, X, torch.zeros_like(X)))
        return coef.t(), None
    return X, None, None, rn, None
