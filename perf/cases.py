"""The workloads whose speed matters: every public operation of the package over
the range of sizes, data types and options that a speculative-decoding server
and its draft-model trainer give it.

``listed()`` names representative calls, ``draw(rng)`` gives more of the same
ranges, ``prepare`` makes a call's inputs on the GPU and the buffers a program
keeps beside them, ``run`` makes the call, and ``exact`` computes what it should
return in 64-bit floating point with plain torch.
"""
from __future__ import annotations

import math

import torch

import paper_2310_07177_gb300 as osd

DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16}

# A Medusa-style static tree of 26 candidates under the root (parent of each node).
MEDUSA = "-1,0,0,0,0,1,1,1,2,2,3,4,5,5,6,7,8,9,11,12,12,13,14,16,18,19,20"
MOST_BYTES = 65536 * 32000 * 8  # the largest listed case; drawn ones stay below it


def _verify(name, B, k, V, dtype, T, std, scale, noise, fresh=False):
    return {"name": name, "op": "verify", "B": B, "k": k, "V": V, "dtype": dtype, "T": T, "std": std,
            "scale": scale, "noise": noise, "fresh": fresh}


def _distill(name, N, V, dtype, kind, beta=0.5, tau=1.0, active=1.0, view=0, noise=2.0, peak=0.0):
    return {"name": name, "op": "distill", "N": N, "V": V, "dtype": dtype, "kind": kind, "beta": beta, "tau": tau,
            "active": active, "view": view, "noise": noise, "peak": peak}


def listed():
    return [
        # One decoding step of a small batch, logits in fp32, results in fresh tensors: latency.
        _verify("verify_tiny", 4, 4, 32000, "f32", 1.0, 2.0, 1.0, 1.0, fresh=True),
        # One decoding step of an ordinary serving batch, results in the server's own buffers.
        _verify("verify_serving", 32, 5, 32000, "bf16", 1.0, 2.5, 0.7, 1.5),
        # The same batch decoded greedily (temperature 0): argmax matching.
        _verify("greedy_serving", 32, 5, 32000, "bf16", 0.0, 2.5, 0.7, 1.5),
        # A large batch with a 128k vocabulary and a draft that is often wrong.
        _verify("verify_large", 256, 8, 128256, "bf16", 0.7, 3.0, 0.5, 2.0),
        # The positions that batch rejected go to the trainer at once, chosen on the device.
        {"name": "rejected_large", "op": "accepted", "B": 256, "k": 8, "V": 128256, "dtype": "bf16", "kind": "fkl",
         "beta": 0.5, "tau": 1.0, "accept": 0.5, "noise": 2.0},
        # Distillation of the few positions of one small step, target rows read in place through strides.
        _distill("distill_tiny", 16, 32000, "f32", "fkl", view=4, noise=1.0),
        # A full distillation buffer flushed: the bulk of the training side's time.
        _distill("flush_rkl", 65536, 32000, "bf16", "rkl"),
        # A flush of a buffer of which 40 % of the positions count, generalised JSD.
        _distill("flush_masked", 16384, 32128, "bf16", "jsd", active=0.4, noise=1.0, peak=8.0),
        # A flush with a vocabulary of odd size (one token added to 32000): rows of no alignment.
        _distill("flush_odd", 4096, 32001, "bf16", "tvd"),
        # A flush with a 128k vocabulary.
        _distill("flush_wide", 2048, 128256, "bf16", "fkl"),
        # Tokens for training data drawn from the mixture of draft and target.
        {"name": "mixed", "op": "mixed", "N": 16384, "V": 32000, "dtype": "bf16", "beta": 0.5, "tau": 1.0, "noise": 2.0},
        # One decoding step with several candidates a position.
        {"name": "tree", "op": "tree", "B": 32, "V": 32000, "dtype": "bf16", "T": 1.0, "noise": 1.0, "parents": MEDUSA},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _vocab(rng):
    v = _log_int(rng, 4000, 160000)
    how = rng.random()
    if how < 0.6:
        return max(64, v // 64 * 64)  # padded, as most models are
    if how < 0.75:
        return max(4, v // 4 * 4)
    return v


def draw(rng):
    op = rng.choice(["verify"] * 4 + ["distill"] * 5 + ["accepted"] * 2 + ["mixed"] * 2 + ["tree"] * 2)
    V, dtype = _vocab(rng), rng.choice(["bf16", "bf16", "bf16", "f32"])
    es = 2 if dtype == "bf16" else 4
    noise = round(rng.uniform(0.2, 2.5), 2)  # how far the draft is from the target: from nearly always right to often wrong
    if op == "verify":
        T = rng.choice([0.0, 0.7, 1.0, 1.0, 1.3])
        c = _verify("", _log_int(rng, 1, 256), rng.randint(1, 8), V, dtype, T, 2.5, rng.choice([0.7, 1.0]), noise,
                    fresh=rng.random() < 0.5)
    elif op == "distill":
        kind = rng.choice(["fkl", "rkl", "jsd", "tvd", "ce"])
        most = max(1, min(65536, MOST_BYTES // (V * (2 * es + 4))))
        c = _distill("", _log_int(rng, 1, most), V, dtype, kind, rng.choice([0.1, 0.5, 0.9]), rng.choice([1.0, 1.0, 0.7, 2.0]),
                     rng.choice([1.0, 1.0, 0.4, 0.8]), rng.choice([0, 0, 4]), noise, rng.choice([0.0, 0.0, 8.0]))
    elif op == "accepted":
        c = {"op": "accepted", "B": _log_int(rng, 1, 256), "k": rng.randint(1, 8), "V": V, "dtype": dtype,
             "kind": rng.choice(["fkl", "rkl", "jsd", "tvd", "ce"]), "beta": 0.5, "tau": rng.choice([1.0, 0.7]),
             "accept": round(rng.uniform(0.3, 0.9), 2), "noise": noise}
    elif op == "mixed":
        most = max(1, min(65536, MOST_BYTES // (2 * V * es)))
        c = {"op": "mixed", "N": _log_int(rng, 1, most), "V": V, "dtype": dtype, "beta": rng.choice([0.1, 0.5, 0.9]),
             "tau": rng.choice([1.0, 0.7]), "noise": noise}
    else:
        n = rng.randint(3, 32)
        parents = [-1]
        for i in range(1, n):  # each node under one of the few before it, so that trees are both wide and deep
            parents.append(rng.randint(max(0, (i - 1) // 4), max(0, (i - 1) // 2)))
        c = {"op": "tree", "B": _log_int(rng, 1, 64), "V": V, "dtype": dtype, "T": rng.choice([0.0, 0.7, 1.0, 1.0]),
             "noise": noise, "parents": ",".join(str(p) for p in parents)}
    c.pop("name", None)
    return c


# ------------------------------------------------------------------ inputs
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _normal(shape, std, g, dtype, base=None, scale=1.0):
    """N(0, std^2) plus scale times base, rounded to dtype; made in pieces to bound the fp32 temporaries."""
    out = torch.empty(shape, dtype=dtype, device="cuda")
    flat = out.view(-1, shape[-1])
    rows = max(1, (1 << 28) // shape[-1])
    for r in range(0, flat.shape[0], rows):
        x = torch.empty(flat[r:r + rows].shape, device="cuda").normal_(0.0, std, generator=g)
        if base is not None:
            x.add_(base.reshape(-1, shape[-1])[r:r + rows].float(), alpha=scale)
        flat[r:r + rows] = x
    return out


def _proposals(z, T, g):
    """One token of each row of z from softmax(z / T), by the Gumbel-max trick."""
    u = torch.rand(z.shape, generator=g, device="cuda").clamp_(min=1e-12)
    return torch.argmax(z.float() / T - torch.log(-torch.log(u)), dim=-1).to(torch.int32)


def _parents(case):
    return [int(p) for p in case["parents"].split(",")]


def prepare(case, seed):
    g, dt, V = _gen(seed), DTYPES[case["dtype"]], case["V"]
    s = dict(case)
    i32, dev = torch.int32, "cuda"
    op = case["op"]
    if op == "verify":
        B, k, T = case["B"], case["k"], case["T"]
        z = _normal((B, k, V), case["std"], g, dt)
        t = torch.empty(B, k + 1, V, dtype=dt, device=dev)
        t[:, :k] = _normal((B, k, V), case["noise"], g, dt, z, case["scale"])
        t[:, k] = _normal((B, V), case["std"], g, dt)
        s["tokens"] = torch.empty(B, k, dtype=i32, device=dev)
        for i in range(k):
            s["tokens"][:, i] = _proposals(z[:, i], T, g) if T > 0 else torch.argmax(z[:, i].float(), dim=-1).to(i32)
        s["u"] = torch.rand(B, k + 1, generator=g, device=dev)
        s["draft"], s["target"] = z, t
        if not case["fresh"]:  # a server's own buffers; it watches the accept margins
            s["workspace"] = torch.empty(osd.osd_verify_workspace_size(B, k, V), dtype=torch.uint8, device=dev)
            margin = torch.zeros(B, k, device=dev) if T > 0 else None
            s["out"] = osd.VerifyResult(torch.zeros(B, dtype=i32, device=dev), torch.zeros(B, k + 1, dtype=i32, device=dev),
                                        torch.zeros(B, k, dtype=torch.uint8, device=dev), margin, None)
    elif op == "tree":
        B, par = case["B"], _parents(case)
        n, T = len(par), case["T"]
        z = _normal((B, n, V), 2.0, g, dt)
        s["draft"], s["target"], s["parent"] = z, _normal((B, n, V), case["noise"], g, dt, z), par
        s["tokens"] = torch.zeros(B, n, dtype=i32, device=dev)
        for i in range(1, n):
            row = z[:, par[i]]
            first = par.index(par[i]) == i
            s["tokens"][:, i] = torch.argmax(row.float(), dim=-1).to(i32) if T == 0 and first else _proposals(row, T or 1.0, g)
        s["u"] = torch.rand(B, n, generator=g, device=dev)
        s["workspace"] = torch.empty(max(16, osd.osd_verify_tree_workspace_size(B, n, V)), dtype=torch.uint8, device=dev)
        margin = torch.zeros(B, n, device=dev) if T > 0 else None
        s["out"] = osd.TreeResult(torch.zeros(B, dtype=i32, device=dev), torch.zeros(B, n, dtype=i32, device=dev),
                                  torch.zeros(B, n, dtype=i32, device=dev), torch.zeros(B, dtype=i32, device=dev), margin, None)
    elif op == "accepted":
        B, k = case["B"], case["k"]
        z = _normal((B, k, V), 2.5, g, dt)
        t = torch.empty(B, k + 1, V, dtype=dt, device=dev)
        t[:, :k] = _normal((B, k, V), case["noise"], g, dt, z)
        t[:, k] = z[:, 0]
        # the leading accepted tokens of each sequence, each accepted with the same probability
        fails = torch.rand(B, k, generator=g, device=dev) >= case["accept"]
        s["accepted"] = torch.where(fails.any(1), fails.int().argmax(1), k).to(i32)
        s["draft"], s["target"] = z, t
        s["out"] = osd.DistillAcceptedResult(torch.zeros(B, device=dev), torch.zeros(B, V, device=dev),
                                             torch.zeros(B, dtype=i32, device=dev), torch.zeros(1, dtype=i32, device=dev))
    elif op == "distill":
        N, p = case["N"], case["view"]  # N rows, or N // p groups of p
        lead = (max(1, N // p), p) if p else (N,)
        z = _normal(lead + (V,), 2.0, g, dt)
        if case["peak"]:
            t = _normal(lead + (V,), case["noise"], g, torch.float32 if math.prod(lead) * V < (1 << 26) else dt)
            hot = torch.randint(0, V, (math.prod(lead), 1), generator=g, device=dev)
            flat = t.view(-1, V)
            flat.scatter_(1, hot, flat.gather(1, hot) + case["peak"])
            t = t.to(dt)
        else:
            t = _normal(lead + (V,), case["noise"], g, dt, z)
        if p:  # rows of a [N, p + 1, V] tensor, as verification reads them
            whole = torch.zeros(lead[0], p + 1, V, dtype=dt, device=dev)
            whole[:, :p] = t
            t = whole[:, :p]
        s["draft"], s["target"], s["mask"] = z, t, None
        if case["active"] < 1.0:
            n = math.prod(lead)
            s["mask"] = torch.zeros(n, dtype=torch.uint8, device=dev)
            s["mask"][torch.randperm(n, generator=g, device=dev)[:max(1, round(case["active"] * n))]] = 1
            s["mask"] = s["mask"].view(lead)
        # the trainer's gradient buffer: inactive rows keep the zeros it put there
        s["loss"], s["dlogits"] = torch.zeros(lead, device=dev), torch.zeros(lead + (V,), device=dev)
    else:
        z = _normal((case["N"], V), 2.0, g, dt)
        s["draft"], s["target"] = z, _normal((case["N"], V), case["noise"], g, dt, z)
        s["u"] = torch.rand(case["N"], generator=g, device=dev)
    return s


def run(s):
    op = s["op"]
    if op == "verify":
        if s["fresh"]:
            return osd.osd_verify(s["draft"], s["target"], s["tokens"], s["u"], s["T"], diagnostics=False)[:3]
        return osd.osd_verify(s["draft"], s["target"], s["tokens"], s["u"], s["T"], workspace=s["workspace"], out=s["out"])[:4]
    if op == "tree":
        return osd.osd_verify_tree(s["draft"], s["target"], s["parent"], s["tokens"], s["u"], s["T"],
                                   workspace=s["workspace"], out=s["out"])[:5]
    if op == "accepted":
        return tuple(osd.osd_distill_accepted(s["draft"], s["target"], s["accepted"], s["kind"], s["beta"],
                                              temperature=s["tau"], out=s["out"]))
    if op == "distill":
        return osd.osd_distill(s["draft"], s["target"], s["mask"], s["kind"], s["beta"], temperature=s["tau"],
                               loss=s["loss"], dlogits=s["dlogits"])
    return osd.osd_mixed_sample(s["draft"], s["target"], s["u"], s["beta"], temperature=s["tau"])[0]


def work(case):
    """Each input read once and each output written once (a masked-out or unchosen row counts nothing); the
    operations are about one exponential's worth (8) and a few sums an entry."""
    V, es, op = case["V"], DTYPES[case["dtype"]].itemsize, case["op"]
    if op == "verify":
        B, k = case["B"], case["k"]
        rows = B * (k + 1) if case["T"] == 0 else B * (2 * k + 1)
        return {"bytes": rows * V * es + B * (4 * k + 4 * (k + 1) * 2 + 4 + k), "flops": 12 * rows * V}
    if op == "tree":
        n = len(_parents(case))
        rows = case["B"] * n * (1 if case["T"] == 0 else 2)
        return {"bytes": rows * V * es + case["B"] * n * 16, "flops": 12 * rows * V}
    if op == "mixed":
        return {"bytes": case["N"] * (2 * V * es + 8), "flops": 24 * case["N"] * V}
    if op == "accepted":
        rows = case["B"] * (1.0 - case["accept"] ** case["k"])  # the expected number of rejecting sequences
    else:
        p = case["view"]
        n = max(1, case["N"] // p) * p if p else case["N"]
        rows = max(1, round(case["active"] * n)) if case["active"] < 1.0 else n
    return {"bytes": int(rows * (V * (2 * es + 4) + 4)), "flops": int(50 * rows * V)}


def tolerance(case):
    op = case["op"]
    if op == "mixed":
        return {"rel": 0.0, "differ": 0.005}
    if op in ("verify", "tree"):
        return {"rel": 1e-5, "differ": 0.01}
    if case["kind"] == "tvd":  # a tie of p and q within rounding may take either sign
        return {"rel": 3e-4, "max": 0.99}
    # the nearer the two rows, the smaller the loss that is left of its cancelling terms
    near = min(1.0, case["noise"] / case["tau"]) if not case.get("peak") else 1.0
    return {"rel": max(1e-5, {"jsd": 3e-5, "fkl": 3e-6, "rkl": 3e-6}.get(case["kind"], 0.0) / near ** 2)}


# ------------------------------------------------------------------ 64-bit results
def _first_argmax(x):
    """The lowest index of the maximum of each row."""
    at = torch.where(x == x.max(-1, keepdim=True).values, torch.arange(x.shape[-1], device=x.device), x.shape[-1])
    return at.min(-1).values


def _draw_token(w, u):
    """min{ j : C_j > u W } of non-negative weights w."""
    C = torch.cumsum(w, -1)
    W = C[..., -1:]
    past = C > u * W
    hit = _first_argmax(past.int())
    last = w.shape[-1] - 1 - _first_argmax((w > 0).flip(-1).int())
    return torch.where(past.any(-1), hit, last)


def _exact_verify(s):
    z, t, T = s["draft"], s["target"], s["T"]
    B, k1, V = t.shape
    k = k1 - 1
    y = s["tokens"].long()
    nan = float("nan")
    acc = torch.full((B,), k, dtype=torch.int32, device="cuda")
    tok = torch.full((B, k + 1), -1, dtype=torch.int32, device="cuda")
    mask = torch.zeros(B, k, dtype=torch.uint8, device="cuda")
    margin = torch.full((B, k), nan, dtype=torch.float64, device="cuda")
    for b in range(B):
        for i in range(k + 1):
            if T == 0:
                best = _first_argmax(t[b, i])
                if i == k or y[b, i] != best:
                    tok[b, i] = best.int()
                    break
            else:
                p = torch.softmax(t[b, i].double() / T, -1)
                if i == k:
                    tok[b, i] = _draw_token(p, s["u"][b, k].double()).int()
                    break
                q = torch.softmax(z[b, i].double() / T, -1)
                r = p[y[b, i]] / q[y[b, i]]
                u = s["u"][b, i].double()
                margin[b, i] = (u - r).abs()
                if not u < r:
                    tok[b, i] = _draw_token((p - q).clamp_(min=0), s["u"][b, k].double()).int()
                    break
            tok[b, i] = y[b, i].int()
        acc[b] = i
        if i < k:
            mask[b, i] = 1
    if s["fresh"]:
        return acc, tok, mask
    return acc, tok, mask, margin if T > 0 else None


def _exact_tree(s):
    z, t, T, par = s["draft"], s["target"], s["T"], s["parent"]
    B, n, V = t.shape
    i32 = torch.int32
    acc, last = torch.zeros(B, dtype=i32, device="cuda"), torch.zeros(B, dtype=i32, device="cuda")
    path, tok = torch.full((B, n), -1, dtype=i32, device="cuda"), torch.full((B, n), -1, dtype=i32, device="cuda")
    margin = torch.full((B, n), float("nan"), dtype=torch.float64, device="cuda")
    ys, us = s["tokens"].tolist(), s["u"].double().tolist()
    for b in range(B):
        node, depth = 0, 0
        while True:
            kids = [c for c in range(n) if par[c] == node]
            go = -1
            if T == 0:
                best = int(_first_argmax(t[b, node]))
                go = next((c for c in kids if ys[b][c] == best), -1)
                if go < 0:
                    tok[b, depth] = best
            else:
                r = torch.softmax(t[b, node].double() / T, -1)
                q = torch.softmax(z[b, node].double() / T, -1)
                for c in kids:
                    ratio = float(r[ys[b][c]] / q[ys[b][c]])
                    margin[b, c] = abs(us[b][c] - ratio)
                    if us[b][c] < ratio:
                        go = c
                        break
                    r = (r - q).clamp_(min=0)
                    r /= r.sum()
                if go < 0:
                    tok[b, depth] = int(_draw_token(r, us[b][0]))
            if go < 0:
                break
            path[b, depth], tok[b, depth] = go, ys[b][go]
            node, depth = go, depth + 1
        acc[b], last[b] = depth, node
    return acc, path, tok, last, margin if T > 0 else None


def _exact_rows(z, t, kind, beta, tau):
    """Loss and gradient of some rows, in 64 bits."""
    lq, lp = torch.log_softmax(z.double() / tau, -1), torch.log_softmax(t.double() / tau, -1)
    q, p = lq.exp(), lp.exp()
    if kind == "fkl":
        return (p * (lp - lq)).sum(-1), (q - p) / tau
    if kind == "rkl":
        d = lq - lp
        loss = (q * d).sum(-1)
        return loss, q * (d - loss[:, None]) / tau
    if kind == "jsd":
        lm = torch.log(beta * p + (1 - beta) * q)
        kp, kq = (p * (lp - lm)).sum(-1), (q * (lq - lm)).sum(-1)
        return beta * kp + (1 - beta) * kq, (1 - beta) * q * (lq - lm - kq[:, None]) / tau
    if kind == "tvd":
        sg = 0.5 * torch.sign(q - p)
        return 0.5 * (q - p).abs().sum(-1), q * (sg - (q * sg).sum(-1, keepdim=True)) / tau
    y = _first_argmax(t)[:, None]
    grad = q.scatter_add(1, y, torch.full_like(y, -1, dtype=torch.float64)) / tau
    return -lq.gather(1, y)[:, 0], grad


def _exact_distill(z, t, rows, kind, beta, tau, n_out, V):
    loss = torch.zeros(n_out, dtype=torch.float64, device="cuda")
    grad = torch.zeros(n_out, V, dtype=torch.float64, device="cuda")
    step = max(1, (1 << 27) // V)
    for r in range(0, len(rows), step):
        zi, ti, out = z(rows[r:r + step]), t(rows[r:r + step]), rows[r:r + step]
        loss[out], grad[out] = _exact_rows(zi, ti, kind, beta, tau)
    return loss, grad


def exact(case, seed):
    s = prepare(case, seed)
    V, op = case["V"], case["op"]
    if op == "verify":
        return _exact_verify(s)
    if op == "tree":
        return _exact_tree(s)
    if op == "mixed":
        out = torch.empty(case["N"], dtype=torch.int32, device="cuda")
        step = max(1, (1 << 27) // V)
        for r in range(0, case["N"], step):
            p = torch.softmax(s["target"][r:r + step].double() / case["tau"], -1)
            q = torch.softmax(s["draft"][r:r + step].double() / case["tau"], -1)
            w = case["beta"] * p + (1 - case["beta"]) * q
            out[r:r + step] = _draw_token(w, s["u"][r:r + step, None].double()).int()
        return out
    if op == "accepted":
        B, k, a = case["B"], case["k"], s["accepted"].long()
        b = torch.arange(B, device="cuda")
        on = a < k
        order = torch.cat([b[on], b[~on]])
        count = int(on.sum())
        z = lambda r: s["draft"][order[r], a[order[r]]]
        t = lambda r: s["target"][order[r], a[order[r]]]
        loss, grad = _exact_distill(z, t, torch.arange(count, device="cuda"), case["kind"], case["beta"], case["tau"], B, V)
        return loss, grad, order.int(), torch.tensor([count], dtype=torch.int32, device="cuda")
    lead = s["draft"].shape[:-1]
    n = math.prod(lead)
    rows = torch.arange(n, device="cuda") if s["mask"] is None else s["mask"].view(-1).nonzero()[:, 0]
    zf = s["draft"].reshape(-1, V)
    if case["view"]:
        p = case["view"]
        t = lambda r: s["target"][r // p, r % p]
    else:
        t = lambda r: s["target"][r]
    s["dlogits"] = None
    loss, grad = _exact_distill(lambda r: zf[r], t, rows, case["kind"], case["beta"], case["tau"], n, V)
    return loss.view(lead), grad.view(*lead, V)
