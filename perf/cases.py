"""The calls that a serving program makes of this framework, with inputs, sizes and tolerances.

Every case goes through the public binding (``paper_2609_09338_gb300.binding`` and the buffer classes of
``session``) the way an engine does: contexts, caches and workspaces are made once, a pass is one call.

Weights.  Matrices are N(0, 0.02^2) as in the repository's synthetic drafters, the embedding is N(0, 1), and each
token t has one or four preferred successors: the LM-head row of a successor carries a multiple of embed[t].  The
draft distribution is then peaked on a few tokens, as a trained drafter's is, and a draw does not hang on the last
bit of a cumulative sum (with a head of pure noise every id has a probability of 1/V, and a change of rounding
moves the draw and, with it, the rest of the chain).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2609_09338_gb300 import binding as ob
from paper_2609_09338_gb300 import workloads as wl
from paper_2609_09338_gb300.session import TreeVerifyBuffers, VerifyBuffers, VerifyHiddenBuffers

DEV = "cuda"
BF = torch.bfloat16
SHAPES = {"d1024-v151936": wl.QWEN3_8B_DRAFTER, "d2048-v128256": wl.LLAMA70B_DRAFTER,
          "d1024-v200064": wl.LARGE_VOCAB_DRAFTER, "d2560-v151936": wl.OSPREY_PAPER_DRAFTER,
          "d4096-v151936": wl.DFLASH_DRAFTER, "d256-v4096": wl.TINY}


# ---------------------------------------------------------------- cases
def _draft(name, shape, B, K, ctx_lo, ctx_hi, max_new, T, out="logits", topk=1):
    return {"name": name, "kind": "draft", "shape": shape, "B": B, "K": K, "ctx_lo": ctx_lo, "ctx_hi": ctx_hi,
            "max_new": max_new, "T": T, "out": out, "topk": topk}


def _verify(name, V, B, K, T, dtype):
    return {"name": name, "kind": "verify", "V": V, "B": B, "K": K, "T": T, "dtype": dtype, "sigma": 0.7}


def listed():
    return [
        # one stream, one new token a call: the interactive step, bound by the LM head and by launch latency
        _draft("draft-b1", "d1024-v151936", 1, 7, 2048, 2048, 1, 1.0),
        # one stream of the paper-shaped two-layer drafter; the call first extends by what the last verify accepted
        _draft("draft-b1-ext8", "d2560-v151936", 1, 7, 2048, 2048, 8, 0.0),
        # a full server in its steady state: ragged numbers of accepted rows (1..8 of max_new 8) for 96 sequences
        _draft("draft-b96-ext8", "d1024-v151936", 96, 7, 1024, 4096, 8, 0.0),
        # long ragged contexts and the large vocabulary, states kept for the logits-free verification
        _draft("draft-b64-long", "d1024-v200064", 64, 8, 1024, 16384, 1, 1.0, out="hidden"),
        # tree drafting: four candidates a step, ragged extend rows, two layers
        _draft("draft-tree-b16", "d2048-v128256", 16, 5, 2048, 8192, 6, 0.0, topk=4),
        # block drafting: 15 proposals a sequence from one forward over anchor and masks
        {"name": "block-b8", "kind": "block", "shape": "d4096-v151936", "B": 8, "block": 16, "ctx_lo": 1024,
         "ctx_hi": 4096, "T": 1.0},
        # verification of one stream: the smallest call, all latency
        _verify("verify-b1", 151936, 1, 7, 1.0, "f32"),
        # a full batch with half-precision logits
        _verify("verify-b64-bf16", 200064, 64, 8, 1.0, "bf16"),
        # a vocabulary that is no multiple of a vector: rows start at odd addresses
        _verify("verify-b32-odd", 151643, 32, 5, 0.7, "f32"),
        # a full batch without draft logits in memory
        {"name": "verify-hidden-b64", "kind": "verify_hidden", "shape": "d1024-v200064", "B": 64, "K": 8, "T": 1.0,
         "dtype": "bf16", "sigma": 0.7},
        # verification of a drafted tree
        {"name": "verify-tree-b8", "kind": "verify_tree", "V": 151936, "B": 8, "K": 5, "topk": 4, "T": 1.0,
         "dtype": "f32", "sigma": 0.7},
        # prefill: the prompt's K/V rows of a batch go to the pages
        {"name": "append-b32", "kind": "append", "shape": "d1024-v151936", "B": 32, "ctx_lo": 128, "ctx_hi": 4096},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _odd(rng, v):
    return v | 1 if rng.random() < 0.5 else v


def draw(rng):
    kind = rng.choice(["draft", "draft", "draft", "draft", "block", "verify", "verify", "verify_hidden", "verify_tree",
                       "append"])
    dtype = rng.choice(["f32", "bf16"])
    if kind == "draft":
        shape, top = rng.choice([("d1024-v151936", 96), ("d2048-v128256", 48), ("d1024-v200064", 64),
                                 ("d2560-v151936", 24), ("d256-v4096", 96)])
        B, K = _log_int(rng, 1, top), rng.randint(1, 8)
        hi = _log_int(rng, 64, min(16384, 64 * 8192 // B))
        max_new = rng.choice([1, K + 1, rng.randint(1, 8)])
        topk = rng.choice([1, 1, rng.randint(2, 8)]) if B <= 80 else 1
        T = rng.choice([0.0, 0.7, 1.0]) if topk == 1 else 0.0
        out = rng.choice(["logits", "hidden"]) if topk == 1 else "logits"
        c = _draft("", shape, B, K, rng.randint(16, hi), hi, max_new, T, out, topk)
    elif kind == "block":
        c = {"kind": kind, "shape": rng.choice(["d4096-v151936", "d1024-v151936"]), "B": _log_int(rng, 1, 16),
             "block": rng.randint(4, 24), "ctx_lo": 64, "ctx_hi": rng.randint(64, 4096), "T": rng.choice([0.0, 1.0])}
    elif kind == "verify":
        V = _odd(rng, _log_int(rng, 4096, 200064))
        c = _verify("", V, _log_int(rng, 1, 256), rng.randint(1, 8), rng.choice([0.0, 0.7, 1.0]), dtype)
    elif kind == "verify_hidden":
        c = {"kind": kind, "shape": rng.choice(["d1024-v151936", "d1024-v200064", "d2048-v128256"]),
             "B": _log_int(rng, 1, 128), "K": rng.randint(1, 8), "T": rng.choice([0.7, 1.0]), "dtype": dtype,
             "sigma": 0.7}
    elif kind == "verify_tree":
        c = {"kind": kind, "V": _odd(rng, _log_int(rng, 4096, 200064)), "B": _log_int(rng, 1, 32),
             "K": rng.randint(1, 6), "topk": rng.randint(2, 8), "T": rng.choice([0.0, 0.7, 1.0]), "dtype": dtype,
             "sigma": 0.7}
    else:
        hi = _log_int(rng, 8, 8192)
        c = {"kind": kind, "shape": rng.choice(["d1024-v151936", "d2048-v128256"]), "B": _log_int(rng, 1, 64),
             "ctx_lo": rng.randint(1, hi), "ctx_hi": hi}
    c.pop("name", None)
    return c


# ---------------------------------------------------------------- inputs
def _gen(seed, salt):
    return torch.Generator(device=DEV).manual_seed((seed * 1000003 + salt) % (1 << 62))


def _normal(g, shape, std=1.0, mean=0.0):
    out = torch.empty(shape, dtype=BF, device=DEV)
    flat, step = out.view(-1), 1 << 26
    for s in range(0, flat.numel(), step):
        part = flat[s:s + step]
        part.copy_(torch.randn(part.numel(), generator=g, device=DEV) * std + mean)
    return out


def _weights(sh, seed, successors):
    g, d, V = _gen(seed, 1), sh.d_model, sh.vocab
    a = sh.n_q_heads * sh.head_dim
    w = {"W_c": _normal(g, (d, sh.feat_dim), 0.02), "embed": _normal(g, (V, d)),
         "final_norm": _normal(g, (d,), 0.02, 1.0), "lm_head": _normal(g, (V, d), 0.02)}
    names = ("attn_norm", "W_qkv", "W_o", "ffn_norm", "W_gate", "W_up", "W_down")
    shapes = ((d,), (sh.qkv_rows, 2 * d), (d, a), (d,), (sh.ffn_dim, d), (sh.ffn_dim, d), (d, sh.ffn_dim))
    for n, s in zip(names, shapes):
        w[n] = [_normal(g, s, 0.02, 1.0 if len(s) == 1 else 0.0) for _ in range(sh.n_layers)]
    for m in w["W_qkv"]:   # the context columns start at zero (Sec. 3.3) and stay small: at 0.02 the fed-back state
        m[:, :d].mul_(0.25)   # makes q and k of random layers so large that a chain amplifies the last bit threefold a step
    # the layers' own contributions dilute the embedding in the residual stream: the gain makes up for it
    dilution = math.sqrt(1 + sh.n_layers * d / 2560)
    gains = [40.0] if successors == 1 else [37.0, 33.0, 32.5, 32.0]
    for gain in (x * dilution for x in gains):
        succ = torch.randperm(V, generator=g, device=DEV)   # succ[j]: the token whose successor is j
        for s in range(0, V, 1 << 15):
            part = w["lm_head"][s:s + (1 << 15)]
            part.copy_(part.float() + w["embed"][succ[s:s + (1 << 15)]].float() * (gain / d))
    return w


def _cpu(seed, salt):
    return np.random.default_rng([seed, salt])


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


def _contexts(case, seed):
    return _cpu(seed, 2).integers(case["ctx_lo"], case["ctx_hi"] + 1, size=case["B"]).astype(np.int32)


def _cache(sh, ctx, reserve, ctx_hi, seed, fill=True):
    B = len(ctx)
    max_pages = -(-(ctx_hi + reserve) // 16)
    table = _cpu(seed, 3).permutation(B * max_pages).reshape(B, max_pages).astype(np.int32)
    kv = ob.alloc_kv(sh, table, B * max_pages, DEV)
    if fill:
        g = _gen(seed, 4)
        for pages in (kv.k_pages, kv.v_pages):
            pages.copy_(_normal(g, tuple(pages.shape)))
        kv.seq_len.copy_(_dev(ctx))
    return kv


def _successors(case):
    """Several where draws stay apart (block and tree candidates) or are few; one where a chain hangs on each of many."""
    few = case["B"] <= 8 and case["T"] > 0
    return 4 if few or case.get("topk", 1) > 1 or case["kind"] == "block" else 1


def _status():
    return torch.zeros(1, dtype=torch.int32, device=DEV)


def _base(V, g):
    b = torch.empty(V, device=DEV)
    b[torch.randperm(V, generator=g, device=DEV)] = -3.3 * torch.log(torch.arange(1, V + 1, device=DEV).float())
    return b


def _randn(g, n):
    return torch.randn(n, generator=g, device=DEV)


def _gumbel(g, z, T, k=1):
    if T == 0.0:
        return torch.topk(z, k).indices
    z = z.double() / T
    return torch.stack([(z - torch.log(-torch.log(torch.rand(z.numel(), generator=g, device=DEV, dtype=torch.float64)
                                                   .clamp_min(1e-300)))).argmax() for _ in range(k)])


def _logits(case, seed):
    """Draft rows q_i, target rows q_i + N(0, sigma^2) and the bonus row of each sequence; tokens drawn from q_i."""
    B, K, V, T = case["B"], case["K"], case["V"], case["T"]
    dt = torch.float32 if case["dtype"] == "f32" else BF
    g = _gen(seed, 5)
    base = _base(V, g)
    zq = torch.empty((B, K, V), dtype=dt, device=DEV)
    zp = torch.empty((B, K + 1, V), dtype=dt, device=DEV)
    tok = torch.empty((B, K), dtype=torch.int32, device=DEV)
    for b in range(B):
        for i in range(K + 1):
            q = (base + _randn(g, V)).to(dt).float()
            zp[b, i] = q + case["sigma"] * _randn(g, V)
            if i < K:
                zq[b, i] = q
                tok[b, i] = _gumbel(g, q, T)[0]
    r = _cpu(seed, 6)
    return zq, zp, tok, _dev(r.random((B, K), dtype=np.float32)), _dev(r.random((B, K + 1), dtype=np.float32))


def _hidden_inputs(case, seed):
    """Kept states, the draft step's q(token) and (M, log S), tokens and target rows for the logits-free verify."""
    sh = SHAPES[case["shape"]]
    B, K, V, T, d = case["B"], case["K"], sh.vocab, case["T"], sh.d_model
    w = _weights(sh, seed, 4)
    g = _gen(seed, 7)
    prev = torch.randint(0, V, (B * K,), generator=g, device=DEV)
    h = w["embed"][prev].float() + 0.5 * torch.randn((B * K, d), generator=g, device=DEV)
    n = h * torch.rsqrt(h.square().mean(-1, keepdim=True) + 1e-6) * w["final_norm"].float()
    dt = torch.float32 if case["dtype"] == "f32" else BF
    zp = torch.empty((B, K + 1, V), dtype=dt, device=DEV)
    tok = torch.empty((B * K,), dtype=torch.int32, device=DEV)
    qx = torch.empty((B * K,), device=DEV)
    stats = torch.empty((B * K, 2), device=DEV)
    head, n64 = w["lm_head"], n.double()
    step = 1 << 14
    for r0 in range(0, B * K, 64):
        z = torch.cat([n64[r0:r0 + 64] @ head[s:s + step].double().t() for s in range(0, V, step)], 1)
        y = z / T
        M = y.max(-1).values
        S = torch.log(torch.exp(y - M[:, None]).sum(-1))
        for r in range(r0, min(r0 + 64, B * K)):
            t = _gumbel(g, z[r - r0].float(), T)[0]
            tok[r], qx[r] = t, torch.exp(y[r - r0, t] - M[r - r0] - S[r - r0])
            stats[r, 0], stats[r, 1] = M[r - r0], S[r - r0]
            zp[r // K, r % K] = z[r - r0].float() + case["sigma"] * _randn(g, V)
            if r % K == K - 1:
                zp[r // K, K] = z[r - r0].float() + _randn(g, V)
    u = _cpu(seed, 6)
    return (w, h.view(B, K, d).contiguous(), qx.view(B, K), stats.view(B, K, 2), tok.view(B, K), zp,
            _dev(u.random((B, K), dtype=np.float32)), _dev(u.random((B, K + 1), dtype=np.float32)))


def _draft_inputs(case, seed):
    sh, r = SHAPES[case["shape"]], _cpu(seed, 8)
    B, K, m, k = case["B"], case["K"], case["max_new"], case["topk"]
    u = r.random((B, K, k) if k > 1 else (B, K), dtype=np.float32)
    return {"n_new": r.integers(1, m + 1, size=B).astype(np.int32),
            "tokens": r.integers(0, sh.vocab, size=(B, m)).astype(np.int32), "u": u,
            "feats": _normal(_gen(seed, 9), (B, m, sh.feat_dim))}


def prepare(case, seed):
    kind = case["kind"]
    if kind == "verify":
        zq, zp, tok, ua, us = _logits(case, seed)
        buf = VerifyBuffers(case["B"], case["K"], case["V"], DEV)
        return {"case": case, "buf": buf, "args": (zp, zq if case["T"] > 0 else None, tok, case["T"], ua, us)}
    if kind == "verify_hidden":
        w, h, qx, stats, tok, zp, ua, us = _hidden_inputs(case, seed)
        ctx = ob.osprey_create(SHAPES[case["shape"]], w)
        buf = VerifyHiddenBuffers(ctx, case["B"], case["K"], DEV)
        return {"case": case, "buf": buf, "args": (zp, h, qx, stats, tok, case["T"], ua, us)}
    if kind == "verify_tree":
        B, K, k, V, T = case["B"], case["K"], case["topk"], case["V"], case["T"]
        dt = torch.float32 if case["dtype"] == "f32" else BF
        g, r = _gen(seed, 10), _cpu(seed, 11)
        base = _base(V, g)
        zq = torch.empty((B, K, V), dtype=dt, device=DEV)
        zp = torch.empty((B, 1 + K * k, V), dtype=dt, device=DEV)
        cand = torch.empty((B, K, k), dtype=torch.int32, device=DEV)
        for b in range(B):
            for i in range(K):
                zq[b, i] = base + _randn(g, V)
                cand[b, i] = _gumbel(g, zq[b, i].float(), T, k)
            zp[b, 0] = zq[b, 0] + case["sigma"] * _randn(g, V)
            for n in range(K * k):
                i, j = divmod(n, k)
                zp[b, 1 + n] = zq[b, i + 1] + case["sigma"] * _randn(g, V) if j == 0 and i + 1 < K \
                    else base + _randn(g, V)
        return {"case": case, "buf": TreeVerifyBuffers(B, K, DEV),
                "args": (zp, zq if T > 0 else None, cand, T, _dev(r.random((B, K, k), dtype=np.float32)),
                         _dev(r.random((B, K + 1), dtype=np.float32)))}
    sh = SHAPES[case["shape"]]
    ctx = _contexts(case, seed)
    if kind == "append":
        n = int(ctx.sum())
        rows = (sh.n_layers, n, sh.n_kv_heads, sh.head_dim)
        g = _gen(seed, 12)
        w = {k: (torch.zeros(s, dtype=BF, device=DEV) if not isinstance(s, list) else
                 [torch.zeros(t, dtype=BF, device=DEV) for t in s]) for k, s in _weight_shapes(sh).items()}
        kv = _cache(sh, ctx, 0, case["ctx_hi"], seed, fill=False)
        return {"case": case, "ctx": ob.osprey_create(sh, w), "kv": kv, "n_rows": _dev(ctx),
                "k": _normal(g, rows), "v": _normal(g, rows), "status": _status()}
    w = _weights(sh, seed, _successors(case))
    st = {"case": case, "ctx": ob.osprey_create(sh, w), "status": _status()}
    if kind == "block":
        B, P = case["B"], case["block"] - 1
        r = _cpu(seed, 13)
        kv = _cache(sh, ctx, P, case["ctx_hi"], seed)
        st.update(kv=kv, seq0=kv.seq_len.clone(), anchors=_dev(r.integers(0, sh.vocab, size=B).astype(np.int32)),
                  mask=int(r.integers(0, sh.vocab)), feats=_normal(_gen(seed, 14), (B, sh.feat_dim)),
                  u=_dev(r.random((B, P), dtype=np.float32)))
        nbytes = ob.osprey_dflash_workspace_bytes(st["ctx"], B, P + 1, kv.max_pages)
        K = P
    else:
        B, K, m = case["B"], case["K"], case["max_new"]
        di = _draft_inputs(case, seed)
        kv = _cache(sh, ctx, m + K, case["ctx_hi"], seed)
        st.update(kv=kv, seq0=kv.seq_len.clone(), n_new=_dev(di["n_new"]), tokens=_dev(di["tokens"]),
                  feats=di["feats"], u=_dev(di["u"]))
        nbytes = ob.osprey_draft_workspace_bytes(st["ctx"], B, K, m, kv.max_pages)
    k = case.get("topk", 1)
    lead = (B, K, k) if k > 1 else (B, K)
    st.update(ws=torch.zeros(nbytes, dtype=torch.uint8, device=DEV), qx=torch.zeros(lead, device=DEV),
              toks=torch.zeros(lead, dtype=torch.int32, device=DEV), stats=torch.zeros((B, K, 2), device=DEV))
    wide = sh.d_model if case.get("out") == "hidden" else sh.vocab
    st["wide"] = torch.zeros((B, K, wide), device=DEV)
    return st


def _weight_shapes(sh):
    d, a, L = sh.d_model, sh.n_q_heads * sh.head_dim, sh.n_layers
    return {"W_c": (d, sh.feat_dim), "embed": (sh.vocab, d), "final_norm": (d,), "lm_head": (sh.vocab, d),
            "attn_norm": [(d,)] * L, "W_qkv": [(sh.qkv_rows, 2 * d)] * L, "W_o": [(d, a)] * L, "ffn_norm": [(d,)] * L,
            "W_gate": [(sh.ffn_dim, d)] * L, "W_up": [(sh.ffn_dim, d)] * L, "W_down": [(d, sh.ffn_dim)] * L}


# ---------------------------------------------------------------- one pass
def run(st):
    kind = st["case"]["kind"]
    if kind in ("verify", "verify_hidden", "verify_tree"):
        b = st["buf"]
        (b.run_hidden if kind == "verify_hidden" else b.run)(*st["args"])
        out = {"out_tokens": b.out_tokens, "n_accepted": b.n_accepted, "flags": b.flags, "status": b.status}
        if kind == "verify_tree":
            out["branch"] = b.branch
        elif st["case"]["T"] > 0:
            out["probs"] = b.probs
        return out
    kv = st["kv"]
    if kind == "append":
        kv.seq_len.zero_()     # the batch's sequences start afresh
        ob.osprey_kv_append(st["ctx"], kv, st["n_rows"], st["k"], st["v"], st["status"])
        return {"k_pages": kv.k_pages, "v_pages": kv.v_pages, "seq_len": kv.seq_len, "status": st["status"]}
    kv.seq_len.copy_(st["seq0"])   # the engine's own bookkeeping: the committed lengths before this call
    T = st["case"]["T"]
    if kind == "block":
        ob.osprey_dflash_step(st["ctx"], kv, st["anchors"], st["mask"], st["feats"], T, st["u"], st["toks"], st["qx"],
                              st["stats"], st["wide"], st["ws"], st["status"])
    elif st["case"]["topk"] > 1:
        ob.osprey_draft_step_topk(st["ctx"], kv, st["n_new"], st["tokens"], st["feats"], T, st["u"], st["toks"],
                                  st["qx"], st["stats"], st["wide"], st["ws"], st["status"])
    elif st["case"]["out"] == "hidden":
        ob.osprey_draft_step_hidden(st["ctx"], kv, st["n_new"], st["tokens"], st["feats"], T, st["u"], st["toks"],
                                    st["qx"], st["stats"], st["wide"], st["ws"], st["status"])
    else:
        ob.osprey_draft_step(st["ctx"], kv, st["n_new"], st["tokens"], st["feats"], T, st["u"], st["toks"], st["qx"],
                             st["stats"], st["wide"], st["ws"], st["status"])
    return {"tokens": st["toks"], "qx": st["qx"], "stats": st["stats"], "wide": st["wide"], "seq_len": kv.seq_len,
            "k_pages": kv.k_pages, "v_pages": kv.v_pages, "status": st["status"]}


# ---------------------------------------------------------------- what a pass cannot do without
def work(case):
    kind, B = case["kind"], case["B"]
    if kind in ("verify", "verify_hidden"):
        K = case["K"]
        V = case["V"] if kind == "verify" else SHAPES[case["shape"]].vocab
        s = 4 if case["dtype"] == "f32" else 2
        if kind == "verify":   # every target row, and every draft row unless greedy
            n = B * (2 * K + 1 if case["T"] > 0 else K + 1) * V
            return {"bytes": n * s, "flops": 4 * n}
        d = SHAPES[case["shape"]].d_model   # the target rows and one pass over the LM head
        return {"bytes": B * (K + 1) * V * s + V * d * 2 + B * d * 4, "flops": 2 * B * V * d}
    if kind == "verify_tree":   # the rows of an average walk: two nodes' target rows, one draft row
        s = 4 if case["dtype"] == "f32" else 2
        n = B * (3 if case["T"] > 0 else 2) * case["V"]
        return {"bytes": n * s, "flops": 4 * n}
    sh = SHAPES[case["shape"]]
    mean_ctx = (case["ctx_lo"] + case["ctx_hi"]) / 2
    kv_row = sh.n_layers * 2 * sh.n_kv_heads * sh.head_dim * 2
    if kind == "append":
        return {"bytes": int(B * mean_ctx * kv_row * 2), "flops": 0}
    # each chain step depends on the token before it, so it reads the layers and the head anew
    steps = 1 if kind == "block" else case["K"]
    ext = B * (case["block"] - 1 if kind == "block" else (1 + case["max_new"]) / 2)
    head_rows = ext if kind == "block" else B * steps
    layers = sh.n_layers * sh.layer_params()
    rows = ext + B * (steps - 1)
    n_bytes = steps * (2 * (layers + sh.vocab * sh.d_model) + B * mean_ctx * kv_row) + 2 * sh.d_model * sh.feat_dim
    n_bytes += 4 * head_rows * (sh.d_model if case.get("out") == "hidden" else sh.vocab)
    flops = 2 * (rows * layers + head_rows * sh.vocab * sh.d_model + ext * sh.d_model * sh.feat_dim)
    flops += 4 * rows * mean_ctx * sh.n_q_heads * sh.head_dim * sh.n_layers
    return {"bytes": int(n_bytes), "flops": int(flops)}


def tolerance(case):
    kind = case["kind"]
    if kind == "append":
        return "exact"
    if kind == "verify_tree":
        return {"rel": 0.0, "differ": 0.01}
    if kind in ("verify", "verify_hidden"):   # 1e-7 against 64 bits, 32-bit sums in another order
        return {"rel": 1e-6, "max": 2e-5, "differ": 0.01}
    # Against 64 bits: logits and states 6e-6, probabilities 1.2e-4 (logits of 40 with operands of 16 bits); a changed
    # last bit of a sum rounds some bf16 K/V rows the other way, and every later row of the sequence sees it.
    return {"rel": 5e-4, "max": 0.04, "differ": 0.01}


# ---------------------------------------------------------------- the same in 64 bits
def _rms(x, gain, eps=1e-6):
    return x * torch.rsqrt(x.square().mean(-1, keepdim=True) + eps) * gain.double()


def _mm(x, w, step=1 << 14):
    return torch.cat([x @ w[s:s + step].double().t() for s in range(0, w.shape[0], step)], -1)


def _rope(x, pos, theta):
    hd = x.shape[-1]
    ang = pos.double()[:, None] * theta ** (-torch.arange(0, hd, 2, device=DEV).double() / hd)[None]
    c, s = torch.cos(ang)[:, None], torch.sin(ang)[:, None]
    a, b = x[..., :hd // 2], x[..., hd // 2:]
    return torch.cat([a * c - b * s, b * c + a * s], -1)


def _layers(sh, w, kv, x, s, seqs, pos):
    """Residual rows x and context rows s of sequences `seqs` (equal ones adjacent) at positions `pos`, through every
    layer; their K/V rows go to the bf16 pages first, so that a row sees itself and the rows before it."""
    pages = kv.page_table.long()[seqs, pos // 16]
    for l in range(sh.n_layers):
        y = _mm(torch.cat([s, _rms(x, w["attn_norm"][l], sh.rms_eps)], -1), w["W_qkv"][l])
        y = y.view(len(seqs), -1, sh.head_dim)
        q = _rope(y[:, :sh.n_q_heads], pos, sh.rope_theta)
        kv.k_pages[l][pages, :, pos % 16] = _rope(y[:, sh.n_q_heads:-sh.n_kv_heads], pos, sh.rope_theta).to(BF)
        kv.v_pages[l][pages, :, pos % 16] = y[:, -sh.n_kv_heads:].to(BF)
        o = torch.empty_like(q)
        for b, at in _runs(seqs):
            n = int(pos[at].max()) + 1
            tab = kv.page_table[b, :-(-n // 16)].long()
            k, v = (p[l][tab].double().permute(1, 0, 2, 3).reshape(sh.n_kv_heads, -1, sh.head_dim)
                    for p in (kv.k_pages, kv.v_pages))
            qb = q[at].view(-1, sh.n_kv_heads, sh.group, sh.head_dim)
            sc = torch.einsum("rhgd,hkd->rhgk", qb, k) / math.sqrt(sh.head_dim)
            sc = sc.masked_fill((torch.arange(k.shape[1], device=DEV) > pos[at][:, None])[:, None, None], -math.inf)
            o[at] = torch.einsum("rhgk,hkd->rhgd", torch.softmax(sc, -1), v).reshape(-1, sh.n_q_heads, sh.head_dim)
        x = x + _mm(o.reshape(len(seqs), -1), w["W_o"][l])
        n = _rms(x, w["ffn_norm"][l], sh.rms_eps)
        x = x + _mm(torch.nn.functional.silu(_mm(n, w["W_gate"][l])) * _mm(n, w["W_up"][l]), w["W_down"][l])
    return x


def _runs(seqs):
    s, out, at = seqs.tolist(), [], 0
    while at < len(s):
        end = at
        while end < len(s) and s[end] == s[at]:
            end += 1
        out.append((s[at], slice(at, end)))
        at = end
    return out


def _head(sh, w, x, T, u, topk=1):
    """Logits, the drawn ids (topk a row), their q and (M, log S) of each row."""
    z = _mm(_rms(x, w["final_norm"], sh.rms_eps), w["lm_head"])
    y = z / T if T > 0 else z
    M = y.max(-1).values
    S = torch.exp(y - M[:, None]).sum(-1)
    if T == 0:
        ids = torch.topk(z, topk).indices
        qx = torch.ones(ids.shape, dtype=torch.float64, device=DEV)
    else:
        C = torch.cumsum(torch.exp(y - M[:, None]), -1)
        ids = torch.searchsorted(C, u.double() * C[:, -1:], right=True).clamp_max(sh.vocab - 1)
        qx = torch.exp(torch.gather(y, 1, ids) - M[:, None]) / S[:, None]
    return z, ids, qx, torch.stack([M, torch.log(S)], -1)


def exact(case, seed):
    kind, B = case["kind"], case["B"]
    if kind in ("append", "verify_tree") or (kind == "verify" and case["T"] == 0):
        return None
    none = {"out_tokens": None, "n_accepted": None, "flags": None, "status": None}
    if kind in ("verify", "verify_hidden"):
        K, T = case["K"], case["T"]
        if kind == "verify":
            zq, zp, tok, _, _ = _logits(case, seed)
        else:
            _, _, qx, _, tok, zp, _, _ = _hidden_inputs(case, seed)
        probs = torch.empty((B, K, 2), dtype=torch.float64, device=DEV)
        for b in range(B):
            at = tok[b].long()[:, None]
            probs[b, :, 0] = torch.gather(torch.softmax(zp[b, :K].double() / T, -1), 1, at)[:, 0]
            probs[b, :, 1] = torch.gather(torch.softmax(zq[b].double() / T, -1), 1, at)[:, 0] if kind == "verify" \
                else qx[b].double()
        return dict(none, probs=probs)
    sh = SHAPES[case["shape"]]
    ctx = _contexts(case, seed)
    w = _weights(sh, seed, _successors(case))
    L0 = _dev(ctx).long()
    if kind == "block":
        P, r = case["block"] - 1, _cpu(seed, 13)
        kv = _cache(sh, ctx, P, case["ctx_hi"], seed)
        tok = _dev(r.integers(0, sh.vocab, size=B)).long()[:, None].repeat(1, P)
        tok[:, 1:] = int(r.integers(0, sh.vocab))
        u = _dev(r.random((B, P), dtype=np.float32))
        s = _mm(_normal(_gen(seed, 14), (B, sh.feat_dim)).double(), w["W_c"]).repeat_interleave(P, 0)
        seqs = torch.arange(B, device=DEV).repeat_interleave(P)
        pos = (L0[:, None] + torch.arange(P, device=DEV)).reshape(-1)
        x = _layers(sh, w, kv, w["embed"][tok.reshape(-1)].double(), s, seqs, pos)
        z, _, qx, stats = _head(sh, w, x, case["T"], u.reshape(-1, 1))
        return {"tokens": None, "qx": qx.view(B, P), "stats": stats.view(B, P, 2), "wide": z.view(B, P, -1),
                "seq_len": None, "k_pages": kv.k_pages, "v_pages": kv.v_pages, "status": None}
    K, m, k = case["K"], case["max_new"], case["topk"]
    di = _draft_inputs(case, seed)
    kv = _cache(sh, ctx, m + K, case["ctx_hi"], seed)
    n_new, u = di["n_new"], _dev(di["u"]).reshape(B, K, k)
    seqs = _dev(np.repeat(np.arange(B), n_new)).long()
    j = _dev(np.concatenate([np.arange(n) for n in n_new])).long()
    x = w["embed"][_dev(di["tokens"]).long()[seqs, j]].double()
    s = _mm(di["feats"][seqs, j].double(), w["W_c"])
    x = _layers(sh, w, kv, x, s, seqs, L0[seqs] + j)
    x = x[_dev(np.cumsum(n_new) - 1).long()]
    one = torch.arange(B, device=DEV)
    wide, qx, stats = [], [], []
    for step in range(K):
        if step:
            x = _layers(sh, w, kv, w["embed"][ids[:, 0]].double(), x, one, L0 + _dev(n_new).long() + step - 1)
        z, ids, q, st = _head(sh, w, x, case["T"], u[:, step], k)
        wide.append((x if case["out"] == "hidden" else z).float() if B > 16 else (x if case["out"] == "hidden" else z))
        qx.append(q)
        stats.append(st)
    qx = torch.stack(qx, 1)
    return {"tokens": None, "qx": qx if k > 1 else qx[..., 0], "stats": torch.stack(stats, 1),
            "wide": torch.stack(wide, 1), "seq_len": None, "k_pages": kv.k_pages, "v_pages": kv.v_pages,
            "status": None}
