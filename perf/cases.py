"""Workloads of the token-tree verification library, for timing it and for comparing two builds of it.

Each case is one call, or one decoding step's worth of calls, as a serving program makes them: its tensors and its
prepared calls exist (``prepare``), and ``run`` goes through the public Python entry points once.  Shapes are those of
``paper_2402_12374_b200.workloads`` and of the test suite; ``draw`` takes more of them over the whole range of each kind.
"""
import math

import numpy as np
import torch

from paper_2402_12374_b200 import binding as B
from paper_2402_12374_b200 import workloads as W

DTYPES = {"fp16": torch.float16, "bf16": torch.bfloat16, "fp32": torch.float32}
D = 128  # head_dim
HEADS = [(32, 32), (40, 40), (52, 52), (64, 8), (32, 8), (40, 8)]  # query heads, kv heads
VOCABS = [32000, 50257, 128256]


def listed():
    return [
        # The smallest decoding step: two layers, a short prompt, a small tree.  Launches and latency count.
        {"name": "step tiny", "kind": "step", "layers": 2, "hq": 32, "hkv": 32, "n": 16, "L": 128, "dtype": "fp16", "V": 32000, "T": 0.6},
        # A whole decoding step of the 7B shape: the attention of all 32 layers, the verification, the cache commit.
        {"name": "step 7b", "kind": "step", "layers": 32, "hq": 32, "hkv": 32, "n": 64, "L": 1024, "dtype": "bf16", "V": 32000, "T": 0.6},
        # One layer's attention with a mid-size tree: the 33B shape.
        {"name": "attention 33b", "kind": "attention", "hq": 52, "hkv": 52, "n": 256, "L": 2048, "dtype": "bf16", "mask": "parent"},
        # The offloading regime: as large a tree as the paper verifies, grouped heads.  Bound by arithmetic.
        {"name": "attention 70b", "kind": "attention", "hq": 64, "hkv": 8, "n": 768, "L": 4096, "dtype": "bf16", "mask": "parent"},
        # Grouped heads whose group (5) does not divide a tile of 128 rows, a ragged tree and prefix.
        {"name": "attention group of 5", "kind": "attention", "hq": 40, "hkv": 8, "n": 100, "L": 1501, "dtype": "bf16", "mask": "bits"},
        # The single-precision mode, for checking a model and for fp32 deployments.
        {"name": "attention fp32", "kind": "attention", "hq": 32, "hkv": 32, "n": 64, "L": 1024, "dtype": "fp32", "mask": "bits"},
        # Serving: eight requests with a prefix length each, stacked as heads, lengths in device memory.
        {"name": "attention of 8 requests", "kind": "attention_batch", "R": 8, "hq": 32, "hkv": 8, "n": 64, "L": 2048, "dtype": "bf16"},
        # Stochastic verification of one request over a large vocabulary and the largest tree.
        {"name": "verify 70b", "kind": "verify", "n": 768, "V": 128256, "T": 0.6, "mode": "sequoia", "logits": "fp32"},
        # Greedy decoding of one request.
        {"name": "verify greedy 13b", "kind": "verify", "n": 128, "V": 32000, "T": 0.0, "mode": "sequoia", "logits": "fp32"},
        # Serving: the verification of sixteen requests in one launch.
        {"name": "verify of 16 requests", "kind": "verify_batch", "R": 16, "n": 64, "V": 32000, "T": 1.0, "mode": "sequoia"},
        # The draft side: children of all internal nodes of the largest tree.
        {"name": "draft sample 70b", "kind": "draft", "rows": 378, "V": 128256, "k": 9, "T": 0.6},
        # Nucleus truncation of the target rows of a 7B-shaped tree.
        {"name": "top-p 7b", "kind": "top_p", "rows": 64, "V": 32000, "T": 0.6, "top_p": 0.9},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case, sizes spread over the logarithm of each kind's range."""
    kind = rng.choice(["step", "attention", "attention", "attention_fp32", "attention_batch", "verify", "verify", "verify_batch", "draft",
                       "draft", "top_p"])
    if kind == "step":
        hq, hkv = rng.choice(HEADS)
        return {"kind": "step", "layers": rng.choice([1, 2, 4, 8]), "hq": hq, "hkv": hkv, "n": _log_int(rng, 4, 128), "L": _log_int(rng, 32, 2048),
                "dtype": rng.choice(["fp16", "bf16"]), "V": 32000, "T": rng.choice([0.0, 0.6, 1.0])}
    if kind == "attention":
        hq, hkv = rng.choice(HEADS)
        n, L = _log_int(rng, 1, 768), _log_int(rng, 16, 8192)
        L = min(L, 768 * 4096 * 64 // (n * hq))  # no more arithmetic than the largest listed one
        return {"kind": "attention", "hq": hq, "hkv": hkv, "n": n, "L": L, "dtype": rng.choice(["fp16", "bf16"]),
                "mask": "bits" if hq // hkv == 5 else rng.choice(["parent", "bits"])}
    if kind == "attention_fp32":
        hq, hkv = rng.choice(HEADS)
        n, L = _log_int(rng, 1, 128), _log_int(rng, 16, 2048)
        L = min(L, 64 * 1024 * 32 // (n * hq) + 1)
        return {"kind": "attention", "hq": hq, "hkv": hkv, "n": n, "L": L, "dtype": "fp32", "mask": "bits"}
    if kind == "attention_batch":
        hq, hkv = rng.choice([(32, 32), (64, 8), (32, 8)])
        return {"kind": "attention_batch", "R": rng.randint(2, 16), "hq": hq, "hkv": hkv, "n": _log_int(rng, 4, 128),
                "L": _log_int(rng, 64, 2048), "dtype": "bf16"}
    if kind == "verify":
        V = rng.choice(VOCABS)
        T = rng.choice([0.0, 0.6, 1.0])
        mode = rng.choice(["sequoia", "sequoia", "specinfer", "target_sample"]) if T > 0 else "sequoia"
        logits = rng.choice(["fp32", "bf16"]) if T > 0 and mode != "target_sample" else "fp32"
        return {"kind": "verify", "n": _log_int(rng, 8, 768), "V": V, "T": T, "mode": mode, "logits": logits}
    if kind == "verify_batch":
        V = rng.choice(VOCABS)
        n = _log_int(rng, 8, 128)
        R = max(1, min(_log_int(rng, 2, 64), 90_000_000 // (n * V)))
        T = rng.choice([0.0, 0.6, 1.0])
        return {"kind": "verify_batch", "R": R, "n": n, "V": V, "T": T, "mode": rng.choice(["sequoia", "target_sample"]) if T > 0 else "sequoia"}
    if kind == "draft":
        return {"kind": "draft", "rows": _log_int(rng, 1, 378), "V": rng.choice(VOCABS), "k": _log_int(rng, 1, 32), "T": rng.choice([0.6, 1.0])}
    V = rng.choice(VOCABS)
    return {"kind": "top_p", "rows": _log_int(rng, 1, 64 * 32000 * 8 // V), "V": V, "T": rng.choice([0.6, 1.0]), "top_p": rng.choice([0.8, 0.9, 0.95])}


# ---------------------------------------------------------------- inputs
def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _tree(n, seed):
    return W.random_tree(n, max(4, min(20, int(2 * math.log2(n + 1)))), 16, np.random.default_rng(seed))


def _rows(shape, g):
    """fp32 normal rows whose stride is a multiple of four elements, as the library asks for."""
    V = shape[-1]
    return torch.randn((*shape[:-1], (V + 3) // 4 * 4), device="cuda", generator=g)[..., :V]


def _logits(shape, g, noise):
    """Target logits N(0, 3^2), draft logits the target's plus noise."""
    target = _rows(shape, g).mul_(3.0)
    draft = _rows(shape, g).mul_(noise).add_(target)
    return target, draft


def _children_tokens(parent, draft, T, g):
    """The k children of a node carry the first k of a draw without replacement from softmax(draft / T), in draw order
    (T = 0: the draft's k best tokens)."""
    n = len(parent)
    rank, count = np.zeros(n, dtype=np.int64), np.zeros(n, dtype=np.int64)
    for i in range(1, n):
        rank[i] = count[parent[i]]
        count[parent[i]] += 1
    if n == 1:
        return torch.zeros(1, dtype=torch.int32, device="cuda")
    keys = draft
    if T > 0:
        keys = torch.empty(draft.shape, device="cuda").exponential_(generator=g).log_().neg_().add_(draft, alpha=1.0 / T)
    top = keys.topk(int(count.max()), dim=1).indices
    tokens = top[torch.from_numpy(np.maximum(parent, 0).astype(np.int64)).cuda(), torch.from_numpy(rank).cuda()].to(torch.int32)
    tokens[0] = 0
    return tokens


def _verify_inputs(n, V, T, seed, g, bf16=False):
    parent = _tree(n, seed)
    target, draft = _logits((n, V), g, 1.5 if V > 100000 else 1.0)
    if bf16:
        pad = (V + 3) // 4 * 4
        target, draft = (torch.empty((n, pad), dtype=torch.bfloat16, device="cuda")[:, :V].copy_(x) for x in (target, draft))
    tokens = _children_tokens(parent, draft.float() if bf16 else draft, T, g)
    return torch.from_numpy(parent).cuda(), tokens, target, draft, torch.rand(n + 1, device="cuda", generator=g)


def _verify_call(parent, tokens, target, draft, T, uniforms, status, mode="sequoia"):
    """One buffer holds what the step brings back to the host: path, path length, bonus token."""
    n = parent.shape[0]
    back = torch.full((n + 2,), -1, dtype=torch.int32, device="cuda")
    call = B.VerifyCall(parent, tokens, target, draft, T, uniforms, path=back[:n], path_len=back[n:n + 1], bonus_token=back[n + 1:],
                        dev_status=status, specinfer=mode == "specinfer", target_sample=mode == "target_sample")
    return call, back


def prepare(case, seed):
    g = _generator(seed)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    s = {"kind": case["kind"], "status": status}
    kind, dt = case["kind"], DTYPES.get(case.get("dtype"))
    if kind == "step":
        layers, hq, hkv, n, L = (case[x] for x in ("layers", "hq", "hkv", "n", "L"))
        q = torch.randn((layers, n, hq, D), device="cuda", generator=g).to(dt)
        k = torch.randn((layers * hkv, L + n, D), device="cuda", generator=g).to(dt)
        v = torch.randn((layers * hkv, L + n, D), device="cuda", generator=g).to(dt)
        parent, tokens, target, draft, uniforms = _verify_inputs(n, case["V"], case["T"], seed, g)
        out = torch.empty_like(q)
        s["attention"] = [B.AttentionCall(q[i], k[i * hkv:(i + 1) * hkv], v[i * hkv:(i + 1) * hkv], None, L, parent=parent, out=out[i], dev_status=status)
                          for i in range(layers)]
        s["verify"], s["back"] = _verify_call(parent, tokens, target, draft, case["T"], uniforms, status)
        s.update(k=k, v=v, L=L, n=n, out=out)
    elif kind in ("attention", "attention_batch"):
        R = case.get("R", 1)
        hq, hkv, n, L = case["hq"] * R, case["hkv"] * R, case["n"], case["L"]
        parent = torch.from_numpy(_tree(n, seed)).cuda()
        mask = B.seq_tree_mask_from_parents(parent)[0] if case.get("mask") == "bits" else None  # once per tree
        q = torch.randn((n, hq, D), device="cuda", generator=g).to(dt)
        k = torch.randn((hkv, L + n, D), device="cuda", generator=g).to(dt)
        v = torch.randn((hkv, L + n, D), device="cuda", generator=g).to(dt)
        lengths = None
        if kind == "attention_batch":  # prefixes between half the longest and the longest
            lengths = torch.randint(L // 2, L + 1, (R,), device="cuda", generator=g, dtype=torch.int32)
        s["call"] = B.AttentionCall(q, k, v, mask, L, parent=parent, dev_status=status, prefix_len_dev=lengths)
    elif kind == "verify":
        parent, tokens, target, draft, uniforms = _verify_inputs(case["n"], case["V"], case["T"], seed, g, case["logits"] == "bf16")
        s["call"], s["back"] = _verify_call(parent, tokens, target, draft, case["T"], uniforms, status, case["mode"])
    elif kind == "verify_batch":
        R, n, V, T = case["R"], case["n"], case["V"], case["T"]
        target, draft = _logits((R, n, V), g, 1.0)
        parents = [_tree(n, seed + 1000 * r) for r in range(R)]
        tokens = torch.stack([_children_tokens(p, draft[r], T, g) for r, p in enumerate(parents)])
        s["args"] = (torch.from_numpy(np.stack(parents)).cuda(), tokens, target, draft, T, torch.rand((R, n + 1), device="cuda", generator=g))
        s.update(next=torch.empty((R, n), dtype=torch.int32, device="cuda"), target_sample=case["mode"] == "target_sample")
    elif kind == "draft":
        logits = _rows((case["rows"], case["V"]), g).mul_(3.2)
        s["args"] = (logits, case["T"], torch.rand(logits.shape, device="cuda", generator=g), case["k"])
    else:
        logits = _rows((case["rows"], case["V"]), g).mul_(3.0)
        out = _rows((case["rows"], case["V"]), g)
        s.update(logits=logits, out=out, kept=torch.empty(case["rows"], dtype=torch.int32, device="cuda"), T=case["T"], top_p=case["top_p"])
    return s


def run(s):
    kind, status = s["kind"], s["status"]
    if kind == "step":
        for layer in s["attention"]:
            layer.run()
        path, path_len, _ = s["verify"].run()
        B.seq_tree_kv_commit(s["k"], s["v"], s["L"], s["n"], path, path_len, dev_status=status)
        return s["out"], s["back"], s["k"], s["v"], status
    if kind in ("attention", "attention_batch"):
        return s["call"].run(), status
    if kind == "verify":
        s["call"].run()
        return s["back"], status
    if kind == "verify_batch":
        # path[r] is written up to path_len[r]; the accepted child of every node says the same and is written whole
        _, path_len, bonus = B.seq_tree_verify_batch(*s["args"], next_child_out=s["next"], dev_status=status, target_sample=s["target_sample"])
        return path_len, bonus, s["next"], status
    if kind == "draft":
        return B.seq_tree_draft_sample(*s["args"], dev_status=status), status
    B.seq_tree_top_p_filter(s["logits"], s["T"], s["top_p"], out=s["out"], kept_out=s["kept"], dev_status=status)
    return s["out"], s["kept"], status


# ---------------------------------------------------------------- what a pass cannot do without
def _attention_work(hq, hkv, n, L, e):
    pairs = n * (L + 0.5 * min(n, 12))  # prefix keys, and a handful of ancestors
    return 2 * (L + n) * hkv * D * e + 2 * n * hq * D * e, 4 * D * hq * pairs


def _verify_work(V, rows, e=4):
    """Three nodes is what a walk visits on these inputs, on the average: their rows once, an exponential and a few
    operations for each entry."""
    return 3 * rows * V * e, 3 * rows * V * 6


def work(case):
    kind = case["kind"]
    if kind == "step":
        b, f = _attention_work(case["hq"], case["hkv"], case["n"], case["L"], 2)
        vb, vf = _verify_work(case["V"], 2 if case["T"] > 0 else 1)
        commit = 2 * 2 * 2 * case["layers"] * case["hkv"] * D * 2  # two rows of every plane, read and written
        b, f = case["layers"] * b + vb + commit, case["layers"] * f + vf
    elif kind in ("attention", "attention_batch"):
        R = case.get("R", 1)
        L = case["L"] if R == 1 else 0.75 * case["L"]
        b, f = _attention_work(case["hq"] * R, case["hkv"] * R, case["n"], L, 4 if case["dtype"] == "fp32" else 2)
    elif kind in ("verify", "verify_batch"):
        b, f = _verify_work(case["V"], 2 if case["T"] > 0 and case["mode"] != "target_sample" else 1, 2 if case.get("logits") == "bf16" else 4)
        b, f = b * case.get("R", 1), f * case.get("R", 1)
    elif kind == "draft":
        b, f = 2 * 4 * case["rows"] * case["V"], 8 * case["rows"] * case["V"]
    else:
        b, f = 2 * 4 * case["rows"] * case["V"], 6 * case["rows"] * case["V"]
    return {"bytes": b, "flops": f}


def tolerance(case):
    """Attention: the output's type (probabilities are rounded to it before the product with V).  Decisions are whole
    numbers: equal but for a uniform on the edge of two tokens."""
    kind = case["kind"]
    if kind in ("step", "attention", "attention_batch"):
        rel = {"fp16": 2e-3, "bf16": 1e-2, "fp32": 1e-5}[case["dtype"]]
        return {"rel": rel, "differ": 0.01}
    return {"rel": 1e-5, "differ": 0.01}
