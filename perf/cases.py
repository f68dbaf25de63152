"""The verification step's performance cases: what a serving program calls, over the sizes it calls it at.

A case is one call of the public API on resident inputs (for ``host`` on pinned host buffers), with
the options, workspace and output buffers such a program allocates once and keeps.  Sizes are the
repository's own workloads and their neighbours: batch 1 to 64, candidate lengths 3 to 20, trees of
up to 100 nodes, vocabularies of 8000 to 256000 entries, whole multiples of 16 bytes a row and not,
both logit types, every divergence, every acceptance rule, both token choices.
"""

from __future__ import annotations

import torch

import paper_2502_20704_b200 as fsd

ELEM = {"bf16": 2, "f32": 4}
TORCH = {"bf16": torch.bfloat16, "f32": torch.float32}
# most logit bytes of one call (the largest listed case)
MAX_BYTES = 2 * 64 * 17 * 152064


def _chain(name, B, gamma, V, dtype="bf16", div="js", mode="fsd", sample="invcdf", T=0.2, call="chain"):
    return {"name": name, "call": call, "B": B, "P": gamma, "V": V, "dtype": dtype, "div": div, "mode": mode,
            "sample": sample, "T": T}


def listed():
    return [
        # one interactive request, short draft, small vocabulary, logits straight from an fp32 head: launches and latency count
        _chain("one_request_f32", 1, 4, 32000, dtype="f32", T=0.05),
        # a small serving batch on a small-vocabulary pair
        _chain("small_batch", 16, 5, 32000, T=1.0 / 7.0),
        # the same kind of batch under the relaxed ratio rule, from a program that owns no scratch memory
        _chain("small_batch_rfsd_static", 12, 6, 32000, mode="rfsd", T=0.05, call="static"),
        # a vocabulary whose rows are not a multiple of 16 bytes (a tokenizer with added tokens)
        _chain("ragged_vocabulary", 8, 5, 50257, T=0.1),
        # an ordinary batch on a 128k vocabulary
        _chain("ordinary_128k", 32, 6, 128256, T=0.1),
        # the headline: a full batch, a 152k vocabulary
        _chain("full_batch_152k", 64, 8, 152064, T=0.2),
        # the strict rule on that shape, the comparison every deployment runs: ratio test and residual draw
        _chain("full_batch_152k_sd", 64, 8, 152064, mode="sd", T=0.0),
        # the largest vocabularies, KL, greedy decoding
        _chain("vocabulary_256k_kl_greedy", 16, 10, 256000, div="kl", sample="greedy", T=0.5),
        # long drafts, fp32 logits, total variation
        _chain("long_draft_f32_tv", 8, 15, 152064, dtype="f32", div="tv", T=0.4),
        # tree drafting: 60 nodes, depth 6
        {"name": "tree_60", "call": "tree", "B": 8, "P": 60, "V": 32000, "dtype": "bf16", "div": "js", "mode": "fsd",
         "sample": "invcdf", "T": 0.05},
        # logits that arrive in host memory (a draft model elsewhere): the copies are part of the call
        _chain("host_buffers", 8, 5, 32000, T=1.0 / 7.0, call="host"),
        # choosing T on a development set's divergences: 64 candidates, the calibration and the labels
        {"name": "threshold_tuning", "call": "tuning", "B": 4096, "P": 8, "K": 64, "target": 3.0},
    ]


def _log_uniform(rng, lo, hi):
    return lo * (hi / lo) ** rng.random()


def draw(rng):
    kind = rng.random()
    if kind < 0.08:
        P = rng.randint(4, 20)
        return {"call": "tuning", "B": int(_log_uniform(rng, 256, 32768)), "P": P, "K": rng.randint(8, 64),
                "target": round(rng.uniform(0.2, 0.7) * P, 2)}
    call = "tree" if kind < 0.20 else "host" if kind < 0.27 else "static" if kind < 0.35 else "chain"
    dtype = rng.choice(["bf16", "bf16", "bf16", "f32"])
    V = int(_log_uniform(rng, 8000, 256000))
    if rng.random() < 0.75:
        V -= V % 64                                   # padded to the head's tile, as most are; the others are ragged
    div = rng.choice(["js", "js", "kl", "tv"])
    sample = rng.choice(["invcdf", "invcdf", "invcdf", "greedy"])
    mode = "fsd" if call == "tree" else rng.choice(["fsd", "fsd", "sd", "rfsd"])
    if call == "tree":
        B, P = int(round(_log_uniform(rng, 1, 16))), rng.randint(16, 100)
    else:
        B, P = int(round(_log_uniform(rng, 1, 64))), rng.randint(3, 20)
    if call == "host":
        B = min(B, 16)
    if call == "static":
        B = min(B, 1024 // P)
    while B > 1 and ELEM[dtype] * B * (2 * P + 1) * V > (MAX_BYTES // 8 if call == "host" else MAX_BYTES):
        B = B * 3 // 4
    T = {"js": 0.1, "kl": 0.5, "tv": 0.35}[div] * rng.choice([0.5, 1.0, 2.0])
    return {"call": call, "B": B, "P": P, "V": V, "dtype": dtype, "div": div, "mode": mode, "sample": sample, "T": T}


# ---- inputs ----------------------------------------------------------------------------------
def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _target_rows(g, n, V):
    """Logit rows of n contexts: small vocabularies 3 N(0, 1) with one spike of 8, large ones
    Zipf-shaped, -1.1 ln(rank) + N(0, 0.5)."""
    noise = torch.randn(n, V, generator=g, device="cuda")
    if V < 60000:
        noise.mul_(3.0)
        at = torch.randint(V, (n, 1), generator=g, device="cuda")
        return noise.scatter_add_(1, at, torch.full((n, 1), 8.0, device="cuda"))
    rank = torch.rand(n, V, generator=g, device="cuda").mul_(V).floor_().add_(1.0)
    return noise.mul_(0.5).add_(rank.log_(), alpha=-1.1)


def _tree_parents(seed, B, N, max_depth):
    """Random draft trees: depth at most max_depth, at most four children a node."""
    import random
    rng = random.Random(int(seed) * 7919 + 11)
    out = []
    for _ in range(B):
        par, depth, kids = [], [], [0] * (N + 1)
        for j in range(N):
            open_ = [i for i in range(-1, j) if kids[i + 1] < 4 and (i < 0 or depth[i] < max_depth)]
            p = rng.choice(open_)
            par.append(p)
            depth.append(1 if p < 0 else depth[p] + 1)
            kids[p + 1] += 1
        out.append(par)
    return out


def _max_depth(case):
    return 6 if case["P"] <= 64 else 8


def _prepare_tuning(case, seed):
    g = _generator(seed)
    B, P, K = case["B"], case["P"], case["K"]
    # divergences as verify calls leave them: mostly small, a tail up to ln 2
    D = torch.rand(B, P, generator=g, device="cuda").pow_(3.0).mul_(0.6931)
    return {"case": case, "D": D, "Ts": torch.linspace(0.01, 0.65, K, device="cuda"),
            "mean": torch.empty(K, device="cuda"), "frac": torch.empty(K, device="cuda"), "T": torch.empty(2, device="cuda"),
            "labels": torch.empty(B, P, dtype=torch.uint8, device="cuda"), "stream": torch.cuda.current_stream().cuda_stream}


def prepare(case, seed):
    if case["call"] == "tuning":
        return _prepare_tuning(case, seed)
    g = _generator(seed)
    B, P, V, tree = case["B"], case["P"], case["V"], case["call"] == "tree"
    dt = TORCH[case["dtype"]]
    target = torch.empty(B, P + 1, V, dtype=dt, device="cuda")
    draft = torch.empty(B, P, V, dtype=dt, device="cuda")
    tokens = torch.empty(B, P, dtype=torch.int32, device="cuda")
    parent = torch.tensor(_tree_parents(seed, B, P, _max_depth(case)), dtype=torch.int32, device="cuda") if tree else None
    for b in range(B):
        rows = _target_rows(g, P + 1, V)
        target[b] = rows
        # the draft model: the target's logits with noise of 0.2 to 1.5, one position in ten unrelated
        base = rows[parent[b].long() + 1] if tree else rows[:P]
        sigma = torch.rand(P, 1, generator=g, device="cuda").mul_(1.3).add_(0.2)
        d = base + sigma * torch.randn(P, V, generator=g, device="cuda")
        other = torch.rand(P, 1, generator=g, device="cuda") < 0.1
        d = torch.where(other, base.roll(V // 3, dims=1), d)
        draft[b] = d
        # candidates drawn from the draft distribution
        d.sub_(torch.rand(P, V, generator=g, device="cuda").clamp_(1e-20, 1.0).log_().neg_().clamp_(1e-20).log_())
        tokens[b] = d.argmax(dim=1)
    u_accept = torch.rand(B, P, generator=g, device="cuda")
    u_sample = torch.rand(B, generator=g, device="cuda")
    opts = fsd.make_opts(div=case["div"], mode=case["mode"], cmp="lt", sample=case["sample"], dtype=case["dtype"], T=case["T"])
    s = {"case": case, "opts": opts, "target": target, "draft": draft, "tokens": tokens, "parent": parent,
         "u_accept": u_accept, "u_sample": u_sample, "stream": torch.cuda.current_stream().cuda_stream}
    on = dict(device="cuda")
    if case["call"] == "host":
        on = dict(pin_memory=True)
        for k in ("target", "draft", "tokens", "u_accept", "u_sample"):
            s[k] = s[k].cpu().pin_memory()
        s["ws_bytes"] = fsd.fsd_host_staging_bytes(B, P, V, opts)
    else:
        s["ws_bytes"] = fsd.fsd_workspace_bytes(B, P, V, opts)
    s["ws"] = torch.empty(s["ws_bytes"], dtype=torch.uint8, device="cuda") if case["call"] != "static" else None
    # accept_len, next_token and row_status in one block, so that a program reads them back in one copy
    s["ints"] = torch.zeros(3, B, dtype=torch.int32, **on)
    s["accept_len"], s["next_token"], s["row_status"] = s["ints"][0], s["ints"][1], s["ints"][2]
    s["divergence"] = torch.zeros(B, P, dtype=torch.float32, **on)
    s["path"] = torch.zeros(B, _max_depth(case), dtype=torch.int32, device="cuda") if tree else None
    return s


# ---- one pass --------------------------------------------------------------------------------
def _ok(rc):
    if rc != 0:
        raise RuntimeError(fsd.fsd_status_string(rc))


def run(s):
    case = s["case"]
    call, B, P = case["call"], case["B"], case["P"]
    if call == "tuning":
        K = case["K"]
        _ok(fsd.fsd_threshold_sweep(s["D"], B, P, s["Ts"], K, 0, s["mean"], s["frac"], s["stream"]))
        _ok(fsd.fsd_calibrate_threshold(s["D"], B, P, case["target"], 0, s["T"][0:1], s["T"][1:2], s["stream"]))
        _ok(fsd.fsd_accept_labels(s["D"], B, P, 0.2, 0, s["labels"], s["stream"]))
        return {"mean": s["mean"], "frac": s["frac"], "T": s["T"], "labels": s["labels"]}
    V = case["V"]
    if call == "tree":
        _ok(fsd.fsd_verify_tree(s["target"], s["draft"], s["parent"], s["u_sample"], B, P, V, _max_depth(case), s["opts"],
                                s["accept_len"], s["path"], s["next_token"], s["divergence"], s["row_status"],
                                s["ws"], s["ws_bytes"], s["stream"]))
        return {"ints": s["ints"], "divergence": s["divergence"], "path": s["path"]}
    if call == "static":
        _ok(fsd.fsd_verify_chain_static(s["target"], s["draft"], s["tokens"], s["u_accept"], s["u_sample"], B, P, V, s["opts"],
                                        s["accept_len"], s["next_token"], s["divergence"], s["row_status"], s["stream"]))
    else:
        fn = fsd.fsd_verify_chain_host if call == "host" else fsd.fsd_verify_chain
        _ok(fn(s["target"], s["draft"], s["tokens"], s["u_accept"], s["u_sample"], B, P, V, s["opts"],
               s["accept_len"], s["next_token"], s["divergence"], s["row_status"], s["ws"], s["ws_bytes"], s["stream"]))
    return {"ints": s["ints"], "divergence": s["divergence"]}


# ---- what a pass cannot do without -----------------------------------------------------------
def work(case):
    B, P = case["B"], case["P"]
    if case["call"] == "tuning":
        # the divergences once, a label each; prefix maxima and one comparison per candidate
        return {"bytes": 5.0 * B * P + 12.0 * case["K"], "flops": float(B * P * (1 + case["K"]))}
    V, es = case["V"], ELEM[case["dtype"]]
    if case["call"] == "tree":
        # every draft row, and the target rows of the nodes that have children (and the root's)
        rows = sum(P + len(set(par)) for par in _tree_parents(0, B, P, _max_depth(case)))
    else:
        rows = B * (2 * P + 1)
    # per position and vocabulary entry: two scaled exponentials, two normalisers, two entropy terms and
    # one s log s of the mean (JS); KL and TV need about half of that
    per_entry = {"js": 16.0, "kl": 9.0, "tv": 9.0}[case["div"]]
    return {"bytes": float(es) * rows * V + 8.0 * B * P + 20.0 * B, "flops": per_entry * B * P * V}


def tolerance(case):
    if case["call"] == "tuning":
        return "exact"
    # Divergences: differences of single-precision entropies of up to ln V = 12 nats, each good to about
    # 2^-22, against divergences of 0.05 and more.  Accepted lengths and tokens are whole numbers; one
    # in a hundred may change where a divergence lies on the threshold or a draw on an interval's end.
    return {"rel": 3e-5, "max": 3e-4, "differ": 0.01}
