"""Performance cases of the copy-and-verify framework: the calls its users make, over the range of
sizes they make them at.

Kinds of case (`kind`):
  search     cs_find_match over token histories that are already on the device
  generate   cs_decode_loop: the whole generation loop for a batch, from the call to its return
  verify     one cs_verify_step with the logits asked for, for callers with a loop of their own
  host_steps a request whose history lives on the host: consecutive cs_step_host calls from pinned
             memory, the first of which uploads the history
  prefill    cs_prefill: context ingestion
  drafted    cs_decode_loop_drafted: the loop merged with a draft model

Model shapes are the package's own: the 8B-class shape (`8b`), the small one (`tiny`), and the
1B-class draft model of the benchmark.  Weights are random (the package's generator), histories
and scripts are built so that every decode step finds a match and accepts a known number of draft
tokens, which fixes the amount of work of a case whatever the seed.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2502_08923_b200 import binding as cs
from paper_2502_08923_b200 import inputs

GAMMA = 3
DRAFT_1B = inputs.ModelConfig(n_layers=16, d_model=2048, n_heads=32, n_kv_heads=8, head_dim=64, d_ffn=8192,
                              vocab=inputs.LLAMA8B.vocab, rope_theta=500000.0, rms_eps=1e-5)
MODELS = {"8b": inputs.LLAMA8B, "tiny": inputs.TINY}


def listed():
    return [
        # one chat session looks for its next draft: the smallest call, launch latency counts
        {"name": "search_b1_4k", "kind": "search", "batch": 1, "tokens": 4097, "gamma": 3, "k": 10, "policy": cs.LATEST},
        # a server's whole batch of long histories in one call
        {"name": "search_b64_32k", "kind": "search", "batch": 64, "tokens": 32768, "gamma": 5, "k": 10, "policy": cs.FIRST},
        # a small model: every kernel is short, so launches and host work set the pace
        {"name": "generate_tiny_b1", "kind": "generate", "model": "tiny", "batch": 1, "context": 512, "k": 10, "steps": 11},
        # plain one-token decoding (no draft), the baseline every speed-up is quoted against
        {"name": "plain_8b_b1_2k", "kind": "generate", "model": "8b", "batch": 1, "context": 2048, "k": 0, "steps": 16},
        # the verification forward on its own at odd sizes: two sequences, five drafted tokens each
        {"name": "verify_8b_b2_1531_k5", "kind": "verify", "model": "8b", "batch": 2, "context": 1531, "k": 5},
        # the usual decode: one sequence, 4k context, ten copied tokens, every accepted length from 0 to 10
        {"name": "generate_8b_b1_4k_k10", "kind": "generate", "model": "8b", "batch": 1, "context": 4096, "k": 10, "steps": 11},
        # a client that keeps its history on the host and asks step by step
        {"name": "host_steps_8b_b1_3001_k10", "kind": "host_steps", "model": "8b", "batch": 1, "context": 3001, "k": 10, "steps": 4},
        # long-context copying (summarising or quoting a long document)
        {"name": "generate_8b_b1_30k_k10", "kind": "generate", "model": "8b", "batch": 1, "context": 30720, "k": 10, "steps": 8},
        # a batch of long contexts with a wide copy window
        {"name": "generate_8b_b8_16k_k20", "kind": "generate", "model": "8b", "batch": 8, "context": 16384, "k": 20, "steps": 6},
        # many multi-turn chats that re-emit earlier answers
        {"name": "generate_8b_b16_8k_k10", "kind": "generate", "model": "8b", "batch": 16, "context": 8192, "k": 10, "steps": 8},
        # ingesting a 4k prompt
        {"name": "prefill_8b_b1_4k", "kind": "prefill", "model": "8b", "batch": 1, "context": 4096},
        # copying merged with a draft model that proposes where nothing matches
        {"name": "drafted_8b_b1_4k_k10_d3", "kind": "drafted", "batch": 1, "context": 4096, "k": 10, "delta": 3, "spans": 2, "span": 25, "fresh": 3},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["search", "search", "generate", "generate", "generate", "tiny", "verify", "verify", "host_steps", "prefill", "drafted"])
    if kind == "search":
        return {"kind": "search", "batch": _log_int(rng, 1, 64), "tokens": _log_int(rng, 1000, 32768), "gamma": rng.choice([2, 3, 5]),
                "k": rng.randint(1, 20), "policy": rng.choice([cs.LATEST, cs.FIRST])}
    if kind == "tiny":
        return {"kind": "generate", "model": "tiny", "batch": rng.randint(1, 8), "context": rng.randint(450, 800), "k": rng.randint(0, 12), "steps": rng.randint(4, 11)}
    if kind == "generate":
        batch = _log_int(rng, 1, 16)
        return {"kind": "generate", "model": "8b", "batch": batch, "context": _log_int(rng, 800, min(30720, 131072 // batch)),
                "k": rng.choice([0, rng.randint(1, 10), min(20, 176 // batch - 1)]), "steps": rng.randint(4, 6)}
    if kind == "verify":
        batch = _log_int(rng, 1, 16)
        return {"kind": "verify", "model": "8b", "batch": batch, "context": _log_int(rng, 300, 30720 // batch), "k": rng.randint(1, min(20, 176 // batch - 1))}
    if kind == "host_steps":
        return {"kind": "host_steps", "model": "8b", "batch": rng.randint(1, 4), "context": _log_int(rng, 800, 8000), "k": rng.randint(1, 12), "steps": rng.randint(2, 4)}
    if kind == "prefill":
        batch = rng.choice([1, 1, 2, 4])
        return {"kind": "prefill", "model": "8b", "batch": batch, "context": _log_int(rng, 200, 4096 // batch)}
    return {"kind": "drafted", "batch": 1, "context": _log_int(rng, 1000, 8000), "k": rng.randint(5, 12), "delta": rng.randint(2, 5), "spans": rng.randint(1, 2),
            "span": rng.randint(15, 25), "fresh": rng.randint(1, 3)}


# ------------------------------------------------------------------------------ what a case holds
def _lengths(case):
    """Tokens whose K/V are cached when the call is made, per sequence: a batch is ragged."""
    n = case["context"]
    return [n - (37 * b) % max(1, n // 8) for b in range(case["batch"])]


def _taus(case):
    """Accepted draft tokens of each step: evenly spread over 0..k."""
    steps, k = case["steps"], case["k"]
    return [round(i * k / max(1, steps - 1)) for i in range(steps)]


def _new_tokens(case):
    return sum(_taus(case)) + case["steps"]


def _drafted_script(case, context, fresh):
    """`spans` times: a verbatim span of the context, then tokens that occur nowhere in it."""
    out, at = [], 0
    for s in range(case["spans"]):
        src = 50 + s * (case["span"] + 20)
        out += context[src:src + case["span"]] + fresh[at:at + case["fresh"]]
        at += case["fresh"]
    return out


def _drafted_counts(case):
    """(target steps, steps that the draft model drafts) of the loop over distinct token ids: the
    search finds a match exactly when the last GAMMA tokens lie inside one copied span."""
    n = case["context"] + 1
    context = list(range(n))
    script = _drafted_script(case, context, list(range(n, n + 4096)))
    where = {tuple(context[i:i + GAMMA]): i for i in range(n - GAMMA + 1)}
    hist, at, steps, drafted = list(context), 0, 0, 0
    while at < len(script):
        p = where.get(tuple(hist[-GAMMA:]), -1)
        tau = 0
        if 0 <= p <= len(hist) - 2 * GAMMA:
            draft = hist[p + GAMMA:p + GAMMA + case["k"]]
            while tau < len(draft) and at + tau < len(script) and draft[tau] == script[at + tau]:
                tau += 1
        else:
            drafted += 1
        take = script[at:at + tau + 1]
        hist += take
        at += len(take)
        steps += 1
    return steps, drafted


def _model(cfg, seed, max_seq, batch, k, lens):
    ctx = cs.Context(cfg, inputs.make_weights(cfg, seed=seed, device="cuda"), max_seq=max_seq, max_batch=batch, k_max=k)
    kv = inputs.synthetic_kv(cfg, batch, max_seq, max(lens), seed=seed + 1, device="cuda") if lens else ctx.alloc_kv()
    return ctx, kv


def _rows(rows, stride):
    """Ragged token rows as one int32 array."""
    h = np.zeros((len(rows), stride), dtype=np.int32)
    for b, r in enumerate(rows):
        h[b, :len(r)] = r
    return h


def prepare(case, seed):
    kind, B = case["kind"], case["batch"]
    rng = np.random.default_rng(seed)
    if kind == "search":
        n = case["tokens"]
        spans = max(1, min(16, n // 2048))
        hi = min(512, (n - 64) // 2 // spans)
        hist, _, _ = inputs.match_search_histories(batch=B, n=n, seed=seed, n_spans=spans, span_lo=min(64, hi), span_hi=hi)
        # the histories of a batch are not equally long
        lens = [n - (137 * b) % max(1, n // 4) for b in range(B)]
        return {"case": case, "hist": torch.from_numpy(hist).cuda(), "len": torch.tensor(lens, dtype=torch.int32, device="cuda")}
    if kind == "drafted":
        n = case["context"] + 1
        cfg = MODELS["8b"]
        ids = rng.permutation(cfg.vocab).astype(np.int32).tolist()
        context = ids[:n]
        script = _drafted_script(case, context, ids[n:n + 4096])
        new = len(script)
        max_seq = n + new + max(case["k"], case["delta"]) + 16
        lens = _lengths(case)
        tctx, tkv = _model(cfg, seed, max_seq, 1, max(case["k"], case["delta"]), lens)
        dctx, dkv = _model(DRAFT_1B, seed + 7, max_seq, 1, 15, lens)
        h = torch.from_numpy(_rows([context], n + new + 16)).cuda()
        start = torch.tensor([n], dtype=torch.int32, device="cuda")
        return {"case": case, "ctx": tctx, "dctx": dctx, "kv": tkv, "dkv": dkv, "hist": h, "len0": start, "kv0": start - 1, "len": start.clone(),
                "kvlen": start.clone(), "dlen": start.clone(), "new": new, "script": torch.tensor([script], dtype=torch.int32, device="cuda")}
    cfg, lens = MODELS[case["model"]], _lengths(case)
    if kind == "prefill":
        ctx, kv = _model(cfg, seed, case["context"] + 64, B, 10, None)
        h = _rows([inputs.zipf_tokens(rng, n + 1, cfg.vocab) for n in lens], case["context"] + 64)
        return {"case": case, "ctx": ctx, "kv": kv, "hist": torch.from_numpy(h).cuda(), "len": torch.tensor(lens, dtype=torch.int32, device="cuda") + 1,
                "kvlen": torch.zeros(B, dtype=torch.int32, device="cuda")}
    k = case["k"]
    if kind == "verify":
        taus = rng.integers(0, k + 1, size=B)
        last, draft, dlen, script = inputs.verify_inputs_with_tau(rng, B, k, taus, cfg.vocab)
        ctx, kv = _model(cfg, seed, case["context"] + 64, B, k, lens)
        kv0 = torch.tensor(lens, dtype=torch.int32, device="cuda")
        return {"case": case, "ctx": ctx, "kv": kv, "kv0": kv0, "kvlen": kv0.clone(), **{n: torch.from_numpy(np.ascontiguousarray(v)).cuda() for n, v in
                (("last", last), ("draft", draft), ("dlen", dlen), ("script", script))},
                "logits": torch.zeros(B, k + 1, cfg.vocab, dtype=torch.float32, device="cuda")}
    new = _new_tokens(case)
    order = [rng.permutation(_taus(case)) for _ in range(B)]
    if kind == "host_steps":
        order = order[:1] * B          # sequences that advance together, so that the script rows of a step are known beforehand
    hists, scripts = zip(*(inputs.tau_controlled_case(rng, o, GAMMA, k, n, cfg.vocab) for o, n in zip(order, lens)))
    stride = (case["context"] + 1 + new + k + 16) // 4 * 4
    ctx, kv = _model(cfg, seed, stride, B, k, lens)
    h, script = torch.from_numpy(_rows(hists, stride)), _rows(scripts, new + k + 1)
    n0 = torch.tensor(lens, dtype=torch.int32) + 1
    if kind == "generate":
        n0 = n0.cuda()
        return {"case": case, "ctx": ctx, "kv": kv, "hist": h.cuda(), "len0": n0, "len": n0.clone(), "kv0": n0 - 1, "kvlen": n0.clone(), "new": new,
                "script": torch.from_numpy(np.ascontiguousarray(script[:, :new])).cuda()}
    at = np.concatenate([[0], np.cumsum(order[0] + 1)])
    rows = [torch.from_numpy(np.ascontiguousarray(script[:, a:a + k + 1])).pin_memory() for a in at[:-1]]
    return {"case": case, "ctx": ctx, "kv": kv, "hist": h.pin_memory(), "len0": n0, "len": n0.clone().pin_memory(), "kv0": (n0 - 1).cuda(),
            "kvlen": n0.cuda(), "hist_dev": torch.zeros(B, stride, dtype=torch.int32, device="cuda"),
            "len_dev": torch.zeros(B, dtype=torch.int32, device="cuda"), "rows": rows, "new": new,
            "tau": torch.zeros(B, dtype=torch.int32).pin_memory(), "out": torch.zeros(B, k + 1, dtype=torch.int32).pin_memory()}


def _appended(s, kv, new):
    """The cache rows that a pass appended, of every sequence."""
    return [kv[:, :, b, :, n:n + new] for b, n in enumerate(_lengths(s["case"]))]


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "search":
        return cs.cs_find_match(s["hist"], s["len"], case["gamma"], case["k"], case["policy"])
    if kind == "prefill":
        s["ctx"].cs_prefill(s["hist"], s["len"], case["context"] + 1, s["kv"], s["kvlen"])
        return {"kv_len": s["kvlen"], "kv": [s["kv"][:, :, b, :, :n] for b, n in enumerate(_lengths(case))]}
    # a pass starts from the cached context again: two small copies
    s["kvlen"].copy_(s["kv0"])
    if kind == "verify":
        accept, out, ids = s["ctx"].cs_verify_step(s["last"], s["draft"], s["dlen"], s["kv"], s["kvlen"], target_script=s["script"], logits_dbg=s["logits"])
        return {"accept": accept, "out": out, "ids": ids, "logits": s["logits"], "kv_len": s["kvlen"], "kv": _appended(s, s["kv"], case["k"] + 1)}
    s["len"].copy_(s["len0"])
    if kind == "generate":
        st = s["ctx"].cs_decode_loop(s["hist"], s["len"], s["kv"], s["kvlen"], GAMMA, case["k"], s["new"], script=s["script"])
    elif kind == "host_steps":
        for rows in s["rows"]:
            s["ctx"].cs_step_host(s["hist"], s["len"], s["hist_dev"], s["len_dev"], s["kv"], s["kvlen"], GAMMA, case["k"], s["tau"], s["out"],
                                  script_host=rows)
        st = {"tau": s["tau"].clone(), "out": s["out"].clone()}
    else:
        s["dlen"].copy_(s["kv0"])
        st = s["ctx"].cs_decode_loop_drafted(s["dctx"], s["hist"], s["len"], s["kv"], s["kvlen"], s["dkv"], s["dlen"], GAMMA, case["k"], case["delta"],
                                             s["new"], script=s["script"])
    if "tau_hist" in st:
        st["tau_hist"] = np.asarray(st["tau_hist"], dtype=np.int64)
    return {"stats": st, "hist": s["hist"], "len": s["len"], "kv_len": s["kvlen"], "kv": _appended(s, s["kv"], s["new"])}


# ------------------------------------------------------------------------------ what a pass costs at least
def _forward(cfg, rows, lens, lm_head=True):
    """(bytes, flops) of one forward of `rows` rows per sequence on top of `lens` cached tokens."""
    params = cfg.streamed_params() if lm_head else cfg.n_layers * cfg.params_per_layer()
    keys = sum(lens) + rows * len(lens)
    nbytes = 2 * params + keys * cfg.kv_bytes_per_token()
    flops = 2 * rows * len(lens) * params + 4 * cfg.n_layers * cfg.q_dim * sum(rows * n + rows * (rows + 1) // 2 for n in lens)
    return nbytes, flops


def work(case):
    kind = case["kind"]
    if kind == "search":
        n, B = case["tokens"], case["batch"]
        tokens = sum(n - (137 * b) % max(1, n // 4) for b in range(B))
        return {"bytes": 4 * tokens + 4 * B * (case["k"] + 3), "flops": tokens}
    lens = _lengths(case)
    if kind == "drafted":
        steps, drafted = _drafted_counts(case)
        t, d = _forward(MODELS["8b"], case["k"] + 1, lens), _forward(DRAFT_1B, 1, lens)
        return {"bytes": steps * t[0] + drafted * case["delta"] * d[0], "flops": steps * t[1] + drafted * case["delta"] * d[1]}
    cfg = MODELS[case["model"]]
    if kind == "prefill":
        # every prompt in one causal forward: the weights once, the cache written once
        nbytes, flops = 2 * cfg.n_layers * cfg.params_per_layer() + sum(lens) * cfg.kv_bytes_per_token(), 0
        for n in lens:
            flops += 2 * n * cfg.n_layers * cfg.params_per_layer() + 4 * cfg.n_layers * cfg.q_dim * n * (n + 1) // 2
        return {"bytes": nbytes, "flops": flops}
    nbytes, flops = _forward(cfg, case["k"] + 1, lens)
    if kind == "verify":
        return {"bytes": nbytes + 4 * cfg.vocab * case["batch"] * (case["k"] + 1), "flops": flops}
    return {"bytes": case["steps"] * nbytes, "flops": case["steps"] * flops}


def tolerance(case):
    """Cached rows are bf16 and every activation is fp32-equivalent, so what another summation order
    changes is which way some rows round: measured by running the same inputs through the three
    attention kernels, which sum in different orders (2-norm 3e-4 of the appended rows, 8e-4 of a
    whole prefilled cache, 4e-5 of the logits; single values move by one bf16 step, 8e-3)."""
    if case["kind"] == "search":
        return "exact"
    if case["kind"] == "prefill":
        return {"rel": 3.5e-3, "max": 0.05, "differ": 1e-3}
    return {"rel": 1.4e-3, "max": 0.035, "differ": 1e-3}
