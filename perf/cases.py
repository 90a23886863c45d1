"""The work that is timed: one pass through the public entry points for each way the library is used.

Five kinds of case, all seeded synthetic stand-ins with the structure of expand-verify-select search:

  step         a whole step on device-resident data (`DevicePipeline.step`): computation deduplication, the gather of
               the unique candidates, tree attention, selection.  Decode (one query token a candidate), verification
               (16 to 128 query tokens a candidate) and steps that mix the two.
  host_step    the same step for data in page-locked host memory (`HostStepPipeline`)
  branch       on-demand branching: the draws of every sequence and their grouping into children
  prefix_tree  the radix tree of candidate paths from raw token ids
  early_prune  pruning while only part of the candidates has been verified
"""
import math

import numpy as np
import torch

from paper_2609_39334_b200 import binding as B
from paper_2609_39334_b200 import synth
from paper_2609_39334_b200.pipeline import DevicePipeline, HostStepPipeline

DEV = "cuda:0"


def _step(name, heads, problems, levels, fanout, leaf, mode, steps=(1, 1), dup=0.0, kind="step"):
    return {"name": name, "kind": kind, "q_heads": heads[0], "kv_heads": heads[1], "problems": problems,
            "levels": " ".join(map(str, levels)), "fanout": " ".join(map(str, fanout)), "leaf_lo": leaf[0],
            "leaf_hi": leaf[1], "mode": mode, "step_lo": steps[0], "step_hi": steps[1], "dup": dup}


def listed():
    return [
        # one user's question with a handful of candidates: nothing but launches and latency
        _step("decode_tiny", (12, 2), 1, [256], [8], (0, 64), "decode", dup=0.125),
        # expansion: every candidate of 16 problems decodes one token (a 1.5 B generator's attention shape)
        _step("decode_expansion", (12, 2), 16, [512], [64], (32, 512), "decode", dup=0.1),
        # expansion from a two-level tree: prompt, then branches, then leaves (an 8 B generator's shape)
        _step("decode_two_level", (32, 8), 4, [2048, 256], [16, 16], (64, 256), "decode", dup=0.3),
        # a lazy-verification batch that has just been released: few candidates, short steps (a 7 B verifier's shape)
        _step("verify_small", (28, 4), 1, [1024], [8], (64, 512), "verify", (16, 128)),
        # a full verification batch
        _step("verify_batch", (28, 4), 8, [1024], [32], (64, 512), "verify", (16, 128)),
        # a large server's step: half of the candidates decode, half are verified, long prompts, 21 GB of KV pages
        _step("mixed_large", (32, 8), 32, [4096], [256], (128, 1024), "mixed", (64, 64), dup=0.2),
        # expansion for a caller whose candidates, queries and scores are produced on the host
        _step("host_decode", (12, 2), 16, [512], [64], (32, 512), "decode", dup=0.1, kind="host_step"),
        # on-demand branching of a few sequences that stand for several candidates each
        {"name": "branch_few", "kind": "branch", "sequences": 16, "vocab": 151936, "most": 8, "temperature": 0.8},
        # ... and of a whole expansion batch, most sequences of which stand for one or two candidates
        {"name": "branch_batch", "kind": "branch", "sequences": 922, "vocab": 151936, "most": 2, "temperature": 0.8},
        # prefix sharing found among the candidates of a few problems ...
        {"name": "tree_few", "kind": "prefix_tree", "problems": 4, "candidates": 16, "prompt": 512, "own_lo": 32,
         "own_hi": 512, "share": 0.25},
        # ... and among those of a large server
        {"name": "tree_large", "kind": "prefix_tree", "problems": 64, "candidates": 256, "prompt": 4096, "own_lo": 128,
         "own_hi": 1024, "share": 0.25},
        # pruning between verification batches, half of the candidates scored so far
        {"name": "early_prune", "kind": "early_prune", "problems": 64, "candidates": 256, "verified": 0.5},
    ]


# ---- cases of the same ranges -------------------------------------------------------------------------------------
def _log(rng, lo, hi):
    """A whole number, spread evenly over the logarithm of the range."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_step(rng, kind):
    heads = rng.choice([(12, 2), (28, 4), (32, 8)])
    mode = "decode" if kind == "host_step" else rng.choice(["decode", "decode", "verify", "verify", "mixed"])
    if rng.random() < 0.3:
        levels = [16 * _log(rng, 16, 192), 16 * _log(rng, 4, 32)]
        fanout = [rng.randint(2, 16), rng.randint(4, 16)]
    else:
        levels = [16 * _log(rng, 16, 256)]
        fanout = [_log(rng, 8, 256)]
    lo = rng.randint(0, 128)
    hi = lo + _log(rng, 64, 896)
    if mode == "mixed":
        step = rng.randint(16, 128)
        steps = (step, step)
    else:
        steps = (1, 1) if mode == "decode" else (16, rng.randint(32, 128))
    problems = _log(rng, 1, 32)
    case = _step("", heads, problems, levels, fanout, (lo, hi), mode, steps, round(rng.choice([0.0, rng.uniform(0.05, 0.3)]), 3),
                 kind)
    del case["name"]
    most = work(listed()[5])
    while True:
        w = work(case)
        if w["bytes"] <= 0.5 * most["bytes"] and w["flops"] <= 0.5 * most["flops"] or case["problems"] == 1:
            return case
        case["problems"] = max(1, case["problems"] // 2)


def draw(rng):
    kind = rng.choice(["step"] * 6 + ["host_step", "branch", "branch", "prefix_tree", "prefix_tree", "early_prune"])
    if kind in ("step", "host_step"):
        return _draw_step(rng, kind)
    if kind == "branch":
        return {"kind": kind, "sequences": _log(rng, 1, 900), "vocab": rng.choice([32000, 128256, 151936]),
                "most": rng.randint(1, 16), "temperature": round(rng.uniform(0.6, 1.2), 3)}
    if kind == "prefix_tree":
        return {"kind": kind, "problems": _log(rng, 1, 60), "candidates": _log(rng, 8, 256), "prompt": _log(rng, 200, 4096),
                "own_lo": rng.randint(16, 128), "own_hi": _log(rng, 160, 1024), "share": round(rng.uniform(0.0, 0.5), 3)}
    return {"kind": kind, "problems": _log(rng, 1, 512), "candidates": _log(rng, 8, 1024),
            "verified": round(rng.uniform(0.1, 1.0), 3)}


# ---- inputs -------------------------------------------------------------------------------------------------------
def _ints(text):
    return [int(x) for x in text.split()]


def _sizes(lo, hi, count, seed):
    """`count` sizes in lo..hi: the same ones for every seed (so that all results have one shape), in the seed's order."""
    return np.random.default_rng(seed).permutation(np.random.default_rng(0).integers(lo, hi + 1, size=count))


def _step_tokens(case, seed):
    lo, hi = case["step_lo"], case["step_hi"]
    if case["mode"] == "decode":
        return lambda i, n, rng: 1
    if case["mode"] == "verify":
        sizes = iter(_sizes(lo, hi, case["problems"] * math.prod(_ints(case["fanout"])), seed).tolist())
        return lambda i, n, rng: next(sizes)
    return lambda i, n, rng: 1 if i < n // 2 else lo


def _prepare_step(case, seed):
    w = synth.build_tree_workload(
        case["kind"], seed, case["q_heads"], case["kv_heads"], _ints(case["levels"]), _ints(case["fanout"]),
        case["problems"], (case["leaf_lo"], case["leaf_hi"]), _step_tokens(case, seed), dup_frac=case["dup"], device=DEV)
    pipe = DevicePipeline(w, DEV)
    for t in (pipe.out, pipe.lse, pipe.unique_paths, pipe.multiplicity):      # only the live rows are written
        t.zero_()
    if case["kind"] == "step":
        return {"pipe": pipe}
    host = HostStepPipeline(pipe, depth=1, compact=True)
    for t in host.sets[0]["h_out"].values():
        t.zero_()
    return {"pipe": pipe, "host": host}


def _prepare_branch(case, seed):
    g = torch.Generator(device=DEV).manual_seed(seed)
    rng = np.random.default_rng(seed)
    S, V = case["sequences"], case["vocab"]
    logits = torch.randn((S, V), generator=g, dtype=torch.float32, device=DEV) * 3
    off = np.concatenate([[0], np.cumsum(_sizes(1, case["most"], S, seed))]).astype(np.int64)
    n = int(off[-1])
    i32 = dict(dtype=torch.int32, device=DEV)
    return {"logits": logits, "off": torch.from_numpy(off).to(DEV), "n": n, "S": S, "V": V, "T": case["temperature"],
            "u": torch.from_numpy(rng.random(n, dtype=np.float32)).to(DEV), "tok": torch.zeros(n, **i32),
            "seq": torch.zeros(n, dtype=torch.int64, device=DEV), "one": torch.arange(n + 1, dtype=torch.int64, device=DEV),
            "canon": torch.zeros(n, **i32), "child": torch.zeros(n, **i32), "first": torch.zeros(n, **i32),
            "potential": torch.zeros(n, **i32), "children": torch.zeros(1, **i32),
            "ws": B.alloc_workspace(B.ss_dedup_workspace_bytes(n), DEV)}


def _prepare_prefix_tree(case, seed):
    g = torch.Generator(device=DEV).manual_seed(seed)
    rng = np.random.default_rng(seed)
    P, F, prompt = case["problems"], case["candidates"], case["prompt"]
    n = P * F
    # a candidate = its problem's prompt, what it has in common with three of its siblings, its own tokens
    own = rng.integers(case["own_lo"], case["own_hi"] + 1, size=n)
    off_np = np.concatenate([[0], np.cumsum(prompt + own)]).astype(np.int64)
    total = int(off_np[-1])
    off = torch.from_numpy(off_np).to(DEV)
    ids = torch.randint(0, synth.VOCAB, (total,), generator=g, dtype=torch.int32, device=DEV)
    prompts = torch.randint(0, synth.VOCAB, (P, prompt), generator=g, dtype=torch.int32, device=DEV)
    pos = torch.arange(prompt, device=DEV)
    for p in range(P):
        ids[(off[p * F:(p + 1) * F, None] + pos).reshape(-1)] = prompts[p].repeat(F)
    common = np.minimum((own * case["share"]).astype(np.int64), own - 1)
    first = (np.arange(n) // F) * F + (np.arange(n) % F) // 4 * 4
    common = np.minimum(common, common[first])
    path = torch.from_numpy(np.repeat(np.arange(n), common)).to(DEV)
    at = torch.from_numpy(np.concatenate([np.arange(c) for c in common]) + prompt).to(DEV)
    ids[off[path] + at] = ids[off[torch.from_numpy(first).to(DEV)[path]] + at]
    i32 = dict(dtype=torch.int32, device=DEV)
    state = {"ids": ids, "off": off, "n": n, "total": total, "order": torch.zeros(n, **i32), "leaf": torch.zeros(n, **i32),
             "num": torch.zeros(1, **i32), "ws": B.alloc_workspace(B.ss_prefix_tree_workspace_bytes(n, total, 16), DEV)}
    state.update({k: torch.zeros(2 * n, **i32) for k in ("parent", "kv_len", "src_path", "src_offset")})
    return state


def _prepare_early_prune(case, seed):
    rng = np.random.default_rng(seed)
    P, F = case["problems"], case["candidates"]
    size = _sizes(max(1, F - F // 8), F, P, seed)                   # some candidates have already been pruned
    seg = np.concatenate([[0], np.cumsum(size)]).astype(np.int32)
    n, k = int(seg[-1]), max(1, F // 4)
    u8 = dict(dtype=torch.uint8, device=DEV)
    return {"scores": torch.from_numpy(np.round(rng.random(n) * 64).astype(np.float32) / 64).to(DEV),
            "verified": torch.from_numpy((rng.random(n) < case["verified"]).astype(np.uint8)).to(DEV),
            "seg": torch.from_numpy(seg).to(DEV), "P": P, "n": n, "k": k, "pruned": torch.zeros(n, **u8),
            "selected": torch.zeros((P, k), dtype=torch.int32, device=DEV), "final": torch.zeros(P, **u8),
            "ws": B.alloc_workspace(B.ss_topk_workspace_bytes(n), DEV)}


def prepare(case, seed):
    make = {"step": _prepare_step, "host_step": _prepare_step, "branch": _prepare_branch,
            "prefix_tree": _prepare_prefix_tree, "early_prune": _prepare_early_prune}[case["kind"]]
    state = make(case, seed)
    state["kind"] = case["kind"]
    return state


# ---- one pass -----------------------------------------------------------------------------------------------------
def run(state):
    s = state
    if s["kind"] == "step":
        p = s["pipe"]
        p.step()
        return {"out": p.out, "lse": p.lse, "canon": p.canon, "path_to_unique": p.path_to_unique,
                "unique_paths": p.unique_paths, "multiplicity": p.multiplicity, "slot_out": p.slot_out,
                "num_unique": p.num_unique, "survivors": p.survivors, "keep": p.keep}
    if s["kind"] == "host_step":
        s["host"].submit(0)
        s["host"].synchronize()
        return dict(s["host"].sets[0]["h_out"])
    if s["kind"] == "branch":
        B.ss_branch_sample(s["logits"], s["off"], s["u"], s["S"], s["V"], s["T"], s["tok"], s["seq"])
        B.ss_dedup_paths(s["tok"], s["one"], s["seq"], None, s["n"], 0, s["canon"], s["child"], s["first"],
                         s["potential"], None, s["children"], s["ws"])
        return {k: s[k] for k in ("tok", "seq", "canon", "child", "first", "potential", "children")}
    if s["kind"] == "prefix_tree":
        B.ss_build_prefix_tree(s["ids"], s["off"], s["n"], s["total"], 16, s["order"], s["leaf"], s["parent"],
                               s["kv_len"], s["src_path"], s["src_offset"], s["num"], s["ws"])
        return {k: s[k] for k in ("order", "leaf", "parent", "kv_len", "src_path", "src_offset", "num")}
    B.ss_early_prune(s["scores"], s["verified"], s["seg"], s["P"], s["n"], s["k"], s["pruned"], s["selected"],
                     s["final"], s["ws"])
    return {k: s[k] for k in ("pruned", "selected", "final")}


# ---- what a pass cannot do without ----------------------------------------------------------------------------------
def _work_step(case):
    """Means over the random lengths: every unique KV token and every unique candidate's query read once, every result
    written once; 4 * 128 operations for each (query row, visible key)."""
    Hq, Hkv = case["q_heads"], case["kv_heads"]
    levels, fanout, P = _ints(case["levels"]), _ints(case["fanout"]), case["problems"]
    nodes, shared = P, 0.0
    for length, f in zip(levels, fanout):
        shared += nodes * length
        nodes *= f
    logical, unique, chain = nodes, nodes * (1 - case["dup"]), sum(levels)
    own = (case["leaf_lo"] + case["leaf_hi"]) / 2
    T = (case["step_lo"] + case["step_hi"]) / 2
    verify = {"decode": 0.0, "verify": 1.0, "mixed": 0.5}[case["mode"]]
    leaf = own + verify * T
    rows = (1 - verify) + verify * T
    keys = (1 - verify) * (chain + own) + verify * T * (chain + own + (T + 1) / 2)
    row_bytes = Hq * 128 * 2
    tokens = shared + unique * leaf
    return {"bytes": tokens * Hkv * 128 * 2 * 2 + unique * rows * (2 * row_bytes + 4 * Hq) + logical * (4 * leaf + 60),
            "flops": 4.0 * 128 * Hq * unique * keys}


def work(case):
    kind = case["kind"]
    if kind in ("step", "host_step"):
        return _work_step(case)
    if kind == "branch":
        draws = case["sequences"] * (1 + case["most"]) / 2
        return {"bytes": 4.0 * case["sequences"] * case["vocab"] + 40 * draws, "flops": 0.0}
    if kind == "prefix_tree":
        n = case["problems"] * case["candidates"]
        return {"bytes": 4.0 * n * (case["prompt"] + (case["own_lo"] + case["own_hi"]) / 2) + 40.0 * n, "flops": 0.0}
    n = case["problems"] * case["candidates"]
    return {"bytes": 7.0 * n, "flops": 0.0}


def tolerance(case):
    # bf16 results, and probabilities rounded to bf16 before they multiply V; everything else is whole numbers.  Measured:
    # 2.3e-3 (max 0.013) against the oracle in 64 bits, 2.6e-3 (0.016) against the library's kernel with fp32
    # probabilities.
    if case["kind"] in ("step", "host_step"):
        return {"rel": 1e-2, "max": 0.06}
    return "exact"
