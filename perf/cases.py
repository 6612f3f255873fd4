"""Workloads this library is timed on: whole passes through its public entry points.

Four kinds of pass, each what a serving program does between two tokens:

  serve    one or more consecutive serving steps: asynclm_plan for the step's lengths and page table,
           then for every layer the append of the new K/V rows and the attention of the new tokens
           (`call`: "calls" = kv_append + attn_mixed, "step" = the one-call form, "rope" = rotary append
           of keys and queries + attn_mixed).  Sequences decode one token, bring an interrupt span or
           are paused; with ctx_hi = 0 they are recomputed from nothing (the trap handler's recompute).
  monitor  constrained greedy selection of the next token of every sequence over its logits
  swap     a paused sequence's KV pages to pinned host memory and back into other pages

Lengths follow from the case alone (`lengths` seeds them), so that its work is a fixed number; page
tables and all values follow from the seed given to prepare().  Values are N(0, 1) in bf16, as queries
and keys are after the normalisations of a trained model's layers.
"""
import math

import numpy as np
import torch

from paper_2412_07017_b200 import binding as B
from paper_2412_07017_b200 import workload as W

PAGE = 16
ROPE_THETA = 500000.0
# (query heads, kv heads, head_dim): the shapes of the configurations and of the parity tests
SHAPES = [(32, 8, 128), (64, 8, 128), (32, 8, 64), (8, 2, 64), (16, 2, 128), (8, 8, 128), (4, 4, 64), (4, 2, 128), (8, 1, 64), (16, 4, 128)]


def _serve(name, shape, batch, ctx, spans=(0, 1, 1), paused=0, layers=1, steps=1, call="calls", lse=True, lengths=1):
    """spans: (sequences that bring one per step, shortest, longest), in new tokens."""
    return {"name": name, "kind": "serve", "q_heads": shape[0], "kv_heads": shape[1], "head_dim": shape[2], "batch": batch,
            "ctx_lo": ctx[0], "ctx_hi": ctx[1], "interrupted": spans[0], "span_lo": spans[1], "span_hi": spans[2],
            "paused": paused, "layers": layers, "steps": steps, "call": call, "lse": lse, "lengths": lengths}


def listed():
    return [
        # the smallest step of all: 4 sequences, one layer, head_dim 64, one 12-token interrupt; all latency
        _serve("tiny_step", (8, 2, 64), 4, (100, 300), (1, 12, 12), lengths=241207018),
        # an interactive server with few users: 4 sequences decode through 32 layers, one call per layer
        _serve("decode_few", (32, 8, 128), 4, (512, 4096), layers=32, call="step", lse=False, lengths=5),
        # decode only, 64 sequences: the ordinary step while no function call returns
        _serve("decode_many", (32, 8, 128), 64, (1024, 3072), layers=8, lengths=11),
        # the mixed batch: 32 sequences, a quarter with a returning call, a whole 32-layer model
        _serve("mixed_layers", (32, 8, 128), 32, (512, 4096), (8, 8, 64), layers=32, call="rope", lse=False, lengths=241207019),
        # large-batch serving with 8 query heads per kv head, a tenth interrupted, some paused by a trap
        _serve("mixed_large", (64, 8, 128), 128, (2048, 8192), (13, 16, 128), paused=6, layers=2, lengths=241207020),
        # long contexts, two long interrupts
        _serve("long_context", (32, 8, 128), 8, (32768, 131072), (2, 256, 256), layers=2, lengths=241207021),
        # interrupt-trace replay: consecutive steps of 256 sequences, each planned anew, about 2 % interrupted
        _serve("replay", (32, 8, 128), 256, (256, 2048), (5, 9, 97), paused=3, steps=4, lengths=241207022),
        # head_dim 64: the mixed batch of a small model
        _serve("mixed_dim64", (32, 8, 64), 32, (512, 4096), (8, 8, 64), layers=16, lengths=31),
        # a burst of returning calls: every sequence brings a span
        _serve("burst", (32, 8, 128), 24, (1024, 3072), (24, 33, 96), layers=4, lengths=12),
        # the trap handler's recompute of one long sequence, rotary append included
        _serve("recompute", (32, 8, 128), 1, (0, 0), (1, 8192, 8192), layers=4, call="rope", lse=False, lengths=7),
        # the token monitor over a full vocabulary
        {"name": "monitor", "kind": "monitor", "batch": 256, "vocab": 128256, "dtype": "bf16"},
        # a trapped sequence of 8192 tokens swapped out and in again (bound by PCIe)
        {"name": "swap", "kind": "swap", "q_heads": 32, "kv_heads": 8, "head_dim": 128, "tokens": 8192},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    what = rng.random()
    if what < 0.12:
        dtype = rng.choice(["bf16", "f32"])
        return {"kind": "monitor", "batch": _log_int(rng, 1, 256), "vocab": rng.choice([128256, 32000, _log_int(rng, 1000, 128256)]),
                "dtype": dtype}
    hq, hkv, d = rng.choice(SHAPES)
    if what < 0.18:
        return {"kind": "swap", "q_heads": hq, "kv_heads": hkv, "head_dim": d, "tokens": _log_int(rng, 100, 8192)}
    if what < 0.32:      # sequences recomputed from nothing
        batch = rng.choice([1, 1, 2, 5])
        hi = _log_int(rng, 128, 6000 // batch)
        case = _serve("", (hq, hkv, d), batch, (0, 0), (batch, max(1, hi // 2), hi), layers=rng.randint(1, 2),
                      call=rng.choice(["calls", "rope", "step"]), lse=rng.random() < 0.5, lengths=rng.randrange(1 << 30))
    else:
        batch = _log_int(rng, 1, 256)
        hi = _log_int(rng, 128, 8192)
        hi = max(128, min(hi, 600_000 // batch))
        interrupted = rng.choice([0, 1, batch // 10, batch // 4, batch])
        interrupted = min(interrupted, batch)
        span_hi = _log_int(rng, 2, 128)
        if interrupted * span_hi > 2048:
            span_hi = max(2, 2048 // interrupted)
        paused = min(batch - interrupted, rng.choice([0, 0, batch // 8]))
        kv_bytes = batch * hi * hkv * d * 4
        layers = max(1, min(rng.choice([1, 4, 16, 32]), int(2.5e9 / kv_bytes)))
        steps = rng.choice([1, 1, 3]) if layers == 1 else 1
        case = _serve("", (hq, hkv, d), batch, (max(1, hi // 8), hi), (interrupted, 2, span_hi), paused=paused, layers=layers,
                      steps=steps, call=rng.choice(["calls", "calls", "rope", "step"]), lse=rng.random() < 0.5,
                      lengths=rng.randrange(1 << 30))
    del case["name"]
    return case


def _lengths(case):
    """(contexts before the first step [B], new tokens per step [steps][B])."""
    g = np.random.Generator(np.random.Philox(key=[case["lengths"], 0]))
    n = case["batch"]
    ctx = g.integers(case["ctx_lo"], case["ctx_hi"] + 1, size=n)
    q_lens = np.ones((case["steps"], n), dtype=np.int64)
    for t in range(case["steps"]):
        who = g.permutation(n)
        spans = who[:case["interrupted"]]
        q_lens[t, spans] = g.integers(case["span_lo"], case["span_hi"] + 1, size=len(spans))
        q_lens[t, who[case["interrupted"]:case["interrupted"] + case["paused"]]] = 0
    return ctx, q_lens


def _normal(gen, *size):
    return torch.empty(size, dtype=torch.bfloat16, device="cuda").normal_(generator=gen)


def _prepare_serve(case, seed):
    shape = W.Shape(case["q_heads"], case["kv_heads"], case["head_dim"], PAGE)
    ctx, q_lens = _lengths(case)
    layers, n = case["layers"], case["batch"]
    need = -(-(ctx + q_lens.sum(axis=0)) // PAGE)
    num_pages = int(need.sum()) + 64
    page_indptr = np.zeros(n + 1, dtype=np.int32)
    page_indptr[1:] = np.cumsum(need)
    ids = np.random.Generator(np.random.Philox(key=[seed, 1])).permutation(num_pages)[:page_indptr[-1]].astype(np.int32)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    pools = _normal(gen, layers, num_pages, 2, shape.num_kv_heads, PAGE, shape.head_dim)
    max_q = int(q_lens.sum(axis=1).max())
    host_bytes, dev_bytes = B.workspace_size(shape, num_pages, n, max_q, int(page_indptr[-1]))
    steps = []
    for t in range(case["steps"]):
        q_indptr = np.zeros(n + 1, dtype=np.int32)
        q_indptr[1:] = np.cumsum(q_lens[t])
        total = int(q_indptr[-1])
        steps.append({
            "q_indptr": q_indptr, "kv_len_before": (ctx + q_lens[:t].sum(axis=0)).astype(np.int32),
            "q": _normal(gen, layers, total, shape.num_q_heads, shape.head_dim),
            "k_new": _normal(gen, layers, total, shape.num_kv_heads, shape.head_dim),
            "v_new": _normal(gen, layers, total, shape.num_kv_heads, shape.head_dim),
            "out": torch.empty((layers, total, shape.num_q_heads, shape.head_dim), dtype=torch.bfloat16, device="cuda"),
            "lse": torch.empty((layers, total, shape.num_q_heads), dtype=torch.float32, device="cuda") if case["lse"] else None})
    # two plan workspaces in turn: the next step is planned on the host while the last one's plan is still
    # being copied or used on the GPU; the event says when a workspace's copy has been made
    slots = [{"host_ws": torch.empty(host_bytes, dtype=torch.uint8).pin_memory(),
              "dev_ws": torch.empty(dev_bytes, dtype=torch.uint8, device="cuda"), "copied": torch.cuda.Event()} for _ in range(2)]
    return {"case": case, "shape": shape, "num_pages": num_pages, "page_indptr": page_indptr, "page_indices": ids, "pools": pools,
            "steps": steps, "slots": slots, "planned": 0}


def _run_serve(state):
    case = state["case"]
    for st in state["steps"]:
        slot = state["slots"][state["planned"] % len(state["slots"])]
        state["planned"] += 1
        slot["copied"].synchronize()      # the host workspace may be written again
        plan = B.asynclm_plan(state["shape"], state["num_pages"], st["q_indptr"], st["kv_len_before"], state["page_indptr"],
                              state["page_indices"], host_ws=slot["host_ws"], dev_ws=slot["dev_ws"])
        slot["copied"].record()
        for layer in range(case["layers"]):
            q, k_new, v_new, pool, out = st["q"][layer], st["k_new"][layer], st["v_new"][layer], state["pools"][layer], st["out"][layer]
            lse = st["lse"][layer] if case["lse"] else None
            if case["call"] == "step":
                B.asynclm_step(plan, q, k_new, v_new, pool, out, lse)
                continue
            if case["call"] == "rope":
                B.asynclm_kv_append_rope(plan, k_new, v_new, pool, q, ROPE_THETA)
            else:
                B.asynclm_kv_append(plan, k_new, v_new, pool)
            B.asynclm_attn_mixed(plan, q, pool, out, lse)
    got = {"pools": state["pools"], "out": [st["out"] for st in state["steps"]]}
    if case["lse"]:
        got["lse"] = [st["lse"] for st in state["steps"]]
    if case["call"] == "rope":
        got["q"] = [st["q"] for st in state["steps"]]      # rotated in place
    return got


def _prepare_monitor(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    n, vocab = case["batch"], case["vocab"]
    stride = -(-vocab // 8) * 8      # rows are 16-byte aligned
    logits = torch.empty((n, stride), dtype=torch.bfloat16 if case["dtype"] == "bf16" else torch.float32, device="cuda")
    logits.normal_(generator=gen).mul_(3.0)
    special = {name: vocab - 250 + k for k, name in enumerate(("CALL", "INTR", "TRAP", "END", "HEAD"))}
    # mostly plain text, some sequences inside a function-call block, a few right after [TRAP]; now and
    # then the model wants a CML token, which its state may or may not allow
    g = np.random.Generator(np.random.Philox(key=[seed, 2]))
    states = torch.from_numpy(g.choice(4, n, p=[0.8, 0.08, 0.1, 0.02]).astype(np.int32)).cuda()
    for b in np.nonzero(g.random(n) < 0.06)[0]:
        logits[int(b), special[str(g.choice(["CALL", "TRAP", "END", "HEAD"]))]] = 20.0
    return {"case": case, "logits": logits[:, :vocab], "special": special, "state_in": states,
            "out": [torch.empty_like(states) for _ in range(3)],
            "ws": torch.zeros(B.token_monitor_workspace_bytes(n), dtype=torch.uint8, device="cuda")}


def _run_monitor(state):
    token, after, flags = state["out"]
    B.asynclm_token_monitor_step(state["logits"], state["special"], state["state_in"], token, after, flags, state["ws"])
    return {"token": token, "state": after, "flags": flags}


def _prepare_swap(case, seed):
    shape = W.Shape(case["q_heads"], case["kv_heads"], case["head_dim"], PAGE)
    n = -(-case["tokens"] // PAGE)
    num_pages = 2 * n + 64
    perm = np.random.Generator(np.random.Philox(key=[seed, 1])).permutation(num_pages).astype(np.int32)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    return {"case": case, "shape": shape, "num_pages": num_pages, "out_pages": perm[:n].copy(), "in_pages": perm[n:2 * n].copy(),
            "pool": _normal(gen, num_pages, 2, shape.num_kv_heads, PAGE, shape.head_dim),
            "staging": torch.empty(B.kv_swap_staging_bytes(shape, num_pages, n), dtype=torch.uint8, device="cuda"),
            "image": torch.empty(n * shape.page_elems, dtype=torch.int16).pin_memory()}


def _run_swap(state):
    B.asynclm_kv_swap_out(state["shape"], state["num_pages"], state["out_pages"], state["pool"], state["staging"], state["image"])
    B.asynclm_kv_swap_in(state["shape"], state["num_pages"], state["in_pages"], state["pool"], state["staging"], state["image"])
    return {"pool": state["pool"], "image": state["image"]}


def prepare(case, seed):
    return {"serve": _prepare_serve, "monitor": _prepare_monitor, "swap": _prepare_swap}[case["kind"]](case, seed)


def run(state):
    return {"serve": _run_serve, "monitor": _run_monitor, "swap": _run_swap}[state["case"]["kind"]](state)


def work(case):
    """Bytes and operations of one pass: cached K/V read, new K/V rows read and written, queries read (and
    written, where they are rotated), outputs written, page ids read; two contractions per visible key."""
    if case["kind"] == "monitor":
        return {"bytes": case["batch"] * case["vocab"] * (2 if case["dtype"] == "bf16" else 4) + 16 * case["batch"], "flops": 0}
    token_bytes = 2 * case["kv_heads"] * case["head_dim"] * 2
    if case["kind"] == "swap":
        pages = -(-case["tokens"] // PAGE)
        return {"bytes": 4 * pages * PAGE * token_bytes, "flops": 0}      # read and written, out and in
    ctx, q_lens = _lengths(case)
    row_bytes = case["q_heads"] * case["head_dim"] * 2
    total_bytes = total_flops = 0
    for t in range(case["steps"]):
        ql = q_lens[t]
        before = ctx + q_lens[:t].sum(axis=0)
        new = int(ql.sum())
        total_bytes += int(before[ql > 0].sum()) * token_bytes + 2 * new * token_bytes + (3 if case["call"] == "rope" else 2) * new * row_bytes
        total_bytes += new * case["q_heads"] * 4 * bool(case["lse"]) + 4 * int((-(-(before + ql) // PAGE))[ql > 0].sum())
        total_flops += 4 * case["head_dim"] * case["q_heads"] * int((ql * before + ql * (ql + 1) // 2).sum())
    return {"bytes": total_bytes * case["layers"], "flops": total_flops * case["layers"]}


def tolerance(case):
    """Attention: bf16 inputs and outputs, probabilities rounded to bf16 for the second contraction.  Against the
    same path in fp64 the serving cases measure rel 2.1e-3 to 2.4e-3 and max 0.6e-2 to 2.4e-2; stated is four times
    that.  The other kinds move or select bits."""
    if case["kind"] == "serve":
        return {"rel": 1e-2, "max": 0.1}
    return "exact"
