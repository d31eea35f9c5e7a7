"""The workloads by which the library's speed is judged: what they are, one pass of each, and what a pass cannot do without.

Every pass goes through the package's public entry points, as a program that embeds the library calls them:

  prefill   one attention layer over a packed batch (`attn_fwd`).  The route depends on the lengths only: a model plans
            it once and its layers share it (`plan` False: it is in hand), a batch with new lengths plans first (`plan`
            True: `plan_route` is part of the pass, into arrays that are kept).
  dense     the same layer with every predecessor block selected (`dense_causal_fwd`): what a layer that was not
            converted runs.
  train     one layer forward and backward (`attn_fwd`, `attn_bwd`), the backward's scratch kept from step to step.
  decode    one token per sequence over a paged KV cache (`decode_fwd`).  A plan serves the 64 tokens of a block; in a
            large batch some sequence crosses a block boundary at nearly every step, so there the plan is part of
            the step (`plan` True: `plan_decode`).

Geometry is `hq` query heads on `hkv` KV heads of dimension `d`; `lens` are the sequence lengths.  Inputs are N(0,1) in
bf16, the first key of every sequence four times as large (an attention sink).
"""
import torch

import paper_2608_20427_b200 as bf1

PAGE = 64


def _case(name, kind, lens, hq, hkv, d, plan=False, block=64, route="bf1"):
    case = {"kind": kind, "lens": " ".join(str(n) for n in lens), "hq": hq, "hkv": hkv, "d": d, "plan": plan,
            "block": block, "route": route}
    if name:
        case["name"] = name
    return case


def listed():
    return [
        # the smallest prompt that is routed at all, a new length every time: launches and host work
        _case("prefill_1k_small", "prefill", [1000], 2, 1, 64, plan=True),
        # a short prompt in the geometry of the benchmark, one of many layers
        _case("prefill_4k", "prefill", [4096], 16, 8, 128),
        # four prompts of unlike, odd lengths in one launch, planned for this batch
        _case("prefill_ragged", "prefill", [3001, 8192, 12345, 16384], 16, 8, 128, plan=True),
        # the long prompt the method is for
        _case("prefill_32k", "prefill", [32768], 16, 8, 128),
        # four query heads per KV head, small heads, blocks of 128 tokens
        _case("prefill_16k_wide_blocks", "prefill", [16384], 32, 8, 64, block=128),
        # a layer that stays dense, at the length where that is still affordable
        _case("dense_8k", "dense", [8192], 16, 8, 128),
        # a training step on one short document
        _case("train_4k", "train", [4096], 16, 8, 128),
        # a training step on packed short documents: other lengths in every batch, four query heads per KV head
        _case("train_packed", "train", [130, 2048, 777, 65, 1, 3333, 512, 1911, 4097, 64, 900, 2547], 8, 2, 128, plan=True),
        # a training step at full context
        _case("train_32k", "train", [32768], 16, 8, 128),
        # one user's next token
        _case("decode_1", "decode", [32768], 16, 8, 128),
        # a few users, context lengths that are no multiple of anything
        _case("decode_8", "decode", [32768, 1000, 20011, 65, 32001, 4097, 9999, 16384], 16, 8, 128),
        # a serving batch; lengths all over the place, so that the plan is renewed with the step
        _case("decode_32", "decode", [65536 - 1777 * i - 13 * (i % 5) for i in range(32)], 16, 8, 128, plan=True),
    ]


def _log_int(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def _split(rng, total, parts):
    """`total` tokens cut into `parts` sequences of unlike lengths."""
    cuts = sorted(rng.sample(range(1, total), parts - 1)) if parts > 1 else []
    return [b - a for a, b in zip([0] + cuts, cuts + [total])]


def draw(rng):
    kind = rng.choice(["prefill", "prefill", "dense", "train", "train", "decode", "decode"])
    hkv = rng.choice([1, 2, 4, 8])
    hq, d = hkv * rng.choice([1, 2, 2, 4]), rng.choice([64, 128, 128])
    plan = rng.random() < 0.5
    if kind == "decode":
        batch = _log_int(rng, 1, 40)
        return _case(None, kind, [_log_int(rng, 20, 65536) for _ in range(batch)], hq, hkv, d, plan=plan)
    block = rng.choice([64, 64, 64, 128]) if kind != "dense" else 64
    route = rng.choice(["bf1", "bf1", "bf1", "sliding"]) if kind != "dense" else "bf1"
    most = 8192 if kind == "dense" else 32768
    if hq * d > 16 * 128 or block == 128:
        most //= 2
    total = _log_int(rng, 100, most)
    lens = _split(rng, total, rng.choice([1, 1, 1, 2, 5, 9]))
    return _case(None, kind, lens, hq, hkv, d, plan=plan and kind != "dense", block=block, route=route)


def _lens(case):
    return [int(x) for x in case["lens"].split()]


def _cfg(case):
    if case["route"] == "sliding":   # a sliding window of about the dyadic route's budget
        return bf1.RouteCfg(case["block"], 9, 0, 0)
    return bf1.RouteCfg(case["block"])


def _listed_blocks(case, j):
    if case["kind"] == "dense":
        return j + 1
    if case["route"] == "sliding":
        return min(j, 9) + 1
    sel = {j, 0} | {j - w for w in (1, 2) if w <= j}
    k = 0
    while (1 << k) <= j:
        sel.add(j - (1 << k))
        k += 1
    return len(sel)


def _pairs(case):
    """(query token, key) pairs that the route selects, per query head."""
    b, total = case["block"], 0
    for n in _lens(case):
        for j in range((n + b - 1) // b):
            rows = min(b, n - j * b)
            total += rows * b * (_listed_blocks(case, j) - 1) + rows * (rows + 1) // 2
    return total


def _packed_inputs(case, gen, dev):
    lens, hq, hkv, d = _lens(case), case["hq"], case["hkv"], case["d"]
    total = sum(lens)
    q = torch.randn((total, hq, d), generator=gen, device=dev).to(torch.bfloat16)
    k = torch.randn((total, hkv, d), generator=gen, device=dev)
    v = torch.randn((total, hkv, d), generator=gen, device=dev).to(torch.bfloat16)
    first = 0
    for n in lens:
        k[first] *= 4.0
        first += n
    return q, k.to(torch.bfloat16), v


def _empty_route(case, total, batch, max_len, dev):
    """Route arrays for the batch, cleared: a batch with many partial blocks does not fill them."""
    cfg = _cfg(case)
    capacity, degree = bf1.route_capacity(batch, total, max_len, cfg)
    route = bf1.Route.empty(capacity, degree, dev, cfg)
    for t in (route.qb_seq, route.qb_block, route.kv_count, route.kv_idx, route.pair_count, route.order):
        t.zero_()
    return route


def prepare(case, seed):
    dev = torch.device("cuda", torch.cuda.current_device())
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed)
    lens, hq, hkv, d = _lens(case), case["hq"], case["hkv"], case["d"]
    state = {"case": case}
    if case["kind"] == "decode":
        used = [(n + PAGE - 1) // PAGE for n in lens]
        pool = sum(used)
        shape = (pool, PAGE, hkv, d)
        state["k"] = torch.empty(shape, dtype=torch.bfloat16, device=dev).normal_(generator=gen)
        state["v"] = torch.empty(shape, dtype=torch.bfloat16, device=dev).normal_(generator=gen)
        state["q"] = torch.randn((len(lens), hq, d), generator=gen, device=dev).to(torch.bfloat16)
        table = torch.full((len(lens), max(used)), -1, dtype=torch.int32)
        where = torch.randperm(pool, generator=gen, device=dev).to(torch.int32).cpu()
        at = 0
        for s, n in enumerate(used):
            table[s, :n] = where[at:at + n]
            at += n
        state["table"] = table.to(dev)
        state["lens"] = torch.tensor(lens, dtype=torch.int32, device=dev)
        state["cfg"] = _cfg(case)
        state["plan"] = bf1.plan_decode(state["lens"], state["table"], state["cfg"])
        state["work"] = bf1.decode_workspace(len(lens), hq, hkv, state["plan"].max_degree, d, dev)
        state["out"] = torch.zeros((len(lens), hq, d), dtype=torch.bfloat16, device=dev)
        state["lse"] = torch.zeros((hq, len(lens)), dtype=torch.float32, device=dev)
        return state
    state["q"], state["k"], state["v"] = _packed_inputs(case, gen, dev)
    state["cu"] = bf1.cu_seqlens_tensor(lens, dev)
    state["max_len"] = max(lens)
    if case["kind"] == "dense":
        state["work"] = torch.zeros(4, dtype=torch.int32, device=dev)
        return state
    route = _empty_route(case, sum(lens), len(lens), max(lens), dev)
    state["cfg"] = _cfg(case)
    state["route"] = bf1.plan_route(state["cu"], max(lens), state["cfg"], route=route)
    if case["kind"] == "train":
        state["grad"] = torch.randn(state["q"].shape, generator=gen, device=dev).to(torch.bfloat16)
        state["work"] = bf1.bwd_workspace(route, sum(lens), hq, hkv, d, dev)
    return state


def run(state):
    case = state["case"]
    q, k, v = state["q"], state["k"], state["v"]
    if case["kind"] == "decode":
        plan = state["plan"]
        if case["plan"]:
            plan = bf1.plan_decode(state["lens"], state["table"], state["cfg"], plan=plan)
        o, lse = bf1.decode_fwd(q, k, v, state["lens"], plan, state["work"], out=state["out"], lse=state["lse"])
        return (o, lse, plan.count, plan.page) if case["plan"] else (o, lse)
    if case["kind"] == "dense":
        return bf1.dense_causal_fwd(q, k, v, state["cu"], state["max_len"], work=state["work"])
    route = state["route"]
    if case["plan"]:
        bf1.plan_route(state["cu"], state["max_len"], state["cfg"], route=route)
    o, lse = bf1.attn_fwd(q, k, v, state["cu"], state["max_len"], route)
    outputs = (o, lse)
    if case["kind"] == "train":
        outputs += bf1.attn_bwd(q, k, v, o, lse, state["grad"], state["cu"], state["max_len"], route, workspace=state["work"])
    if case["plan"]:
        outputs += (route.kv_idx, route.kv_count, route.pair_count, route.total_pairs)
    return outputs


def work(case):
    lens, hq, hkv, d = _lens(case), case["hq"], case["hkv"], case["d"]
    total = sum(lens)
    if case["kind"] == "decode":
        keys = 0
        for n in lens:
            j = (n - 1) // PAGE
            keys += (_listed_blocks(case, j) - 1) * PAGE + n - j * PAGE
        return {"bytes": 4 * keys * hkv * d + len(lens) * hq * (4 * d + 4), "flops": 4 * d * keys * hq}
    flops = 4 * d * _pairs(case) * hq
    moved = 4 * total * hq * d + 4 * total * hkv * d + 4 * total * hq   # q, o; k, v; lse
    if case["kind"] == "train":   # dS = P (dP - D) needs S and dP again: five contractions; do, dq; dk, dv
        flops += 10 * d * _pairs(case) * hq
        moved += 4 * total * hq * d + 4 * total * hkv * d
    return {"bytes": moved, "flops": flops}


def tolerance(case):
    # About four times the distance from the same path in 64 bits (bf16 results of sums whose weights are rounded to
    # bf16 as well): 1.9e-3 and, element by element, 1.6e-2 for o; 4.3e-3 and 0.36 for the gradients, whose largest
    # differences sit in the first tokens of a sequence, where the terms that cancel are many times the typical gradient.
    if case["kind"] == "train":
        return {"rel": 1.6e-2, "max": 1.4}
    return {"rel": 7e-3, "max": 6e-2}
