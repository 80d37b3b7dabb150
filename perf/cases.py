"""The work that a program has libfvar do, as cases that can be timed and compared.

Six kinds, all through the binding's public calls (paper_2512_16483_b200.binding):
  dense       scale steps without approximation, both branches of every CFG pair, KV rows appended after each
  late        late scale steps under the paper's approximation (null-prompt branch alone, random projection to r
              rows, representative-token restoration) over the cache that earlier scales left
  late_host   the same with the tokens and the results in pinned host memory (the pipelined host entry point)
  generate    the transformer part of a generation: conditioning, projections drawn from a seed, every scale from the
              first token on dense with both branches, the last one approximated
  transition  between the steps: guidance on the two branches, nearest codeword, Up-accumulate, area Down
  rows        the method's row kernels on a caller's own buffers: score, selection, LayerNorm + modulation, fill

Shapes are the stacks this repository measures (VAR-d16, VAR-d30, Infinity-2B); weights, tokens and caches are seeded
draws of the distributions its tests use.  Ranks are equal in all block groups of a step, or rise with depth: a group
that keeps fewer rows than the group before it ranks projected rows of nearly equal norms, and there two correct
programs take different rows after the first rounding difference.
"""
from __future__ import annotations

import math

import torch

from paper_2512_16483_b200 import binding as fv
from paper_2512_16483_b200 import schedule

VAR_SIDES = (1, 2, 3, 4, 5, 6, 8, 10, 13, 16)
INFINITY_SIDES = (1, 2, 4, 6, 8, 12, 16, 20, 24, 32, 40, 48, 64)

# blocks, blocks per group, width, heads, head width, FFN width, sides of the scales, context tokens (0: none)
STACKS = {
    "var_d16": (16, 1, 1024, 16, 64, 4096, VAR_SIDES, 0),
    "var_d30": (30, 1, 1920, 30, 64, 7680, VAR_SIDES, 0),
    "infinity_2b": (32, 4, 2048, 16, 128, 8192, INFINITY_SIDES, 256),
}
FIRST_LATE = {"var_d16": 7, "var_d30": 8, "infinity_2b": 10}
GUIDANCE = 3.0


def listed():
    return [
        # the first scales of a generation: 1 to 25 tokens a branch, where launches and latency are everything
        {"name": "var_d16_start_b2", "kind": "dense", "stack": "var_d16", "batch": 2, "first": 0, "last": 4},
        # the last scales of a batch of eight images, nothing approximated
        {"name": "var_d16_dense3_b16", "kind": "dense", "stack": "var_d16", "batch": 16, "first": 7, "last": 9},
        # one late scale of that batch at half of the rows: 85 of 169 rows, an odd size
        {"name": "var_d16_13x13_half_b16", "kind": "late", "stack": "var_d16", "batch": 16, "first": 8, "last": 8, "keep": 0.5},
        # the same method on the wider stack (1920 columns, 30 heads) and the largest batch it is run at
        {"name": "var_d30_16x16_half_b32", "kind": "late", "stack": "var_d30", "batch": 32, "first": 9, "last": 9, "keep": 0.5},
        # the one approximated step of the paper's schedule for the Infinity stack, at its tabulated ranks
        {"name": "infinity_40_table_b2", "kind": "late", "stack": "infinity_2b", "batch": 2, "first": 10, "last": 10, "keep": "table"},
        # all three late scales at their mean tabulated rank, fed from host memory as a server does
        {"name": "infinity_late3_host_b2", "kind": "late_host", "stack": "infinity_2b", "batch": 2, "first": 10, "last": 12, "keep": "mean"},
        # the last scale at the smallest rank of the table: weights streamed for 16 rows
        {"name": "infinity_64_r16_b2", "kind": "late", "stack": "infinity_2b", "batch": 2, "first": 12, "last": 12, "keep": 16},
        # four images at a quarter of the rows
        {"name": "infinity_64_r1024_b8", "kind": "late", "stack": "infinity_2b", "batch": 8, "first": 12, "last": 12, "keep": 1024},
        # the late scales of one image without approximation: the largest step there is
        {"name": "infinity_dense3_b2", "kind": "dense", "stack": "infinity_2b", "batch": 2, "first": 10, "last": 12},
        # one image from its prompt to the end of the paper's schedule (scales 48 and 64 are skipped there)
        {"name": "infinity_generate_b2", "kind": "generate", "stack": "infinity_2b", "batch": 2, "last": 10, "keep": "mean"},
        # everything between the steps of that generation, one image at a time
        {"name": "infinity_transition_b1", "kind": "transition", "stack": "infinity_2b", "batch": 1, "codes": 8192, "last": 10},
        # selection and restoration around somebody else's blocks, at the size of one VAR scale
        {"name": "rows_16x16_b16", "kind": "rows", "batch": 16, "h0": 13, "w0": 13, "h1": 16, "w1": 16, "width": 1024, "keep": 0.5},
    ]


def _log(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _draw_once(rng):
    kind = rng.choice(("dense", "dense", "late", "late", "late", "late_host", "generate", "transition", "rows"))
    if kind == "rows":
        h0, w0 = _log(rng, 4, 48), _log(rng, 4, 48)
        return {"kind": kind, "batch": _log(rng, 1, 16), "h0": h0, "w0": w0, "h1": _log(rng, h0, 64), "w1": _log(rng, w0, 64),
                "width": 64 * rng.randint(8, 32), "keep": round(rng.uniform(0.02, 0.6), 3)}
    stack = rng.choice(("var_d16", "var_d30", "infinity_2b", "infinity_2b"))
    last = len(STACKS[stack][6]) - 1
    inf = stack == "infinity_2b"
    if kind == "dense":
        a = rng.randint(0, last)
        return {"kind": kind, "stack": stack, "batch": _log(rng, 1, 4 if inf else 32), "first": a, "last": min(last, a + rng.randint(0, 3))}
    if kind == "transition":
        return {"kind": kind, "stack": stack, "batch": _log(rng, 1, 8), "codes": _log(rng, 1024, 16384), "last": rng.randint(FIRST_LATE[stack], last)}
    a = rng.randint(FIRST_LATE[stack], last)
    side = STACKS[stack][6][a]
    if inf:
        keep = rng.choice(("table", "mean", 0)) if kind != "generate" else rng.choice(("mean", 0))
        keep = keep or _log(rng, 8, side * side // 4)
    else:
        keep = round(rng.uniform(0.1, 0.5), 3)
    if kind == "generate":
        return {"kind": kind, "stack": stack, "batch": 2 * _log(rng, 1, 2 if inf else 8), "last": a, "keep": keep}
    b = last if keep == "mean" else a        # the three late scales in sequence at the mean ranks, else one of them
    return {"kind": kind, "stack": stack, "batch": 2 * _log(rng, 1, 4 if inf else 16), "first": 10 if keep == "mean" else a, "last": b, "keep": keep}


def draw(rng):
    top = [work(c) for c in listed()]
    flops, bytes_ = max(w["flops"] for w in top), max(w["bytes"] for w in top)
    while True:
        case = _draw_once(rng)
        w = work(case)
        if w["flops"] <= flops and w["bytes"] <= bytes_:
            return case


# ------------------------------------------------------------------------------------------------ sizes of a case

def _tokens(stack):
    return [s * s for s in STACKS[stack][6]]


def _ranks(stack, k, keep):
    """Rank of every block group at scale k."""
    blocks, per_group, width = STACKS[stack][:3]
    groups, M = blocks // per_group, _tokens(stack)[k]
    if keep in ("table", "mean"):
        table = schedule.infinity_group_ranks(STACKS[stack][6][k], width, groups)
        if keep == "mean":
            return [int(round(sum(table) / groups))] * groups
        return [max(table[: g + 1]) for g in range(groups)]          # never below the group before
    return [keep if keep >= 1 else schedule.rank_from_keep_ratio(M, keep)] * groups


def _plan(case):
    """[(scale, null-prompt branch alone?, rank per group or None)] of the steps of a pass."""
    stack, late = case["stack"], FIRST_LATE[case["stack"]]
    if case["kind"] == "dense":
        return [(k, False, None) for k in range(case["first"], case["last"] + 1)]
    first = 0 if case["kind"] == "generate" else case["first"]
    return [(k, True, _ranks(stack, k, case["keep"])) if k >= late and (case["kind"] != "generate" or k == case["last"])
            else (k, False, None) for k in range(first, case["last"] + 1)]


def work(case):
    if case["kind"] == "rows":
        B, M, C = case["batch"], case["h1"] * case["w1"], case["width"]
        r = schedule.rank_from_keep_ratio(M, case["keep"])
        # rows scored and the cached map read, every row written once (r of them from the caller's rows), the r rows
        # normalised to bf16, lists written
        return {"bytes": B * (4.0 * M * C + 4.0 * case["h0"] * case["w0"] * C + 4.0 * (M - r) * C + 6.0 * r * C + 8.0 * C + 8.0 * M + 4.0 * r),
                "flops": B * (2.0 * M * C + 8.0 * r * C + 7.0 * (M - r) * C)}
    blocks, per_group, C, H, D, F, sides, ctx = STACKS[case["stack"]]
    groups, Ms, B = blocks // per_group, _tokens(case["stack"]), case["batch"]
    if case["kind"] == "transition":
        V, flops, bytes_ = case["codes"], 0.0, 2.0 * case["codes"] * C
        for k in range(case["last"] + 1):
            nxt = Ms[k + 1] if k < case["last"] else 0
            flops += B * (2.0 * Ms[k] * V * C + 9.0 * Ms[-1] * C)
            # both branches and the codebook read, the map read (after the first) and written, both branches' tokens written
            bytes_ += B * (4.0 * Ms[k] * C + (4.0 if k else 0.0) * Ms[-1] * C + 4.0 * Ms[-1] * C + 4.0 * Ms[k] + 4.0 * nxt * C)
        return {"bytes": bytes_, "flops": flops}
    P = 4 * C * C + 2 * C * F + (2 * C * C if ctx else 0)          # weights of a block that a row meets
    plan = _plan(case)
    L = [0 if case["kind"] == "generate" else sum(Ms[: plan[0][0]])] * groups
    flops = bytes_ = 0.0
    if case["kind"] == "generate":
        flops += blocks * (12.0 * B * C * C + (4.0 * B * ctx * C * C))
        bytes_ += blocks * (12.0 * C * C + 24.0 * B * C + (4.0 * C * C + 4.0 * B * ctx * C if ctx else 0.0)) + 2.0 * B * ctx * C
    for k, null_only, ranks in plan:
        E, M = (B // 2 if null_only else B), Ms[k]
        for g in range(groups):
            r = ranks[g] if ranks else M
            late = r < M
            flops += E * per_group * (2.0 * r * P + 4.0 * r * (L[g] + r) * C + 4.0 * r * ctx * C) + (2.0 * E * M * r * C if late else 0.0)
            # weights once, the cache and the context, the group's input and output, for a late group Q and the cached output
            bytes_ += 2.0 * per_group * P + E * (4.0 * per_group * (L[g] + r + ctx) * C + 4.0 * M * C)
            bytes_ += (2.0 * M * r + 2.0 * E * (M + Ms[max(k - 1, 0)]) * C) if late else 0.0
            L[g] += r
    return {"bytes": bytes_, "flops": flops}


def tolerance(case):
    if case["kind"] == "rows":
        return {"rel": 1e-3, "max": 1e-2, "differ": 0.0}      # fp32 sums; the modulated rows are bf16 (2^-9 each)
    if case["kind"] == "transition":
        return {"rel": 1e-3, "max": 1e-2, "differ": 0.0}      # fp32 map, bf16 tokens; codewords well apart
    # a stack of bf16 blocks on an fp32 residual stream, the result rounded to bf16: two summation orders of the same
    # precision are 1e-3 to 5e-3 apart over a whole stack
    return {"rel": 1.2e-2, "max": 1e-1}


# ------------------------------------------------------------------------------------------------ inputs

def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _randn(g, *shape, std=1.0, dtype=torch.bfloat16):
    t = torch.randn(shape, generator=g, device="cuda", dtype=dtype)
    return t if std == 1.0 else t.mul_(std)


def _spread(g, B, M, C, dtype=torch.bfloat16):
    """Rows whose norms are well separated (log-normal), as the rows of a real feature map are."""
    x = torch.randn((B, M, C), generator=g, device="cuda")
    return x.mul_(torch.exp(0.5 * torch.randn((B, M, 1), generator=g, device="cuda"))).to(dtype)


def _weights(g, stack):
    """Every parameter N(0, 0.02^2), cut out of one draw a block."""
    blocks, _, C, _, _, F, _, ctx = STACKS[stack]
    dims = {"w_qkv": (3 * C, C), "b_qkv": (3 * C,), "w_o": (C, C), "b_o": (C,), "w_fc1": (F, C), "b_fc1": (F,), "w_fc2": (C, F),
            "b_fc2": (C,), "w_ada": (6 * C, C), "b_ada": (6 * C,)}
    if ctx:
        dims.update({"w_cq": (C, C), "w_ckv": (2 * C, C), "w_co": (C, C)})
    out = []
    for _ in range(blocks):
        flat, at, blk = _randn(g, sum(math.prod(d) for d in dims.values()), std=0.02), 0, {}
        for name, d in dims.items():
            blk[name] = flat[at : at + math.prod(d)].view(d)
            at += math.prod(d)
        if ctx:
            blk["ln_c_gamma"] = 1.0 + _randn(g, C, std=0.1)
        out.append(blk)
    return out


def _context(stack, batch, weights):
    _, per_group, C, H, D, F, sides, ctx = STACKS[stack]
    return fv.Fvar(weights, blocks_per_group=per_group, n_heads=H, head_dim=D, ffn_dim=F, scale_hw=[(s, s) for s in sides],
                   max_batch=batch, ctx_len=ctx, ctx_width=C if ctx else 0)


def prepare(case, seed):
    g, kind = _generator(seed), case["kind"]
    if kind == "rows":
        B, C = case["batch"], case["width"]
        M = case["h1"] * case["w1"]
        r = schedule.rank_from_keep_ratio(M, case["keep"])
        return {"kind": kind, "r": r, "hw0": (case["h0"], case["w0"]), "hw1": (case["h1"], case["w1"]), "x": _spread(g, B, M, C, torch.float32),
                "prev": _randn(g, B, case["h0"] * case["w0"], C, dtype=torch.float32), "kept": _randn(g, B, r, C, dtype=torch.float32),
                "out": _randn(g, B, M, C, dtype=torch.float32), "shift": _randn(g, B, C, std=0.5, dtype=torch.float32),
                "scale": _randn(g, B, C, std=0.5, dtype=torch.float32)}
    stack, B = case["stack"], case["batch"]
    blocks, per_group, C, _, _, _, _, ctx = STACKS[stack]
    groups, Ms = blocks // per_group, _tokens(stack)
    ctx_obj = _context(stack, B, _weights(g, stack))
    if kind == "transition":
        Z = _randn(g, case["codes"], C)
        ctx_obj.set_codebook(Z)
        pairs = []
        for k in range(case["last"] + 1):
            pick = torch.randint(case["codes"], (B, Ms[k]), generator=g, device="cuda")
            # a codeword plus noise in each branch: tokens near the codebook, as a trained stack puts them out
            near = Z[pick].float().unsqueeze(1) + 0.1 * torch.randn((B, 2, Ms[k], C), generator=g, device="cuda")
            pairs.append(near.to(torch.bfloat16).view(2 * B, Ms[k], C))
        return {"kind": kind, "ctx": ctx_obj, "pairs": pairs, "Ms": Ms, "last": case["last"]}
    plan = _plan(case)
    state = {"kind": kind, "ctx": ctx_obj, "plan": plan, "seed": seed, "groups": groups,
             "cond": _randn(g, B, C), "context": _randn(g, B, ctx, C) if ctx else None}
    ctx_obj.set_cond(state["cond"], state["context"])
    k0 = plan[0][0]
    state["loaded"] = k0 > 0
    if k0 > 0:                                   # what the earlier scales left: their K / V rows and group outputs
        L = sum(Ms[:k0])
        ctx_obj.load_kv(_randn(g, blocks, B, L, C), _randn(g, blocks, B, L, C))
        ctx_obj.load_group_cache(k0 - 1, _randn(g, groups, B, Ms[k0 - 1], C, dtype=torch.float32))
    single = len(plan) == 1
    state["tokens"], state["outs"] = {}, {}
    for k, null_only, ranks in plan:
        state["tokens"][k] = _spread(g, B, Ms[k], C) if ranks and single else _randn(g, B, Ms[k], C)
        state["outs"][k] = torch.empty((B // 2 if null_only else B, Ms[k], C), dtype=torch.bfloat16, device="cuda")
        if ranks and kind != "generate":
            for i, r in enumerate(ranks):
                if r < Ms[k]:
                    ctx_obj.set_projection(k, i, _randn(g, r, Ms[k], std=1.0 / math.sqrt(r)))
    if kind == "late_host":
        state["tokens"] = {k: t.cpu().pin_memory() for k, t in state["tokens"].items()}
        state["outs"] = {k: t.cpu().pin_memory() for k, t in state["outs"].items()}
    return state


# ------------------------------------------------------------------------------------------------ passes

def _run_rows(s):
    scores = fv.fvar_row_scores(s["x"])
    idx, inv = fv.fvar_select_topr(scores, s["r"])
    y = fv.fvar_ln_modulate(s["kept"], s["shift"], s["scale"], 1e-6)
    fv.fvar_rtr_fill(s["prev"], s["hw0"], s["hw1"], inv, s["out"])
    return {"scores": scores, "idx": idx, "inv": inv, "y": y, "out": s["out"]}


def _run_transition(s):
    ctx, last, out = s["ctx"], s["last"], {}
    for k in range(last + 1):
        fo = fv.fvar_cfg_combine(s["pairs"][k], GUIDANCE)
        out["codes%d" % k], nxt = ctx.scale_transition(fo, k, s["Ms"][k + 1] if k < last else None, pairs=True)
        if nxt is not None:
            out["tokens%d" % (k + 1)] = nxt
    out["feature"] = ctx.get_feature(s["pairs"][0].shape[0] // 2, s["Ms"][-1], s["pairs"][0].shape[2])
    return out


def run(state):
    kind = state["kind"]
    if kind == "rows":
        return _run_rows(state)
    if kind == "transition":
        return _run_transition(state)
    ctx = state["ctx"]
    if kind == "generate":                       # a new prompt: conditioning, and the paper draws Q anew for each generation
        ctx.set_cond(state["cond"], state["context"])
        for k, _, ranks in state["plan"]:
            for i, r in enumerate(ranks or ()):
                ctx.generate_projection(k, i, r, state["seed"])
    elif state["loaded"]:
        ctx.restore_loaded()
    else:
        ctx.reset()
    step = ctx.scale_step_host_async if kind == "late_host" else None
    for k, null_only, ranks in state["plan"]:
        how = {"mode": fv.LOWRANK_RTR if ranks else fv.DENSE, "cfg_mode": fv.CFG_NULL_ONLY if null_only else fv.CFG_PAIR, "rank_per_group": ranks}
        if step:
            step(state["tokens"][k], k, state["outs"][k], **how)
        else:
            ctx.scale_step(state["tokens"][k], k, out=state["outs"][k], **how)
        ctx.kv_append(k)
    if step:
        ctx.host_sync()
    return {"out%d" % k: t for k, t in state["outs"].items()}
