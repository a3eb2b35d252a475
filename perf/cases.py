"""Performance cases of the paged-KV engine: the steps that a rollout program has it do, through `tide.TideKV`.

A case is a dict of plain values.  `kind` names the calls of one pass:

  step    append + attend: one engine step of a one-layer cache (decode rows, resume rows, prompts from scratch)
  layers  step_begin + step_layer for every layer of a model
  host    step_host: the same step from pinned host buffers, results back in host memory
  group   append + attend of decode rows whose tasks were forked from a few prompts and share those pages
  prune   one turn under a sliding window: prune the oldest observation, append the new one, attend

Lengths are drawn from the case's own `lens` number (so that the work of a case is known), values from the seed.  A
pass is repeatable: what it appends is rolled back (`truncate`, host only) at the start of the next pass, as a program
does that retries a turn; decode-only batches grow for `WINDOW` steps before they are rolled back, as in a decode loop.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2608_10402_b200 import tide

WINDOW = 32          # steps that a decode-only batch grows before it is rolled back
K = 1024

TEXT = {"q_heads": 28, "kv_heads": 4, "head_dim": 128, "page": 16}      # 7B-class layer
IMAGE = {"q_heads": 32, "kv_heads": 8, "head_dim": 128, "page": 16}     # multimodal agent
SMALL = {"q_heads": 8, "kv_heads": 2, "head_dim": 64, "page": 16}       # the smallest layer of the tests
NARROW = {"q_heads": 32, "kv_heads": 8, "head_dim": 64, "page": 16}     # the other head size at a serving width
GEOMETRIES = [TEXT, TEXT, IMAGE, dict(TEXT, page=32), SMALL, NARROW,
              {"q_heads": 16, "kv_heads": 1, "head_dim": 128, "page": 16}, {"q_heads": 8, "kv_heads": 1, "head_dim": 128, "page": 32},
              {"q_heads": 12, "kv_heads": 4, "head_dim": 64, "page": 16}, {"q_heads": 6, "kv_heads": 2, "head_dim": 128, "page": 16}]


def listed():
    return [
        # The smallest step: four short tasks of a small layer, two of them resuming; launches and latency count.
        dict(SMALL, name="tiny_mixed", kind="step", tasks=4, resume=2, dist="uniform", ctx_lo=200, ctx_hi=600, new_lo=32, new_hi=64,
             sigma=1.0, lens=1),
        # One task decoding alone: the latency of the tail of a rollout, when the other tasks wait for their environments.
        dict(TEXT, name="decode_one", kind="step", tasks=1, resume=0, dist="uniform", ctx_lo=3971, ctx_hi=3971, new_lo=0, new_hi=0,
             sigma=1.0, lens=2),
        # The decode step of an ordinary continuous batch.
        dict(TEXT, name="decode_64", kind="step", tasks=64, resume=0, dist="lognormal", ctx_mid=4 * K, ctx_lo=1 * K, ctx_hi=32 * K,
             new_lo=0, new_hi=0, sigma=1.0, lens=3),
        # Multi-turn text rollouts: decode rows next to tasks that come back with their observations.
        dict(TEXT, name="mixed_text", kind="step", tasks=128, resume=32, dist="lognormal", ctx_mid=8 * K, ctx_lo=2 * K, ctx_hi=32 * K,
             new_lo=200, new_hi=2000, sigma=1.0, lens=4),
        # Multimodal agents: every task resumes with an image and some text; the largest step.
        dict(IMAGE, name="multimodal", kind="step", tasks=32, resume=32, dist="lognormal", ctx_mid=16 * K, ctx_lo=4 * K, ctx_hi=64 * K,
             new_lo=1050, new_hi=3200, sigma=1.5, lens=5),
        # Long-horizon rollouts: heavy-tailed contexts up to 128k, mostly decoding, larger pages.
        dict(TEXT, name="long_horizon", kind="step", page=32, tasks=256, resume=26, dist="pareto", ctx_lo=1 * K, ctx_hi=128 * K,
             new_lo=500, new_hi=4000, sigma=1.0, lens=6),
        # The other head size in earnest: a mixed batch of a layer with 64-wide heads.
        dict(NARROW, name="mixed_d64", kind="step", tasks=24, resume=12, dist="lognormal", ctx_mid=8 * K, ctx_lo=2 * K, ctx_hi=32 * K,
             new_lo=200, new_hi=2000, sigma=1.0, lens=7),
        # Prompts from scratch (new tasks are admitted): no prefix, ragged lengths.
        dict(TEXT, name="prefill", kind="step", tasks=16, resume=16, dist="uniform", ctx_lo=0, ctx_hi=0, new_lo=200, new_hi=4000,
             sigma=1.0, lens=8),
        # A decode step of a model with several layers: planned once, then layer by layer.
        dict(TEXT, name="layers_decode", kind="layers", layers=8, tasks=48, resume=0, dist="lognormal", ctx_mid=2 * K, ctx_lo=256,
             ctx_hi=16 * K, new_lo=0, new_hi=0, sigma=1.0, lens=9),
        # A mixed step whose inputs and results live in host memory.
        dict(TEXT, name="host_mixed", kind="host", tasks=32, resume=8, dist="lognormal", ctx_mid=8 * K, ctx_lo=2 * K, ctx_hi=32 * K,
             new_lo=200, new_hi=2000, sigma=1.0, lens=10),
        # Decode step of eight groups of rollouts, each group forked from one long prompt.
        dict(TEXT, name="group_decode", kind="group", groups=8, members=8, shared=6 * K + 5, own_lo=900, own_hi=3100, sigma=1.0, lens=11),
        # One turn of agents that keep only their latest observations.
        dict(TEXT, name="prune_turn", kind="prune", tasks=8, resume=8, dist="lognormal", ctx_mid=8 * K, ctx_lo=4 * K, ctx_hi=16 * K,
             new_lo=200, new_hi=1200, keep_lo=100, keep_hi=700, sigma=1.0, lens=12),
    ]


def _spread(rng, lo, hi):
    """A whole number between lo and hi, spread over its logarithm."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw(rng):
    kind = rng.choice(["decode", "decode", "mixed", "mixed", "resume", "prefill", "layers", "host", "group", "prune"])
    case = dict(rng.choice(GEOMETRIES), kind="step", dist="lognormal", sigma=rng.choice([1.0, 1.5]), lens=rng.randrange(1, 1 << 20))
    mid = _spread(rng, 256, 24 * K)
    ctx = dict(ctx_mid=mid, ctx_lo=max(1, mid // 4), ctx_hi=min(64 * K, mid * 4))
    new_hi = _spread(rng, 12, 4000)
    new = dict(new_lo=max(2, new_hi // rng.choice([2, 5, 10])), new_hi=new_hi)
    if kind == "decode":
        return dict(case, **ctx, tasks=_spread(rng, 1, 256), resume=0, new_lo=0, new_hi=0)
    if kind == "mixed":
        tasks = _spread(rng, 2, 160)
        return dict(case, **ctx, **new, tasks=tasks, resume=rng.randint(1, max(1, tasks // 2)))
    if kind == "resume":
        tasks = _spread(rng, 1, 48)
        return dict(case, **ctx, **new, tasks=tasks, resume=tasks)
    if kind == "prefill":
        tasks = _spread(rng, 1, 48)
        return dict(case, **new, dist="uniform", ctx_lo=0, ctx_hi=0, tasks=tasks, resume=tasks)
    if kind == "layers":
        tasks = _spread(rng, 1, 64)
        resume = rng.choice([0, 0, max(1, tasks // 8)])
        return dict(case, **ctx, kind="layers", layers=rng.randint(2, 12), tasks=tasks, resume=resume,
                    new_lo=new["new_lo"] if resume else 0, new_hi=new["new_hi"] if resume else 0)
    if kind == "host":
        tasks = _spread(rng, 1, 64)
        return dict(case, **ctx, **new, kind="host", tasks=tasks, resume=rng.randint(0, max(1, tasks // 4)))
    if kind == "group":
        own = _spread(rng, 64, 3 * K)
        return {**{k: case[k] for k in ("q_heads", "kv_heads", "head_dim", "page", "sigma", "lens")}, "kind": "group",
                "groups": rng.randint(1, 12), "members": rng.randint(2, 12), "shared": _spread(rng, 300, 12 * K),
                "own_lo": max(1, own // 3), "own_hi": own}
    tasks = _spread(rng, 1, 16)
    keep = _spread(rng, 16, 700)
    mid = max(mid, 4 * (keep + new_hi))
    return dict(case, **new, kind="prune", ctx_mid=mid, ctx_lo=max(mid // 2, keep + new_hi + 1), ctx_hi=2 * mid, tasks=tasks, resume=tasks,
                keep_lo=max(1, keep // 4), keep_hi=keep)


def _cost(case):
    w = work(case)
    return max(w["bytes"] / 6.5e12, w["flops"] / 1.4e15)


def draw(rng):
    top = max(_cost(c) for c in listed() if c["kind"] == "step")
    while True:
        case = _draw(rng)
        w = work(case)
        # a step of every kind stays below the largest listed one; several layers and two copies of host data included
        if _cost(case) <= top and w["bytes"] <= 12e9:
            return case


def _lengths(case):
    """Per task: context before the pass, new tokens of the pass (1 for a decode row), kept prefix (prune)."""
    rng = np.random.default_rng(case["lens"])
    if case["kind"] == "group":
        n = case["groups"] * case["members"]
        return case["shared"] + rng.integers(case["own_lo"], case["own_hi"] + 1, n), np.ones(n, np.int64), np.zeros(n, np.int64)
    n, lo, hi = case["tasks"], case["ctx_lo"], case["ctx_hi"]
    if case["dist"] == "uniform":
        ctx = rng.integers(lo, hi + 1, n)
    elif case["dist"] == "lognormal":
        ctx = np.clip(np.rint(case["ctx_mid"] * np.exp(rng.standard_normal(n))), lo, hi).astype(np.int64)
    else:
        ctx = np.clip(np.rint(lo * (1.0 - rng.random(n)) ** (-1.0 / 1.5)), lo, hi).astype(np.int64)
    if case["dist"] != "uniform" and n > 4:
        ctx[0] = hi                                           # the longest context is always there
    new = np.ones(n, np.int64)
    if case["resume"]:
        new[n - case["resume"]:] = rng.integers(case["new_lo"], case["new_hi"] + 1, case["resume"])
    keep = np.zeros(n, np.int64)
    if case["kind"] == "prune":
        keep = rng.integers(case["keep_lo"], case["keep_hi"] + 1, n)
    order = rng.permutation(n)
    return ctx[order], new[order], keep[order]


def work(case):
    ctx, new, keep = _lengths(case)
    hq, hkv, d = case["q_heads"], case["kv_heads"], case["head_dim"]
    token = hkv * d * 4                                       # K and V of one token
    layers = case.get("layers", 1)
    n = new.astype(float)
    prefix = ctx.astype(float)
    if case["kind"] == "prune":
        prefix = prefix - n                                   # the turn drops as much as it appends
    pairs = float((n * prefix + n * (n + 1) / 2).sum())
    read = float((prefix + n).sum()) * token
    if case["kind"] == "group":
        read -= (case["members"] - 1) * case["groups"] * float(case["shared"]) * token     # a prompt is read once per group
    total = float(n.sum())
    moved = total * token * 2 + total * hq * d * 4 + total * hq * 4      # new K/V in and into the pages, q, out, lse
    if case["kind"] == "prune":
        moved += 2 * float((ctx - keep - new).sum()) * token             # the tail moves down
    return {"bytes": layers * (read + moved), "flops": layers * 4.0 * d * hq * pairs}


def tolerance(case):
    # bf16 results and bf16 weights of the second product.  Measured against 64-bit sums: relative error 2.1e-3 to 2.4e-3,
    # largest difference 0.006 to 0.025 of the root mean square; about four times that.
    return {"rel": 1e-2, "max": 0.1}


class _State:
    pass


def _normal(gen, shape, sigma, device="cuda"):
    x = torch.randn(shape, device=device, generator=gen)
    return (x * sigma if sigma != 1.0 else x).to(torch.bfloat16)


def prepare(case, seed):
    ctx, new, keep = _lengths(case)
    hq, hkv, d, page = case["q_heads"], case["kv_heads"], case["head_dim"], case["page"]
    n, total, layers = len(ctx), int(new.sum()), case.get("layers", 1)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    most = ctx + new * (WINDOW if (new == 1).all() else 1)
    pages = int(((most + page - 1) // page).sum() * 1.25) + n + 64
    group = case["kind"] == "group"
    members = case["members"] if group else 1
    parents = case["groups"] if group else 0
    s = _State()
    s.kind, s.layers, s.scale = case["kind"], layers, 1.0 / math.sqrt(d)
    s.kv = kv = tide.TideKV(hq, hkv, d, page, pages, n + parents, int((most.max() + page - 1) // page) + 2, n, max(total, 4096),
                            free_order=np.random.default_rng(seed).permutation(pages), num_layers=layers)

    def fill(tasks, counts):
        """Resident context: values appended in calls of bounded size."""
        per_token = 2 * hkv * d
        at = 0
        while at < len(tasks):
            to, size = at, 0
            while to < len(tasks) and (to == at or size + int(counts[to]) * per_token <= 1 << 28):
                size += int(counts[to]) * per_token
                to += 1
            ids, indptr = tasks[at:to], np.concatenate([[0], np.cumsum(counts[at:to])])
            rows = int(indptr[-1])
            kv.extend(ids, indptr)
            for layer in range(layers):
                kv.write(layer, ids, indptr, _normal(gen, (rows, hkv, d), 1.0), _normal(gen, (rows, hkv, d), 1.0))
            at = to

    tasks = list(range(n))
    if group:
        roots = list(range(n, n + parents))
        for t in roots:
            kv.alloc(t)
        fill(roots, np.full(parents, case["shared"], np.int64))
        for t in tasks:
            kv.fork(roots[t // members], t)
        fill(tasks, ctx - case["shared"])
        kv.release_many(roots)
    else:
        for t in tasks:
            kv.alloc(t)
        fill(tasks, ctx)

    shape = (layers, total) if s.kind == "layers" else (total,)
    s.new_k = _normal(gen, (*shape, hkv, d), case["sigma"])
    s.new_v = _normal(gen, (*shape, hkv, d), case["sigma"])
    s.q = _normal(gen, (*shape, hq, d), 1.0)
    s.out = torch.empty_like(s.q)
    s.lse = torch.empty((*shape, hq), dtype=torch.float32, device="cuda")
    if s.kind == "host":
        s.new_k, s.new_v, s.q, s.out, s.lse = (x.cpu().pin_memory() for x in (s.new_k, s.new_v, s.q, s.out, s.lse))
    s.ids = np.asarray(tasks, np.int32)
    s.indptr = np.concatenate([[0], np.cumsum(new)]).astype(np.int32)
    s.base, s.new, s.keep = ctx.tolist(), new, keep.tolist()
    s.rows = tide.rows_array([(t, int(new[t]), 0) for t in tasks])
    s.ctx_len = np.frombuffer(s.rows, np.int32).reshape(n, 3)[:, 2]      # the rows' ctx_len column, updated in place
    s.window = WINDOW if (new == 1).all() else 1
    s.steps = 0
    s.length = ctx.astype(np.int32)
    return s


def run(s):
    kv = s.kv
    if s.kind == "prune":
        for t, keep in enumerate(s.keep):
            kv.prune(t, keep, keep + int(s.new[t]))
        s.ctx_len[:] = s.base
        kv.append(s.ids, s.indptr, s.new_k, s.new_v)
        kv.attend(s.rows, s.q, s.scale, s.out, s.lse)
        return s.out, s.lse
    if s.steps == s.window:                                   # back to the start of the turn, last page first
        for t in range(len(s.base) - 1, -1, -1):
            kv.truncate(t, s.base[t])
        s.steps = 0
        s.length[:] = s.base
    s.steps += 1
    s.length += s.new
    s.ctx_len[:] = s.length
    if s.kind == "layers":
        kv.step_begin(s.rows)
        for layer in range(s.layers):
            kv.step_layer(layer, s.new_k[layer], s.new_v[layer], s.q[layer], s.scale, s.out[layer], s.lse[layer])
    elif s.kind == "host":
        kv.step_host(s.rows, s.new_k, s.new_v, s.q, s.scale, s.out, s.lse)
    else:
        kv.append(s.ids, s.indptr, s.new_k, s.new_v)
        kv.attend(s.rows, s.q, s.scale, s.out, s.lse)
    return s.out, s.lse
