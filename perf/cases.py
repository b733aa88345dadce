"""What this library is used for, as cases that can be timed and compared.

Three kinds of pass, each through the calls that a serving program makes:

- ``prompt``: a prompt is ingested in sub-sequences; every one is written to the KVCache and attends to all rows before it
  and to itself (``chunk_prefill_append_attn``, one call per sub-sequence).
- ``step``: one decoding or verification step of several branches that share a prompt's KVCache, for one layer
  (``branch_append_attn``), for the layers of a pipeline stage (``branch_append_attn_layers``), or with a token tree
  (``kv_append``, ``branch_attn_tree``, ``kv_compact``).
- ``ingest``: every branch ingests its own instruction on top of the shared prompt (``kv_append``,
  ``branch_prefill_attn``).
"""
import math
import random

import numpy as np
import torch

import paper_2504_08242_b200 as J

BF16 = torch.bfloat16


def listed():
    return [
        # The smallest prompt of the benchmark's configurations: head_dim 64, four short calls.
        prompt("tiny_prompt_d64", 1, 4, 4, 64, 256, 64, 256),
        # A question of ordinary length (260 tokens is the paper's average prompt) in four sub-sequences of 65, with the
        # log-sum-exps returned as a caller needs them who merges the result with another segment.
        prompt("short_prompt", 1, 32, 32, 128, 260, 65, 512, lse=True),
        # The benchmark's 7B-shaped prompt: 2048 tokens in sub-sequences of 256.
        prompt("prompt_7b", 1, 32, 32, 128, 2048, 256, 4096),
        # The benchmark's long GQA prompts, four at a time, at its default sub-sequence length and at its shortest one.
        prompt("long_prompt_c512", 4, 32, 8, 128, 8192, 512, 8192),
        prompt("long_prompt_c128", 4, 32, 8, 128, 8192, 128, 8192),
        # One head_dim-64 GQA prompt of a few thousand tokens, the length no multiple of the sub-sequence.
        prompt("prompt_d64", 1, 32, 8, 64, 3000, 448, 4096),
        # One layer of the benchmark's outline decoding: eight branches, one token each.  The smallest step.
        step("decode_layer", 1, 8, 32, 32, 128, 1024, 1, 257, 1, 320),
        # The same step for the 32 layers of a 7B-shaped model, in one call.
        step("decode_32_layers", 32, 8, 32, 32, 128, 1024, 1, 257, 1, 320),
        # The benchmark's speculative verification (16 branches, five drafts, GQA) in the eight layers of a pipeline stage.
        step("verify_8_layers", 8, 16, 32, 8, 128, 2048, 69, 517, 5, 520),
        # One layer of token-tree verification: write the block, verify the tree, compact the accepted path.
        step("verify_tree", 1, 6, 32, 8, 128, 1000, 8, 400, 8, 512, tree=True, lse=True),
        # Verification with head_dim 64.
        step("verify_d64", 1, 16, 32, 8, 64, 1500, 69, 400, 5, 512),
        # Every branch of an outline ingests its own instruction behind the shared prompt.
        ingest("branch_ingest", 8, 32, 8, 128, 1024, 0, 150, 512),
    ]


def prompt(name, batch, q_heads, kv_heads, head_dim, length, chunk, capacity, lse=False):
    return named(name, kind="prompt", batch=batch, q_heads=q_heads, kv_heads=kv_heads, head_dim=head_dim, length=length,
                 chunk=chunk, capacity=capacity, lse=lse)


def step(name, layers, branches, q_heads, kv_heads, head_dim, prefix, shortest, longest, drafts, capacity, tree=False,
         lse=False):
    """``shortest`` and ``longest``: the branches' lengths with this step's rows."""
    return named(name, kind="step", layers=layers, branches=branches, q_heads=q_heads, kv_heads=kv_heads,
                 head_dim=head_dim, prefix=prefix, shortest=shortest, longest=longest, drafts=drafts, capacity=capacity,
                 tree=tree, lse=lse)


def ingest(name, branches, q_heads, kv_heads, head_dim, prefix, pos, length, capacity, lse=False):
    return named(name, kind="ingest", branches=branches, q_heads=q_heads, kv_heads=kv_heads, head_dim=head_dim,
                 prefix=prefix, pos=pos, length=length, capacity=capacity, lse=lse)


def named(name, **case):
    return dict({"name": name} if name else {}, **case)


def draw(rng):
    def spread(lo, hi):  # over the logarithm
        return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))

    def heads(choices):
        q, kv = rng.choice(choices)
        return q, kv

    shapes = [(32, 32), (32, 8), (16, 16), (16, 4), (8, 2), (4, 4), (64, 8)]
    lse = rng.random() < 0.25
    kind = rng.choice(["prompt", "prompt", "prompt", "step", "step", "step", "step", "ingest"])
    if kind == "prompt":
        head_dim = rng.choice([64, 128, 128])
        q_heads, kv_heads = heads(shapes)
        batch = rng.choice([1, 1, 2, 3, 4])
        length = spread(64, 8192)
        while batch * q_heads * length * length > 4 * 32 * 8192 * 8192 // (2 if head_dim == 64 else 1):
            length -= length // 3
        chunk = min(length, spread(max(32, -(-length // 64)), 1024))
        return prompt(None, batch, q_heads, kv_heads, head_dim, length, chunk, length + rng.randrange(0, 300), lse)
    if kind == "step":
        what = rng.choice(["decode", "decode", "verify", "verify", "tree"])
        head_dim = rng.choice([64, 128, 128, 128])
        q_heads, kv_heads = heads(shapes)
        branches = rng.randint(1, 16)
        drafts = 1 if what == "decode" else rng.randint(2, 8) if what == "verify" else rng.randint(4, 16)
        prefix = spread(64, 4096)
        longest = drafts + spread(16, 512)
        shortest = drafts + rng.randrange(0, (longest - drafts) // 2 + 1)
        capacity = longest + rng.randrange(0, 100)
        layers = 1 if what == "tree" else rng.choice([1, 4, 8, 32])
        while layers > 1 and layers * kv_heads * head_dim * (prefix + branches * capacity) > 600_000_000:
            layers //= 2
        return step(None, layers, branches, q_heads, kv_heads, head_dim, prefix, shortest, longest, drafts, capacity,
                    what == "tree", lse)
    q_heads, kv_heads = heads(shapes)
    pos, length = rng.choice([0, 0, rng.randrange(1, 200)]), spread(16, 512)
    return ingest(None, rng.randint(1, 16), q_heads, kv_heads, 128, spread(64, 4096), pos, length,
                  pos + length + rng.randrange(0, 200), lse)


def chunks(case):
    return [(p, min(case["chunk"], case["length"] - p)) for p in range(0, case["length"], case["chunk"])]


def lengths(case):
    """The branches' lengths, evenly over their range (which branch has which one depends on the seed)."""
    n, lo, hi = case["branches"], case["shortest"], case["longest"]
    return [hi] if n == 1 else [lo + (hi - lo) * i // (n - 1) for i in range(n)]


class Source:
    """Seeded inputs on the GPU."""

    def __init__(self, seed):
        self.gen = torch.Generator(device="cuda").manual_seed(seed)

    def normal(self, *shape):
        return torch.randn(*shape, generator=self.gen, device="cuda", dtype=torch.float32).to(BF16)

    def queries(self, *shape):
        """Queries whose heads look about in different widths: the scores' standard deviation is 0.5 to 2.5 by the head."""
        gain = 0.5 + 2.0 * torch.rand(shape[-2], 1, generator=self.gen, device="cuda")
        x = torch.randn(*shape, generator=self.gen, device="cuda", dtype=torch.float32)
        return x.mul_(gain).to(BF16)


def floats(*shape):
    return torch.zeros(*shape, device="cuda", dtype=torch.float32)


def zeros(*shape):
    return torch.zeros(*shape, device="cuda", dtype=BF16)


def prepare(case, seed):
    state = {"case": case, "ctx": J.Context(torch.cuda.current_device()), "scale": 1.0 / math.sqrt(case["head_dim"])}
    fill = {"prompt": prepare_prompt, "step": prepare_step, "ingest": prepare_ingest}[case["kind"]]
    fill(case, Source(seed), random.Random(seed), state)
    return state


def prepare_prompt(case, src, rng, state):
    batch, q_heads, kv_heads, dim = case["batch"], case["q_heads"], case["kv_heads"], case["head_dim"]
    cache = zeros(2, batch, kv_heads, case["capacity"], dim)
    # the sub-sequences' results lie one after the other, each dense
    out = floats(batch * case["length"], q_heads, dim)
    lse = floats(batch * case["length"] * q_heads) if case["lse"] else None
    state["calls"] = []
    for pos, n in chunks(case):
        first, last = batch * pos, batch * (pos + n)
        state["calls"].append((src.queries(batch, n, q_heads, dim), src.normal(batch, n, kv_heads, dim),
                               src.normal(batch, n, kv_heads, dim), n, pos, out[first:last],
                               lse[first * q_heads:last * q_heads] if case["lse"] else None))
    state["cache"], state["desc"], state["out"], state["lse"] = cache, J.cache_desc(cache[0], cache[1]), out, lse


def prepare_step(case, src, rng, state):
    layers, branches, drafts = case["layers"], case["branches"], case["drafts"]
    q_heads, kv_heads, dim = case["q_heads"], case["kv_heads"], case["head_dim"]
    lens = lengths(case)
    rng.shuffle(lens)
    state["prefix"] = src.normal(layers, 2, 1, kv_heads, case["prefix"], dim)
    state["suffix"] = src.normal(layers, 2, branches, kv_heads, case["capacity"], dim)
    state["q"] = torch.stack([src.queries(branches, drafts, q_heads, dim) for _ in range(layers)])
    state["k"] = src.normal(layers, branches, drafts, kv_heads, dim)
    state["v"] = src.normal(layers, branches, drafts, kv_heads, dim)
    state["out"] = floats(layers, branches, drafts, q_heads, dim)
    state["lse"] = floats(layers, branches, q_heads, drafts) if case["lse"] else None
    state["lens"] = torch.tensor(lens, dtype=torch.int32, device="cuda")
    state["layers"] = [(state["q"][i], state["k"][i], state["v"][i],
                        J.cache_desc(state["prefix"][i, 0], state["prefix"][i, 1]),
                        J.cache_desc(state["suffix"][i, 0], state["suffix"][i, 1]), state["out"][i],
                        state["lse"][i] if case["lse"] else None) for i in range(layers)]
    if case["tree"]:
        masks, paths, counts = zip(*(tree(drafts, rng) for _ in range(branches)))
        state["masks"] = torch.from_numpy(np.array(masks, np.uint32).view(np.int32)).cuda()
        state["paths"] = torch.tensor(paths, dtype=torch.int32, device="cuda")
        state["counts"] = torch.tensor(counts, dtype=torch.int32, device="cuda")
        state["pos"] = state["lens"] - drafts


def tree(n, rng):
    """A random token tree of n nodes: each node's mask of ancestors and itself, and a root-to-leaf path that is accepted."""
    parent = [-1] + [rng.randrange(max(0, i - 4), i) for i in range(1, n)]
    masks, path = [], []
    for i in range(n):
        masks.append((masks[parent[i]] if i else 0) | 1 << i)
    at = rng.randrange(n)
    while at >= 0:
        path.append(at)
        at = parent[at]
    path.reverse()
    return masks, path + [0] * (n - len(path)), len(path)


def prepare_ingest(case, src, rng, state):
    branches, n, q_heads, kv_heads, dim = (case[k] for k in ("branches", "length", "q_heads", "kv_heads", "head_dim"))
    state["prefix"] = src.normal(2, 1, kv_heads, case["prefix"], dim)
    state["suffix"] = src.normal(2, branches, kv_heads, case["capacity"], dim)
    state["q"], state["out"] = src.queries(branches, n, q_heads, dim), floats(branches, n, q_heads, dim)
    state["k"], state["v"] = src.normal(branches, n, kv_heads, dim), src.normal(branches, n, kv_heads, dim)
    state["lse"] = floats(branches, q_heads, n) if case["lse"] else None
    state["descs"] = (J.cache_desc(state["prefix"][0], state["prefix"][1]),
                      J.cache_desc(state["suffix"][0], state["suffix"][1]))


def run(state):
    return {"prompt": run_prompt, "step": run_step, "ingest": run_ingest}[state["case"]["kind"]](state)


def run_prompt(state):
    ctx, desc, q_heads, scale = state["ctx"], state["desc"], state["case"]["q_heads"], state["scale"]
    for q, k, v, n, pos, out, lse in state["calls"]:
        ctx.chunk_prefill_append_attn(q, k, v, desc, q_heads, n, pos, scale, out, lse)
    return {"out": state["out"], "lse": state["lse"], "cache": state["cache"]}


def run_step(state):
    case, ctx, scale = state["case"], state["ctx"], state["scale"]
    prefix, longest, branches, q_heads, drafts = (case[k] for k in ("prefix", "longest", "branches", "q_heads", "drafts"))
    if case["tree"]:
        q, k, v, pfx, sfx, out, lse = state["layers"][0]
        ctx.kv_append(sfx, k, v, drafts, 0, state["pos"])
        ctx.branch_attn_tree(q, pfx, prefix, sfx, state["lens"], state["masks"], longest, branches, q_heads, drafts, scale,
                             out, lse)
        ctx.kv_compact(sfx, drafts, state["pos"], state["paths"], state["counts"])
    elif case["layers"] == 1:
        q, k, v, pfx, sfx, out, lse = state["layers"][0]
        ctx.branch_append_attn(q, k, v, pfx, prefix, sfx, state["lens"], longest, branches, q_heads, drafts, scale, out, lse)
    else:
        ctx.branch_append_attn_layers(state["layers"], prefix, state["lens"], longest, branches, q_heads, drafts, scale)
    return {"out": state["out"], "lse": state["lse"], "suffix": state["suffix"]}


def run_ingest(state):
    case, ctx = state["case"], state["ctx"]
    pfx, sfx = state["descs"]
    ctx.kv_append(sfx, state["k"], state["v"], case["length"], case["pos"])
    ctx.branch_prefill_attn(state["q"], pfx, case["prefix"], sfx, case["q_heads"], case["length"], case["pos"],
                            state["scale"], state["out"], state["lse"])
    return {"out": state["out"], "lse": state["lse"], "suffix": state["suffix"]}


def work(case):
    """Inputs read once and results written once; 4 * head_dim operations per (query, key) pair that the mask leaves."""
    q_heads, kv_heads, dim = case["q_heads"], case["kv_heads"], case["head_dim"]
    if case["kind"] == "prompt":
        rows, new = case["batch"] * case["length"], case["batch"] * case["length"]
        pairs, cached = case["batch"] * case["length"] * (case["length"] + 1) // 2, 0
    elif case["kind"] == "ingest":
        n, pos = case["length"], case["pos"]
        rows, new = case["branches"] * n, case["branches"] * n
        pairs = case["branches"] * (n * (case["prefix"] + pos) + n * (n + 1) // 2)
        cached = case["prefix"] + case["branches"] * pos
    else:
        n, layers, lens = case["drafts"], case["layers"], lengths(case)
        rows, new = layers * len(lens) * n, layers * len(lens) * n
        # a chain sees i + 1 rows of its block; a tree's nodes see fewer, which depends on the seed
        pairs = layers * sum(n * (case["prefix"] + length - n) + n * (n + 1) // 2 for length in lens)
        cached = layers * (case["prefix"] + sum(length - n for length in lens))
    kv_row = 2 * kv_heads * dim * 2
    return {"bytes": rows * q_heads * (dim * (2 + 4) + (4 if case["lse"] else 0)) + kv_row * (2 * new + cached),
            "flops": 4 * dim * q_heads * pairs}


def tolerance(case):
    # bf16 weights times bf16 values, sums in 32 bits.  Against the same attention in 64 bits the results are off by up to
    # 1.6e-3 (2-norm) and by up to 1.9e-2 of the root mean square at the worst element: four times that.
    return {"rel": 6e-3, "max": 0.08}
