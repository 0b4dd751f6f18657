"""The work that users of this library have it do, as cases that can be timed.

A case is one draft-and-verify step (or a few) on one GPU: a draft token tree is grown layer by layer from the
draft model's logits, the target model's attention runs over that tree, and the accepted path is walked.  The
model forwards are the caller's, so seeded logits and Q/K/V stand in for them: draft rows are noise plus, on
some rows, one confident token (the mix of ``synth.CONFIGS``), target rows are the draft rows plus noise of
their own, so that part of what was drafted is accepted.

``path`` says which of the public entry points the step goes through:

  step    ``Talon.step``: everything device-resident, one call (a serving loop that replays its step)
  calls   one call per stage, as a program does whose draft model runs between two layers; a layer's logits
          come packed, the frontier's rows only, from the place where its draft pass wrote them
  sample  one call per stage at temperature 1 on a paged cache, with the commit that ends such a step
  static  the fixed-width tree that the method is compared with: Top-K in every layer, then pruned
  loop    ``Talon.loop``: several steps with the commit between them, one call
  host    ``Talon.step_host``: pinned host buffers in, host results out

and ``stream`` whether the caller works on torch's default stream or on one of its own.
"""
from __future__ import annotations

import math

import torch

from paper_2601_07353_b200.talon import PAGE_TOKENS, ROWS_BY_NODE, ROWS_PACKED, Talon

HEAD_DIM = 128
_STREAM = None


def _case(name, path, batch, vocab, budget, topk, depth, q_heads, kv_heads, prefix_min, prefix_max, *, cand=-1,
          stream="default", mu=0.03, temp=0.5, confident=0.5, steps=1, keep=0):
    """cand: candidates kept per parent, -1 = topk, 0 = the whole-vocabulary pool; confident: share of rows with one
    dominant token; keep: nodes a static tree is pruned to."""
    return {"name": name, "path": path, "batch": batch, "vocab": vocab, "budget": budget, "topk": topk, "depth": depth,
            "q_heads": q_heads, "kv_heads": kv_heads, "prefix_min": prefix_min, "prefix_max": prefix_max,
            "cand": topk if cand < 0 else cand, "stream": stream, "mu": mu, "temp": temp, "confident": confident,
            "steps": steps, "keep": keep}


def listed():
    return [
        # a small draft head and one short conversation: launches and latency are all there is
        _case("tiny_step", "step", 1, 32000, 16, 4, 8, 32, 8, 512, 512, confident=0.33),
        # one user, an 8B-shaped target: the interactive case, replayed on the server's own stream
        _case("single_step", "step", 1, 128256, 60, 8, 12, 32, 8, 2048, 2048, stream="own"),
        # the same user in a program that runs its draft model between the layers
        _case("single_calls", "calls", 1, 128256, 60, 8, 12, 32, 8, 2048, 2048),
        # the paper's own pool (every token of every frontier row competes) at its defaults N 60, K 10
        _case("full_pool_calls", "calls", 2, 128256, 60, 10, 10, 32, 8, 1500, 1500, cand=0),
        # a batch of conversations of different lengths
        _case("batched_step", "step", 16, 128256, 60, 8, 12, 32, 8, 1024, 4096, stream="own"),
        # a larger vocabulary and more query heads, fewer confident rows: wide, shallow trees
        _case("wide_step", "step", 8, 151936, 60, 10, 16, 64, 8, 8192, 8192, temp=0.7, confident=0.3),
        # the largest: long prompts, the largest budget
        _case("long_step", "step", 32, 128256, 128, 8, 24, 32, 8, 32768, 32768, stream="own", confident=0.6),
        # query heads in groups of five, an odd vocabulary, ragged prompts
        _case("group5_calls", "calls", 4, 50001, 48, 6, 10, 40, 8, 700, 3000),
        # serving at temperature 1 on a paged cache, with the commit
        _case("sampled_paged", "sample", 8, 50001, 60, 8, 12, 32, 8, 1000, 5000, stream="own"),
        # the static tree (Top-10 in eight layers, pruned to 60 nodes) on the same kernels
        _case("static_calls", "static", 4, 128256, 91, 10, 9, 32, 8, 2048, 2048, cand=10, keep=60),
        # four steps of a generation loop with the cache growing between them
        _case("generation_loop", "loop", 2, 128256, 60, 8, 12, 32, 8, 2000, 2300, stream="own", steps=4),
        # everything comes from and goes back to host memory
        _case("host_step", "host", 1, 128256, 60, 8, 12, 32, 8, 2048, 2048),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    path = rng.choice(("step", "step", "calls", "calls", "sample", "static", "loop", "host"))
    batch = _log_uniform(rng, 1, 4 if path == "host" else 8 if path == "loop" else 32)
    vocab = _log_uniform(rng, 8000, 152000)
    budget = _log_uniform(rng, 12, 128)
    topk = rng.randint(2, 10)
    depth = rng.randint(4, 24)
    cand, keep, steps = -1, 0, 1
    heads = [(32, 8), (64, 8), (16, 8), (32, 4), (8, 8)]
    if path in ("step", "calls"):
        heads += [(40, 8), (28, 4), (24, 8)]
    q_heads, kv_heads = rng.choice(heads)
    longest = _log_uniform(rng, 64, 32768)
    shortest = longest if rng.random() < 0.4 else max(1, int(longest * rng.uniform(0.2, 0.9)))
    if path == "host":
        vocab -= vocab % 4                       # dense host rows have to start on 16 bytes
        longest, shortest = min(longest, 8192), min(shortest, 8192)
    if path == "calls" and rng.random() < 0.3:
        cand = 0
    if path == "static":
        topk = rng.randint(4, 10)
        depth = rng.randint(4, 10)
        budget = 1 + topk * depth                # Top-K in `depth` layers
        cand, keep = topk, rng.randint(max(2, budget // 2), budget)
    if path == "loop":
        steps = rng.randint(2, 6)
    # no more logits, keys or products than the largest listed case (the stages called one by one: an eighth of it)
    share = {"step": 1.0, "host": 1.0 / 32}.get(path, 1.0 / 8)
    while batch > 1 and (steps * batch * budget * vocab > share * 32 * 128 * 128256 or
                         steps * batch * (longest + budget) * q_heads * budget > share * 32 * 32768 * 32 * 128):
        batch -= 1
    return {k: v for k, v in _case("", path, batch, vocab, budget, topk, depth, q_heads, kv_heads, shortest, longest, cand=cand,
                                   stream=rng.choice(("default", "own")), mu=rng.choice((0.01, 0.03, 0.03, 0.1)),
                                   temp=rng.choice((0.5, 0.7)), confident=rng.choice((0.3, 0.5, 0.7)), steps=steps,
                                   keep=keep).items() if k != "name"}


def _rows(shape, vocab, dev):
    """[*shape, vocab] fp32 logit rows; each starts on 16 bytes, as the library asks."""
    return torch.empty(*shape, (vocab + 3) // 4 * 4, dtype=torch.float32, device=dev)[..., :vocab]


def _logits(case, dev, gen):
    """Draft and target rows [steps, batch, budget, vocab] of every node slot; packed draft rows are twice as many, so that
    each layer starts at rows of its own."""
    N = case["budget"]
    n_draft = 2 * N if case["path"] == "calls" else N
    shape = (case["steps"], case["batch"], n_draft)
    draft, target = _rows(shape, case["vocab"], dev), _rows((*shape[:2], N), case["vocab"], dev)
    tok = torch.randint(0, case["vocab"], (*shape, 1), device=dev, generator=gen)
    u = torch.rand(*shape, 1, device=dev, generator=gen)
    c = case["confident"]
    h = torch.where(u < c, 8.0, torch.where(u < c + 0.5 * (1.0 - c), 2.0, 0.0))
    for s in range(shape[0]):
        for b in range(shape[1]):
            noise = torch.randn(n_draft, case["vocab"], device=dev, generator=gen)
            draft[s, b] = noise.mul_(case["temp"]).scatter_add_(1, tok[s, b], h[s, b])
            # a sampled target is as sharp as a trained model's posterior, a greedy one only needs its maximum
            if case["path"] == "sample":
                target[s, b] = draft[s, b, :N] * 4.0
            else:
                target[s, b] = draft[s, b, :N] + noise[:N].normal_(generator=gen).mul_(0.5)
    return draft, target


def _qkv(dev, gen, *shape):
    """bf16 N(0, 1), made a part at a time so that the fp32 numbers behind it stay small."""
    out = torch.empty(shape, dtype=torch.bfloat16, device=dev)
    flat = out.view(-1)
    for at in range(0, flat.numel(), 1 << 26):
        flat[at:at + (1 << 26)].normal_(generator=gen)
    return out


def _prefix_lens(case, gen, dev):
    lo, hi = case["prefix_min"], case["prefix_max"]
    return torch.randint(lo, hi + 1, (case["batch"],), device=dev, generator=gen).tolist()


def prepare(case, seed):
    global _STREAM
    dev = torch.device("cuda", torch.cuda.current_device())
    gen = torch.Generator(device=dev).manual_seed(seed)
    path, B, N, D = case["path"], case["batch"], case["budget"], case["depth"]
    Hq, Hkv = case["q_heads"], case["kv_heads"]
    if _STREAM is None:
        _STREAM = torch.cuda.Stream(dev)
    talon = Talon(batch_max=B, vocab=case["vocab"], budget=N, root_topk=case["topk"], cand_topk=case["cand"], max_depth=D,
                  n_q_heads=Hq, n_kv_heads=Hkv, head_dim=HEAD_DIM, mu=case["mu"],
                  init_layers=D if path == "static" else 1, device=dev.index)
    st = {"case": case, "talon": talon, "stream": _STREAM if case["stream"] == "own" else None,
          "scale": 1.0 / math.sqrt(HEAD_DIM)}
    lens = _prefix_lens(case, gen, dev)
    roots = torch.randint(0, case["vocab"], (B,), device=dev, generator=gen).tolist()
    draft, target = _logits(case, dev, gen)
    S = case["steps"]
    grows = path in ("loop", "sample")           # the commit appends to the cache
    room = S * (D + 1) if grows else 0
    i32 = dict(dtype=torch.int32, device=dev)
    lead = (S,) if path == "loop" else ()
    st["q"] = _qkv(dev, gen, *lead, B, N, Hq, HEAD_DIM)
    st["k_tree"], st["v_tree"] = (_qkv(dev, gen, *lead, B, N, Hkv, HEAD_DIM) for _ in range(2))
    if path == "sample":                         # pages of every sequence, shuffled over the pool
        blocks = [(n + room + PAGE_TOKENS - 1) // PAGE_TOKENS for n in lens]
        pool = B * ((case["prefix_max"] + room + PAGE_TOKENS - 1) // PAGE_TOKENS)
        pages = torch.randperm(pool, device=dev, generator=gen).to(torch.int32)
        st["block_table"] = torch.zeros(B, max(blocks), **i32)
        at = 0
        for b, n in enumerate(blocks):
            st["block_table"][b, :n] = pages[at:at + n]
            at += n
        st["n_blocks"], st["n_pages"] = torch.tensor(blocks, **i32), pool
        tokens = st["n_pages"] * PAGE_TOKENS
        st["u_accept"] = torch.rand(B, N, dtype=torch.float64, device=dev, generator=gen)
        st["u_sample"] = torch.rand(B, dtype=torch.float64, device=dev, generator=gen)
    else:                                        # back to back; a cache that grows has a block of its own per sequence
        starts = [0]
        for n in lens:
            starts.append(starts[-1] + (case["prefix_max"] if grows else n) + room)
        tokens = starts[-1]
        st["kv_start"] = torch.tensor(starts[:-1], dtype=torch.int64, device=dev)
        st["kv_limit"] = torch.tensor(starts[1:], dtype=torch.int64, device=dev)
    st["kv_tokens"] = tokens
    st["k_cache"], st["v_cache"] = (_qkv(dev, gen, tokens, Hkv, HEAD_DIM) for _ in range(2))
    st["max_len"] = max(lens) + room
    st["first"] = torch.tensor([lens, roots], **i32)      # prefix lengths and roots as the step finds them
    st["now"] = st["first"].clone()
    st["prefix_len"], st["root_tok"] = st["now"][0], st["now"][1]
    st["draft"], st["target"] = (draft, target) if path == "loop" else (draft[0], target[0])
    if path == "calls":
        st["layers"] = [st["draft"][:, d * N // D:] for d in range(D)]
    if path == "host":
        return _on_host(st, lens, roots)
    st["tree"] = talon.alloc_tree(B)
    st["out"] = torch.zeros(B, N, Hq, HEAD_DIM, dtype=torch.bfloat16, device=dev)
    st["target_tok"] = torch.zeros(B, N, **i32)
    st["accept_len"], st["next_tok"] = torch.zeros(*lead, B, **i32), torch.zeros(*lead, B, **i32)
    st["accept_nodes"] = torch.zeros(*lead, B, D + 1, **i32)
    st["counters"] = torch.zeros(B, 3, dtype=torch.int64, device=dev)
    torch.cuda.synchronize()
    return st


def _on_host(st, lens, roots):
    """The same inputs in pinned host memory, and host arrays for the results."""
    case = st["case"]
    B, N, D = case["batch"], case["budget"], case["depth"]

    def pinned(x):
        return torch.empty(x.shape, dtype=x.dtype, pin_memory=True).copy_(x)

    host = {k: pinned(st[k]) for k in ("draft", "target", "q", "k_cache", "v_cache", "k_tree", "v_tree")}
    i32 = dict(dtype=torch.int32, pin_memory=True)
    host["prefix_len"], host["root_tok"] = torch.tensor(lens, **i32), torch.tensor(roots, **i32)
    host["out"] = torch.zeros(B, N, case["q_heads"], HEAD_DIM, dtype=torch.bfloat16, pin_memory=True)
    for k, shape in (("n_nodes", (B,)), ("token", (B, N)), ("parent", (B, N)), ("depth", (B, N)), ("position", (B, N)),
                     ("accept_len", (B,)), ("accept_nodes", (B, D + 1)), ("bonus", (B,))):
        host[k] = torch.zeros(shape, **i32)
    torch.cuda.synchronize()
    return {"case": case, "talon": st["talon"], "stream": st["stream"], "scale": st["scale"], "host": host}


def _tree_out(st):
    t = st["tree"]
    return [t.n_nodes, t.token, t.parent, t.depth, t.position, t.layer_off, t.score, t.mask]


def _grow(st):
    """The draft phase, a call per layer."""
    talon, tree, case = st["talon"], st["tree"], st["case"]
    talon.reset(tree, st["root_tok"], st["prefix_len"])
    for d in range(case["depth"]):
        if case["path"] == "calls":
            talon.expand_layer(tree, st["layers"][d], rows_per_seq=2 * case["budget"], layout=ROWS_PACKED)
        else:
            talon.expand_layer(tree, st["draft"], layout=ROWS_BY_NODE)


def _attend(st):
    h = st["case"]["kv_heads"] * HEAD_DIM
    st["talon"].tree_attention(st["tree"], st["q"], st["k_cache"], st["v_cache"], st["k_tree"], st["v_tree"], st["kv_start"],
                               st["kv_tokens"], h, HEAD_DIM, st["max_len"], st["scale"], st["out"])


def _step(st):
    h = st["case"]["kv_heads"] * HEAD_DIM
    st["talon"].step(st["tree"], st["root_tok"], st["prefix_len"], st["draft"], st["case"]["depth"], st["q"], st["k_cache"],
                     st["v_cache"], st["k_tree"], st["v_tree"], st["kv_start"], st["kv_tokens"], h, HEAD_DIM, st["max_len"],
                     st["scale"], st["out"], st["target"], st["target_tok"], st["accept_len"], st["accept_nodes"],
                     st["next_tok"])
    return _tree_out(st) + [st["out"], st["target_tok"], st["accept_len"], st["accept_nodes"], st["next_tok"]]


def _calls(st):
    talon, tree = st["talon"], st["tree"]
    _grow(st)
    if st["case"]["path"] == "static":
        talon.prune_tree(tree, st["case"]["keep"])
    talon.build_tree(tree)
    _attend(st)
    talon.accept(tree, st["target"], st["accept_len"], st["accept_nodes"], st["next_tok"], st["target_tok"])
    return _tree_out(st) + [st["out"], st["target_tok"], st["accept_len"], st["accept_nodes"], st["next_tok"]]


def _sample(st):
    talon, tree, h = st["talon"], st["tree"], st["case"]["kv_heads"] * HEAD_DIM
    st["now"].copy_(st["first"])                 # the next request takes this slot of the batch
    _grow(st)
    talon.build_tree(tree)
    talon.tree_attention_paged(tree, st["q"], st["k_cache"], st["v_cache"], st["k_tree"], st["v_tree"], st["block_table"],
                               st["n_pages"], h, HEAD_DIM, st["max_len"], st["scale"], st["out"])
    talon.accept_sample(tree, st["target"], 1.0, st["u_accept"], st["u_sample"], st["accept_len"], st["accept_nodes"],
                        st["next_tok"])
    talon.commit_paged(tree, st["accept_len"], st["accept_nodes"], st["next_tok"], st["k_tree"], st["v_tree"], st["k_cache"],
                       st["v_cache"], st["block_table"], st["n_blocks"], st["n_pages"], h, HEAD_DIM, st["prefix_len"],
                       st["root_tok"], st["counters"])
    return _tree_out(st) + [st["out"], st["accept_len"], st["accept_nodes"], st["next_tok"], st["now"], st["counters"],
                            st["k_cache"], st["v_cache"]]


def _loop(st):
    h = st["case"]["kv_heads"] * HEAD_DIM
    st["now"].copy_(st["first"])
    st["talon"].loop(st["tree"], st["case"]["steps"], st["root_tok"], st["prefix_len"], st["draft"], st["case"]["depth"],
                     st["q"], st["k_cache"], st["v_cache"], st["k_tree"], st["v_tree"], st["kv_start"], st["kv_limit"],
                     st["kv_tokens"], h, HEAD_DIM, st["max_len"], st["scale"], st["out"], st["target"], st["target_tok"],
                     st["accept_len"], st["accept_nodes"], st["next_tok"], st["counters"])
    return _tree_out(st) + [st["out"], st["target_tok"], st["accept_len"], st["accept_nodes"], st["next_tok"], st["now"],
                            st["counters"], st["k_cache"], st["v_cache"]]


def _host(st):
    h = st["host"]
    status = st["talon"].step_host(h["root_tok"], h["prefix_len"], h["draft"], h["target"], h["q"], h["k_cache"], h["v_cache"],
                                   h["k_tree"], h["v_tree"], st["scale"], h["out"], h["n_nodes"], h["token"], h["parent"],
                                   h["depth"], h["position"], h["accept_len"], h["accept_nodes"], h["bonus"])
    return [int(status)] + [h[k] for k in ("out", "n_nodes", "token", "parent", "depth", "position", "accept_len",
                                           "accept_nodes", "bonus")]


_RUN = {"step": _step, "calls": _calls, "static": _calls, "sample": _sample, "loop": _loop, "host": _host}


def run(state):
    fn = _RUN[state["case"]["path"]]
    if state["stream"] is None:
        return fn(state)
    with torch.cuda.stream(state["stream"]):
        return fn(state)


def work(case):
    """How large a tree grows depends on its logits: on these it takes about 0.85 of its budget, or as much as its depth
    allows at three quarters of K nodes a layer, and expands about 0.85 of its nodes; with the whole-vocabulary pool it is
    full after three or four layers, a quarter of its nodes expanded."""
    B, N, D, V, S = case["batch"], case["budget"], case["depth"], case["vocab"], case["steps"]
    Hq, Hkv = case["q_heads"], case["kv_heads"]
    if case["path"] == "static":
        nodes, rows = case["keep"], 1 + case["topk"] * (D - 1)
    elif case["cand"] == 0:
        nodes, rows = N, 1 + N // 4
    else:
        nodes = int(min(0.85 * N, 1 + 0.75 * case["topk"] * D))
        rows = int(0.85 * nodes)
    length = 0.5 * (case["prefix_min"] + case["prefix_max"])
    kv = 2 * 2 * HEAD_DIM * Hkv * (length + nodes)
    qo = 2 * 2 * HEAD_DIM * Hq * nodes
    mask = 8 * ((N + 63) // 64) * nodes
    per_seq = 4 * V * (rows + nodes) + kv + qo + mask
    return {"bytes": float(S * B * per_seq), "flops": float(S * B * 4 * HEAD_DIM * Hq * nodes * (length + nodes))}


def tolerance(case):
    """The attention output is bf16 and its probabilities are rounded to bf16 before the product with V: a few times 2^-9 of
    its norm, and of the larger of a value and the rms.  Scores (sums of fp32 log-softmax) are far inside that.  Tokens,
    parents, masks and paths are whole numbers and the same, but for a candidate that ties with the last one taken."""
    return {"rel": 6e-3, "max": 0.06, "differ": 0.005}
