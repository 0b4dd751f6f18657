#!/usr/bin/env python
"""Benchmark of the Talon hot path: draft-and-verify steps per second on synthetic inputs.

    python bench.py [--gpus N] [--steps K] [--warmup W] [--config NAME] [--impl talon|reference]

A *step* is one pass of the whole path over one batch: tree reset, D_max expansion-layer calls
(Algorithm 2; layers after the budget is spent read nothing), tree finalisation, tree attention of
the N tree tokens against the prefix KV cache, target argmax and the greedy accept walk.  The draft
and target model forwards are not part of the path: their outputs (fp32 logits, bf16 Q/K/V) are
seeded synthetic tensors, resident in HBM before the timed region starts.

Without ``--config`` the headline is the largest workload that fits one GPU (``longctx``) and the
other four workloads are measured in the same invocation and reported under ``configs``.

The timed region is K back-to-back ``talon_step`` calls that rotate over enough distinct input sets
that the bytes touched between two uses of a set exceed the L2 capacity several times over, so
every step reads its inputs from HBM.  It is bracketed by a barrier and a device synchronisation on
both sides, timed with CUDA events, and reported as the maximum over ranks.  When K steps take less
than half a second the region is repeated and the median repeat is reported (``repeats``,
``spread``), so that clock samples fall inside it.  With more than one GPU every rank runs its own
replicas (sequences are independent: no data-path collective).

Rank 0 prints one JSON line.  Beside the contract's keys it carries ``kernels`` (each kernel family of
the single calls timed alone: one event pair around at least 20 back-to-back graph replays of just
those launches, inputs rotated, so no event bracket sits between two kernels; ``rows_and_growth``,
what a whole step launches instead of the expansion layers, by difference), ``roofline`` (algorithmic
bytes or flops over that duration of the dominant family of the timed step, against the measured peaks),
``cpu_baseline`` (the
fp64 CPU oracle on all host cores, one core beside it, with its per-stage split and the count of
tolerated selection ties), ``e2e`` (the same step through ``talon_step_host`` with pinned host
buffers), ``tree_shapes`` and ``configs``.  ``--impl reference`` times the CPU oracle alone.
"""
from __future__ import annotations

import argparse
import json
import math
import os
import statistics
import subprocess
import sys
import threading
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

import numpy as np  # noqa: E402

METRIC = "draft+verify steps/sec"
UNIT = "steps/s"
L2_BYTES = 126 * 1024 * 1024
ROTATION_FACTOR = 3.0            # bytes between two uses of an input set, in units of L2
MIN_REGION_S = 0.5               # a timed region shorter than this is repeated
KERNEL_REPLAYS = 24              # back-to-back replays per kernel-alone measurement (at least 20)
HEADLINE = "longctx"
SUB_CONFIGS = ["tiny", "llama8b", "llama8b_batched", "qwen32b"]
LOOP_CONFIG = "llama8b"          # the workload the multi-step generation loop is run on as an extra
ORACLE_PREFIX_SAMPLE = 4096      # prefix tokens the oracle's attention is timed on when the prefix is longer
DTYPE = "f32 logits, f64 path scores, bf16 attention (f32 accumulate)"


# --------------------------------------------------------------------------------------------
# clocks
# --------------------------------------------------------------------------------------------
class ClockSampler:
    """Polls nvidia-smi for SM clock and throttle reasons of one GPU while work is running."""
    QUERY = ("clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.hw_slowdown,"
             "clocks_event_reasons.hw_thermal_slowdown,clocks_event_reasons.sw_thermal_slowdown,"
             "clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index: int, period_ms: int = 50):
        self.samples = []            # (t, sm, max_sm, power, [reasons])
        self.proc = None
        self.thread = None
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", f"--query-gpu={self.QUERY}", "--format=csv,noheader,nounits",
                 "-lms", str(period_ms), "-i", str(gpu_index)],
                stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
        except OSError:
            return
        self.thread = threading.Thread(target=self._read, daemon=True)
        self.thread.start()

    def _read(self):
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for line in self.proc.stdout:
            parts = [p.strip() for p in line.split(",")]
            if len(parts) < 7:
                continue
            try:
                sm, mx = float(parts[0]), float(parts[1])
                power = float(parts[2]) if parts[2].replace(".", "", 1).isdigit() else float("nan")
            except ValueError:
                continue
            reasons = [n for n, p in zip(names, parts[3:7]) if p.lower().startswith("active")]
            self.samples.append((time.time(), sm, mx, power, reasons))

    def stop(self):
        if self.proc is not None:
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except subprocess.TimeoutExpired:
                self.proc.kill()
        if self.thread is not None:
            self.thread.join(timeout=5)

    def summary(self, t0: float, t1: float):
        inside = [s for s in self.samples if t0 <= s[0] <= t1]
        window = "timed region"
        if len(inside) < 3:          # too few samples inside: take the whole busy span and say so
            inside = list(self.samples)
            window = "warm-up to end of run"
        if not inside:
            return None
        reasons = sorted({r for s in inside for r in s[4]})
        return {"sm_mhz": statistics.median(s[1] for s in inside), "sm_max_mhz": inside[0][2],
                "reasons": reasons, "samples": len(inside), "window": window,
                "power_w_max": max((s[3] for s in inside if s[3] == s[3]), default=None)}


# --------------------------------------------------------------------------------------------
# the oracle as a timed CPU baseline (the only place outside tests/ and smoke that runs it)
# --------------------------------------------------------------------------------------------
def oracle_heads(cfg):
    """Attention heads the oracle is timed on: all of them when that stays within seconds, else
    three (first, middle, last), scaled to all."""
    all_heads = cfg.n_q_heads * (min(cfg.prefix_max, ORACLE_PREFIX_SAMPLE) + cfg.budget) <= 32 * 4300
    return list(range(cfg.n_q_heads)) if all_heads else [0, cfg.n_q_heads // 2, cfg.n_q_heads - 1]


class OracleStep:
    """One draft-and-verify step of one sequence through the CPU oracle, inputs prepared up front.
    A prefix longer than ORACLE_PREFIX_SAMPLE tokens is cut to that length for the attention stage
    and the stage's time scaled by the key count (attention is linear in it)."""

    def __init__(self, cfg, seed: int, seq_id: int):
        from oracle import talon_oracle as O
        from paper_2601_07353_b200 import synth
        self.O, self.cfg, self.seed, self.seq_id = O, cfg, seed, seq_id
        self.heads = oracle_heads(cfg)
        self.p = O.Params(cfg.budget, cfg.topk, cfg.topk, cfg.mu, cfg.max_depth)
        self.root = synth.root_token(cfg, seed, seq_id)
        self.L = synth.prefix_len(cfg, seed, seq_id)
        self.L_used = min(self.L, ORACLE_PREFIX_SAMPLE)
        self.rows = {}

        def cached(path):
            key = tuple(path)
            if key not in self.rows:
                self.rows[key] = synth.draft_logits_row(cfg, seed, seq_id, path)
            return self.rows[key]
        self.logits_fn = cached
        tree = O.expand(self.root, cached, self.p)        # untimed pass: fills the row cache
        self.tree = tree
        n, N = tree.n_nodes, cfg.budget
        self.target = np.zeros((N, cfg.vocab), np.float32)
        for i in range(n):
            self.target[i] = synth.target_logits_row(cfg, seed, seq_id, O.path_tokens(tree, i))
        Hq, Hkv, Dh = cfg.n_q_heads, cfg.n_kv_heads, cfg.head_dim
        self.q = synth.qkv_block(seed, synth.STREAM_Q, seq_id, N * Hq * Dh).reshape(N, Hq, Dh)
        self.kt = synth.qkv_block(seed, synth.STREAM_KT, seq_id, N * Hkv * Dh).reshape(N, Hkv, Dh)
        self.vt = synth.qkv_block(seed, synth.STREAM_VT, seq_id, N * Hkv * Dh).reshape(N, Hkv, Dh)
        cnt = self.L_used * Hkv * Dh
        self.kp = synth.qkv_block(seed, synth.STREAM_K, seq_id, cnt).reshape(-1, Hkv, Dh) if cnt else np.zeros((0, Hkv, Dh), np.float32)
        self.vp = synth.qkv_block(seed, synth.STREAM_V, seq_id, cnt).reshape(-1, Hkv, Dh) if cnt else np.zeros((0, Hkv, Dh), np.float32)

    def run(self):
        """Seconds per stage for one step of this sequence: expansion, finalise, argmax + accept walk,
        attention (scaled to all heads and to the full prefix)."""
        O, cfg = self.O, self.cfg
        t0 = time.perf_counter()
        tree = O.expand(self.root, self.logits_fn, self.p)
        t1 = time.perf_counter()
        O.finalize(tree, self.L)
        t2 = time.perf_counter()
        tt = O.target_argmax(self.target, tree.n_nodes)
        O.accept(tree, tt)
        t3 = time.perf_counter()
        g = cfg.group
        for h in self.heads:
            kv = h // g
            O.tree_attention(self.q[:, h:h + 1], self.kp[:, kv:kv + 1], self.vp[:, kv:kv + 1],
                             self.kt[:, kv:kv + 1], self.vt[:, kv:kv + 1], tree, 1.0 / math.sqrt(cfg.head_dim))
        t4 = time.perf_counter()
        scale = (cfg.n_q_heads / len(self.heads)) * ((self.L + cfg.budget) / (self.L_used + cfg.budget))
        return dict(expand=t1 - t0, finalize=t2 - t1, accept=t3 - t2, attention=(t4 - t3) * scale)


def _oracle_worker(job):
    """One host core: prepares and times the oracle on one sequence; optionally checks a tree the
    CUDA path produced for that sequence against the oracle, layer by layer (runs in a child process)."""
    cfg_name, seed, seq_id, steps, budget_s, gpu_tree = job
    try:
        from threadpoolctl import threadpool_limits
        threadpool_limits(limits=1)
    except Exception:                                     # pragma: no cover
        pass
    from paper_2601_07353_b200 import synth
    cfg = synth.CONFIGS[cfg_name]
    st = OracleStep(cfg, seed, seq_id)
    acc, n = dict(expand=0.0, finalize=0.0, accept=0.0, attention=0.0), 0
    t_start = time.perf_counter()
    for _ in range(steps):
        r = st.run()
        for k in acc:
            acc[k] += r[k]
        n += 1
        if time.perf_counter() - t_start > budget_s:
            break
    out = {k: v / n for k, v in acc.items()}
    out["steps"] = n
    out["ties"] = None
    if gpu_tree is not None:
        # selection differences between candidates whose fp64 scores lie within 1e-5 are tolerated
        # and counted; anything else is a mismatch
        from tests import parity_util as PU
        try:
            _, tol = PU.follow_tree(cfg, st.p, st.root, st.logits_fn, gpu_tree["token"], gpu_tree["parent"],
                                    gpu_tree["n_nodes"], gpu_tree["layer_off"], f"{cfg.name}[seq {seq_id}]")
            out["ties"] = (tol, 0)
        except AssertionError:
            out["ties"] = (0, 1)
    return out


def time_oracle(cfg, seed: int, seq_ids, steps: int, budget_s: float, workers: int, gpu_trees=None):
    """Times the oracle on ``seq_ids``, one sequence per host core at a time.  Returns the all-cores
    figure (sequences run side by side), the one-core figure (mean sequence time), the per-stage
    split and the tie count, as steps/s of a whole batch."""
    import multiprocessing as mp
    jobs = [(cfg.name, seed, s, steps, budget_s, None if gpu_trees is None else gpu_trees.get(s)) for s in seq_ids]
    workers = max(1, min(workers, len(jobs)))
    t0 = time.perf_counter()
    if workers == 1:
        res = [_oracle_worker(j) for j in jobs]
    else:
        with mp.get_context("spawn").Pool(workers) as pool:
            res = pool.map(_oracle_worker, jobs)
    wall = time.perf_counter() - t0
    stages = {k: float(np.mean([r[k] for r in res])) for k in ("expand", "finalize", "accept", "attention")}
    per_seq = sum(stages.values())                     # one core, one sequence, one step
    one_core = 1.0 / (per_seq * cfg.batch)
    all_cores = one_core * workers                     # `workers` sequences side by side, one core each
    ties = [r["ties"] for r in res if r["ties"] is not None]
    heads = oracle_heads(cfg)
    sample = (f"{len(jobs)} sequences ({workers} at a time, one per core), {res[0]['steps']} oracle step(s) each; attention on "
              f"{'all' if len(heads) == cfg.n_q_heads else len(heads)} of {cfg.n_q_heads} heads"
              f"{'' if cfg.prefix_max <= ORACLE_PREFIX_SAMPLE else f' and the first {ORACLE_PREFIX_SAMPLE} prefix tokens'}"
              f", scaled to the whole; x batch {cfg.batch}")
    return dict(value=all_cores, unit=UNIT, cores=workers, kind="oracle", sample=sample,
                one_core={"value": one_core, "cores": 1, "ms_per_step": per_seq * cfg.batch * 1e3},
                stage_ms_per_sequence={k: v * 1e3 for k, v in stages.items()},
                ties=None if not ties else {"sequences_checked": len(ties), "tolerated_within_1e-5": sum(t[0] for t in ties),
                                            "mismatches": sum(t[1] for t in ties)},
                setup_and_run_wall_s=wall)


def workload_text(cfg) -> str:
    pl = f"{cfg.prefix_min}" if cfg.prefix_min == cfg.prefix_max else f"U[{cfg.prefix_min},{cfg.prefix_max}]"
    return (f"{cfg.name}: batch {cfg.batch}, vocab {cfg.vocab}, budget N={cfg.budget} (root included), D_max "
            f"{cfg.max_depth}, K {cfg.topk}, mu {cfg.mu}, {cfg.n_q_heads}/{cfg.n_kv_heads} heads, Dh {cfg.head_dim}, "
            f"prefix {pl}, spike mix '{cfg.spike}', T {cfg.temp}")


# --------------------------------------------------------------------------------------------
# reference arm: the oracle on host cores
# --------------------------------------------------------------------------------------------
def run_reference(args, cfg):
    from paper_2601_07353_b200 import dist
    info = dist.env_rank_info()
    if not info.is_main:
        return 0
    cores = os.cpu_count() or 1
    r = time_oracle(cfg, args.seed, list(range(min(cores, cfg.batch))), max(1, args.steps), 60.0, cores)
    line = {
        "impl": "reference", "metric": METRIC, "value": r["value"], "unit": UNIT, "n_gpus": args.gpus,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1e3 / r["value"],
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": {"workload": workload_text(cfg)},
        "cpu_baseline": {k: r[k] for k in ("value", "unit", "cores", "kind", "sample", "one_core", "stage_ms_per_sequence")},
        "e2e": {"value": r["value"], "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
        "gpu_launches": 0,
    }
    print(json.dumps(line))
    return 0


# --------------------------------------------------------------------------------------------
# the CUDA arm
# --------------------------------------------------------------------------------------------
def set_bytes(wl) -> int:
    """HBM bytes one step touches in one input set (upper bound: every draft row counted)."""
    t = wl.draft.numel() * 4 + wl.target.numel() * 4
    for x in (wl.q, wl.k_prefix, wl.v_prefix, wl.k_tree, wl.v_tree, wl.out):
        t += x.numel() * 2
    return t


def tree_statistics(cfg, sets, roofline):
    """Algorithmic work per step and the shapes of the trees the input sets produce."""
    B, N, V, D = cfg.batch, cfg.budget, cfg.vocab, cfg.max_depth
    exp_b = arg_b = att_b = att_f = 0
    n_nodes, depths, rows_per_seq = [], [], []
    per_depth = np.zeros(D + 1)
    for wl in sets:
        lo = wl.tree.layer_off.cpu().numpy()
        nn = wl.tree.n_nodes.cpu().numpy()
        pl = wl.prefix_len.cpu().numpy()
        dep = wl.tree.depth.cpu().numpy()
        for b in range(B):
            rows = roofline.expanded_rows(lo[b], N, D)
            exp_b += roofline.expand_bytes(rows, V)
            arg_b += roofline.argmax_bytes(int(nn[b]), V)
            att_b += roofline.attention_bytes(int(pl[b]), int(nn[b]), cfg.n_q_heads, cfg.n_kv_heads, cfg.head_dim, N)
            att_f += roofline.attention_flops(int(pl[b]), int(nn[b]), cfg.n_q_heads, cfg.head_dim)
            n_nodes.append(int(nn[b])); depths.append(int(dep[b, :nn[b]].max())); rows_per_seq.append(rows)
            per_depth += np.bincount(dep[b, :nn[b]], minlength=D + 1)[:D + 1]
    n = len(sets)
    work = dict(expand_rows=exp_b / n, accept=arg_b / n, tree_attention=att_b / n, attention_flops=att_f / n)
    shapes = {"n_nodes_min": min(n_nodes), "n_nodes_max": max(n_nodes), "n_nodes_mean": float(np.mean(n_nodes)),
              "max_depth_min": min(depths), "max_depth_max": max(depths),
              "expanded_rows_per_seq_mean": float(np.mean(rows_per_seq)),
              "nodes_per_depth_mean": [round(float(x), 2) for x in per_depth / len(n_nodes)]}
    return work, shapes


def time_replays(graphs, replays: int):
    """Milliseconds per replay: one event pair around ``replays`` back-to-back graph launches that
    rotate over ``graphs`` (one per input set)."""
    import torch
    for i in range(min(3, replays)):
        graphs[i % len(graphs)].replay()
    torch.cuda.synchronize()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record()
    for i in range(replays):
        graphs[i % len(graphs)].replay()
    e1.record()
    torch.cuda.synchronize()
    return e0.elapsed_time(e1) / replays


def kernel_pass(t, cfg, sets, stream):
    """Times each kernel family alone.  For every input set the launches of one family are captured
    in a CUDA graph of their own (expansion: the reset plus the D_max layer launches, since a layer
    needs the tree the previous one left; the reset's own time is measured and subtracted); the
    graphs are replayed back to back, rotating over the sets, between one pair of events."""
    import torch
    from paper_2601_07353_b200 import workload
    D = cfg.max_depth
    scale = 1.0 / math.sqrt(cfg.head_dim)
    fam = {
        "reset": lambda wl: t.reset(wl.tree, wl.root_tok, wl.prefix_len),
        "reset+expand": lambda wl: (t.reset(wl.tree, wl.root_tok, wl.prefix_len),
                                    [t.expand_layer(wl.tree, wl.draft) for _ in range(D)]),
        "tree_attention": lambda wl: t.tree_attention(wl.tree, wl.q, wl.k_prefix, wl.v_prefix, wl.k_tree, wl.v_tree,
                                                      wl.kv_start, wl.k_prefix.shape[0], cfg.n_kv_heads * cfg.head_dim,
                                                      cfg.head_dim, wl.max_prefix_len, scale, wl.out),
        # the tail of a step: the accept walk also closes the tree (no separate build launch)
        "accept": lambda wl: t.close_and_accept(wl.tree, wl.target, wl.accept_len, wl.accept_nodes, wl.bonus_tok,
                                                wl.target_tok),
    }
    for wl in sets:                                   # every family runs on a finished tree
        workload.run_step(t, wl)
    torch.cuda.synchronize()
    out, launches = {}, {}
    replays = max(KERNEL_REPLAYS, 2 * len(sets))
    with torch.cuda.stream(stream):
        for name, fn in fam.items():
            graphs = []
            l0 = t.launch_count()
            for wl in sets:
                g = torch.cuda.CUDAGraph()
                with torch.cuda.graph(g, stream=stream):
                    fn(wl)
                graphs.append(g)
            launches[name] = (t.launch_count() - l0) / len(sets)
            out[name] = time_replays(graphs, replays)
            del graphs
        for wl in sets:                               # leave every set with a complete step behind it
            workload.run_step(t, wl)
    torch.cuda.synchronize()
    return out, launches, replays


def generation_loop_extra(t, cfg, args, dev, steps: int = 4):
    """Section 5.3's loop as an extra: ``steps`` draft-and-verify steps with the commit between them as
    ONE ``talon_loop`` call captured in one CUDA graph; delta, tau and R from the library's counters.
    The steps' inputs are built one after the other (a step starts from its predecessor's correction
    token and prefix length), then the whole loop is replayed from the same start."""
    import torch
    from paper_2601_07353_b200 import synth, talon, workload
    B, N, D, Hq, Hkv, Dh = cfg.batch, cfg.budget, cfg.max_depth, cfg.n_q_heads, cfg.n_kv_heads, cfg.head_dim
    seqs = list(range(B))
    scale = 1.0 / math.sqrt(Dh)
    room = steps * (D + 1)
    lens = [synth.prefix_len(cfg, args.seed, s) for s in seqs]
    roots = [synth.root_token(cfg, args.seed, s) for s in seqs]
    blocks = [L + room for L in lens]
    starts = np.concatenate([[0], np.cumsum(blocks)[:-1]]).astype(np.int64)
    total = int(starts[-1] + blocks[-1])
    i64 = lambda x: torch.tensor(np.asarray(x), dtype=torch.int64, device=dev)
    kv_start, kv_limit = i64(starts), i64(starts + np.asarray(blocks, np.int64))
    kc = torch.zeros(total, Hkv, Dh, dtype=torch.bfloat16, device=dev)
    vc = torch.zeros(total, Hkv, Dh, dtype=torch.bfloat16, device=dev)
    plen = torch.tensor(lens, dtype=torch.int32, device=dev)
    root = torch.tensor(roots, dtype=torch.int32, device=dev)
    counters = torch.zeros(B, 3, dtype=torch.int64, device=dev)
    built = []
    for s in range(steps):
        wl = workload.build_workload(cfg, t, args.seed + 1000 + s, seqs, prefix_lens=plen.cpu().tolist(),
                                     root_tokens=root.cpu().tolist())
        if s == 0:
            ws = wl.kv_start.cpu().numpy()
            for b in range(B):
                kc[starts[b]:starts[b] + lens[b]] = wl.k_prefix[int(ws[b]):int(ws[b]) + lens[b]]
                vc[starts[b]:starts[b] + lens[b]] = wl.v_prefix[int(ws[b]):int(ws[b]) + lens[b]]
        t.reset(wl.tree, root, plen)
        for _ in range(D):
            t.expand_layer(wl.tree, wl.draft)
        t.build_tree(wl.tree)
        t.tree_attention(wl.tree, wl.q, kc, vc, wl.k_tree, wl.v_tree, kv_start, total, Hkv * Dh, Dh, int(plen.max()), scale, wl.out)
        t.accept(wl.tree, wl.target, wl.accept_len, wl.accept_nodes, wl.bonus_tok, wl.target_tok)
        t.commit(wl.tree, wl.accept_len, wl.accept_nodes, wl.bonus_tok, wl.k_tree, wl.v_tree, kc, vc, kv_start, kv_limit,
                 total, Hkv * Dh, Dh, plen, root, counters)
        built.append(wl)
    assert t.poll_status() == talon.OK
    draft = torch.stack([w.draft for w in built]); target = torch.stack([w.target for w in built])
    q = torch.stack([w.q for w in built]); kt = torch.stack([w.k_tree for w in built]); vt = torch.stack([w.v_tree for w in built])
    tree, out = built[0].tree, built[0].out
    al = torch.zeros(steps, B, dtype=torch.int32, device=dev); an = torch.zeros(steps, B, D + 1, dtype=torch.int32, device=dev)
    bo = torch.zeros(steps, B, dtype=torch.int32, device=dev); tt = torch.zeros(B, N, dtype=torch.int32, device=dev)
    plen0, root0 = torch.tensor(lens, dtype=torch.int32, device=dev), torch.tensor(roots, dtype=torch.int32, device=dev)
    side = torch.cuda.Stream(dev)
    with torch.cuda.stream(side):
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=side):
            plen.copy_(plen0); root.copy_(root0); counters.zero_()       # every replay starts from the same state
            t.loop(tree, steps, root, plen, draft, D, q, kc, vc, kt, vt, kv_start, kv_limit, total, Hkv * Dh, Dh,
                   max(lens) + room, scale, out, target, tt, al, an, bo, counters)
        ms = time_replays([g], KERNEL_REPLAYS)
    assert t.poll_status() == talon.OK
    m5, m10 = talon.loop_metrics(counters, 0.05), talon.loop_metrics(counters, 0.10)
    return {"steps_per_call": steps, "ms_per_call": ms, "value": steps / (ms * 1e-3), "unit": UNIT,
            "delta": m5["delta"], "tau": m5["tau"], "speedup_R_at_c_0.05": m5["speedup"], "speedup_R_at_c_0.10": m10["speedup"],
            "note": "talon_loop (step + commit per step) captured in one CUDA graph; delta = N_q/N_p, tau = L/N_p, "
                    "R = tau/(1 + c delta) from the library's counters; the acceptance statistics are those of the synthetic "
                    "target logits, not of a model"}


def measure(cfg, args, info, dev, dev_index, peaks, headline: bool, sampler=None):
    """Builds the workload of ``cfg`` and measures it.  Returns the fields of a result line."""
    import torch
    from paper_2601_07353_b200 import dist, roofline, synth, talon, workload

    B, N, V, D = cfg.batch, cfg.budget, cfg.vocab, cfg.max_depth
    t = workload.make_talon(cfg, device=dev_index)
    probe = workload.build_workload(cfg, t, args.seed, dist.rank_sequence_ids(info, 1, B)[0])
    per_set = set_bytes(probe)
    n_sets = max(1, math.ceil(ROTATION_FACTOR * L2_BYTES / per_set)) if args.sets is None else args.sets
    free_b, _ = torch.cuda.mem_get_info(dev)
    n_sets = max(1, min(n_sets, int(0.6 * free_b // per_set) + 1))
    ids = dist.rank_sequence_ids(info, n_sets, B)
    sets = [probe] + [workload.build_workload(cfg, t, args.seed, ids[s]) for s in range(1, n_sets)]
    torch.cuda.synchronize()
    assert t.poll_status() == talon.OK
    work, shapes = tree_statistics(cfg, sets, roofline)

    step = lambda i: workload.run_step_fused(t, sets[i % n_sets])
    # Everything below runs on a stream of its own: talon_step replays a captured graph of its
    # launches from the second call with the same arguments, which the legacy default stream cannot do.
    torch.cuda.synchronize()
    main_stream = torch.cuda.Stream(dev)
    torch.cuda.set_stream(main_stream)

    # ---- warm-up: every input set at least twice, so that each set's step has been captured ----
    warm = max(args.warmup, 3, 2 * n_sets)
    for i in range(warm):
        step(i)
    torch.cuda.synchronize()

    # ---- the timed region: K steps, repeated until half a second has been measured ----
    K = args.steps
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    launches0 = t.launch_count()
    reps, total, wall0 = [], 0.0, time.time()
    max_reps = 1 if args.no_repeat else 200
    while len(reps) < max_reps and (not reps or total < MIN_REGION_S):
        torch.cuda.synchronize()
        dist.barrier(info)
        ev0.record()
        for i in range(K):
            step(len(reps) * K + i)
        ev1.record()
        torch.cuda.synchronize()
        dist.barrier(info)
        s = dist.max_over_ranks(ev0.elapsed_time(ev1) * 1e-3, info, dev)
        reps.append(s)
        total += s
    wall1 = time.time()
    gpu_launches = (t.launch_count() - launches0) // len(reps)
    assert t.poll_status() == talon.OK
    seconds = statistics.median(reps)
    value = dist.whole_job_rate(K, seconds, info)
    res = {
        "value": value, "ms_per_step": seconds / K * 1e3, "steps": K, "repeats": len(reps),
        "spread": (max(reps) - min(reps)) / seconds if len(reps) > 1 else 0.0,
        "warmup": warm, "warmup_requested": args.warmup, "gpu_launches": int(gpu_launches),
        "launches_per_step": gpu_launches / K, "sequence_steps_per_s": value * B, "tree_shapes": shapes, "algorithmic_per_step": work,
        "l2": f"inputs larger than L2: steps rotate over {n_sets} input sets of {per_set / 1e6:.1f} MB "
              f"({n_sets * per_set / 1e6:.0f} MB vs 126 MB L2)",
        "input_sets": n_sets, "timed_wall": (wall0, wall1),
    }

    if args.no_kernel_pass:
        t.close()
        res.update({"kernels": {}, "kernels_sum_over_step": None, "kernel_timing": "skipped", "roofline": None})
        return res
    # ---- each kernel family alone ----
    ms, launches, replays = kernel_pass(t, cfg, sets, main_stream)
    exp_ms = max(ms["reset+expand"] - ms["reset"], 1e-6)
    gbs = lambda b, m: b / (m * 1e-3) / 1e9
    kernels = {
        "reset": {"ms_per_step": ms["reset"], "launches_per_step": launches["reset"]},
        "expand_rows": {"ms_per_step": exp_ms, "launches_per_step": launches["reset+expand"] - launches["reset"],
                        "avg_launch_us": exp_ms * 1e3 / max(1.0, launches["reset+expand"] - launches["reset"]),
                        "algorithmic_gbs": gbs(work["expand_rows"], exp_ms)},
        "build_tree": {"ms_per_step": 0.0, "launches_per_step": 0.0,
                       "note": "inside a step the accept walk closes the tree: no launch of its own"},
        "tree_attention": {"ms_per_step": ms["tree_attention"], "launches_per_step": launches["tree_attention"],
                           "algorithmic_gbs": gbs(work["tree_attention"], ms["tree_attention"]),
                           "tflops": work["attention_flops"] / (ms["tree_attention"] * 1e-3) / 1e12},
        "accept": {"ms_per_step": ms["accept"], "launches_per_step": launches["accept"],
                   "algorithmic_gbs": gbs(work["accept"], ms["accept"]),
                   "note": "target argmax (the bytes) plus the accept walk, which also closes the tree (a few microseconds)"},
    }
    for k in ("expand_rows", "tree_attention", "accept"):
        kernels[k]["frac_of_hbm_peak"] = kernels[k]["algorithmic_gbs"] / peaks["hbm_gbs"]
        kernels[k]["frac_of_nominal_8tbs"] = kernels[k]["algorithmic_gbs"] / 8000.0
    kernels["tree_attention"]["frac_of_bf16_sustained"] = kernels["tree_attention"]["tflops"] / peaks["bf16_tflops_sustained"]
    ksum = ms["reset+expand"] + ms["tree_attention"] + ms["accept"]
    res["kernels"] = kernels
    res["kernels_sum_ms"] = ksum
    res["kernel_timing"] = (f"each family of the single calls alone: one event pair around {replays} back-to-back graph replays of its "
                            "launches, inputs rotated over the input sets; layers that find the tree full are launched and counted")
    # A whole step whose rows are prepared at once launches none of the expansion layers; what it launches instead (row pass,
    # growth, an arg-max where the target rows do not ride along) is the step less the attention.
    families = ["expand_rows", "tree_attention", "accept"]
    if res["launches_per_step"] < D + 3:
        rows_ms = max(res["ms_per_step"] - ms["tree_attention"], 1e-6)
        work["rows_and_growth"] = work["expand_rows"] + work["accept"]
        kernels["rows_and_growth"] = {
            "ms_per_step": rows_ms, "launches_per_step": res["launches_per_step"] - launches["tree_attention"],
            "algorithmic_gbs": gbs(work["rows_and_growth"], rows_ms),
            "note": "row_pass_kernel + grow_kernel, and the arg-max where it is a launch of its own: the step less the attention "
                    "alone (part of which runs beside the growth); bytes of the rows the trees need, not of all rows read"}
        kernels["rows_and_growth"]["frac_of_hbm_peak"] = kernels["rows_and_growth"]["algorithmic_gbs"] / peaks["hbm_gbs"]
        families = ["rows_and_growth", "tree_attention"]
        res["kernels_sum_over_step"] = None
        res["kernel_timing"] += "; rows_and_growth by difference; expand_rows and accept are not what the timed step launches"
    else:
        res["kernels_sum_over_step"] = ksum / res["ms_per_step"]

    # ---- roofline of the dominant kernel ----
    dominant = max(families, key=lambda k: kernels[k]["ms_per_step"])
    kd = kernels[dominant]
    intensity = work["attention_flops"] / max(1.0, work["tree_attention"])
    ridge = peaks["bf16_tflops_sustained"] * 1e12 / (peaks["hbm_gbs"] * 1e9)
    n_launch = max(1.0, kd["launches_per_step"])
    ratio = roofline.captured_traffic_ratio(ROOT, dominant, cfg.name)
    roof = {"kernel": dominant, "bound": "hbm", "achieved": kd["algorithmic_gbs"], "peak": peaks["hbm_gbs"], "unit": "GB/s",
            "frac": kd["frac_of_hbm_peak"], "peak_source": f"of {peaks['source']}",
            "avg_launch_us": kd["ms_per_step"] * 1e3 / n_launch, "launches_per_step": n_launch,
            "algorithmic_bytes_per_launch": work[dominant] / n_launch,
            "traffic": None if ratio is None else ratio * work[dominant] / n_launch,
            "traffic_source": None if ratio is None else "profiles/traffic_capture.json: DRAM bytes per algorithmic byte from the "
                                                          "last ncu capture of this kernel source on this workload x this run's bytes per launch"}
    if dominant == "tree_attention" and intensity > ridge:
        roof.update({"bound": "tensor", "achieved": kd["tflops"], "peak": peaks["bf16_tflops_sustained"], "unit": "TFLOP/s",
                     "frac": kd["frac_of_bf16_sustained"], "flop_per_byte": intensity, "ridge_flop_per_byte": ridge})
    res["roofline"] = roof

    if cfg.name == LOOP_CONFIG and not args.no_loop:
        try:
            res["generation_loop"] = generation_loop_extra(t, cfg, args, dev)
        except Exception as e:                           # an extra, never the headline
            res["generation_loop"] = {"error": str(e).splitlines()[0][:200]}
            torch.cuda.synchronize()
    if not headline:
        t.close()
        del sets
        torch.cuda.empty_cache()
        return res

    # ---- the same steps as one CUDA graph replay each (no library entry, no launch gaps from the host) ----
    if not args.no_graph:
        try:
            graphs = []
            side = torch.cuda.Stream(dev)
            with torch.cuda.stream(side):
                for s in range(n_sets):
                    gph = torch.cuda.CUDAGraph()
                    with torch.cuda.graph(gph, stream=side):
                        workload.run_step_fused(t, sets[s])
                    graphs.append(gph)
                torch.cuda.synchronize()
                gms = time_replays(graphs, max(K, 3 * n_sets))
            res["graph_replay"] = {"value": dist.whole_job_rate(1, dist.max_over_ranks(gms * 1e-3, info, dev), info),
                                   "unit": UNIT, "ms_per_step": gms}
            del graphs
        except Exception as e:                           # graph capture is an extra, never the headline
            res["graph_replay"] = {"error": str(e).splitlines()[0][:200]}
            torch.cuda.synchronize()

    # ---- the sampling verification (the paper's temperature-1 setting) on the same trees: an extra ----
    if not args.no_sampling:
        Ks = min(K, 64)
        dev_t = sets[0].target.device
        uas = [torch.from_numpy(np.stack([synth.verify_uniforms(args.seed, sid, N, 0)[0] for sid in wl.seq_ids])).to(dev_t)
               for wl in sets]
        uss = [torch.tensor([synth.verify_uniforms(args.seed, sid, N, 0)[1] for sid in wl.seq_ids], dtype=torch.float64,
                            device=dev_t) for wl in sets]
        s_tok = torch.zeros(B, dtype=torch.int32, device=dev_t)

        def sample_step(i):
            wl = sets[i % n_sets]
            t.accept_sample(wl.tree, wl.target, 1.0, uas[i % n_sets], uss[i % n_sets], wl.accept_len, wl.accept_nodes, s_tok)

        for i in range(3):
            sample_step(i)
        torch.cuda.synchronize()
        t.timing_enable(2 * Ks + 8, ["target_softmax_stats", "accept_sample"])
        for i in range(Ks):
            sample_step(i)
        st = t.timing_read()
        t.timing_enable(0)
        assert t.poll_status() == talon.OK
        sm_ms, sm_n = st["target_softmax_stats"]
        wk_ms, wk_n = st["accept_sample"]
        if sm_n and wk_n:
            g = work["accept"] / (sm_ms / sm_n * 1e-3) / 1e9
            res["sampling_verify"] = {"temperature": 1.0, "calls": Ks,
                                      "target_softmax_stats": {"ms_per_call": sm_ms / sm_n, "algorithmic_gbs": g,
                                                               "frac_of_hbm_peak": g / peaks["hbm_gbs"],
                                                               "note": "bracketed by events per launch"},
                                      "accept_sample": {"ms_per_call": wk_ms / wk_n}}

    # ---- end to end: host buffers in, host results out, copies inside the timed region ----
    if not args.no_e2e:
        pin = lambda x: x.cpu().pin_memory()
        hi32 = lambda *s: torch.zeros(*s, dtype=torch.int32).pin_memory()
        n_host = max(1, min(n_sets, int((10 << 30) // per_set)))
        host = []
        for wl in sets[:n_host]:
            host.append((pin(wl.root_tok), pin(wl.prefix_len), pin(wl.draft), pin(wl.target), pin(wl.q),
                         pin(wl.k_prefix), pin(wl.v_prefix), pin(wl.k_tree), pin(wl.v_tree)))
        out_h = torch.zeros(B, N, cfg.n_q_heads, cfg.head_dim, dtype=torch.bfloat16).pin_memory()
        hres = (hi32(B), hi32(B, N), hi32(B, N), hi32(B, N), hi32(B, N), hi32(B), hi32(B, D + 1), hi32(B))
        h2d = sum(x.numel() * x.element_size() for x in host[0]) + 8 * B
        d2h = out_h.numel() * 2 + sum(x.numel() * 4 for x in hres)
        Ke = max(3, min(K, int(8.0 / max(1e-4, h2d / 20e9))))       # keep this leg within ~10 s
        scale = 1.0 / math.sqrt(cfg.head_dim)
        for i in range(2):
            assert t.step_host(*host[i % n_host], scale, out_h, *hres) == talon.OK
        torch.cuda.synchronize()
        dist.barrier(info)
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        w0 = time.perf_counter()
        e0.record()
        for i in range(Ke):
            t.step_host(*host[i % n_host], scale, out_h, *hres)
        e1.record()
        torch.cuda.synchronize()
        w1 = time.perf_counter()
        dist.barrier(info)
        es = dist.max_over_ranks(max(e0.elapsed_time(e1) * 1e-3, 0.0), info, dev)
        res["e2e"] = {"value": dist.whole_job_rate(Ke, es, info), "unit": UNIT, "h2d_bytes_per_step": h2d,
                      "d2h_bytes_per_step": d2h, "steps": Ke, "ms_per_step": es / Ke * 1e3,
                      "host_wall_ms_per_step": (w1 - w0) / Ke * 1e3,
                      "api": "talon_step_host (pinned host buffers in, host results out)"}
        del host

    # ---- the oracle beside it, on the machine's host cores, and the tie count against the CUDA trees ----
    if info.is_main and info.world == 1 and not args.no_cpu_baseline:
        cores = os.cpu_count() or 1
        gpu_trees, seqs = {}, []
        for wl in sets:
            tok, par = wl.tree.token.cpu().numpy(), wl.tree.parent.cpu().numpy()
            nn, lo = wl.tree.n_nodes.cpu().numpy(), wl.tree.layer_off.cpu().numpy()
            for bi, sid in enumerate(wl.seq_ids):
                if len(seqs) < cores:
                    seqs.append(sid)
                    gpu_trees[sid] = dict(token=tok[bi], parent=par[bi], n_nodes=int(nn[bi]), layer_off=lo[bi])
        r = time_oracle(cfg, args.seed, seqs, 1, 20.0, cores, gpu_trees)
        res["cpu_baseline"] = {k: r[k] for k in ("value", "unit", "cores", "kind", "sample", "one_core",
                                                 "stage_ms_per_sequence", "setup_and_run_wall_s")}
        res["selection_ties"] = r["ties"]
    t.close()
    del sets
    torch.cuda.empty_cache()
    return res


def run_talon(args):
    import torch
    from paper_2601_07353_b200 import dist, roofline, synth

    info = dist.env_rank_info()
    if not torch.cuda.is_available():
        raise SystemExit("bench.py needs a CUDA device: the path has no CPU fallback")
    dev_index = info.local_rank % torch.cuda.device_count()
    torch.cuda.set_device(dev_index)
    dev = torch.device("cuda", dev_index)
    dist.init(info, "nccl")
    peaks = roofline.load_peaks(ROOT)
    head_name = args.config or HEADLINE
    subs = [] if (args.config or args.no_sub_configs or info.world > 1) else SUB_CONFIGS

    sampler = ClockSampler(dev_index) if info.is_main else None
    head_cfg = synth.CONFIGS[head_name]
    if args.batch is not None:
        head_cfg = head_cfg.scaled(batch=args.batch)
    head = measure(head_cfg, args, info, dev, dev_index, peaks, True)
    wall0, wall1 = head.pop("timed_wall")
    clocks = sampler.summary(wall0, wall1) if sampler is not None else None
    others = {}
    for name in subs:
        torch.cuda.set_stream(torch.cuda.default_stream(dev))
        r = measure(synth.CONFIGS[name], args, info, dev, dev_index, peaks, False)
        r.pop("timed_wall")
        others[name] = {"workload": workload_text(synth.CONFIGS[name]),
                        **{k: r[k] for k in ("value", "ms_per_step", "steps", "repeats", "spread", "roofline", "kernels",
                                             "kernels_sum_over_step", "tree_shapes", "input_sets", "gpu_launches", "algorithmic_per_step")},
                        **({"generation_loop": r["generation_loop"]} if "generation_loop" in r else {})}
    if sampler is not None:
        sampler.stop()

    if info.is_main:
        cfg = head_cfg
        line = {
            "metric": METRIC, "value": head["value"], "unit": UNIT, "n_gpus": info.world, "steps": head["steps"],
            "warmup": head["warmup"], "warmup_requested": head["warmup_requested"], "ms_per_step": head["ms_per_step"],
            "repeats": head["repeats"], "spread": head["spread"],
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": DTYPE, "data": "synthetic",
            "config": {"workload": workload_text(cfg), "l2": head["l2"],
                       "step": f"talon_step, {head['launches_per_step']:.0f} launches: "
                               + ("draft rows of all node slots in one pass or two, trees grown in a kernel of their own, tree attention, "
                                  "target arg-max and walk (in the pass and the growth kernel where one pass does)"
                                  if head["launches_per_step"] < cfg.max_depth + 3 else
                                  f"reset + {cfg.max_depth} expansion layers + tree attention + accept (whose walk closes the tree)")
                               + " (the library replays its own captured graph of these launches)",
                       "sequences_per_rank": cfg.batch, "input_sets": head["input_sets"]},
            "clocks": clocks, "e2e": head.get("e2e"), "gpu_launches": head["gpu_launches"], "roofline": head["roofline"],
            "cpu_baseline": head.get("cpu_baseline"), "selection_ties": head.get("selection_ties"),
            "graph_replay": head.get("graph_replay"), "kernels": head["kernels"], "kernel_timing": head["kernel_timing"],
            "kernels_sum_over_step": head["kernels_sum_over_step"], "sampling_verify": head.get("sampling_verify"),
            "tree_shapes": head["tree_shapes"], "sequence_steps_per_s": head["sequence_steps_per_s"],
            "algorithmic_per_step": head["algorithmic_per_step"],
            "generation_loop": head.get("generation_loop"),
            "configs": others,
        }
        print(json.dumps(line))
    dist.shutdown()
    return 0


# --------------------------------------------------------------------------------------------
# the paper's own on-path experiment: single-layer tree-expansion latency on Zipf rows
# --------------------------------------------------------------------------------------------
def run_zipf_micro(args):
    """Latency of one expansion layer (the K children of the root as frontier, batch 1) on rows with
    P(rank r) ~ r^-alpha, for the paper's vocabularies and exponents: 20 warm-up runs, mean of 100,
    as in the appendix's tree-construction micro-benchmark.  Two strategies run on the same rows and
    the same kernel: Talon's gated layer (Algorithm 2) and the static method's dual Top-K layer
    (Algorithm 1: per-parent Top-K, then the Top-K of the K x K pool).  Extra mode; prints its own
    JSON line."""
    import torch
    from paper_2601_07353_b200 import roofline, synth, talon

    if not torch.cuda.is_available():
        raise SystemExit("bench.py needs a CUDA device: the path has no CPU fallback")
    dev = torch.device("cuda", 0)
    torch.cuda.set_device(0)
    peaks = roofline.load_peaks(ROOT)
    N, K, D = 60, 10, 8
    results = []

    def timed_layer(t, tree, root, plen, draft):
        e0 = [torch.cuda.Event(enable_timing=True) for _ in range(120)]
        e1 = [torch.cuda.Event(enable_timing=True) for _ in range(120)]
        for it in range(120):
            t.reset(tree, root, plen)
            t.expand_layer(tree, draft)           # root layer (Top-K in both strategies): untimed
            e0[it].record()
            t.expand_layer(tree, draft)           # the timed layer: K frontier rows
            e1[it].record()
        torch.cuda.synchronize()
        assert t.poll_status() == talon.OK
        us = [a.elapsed_time(b) * 1e3 for a, b in zip(e0[20:], e1[20:])]
        lo = tree.layer_off[0].cpu().tolist()
        return sum(us) / len(us), min(us), lo[2] - lo[1], lo[3] - lo[2]

    for V in (32000, 128256, 151936):
        mk = lambda init: talon.Talon(batch_max=1, vocab=V, budget=N, root_topk=K, cand_topk=K, max_depth=D, mu=0.03,
                                      n_q_heads=32, n_kv_heads=8, head_dim=128, init_layers=init, device=0)
        t_gate, t_static = mk(1), mk(D)
        tree = t_gate.alloc_tree(1)
        root = torch.zeros(1, dtype=torch.int32, device=dev)
        plen = torch.zeros(1, dtype=torch.int32, device=dev)
        draft = torch.zeros(1, N, V, dtype=torch.float32, device=dev)
        for alpha in (0.7, 1.35, 5.0):
            for i in range(K + 1):                    # the root's row and the rows of its K children
                draft[0, i] = synth.zipf_logits_row(V, alpha, args.seed, i, device=dev)
            mean, best, rows, added = timed_layer(t_gate, tree, root, plen, draft)
            s_mean, s_best, s_rows, s_added = timed_layer(t_static, tree, root, plen, draft)
            results.append({"vocab": V, "alpha": alpha, "frontier_rows": rows, "talon_nodes_added": added,
                            "talon_us_mean": mean, "talon_us_min": best, "static_nodes_added": s_added,
                            "static_us_mean": s_mean, "static_us_min": s_best, "static_over_talon": s_mean / mean,
                            "algorithmic_gbs": 4.0 * V * rows / (mean * 1e-6) / 1e9})
        t_gate.close()
        t_static.close()
    print(json.dumps({"metric": "single-layer tree-expansion latency (Zipf rows, warm caches)", "unit": "us",
                      "higher_is_better": False, "n_gpus": 1, "data": "synthetic",
                      "config": {"workload": "batch 1, budget 60, K 10, frontier = the root's children; "
                                             "20 warm-up runs, mean of 100, events around the launch; gated layer "
                                             "(Algorithm 2) and dual Top-K layer (Algorithm 1) on the same fused kernel"},
                      "paper": "Talon 1.18x-1.44x faster than the dual Top-K layer (one H200, PyTorch ops: two sorts "
                               "against masking + nonzero); context, not the target",
                      "peak_hbm_gbs": peaks["hbm_gbs"], "results": results}))
    return 0


def main(argv=None):
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=None)
    ap.add_argument("--warmup", type=int, default=None)
    ap.add_argument("--impl", choices=["talon", "reference"], default="talon")
    ap.add_argument("--config", default=None,
                    help=f"measure this workload only (default: {HEADLINE} as the headline, the others under 'configs')")
    ap.add_argument("--seed", type=int, default=None)
    ap.add_argument("--sets", type=int, default=None, help="input sets to rotate over (default: enough to defeat L2)")
    ap.add_argument("--no-graph", action="store_true")
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-sampling", action="store_true", help="skip the sampling-verification extra")
    ap.add_argument("--no-sub-configs", action="store_true", help="skip the other workloads")
    ap.add_argument("--no-repeat", action="store_true", help="time the K steps once, however short")
    ap.add_argument("--no-loop", action="store_true", help="skip the multi-step generation-loop extra")
    ap.add_argument("--no-kernel-pass", action="store_true",
                    help="skip the per-kernel timing pass (for profiler captures of the timed steps alone)")
    ap.add_argument("--batch", type=int, default=None,
                    help="override the workload's batch size (smaller captures of the same kernel shapes)")
    ap.add_argument("--zipf-micro", action="store_true",
                    help="instead of the step benchmark: single-layer expansion latency on Zipf rows")
    args = ap.parse_args(argv)
    from paper_2601_07353_b200 import synth
    if args.seed is None:
        args.seed = synth.DEFAULT_SEED
    if args.zipf_micro:
        return run_zipf_micro(args)
    if args.impl == "reference":
        args.steps = 1 if args.steps is None else args.steps
        args.warmup = 0 if args.warmup is None else args.warmup
        return run_reference(args, synth.CONFIGS[args.config or HEADLINE])
    args.steps = 100 if args.steps is None else args.steps
    args.warmup = 5 if args.warmup is None else args.warmup
    return run_talon(args)


if __name__ == "__main__":
    sys.exit(main())
