"""The kernels behind whole steps and behind odd sizes of single calls: the row pass with the growth
kernel (talon_step, talon_loop), the host step's layer by layer copies, wide candidate lists, chunks at the
edges of what stays resident, and the tensor-core attention with one and two query tiles per CTA."""
import math

import numpy as np
import pytest
import torch

from oracle import talon_oracle as O

pytestmark = pytest.mark.gpu

DH = 128
# A score is a sum of log-probabilities, one per level; each carries the fp32 rounding of its row's sum
# of exponentials (relative 2^-24 per addition in chains of at most a few dozen) and of the maximum's
# exponentials: some 1e-6 a level, below 2e-5 at the depths used here.
SCORE_TOL = 2e-5
# bf16 outputs of order one, P rounded to bf16 before P.V: 2^-9 relative each, summed over keys.
ATT_TOL = 1e-2


def _talon(B, V, N, K, D, cand=None, hq=8, hkv=2, **kw):
    from paper_2601_07353_b200 import talon
    return talon, talon.Talon(batch_max=B, vocab=V, budget=N, root_topk=K, cand_topk=K if cand is None else cand, max_depth=D,
                              n_q_heads=hq, n_kv_heads=hkv, head_dim=DH, mu=0.03, **kw)


def _rows(gen, *shape, spread=4.0):
    """Logit rows with a stride of whole 16-byte units; NaN in the padding."""
    V = shape[-1]
    x = torch.full((*shape[:-1], (V + 3) // 4 * 4), float("nan"), device="cuda")
    x[..., :V] = torch.randn(*shape, device="cuda", generator=gen) * spread
    return x[..., :V]


def _bf16(gen, *shape):
    return torch.randn(*shape, device="cuda", generator=gen).to(torch.bfloat16)


class Step:
    """Random inputs of one step (or S steps of a loop) and room for its results."""

    def __init__(self, t, B, V, N, D, hq, hkv, prefix, seed, steps=None):
        gen = torch.Generator(device="cuda").manual_seed(seed)
        lead = () if steps is None else (steps,)
        room = 0 if steps is None else steps * (D + 1)
        i32 = dict(dtype=torch.int32, device="cuda")
        self.B, self.D, self.hkv, self.prefix = B, D, hkv, prefix
        self.draft, self.target = _rows(gen, *lead, B, N, V), _rows(gen, *lead, B, N, V)
        self.q, self.kt, self.vt = _bf16(gen, *lead, B, N, hq, DH), _bf16(gen, *lead, B, N, hkv, DH), _bf16(gen, *lead, B, N, hkv, DH)
        self.tokens = sum(p + room for p in prefix)
        self.kp, self.vp = _bf16(gen, max(self.tokens, 1), hkv, DH), _bf16(gen, max(self.tokens, 1), hkv, DH)
        ends = np.cumsum([p + room for p in prefix])
        self.start = torch.tensor([0, *ends[:-1]], dtype=torch.int64, device="cuda")
        self.limit = torch.tensor(ends, dtype=torch.int64, device="cuda")
        self.plen = torch.tensor(prefix, **i32)
        self.root = torch.randint(0, V, (B,), device="cuda", generator=gen).to(torch.int32)
        self.max_len = max(prefix) + room
        self.tree = t.alloc_tree(B)
        self.out = torch.zeros(B, N, hq, DH, dtype=torch.bfloat16, device="cuda")
        self.tok = torch.zeros(B, N, **i32)
        self.alen, self.bonus = torch.zeros(*lead, B, **i32), torch.zeros(*lead, B, **i32)
        self.anodes = torch.zeros(*lead, B, D + 1, **i32)
        self.counters = torch.zeros(B, 3, dtype=torch.int64, device="cuda")

    def calls(self, t):
        t.reset(self.tree, self.root, self.plen)
        for _ in range(self.D):
            t.expand_layer(self.tree, self.draft)
        t.build_tree(self.tree)
        t.tree_attention(self.tree, self.q, self.kp, self.vp, self.kt, self.vt, self.start, self.tokens, self.hkv * DH, DH,
                         self.max_len, 1 / math.sqrt(DH), self.out)
        t.accept(self.tree, self.target, self.alen, self.anodes, self.bonus, self.tok)

    def step(self, t):
        t.step(self.tree, self.root, self.plen, self.draft, self.D, self.q, self.kp, self.vp, self.kt, self.vt, self.start,
               self.tokens, self.hkv * DH, DH, self.max_len, 1 / math.sqrt(DH), self.out, self.target, self.tok, self.alen,
               self.anodes, self.bonus)

    def whole(self):
        tr = self.tree
        return [x.clone() for x in (tr.n_nodes, tr.token, tr.parent, tr.depth, tr.position, tr.layer_off, tr.mask, self.tok,
                                    self.alen, self.anodes, self.bonus)]


def _check_tree(tree, b, draft, root, p, label):
    """The oracle's tree on rows given by node."""
    ref = O.new_tree(root, p.budget, p.max_depth)
    while O.is_active(ref):
        O.expand_layer(ref, [draft[i] for i in ref.frontier], p)
    n = ref.n_nodes
    assert int(tree.n_nodes[b]) == n, label
    assert (tree.token[b, :n].cpu().numpy() == ref.token[:n]).all() and (tree.parent[b, :n].cpu().numpy() == ref.parent[:n]).all(), label
    assert np.abs(tree.score[b, :n].cpu().numpy() - ref.score[:n]).max() <= SCORE_TOL, label
    return ref


# (sequences, vocabulary, budget, K): budgets around one and two mask words, lists of 8, 16 and 32 keys,
# rows one short of and one past whole tiles, a vocabulary of several arg-max chunks, batches around 32
STEPS = [(1, 4096, 2, 1), (1, 4097, 33, 8), (3, 8191, 34, 9), (2, 4095, 65, 16), (1, 12289, 128, 17), (2, 5000, 128, 32),
         (33, 1003, 24, 8), (32, 1000, 24, 8), (1, 140001, 20, 6)]


@pytest.mark.parametrize("first_rows", ["", "3"])
@pytest.mark.parametrize("B,V,N,K", STEPS)
def test_whole_step_equals_single_calls_and_the_oracle(B, V, N, K, first_rows, monkeypatch):
    if first_rows:
        if N < 33 or B > 3:
            pytest.skip("two rounds of the row pass: a few shapes")
        monkeypatch.setenv("TALON_STEP_FIRST_ROWS", first_rows)       # read when the context is made
    D = 5
    talon, t = _talon(B, V, N, K, D)
    s = Step(t, B, V, N, D, 8, 2, [37 + 11 * (b % 40) for b in range(B)], 100 + V + N)
    s.calls(t)
    torch.cuda.synchronize()
    want, score, out = s.whole(), s.tree.score.clone(), s.out.clone()
    p = O.Params(N, K, K, 0.03, D)
    for b in range(min(B, 2)):
        _check_tree(s.tree, b, s.draft[b].cpu().numpy(), int(s.root[b]), p, f"calls [{b}]")
    for x in (s.tree.token, s.out, s.tok, s.alen, s.anodes):
        x.zero_()
    for call in range(3):
        s.step(t)
        torch.cuda.synchronize()
        assert t.poll_status() == talon.OK
        for a, g in zip(want, s.whole()):
            assert torch.equal(a, g), f"call {call}"
        for b in range(B):
            n = int(want[0][b])
            assert (s.tree.score[b, :n] - score[b, :n]).abs().max() <= SCORE_TOL
            assert torch.equal(s.tok[b, :n].long(), s.target[b, :n].argmax(-1))
        assert (s.out.float() - out.float()).abs().max() <= ATT_TOL
    t.close()


@pytest.mark.parametrize("bad", [[(1, 0)], [(0, 0), (2, 3)], [(1, 6)]])
def test_rows_that_are_not_finite_in_a_whole_step(bad):
    """A NaN row counts only if the tree reaches it: the same trees and the same status as single calls."""
    B, V, N, K, D = 3, 3001, 30, 6, 4
    talon, t = _talon(B, V, N, K, D)
    s = Step(t, B, V, N, D, 8, 2, [50, 0, 130], 7)
    for b, row in bad:
        s.draft[b, row, 17] = float("nan")
    s.calls(t)
    torch.cuda.synchronize()
    status, want = t.poll_status(), s.whole()[:6]
    assert status != talon.OK
    s.step(t)
    torch.cuda.synchronize()
    assert t.poll_status() == status
    for a, g in zip(want, s.whole()):
        assert torch.equal(a, g)
    t.close()


def test_loop_longer_than_the_rows_prepared_at_once():
    """Eleven steps in one call (rows are prepared eight steps at a time) against eleven calls of one."""
    B, V, N, K, D, S = 2, 2003, 20, 5, 4, 11
    talon, t = _talon(B, V, N, K, D)

    def loop(s, first, n):
        at = slice(first, first + n)
        t.loop(s.tree, n, s.root, s.plen, s.draft[at], D, s.q[at], s.kp, s.vp, s.kt[at], s.vt[at], s.start, s.limit, s.tokens,
               s.hkv * DH, DH, s.max_len, 1 / math.sqrt(DH), s.out, s.target[at], s.tok, s.alen[at], s.anodes[at], s.bonus[at],
               s.counters)

    res = []
    for calls in ([S], [1] * S):
        s = Step(t, B, V, N, D, 8, 2, [90, 33], 21, steps=S)
        at = 0
        for n in calls:
            loop(s, at, n)
            at += n
        torch.cuda.synchronize()
        assert t.poll_status() == talon.OK
        res.append(s)
    a, b = res
    for x, y in zip(a.whole() + [a.plen, a.root, a.counters, a.kp, a.vp], b.whole() + [b.plen, b.root, b.counters, b.kp, b.vp]):
        assert torch.equal(x, y)
    assert (a.out.float() - b.out.float()).abs().max() <= ATT_TOL
    t.close()


@pytest.mark.parametrize("B,K,N", [(3, 8, 40), (2, 40, 50), (1, 16, 128)])
def test_host_step_copies_every_row_the_tree_reads(B, K, N):
    """Rows are fetched as the tree grows, for lists of any length."""
    V, D = 3001, 5
    talon, t = _talon(B, V, N, K, D)
    s = Step(t, B, V, N, D, 8, 2, [70 + 50 * b for b in range(B)], 5)
    s.draft, s.target = s.draft.contiguous()[..., :3000].contiguous(), s.target[..., :3000].contiguous()
    t.close()
    talon, t = _talon(B, 3000, N, K, D)
    s.tree = t.alloc_tree(B)
    s.root %= 3000
    s.calls(t)
    torch.cuda.synchronize()
    pin = lambda x: x.cpu().contiguous().pin_memory()
    z = lambda *shape: torch.zeros(*shape, dtype=torch.int32).pin_memory()
    out, n_nodes, token, parent = pin(torch.zeros_like(s.out)), z(B), z(B, N), z(B, N)
    depth, position, alen, anodes, bonus = z(B, N), z(B, N), z(B), z(B, D + 1), z(B)
    for _ in range(2):
        st = t.step_host(pin(s.root), pin(s.plen), pin(s.draft), pin(s.target), pin(s.q), pin(s.kp), pin(s.vp), pin(s.kt),
                         pin(s.vt), 1 / math.sqrt(DH), out, n_nodes, token, parent, depth, position, alen, anodes, bonus)
        assert st == talon.OK
        for got, want in ((n_nodes, s.tree.n_nodes), (token, s.tree.token), (parent, s.tree.parent), (depth, s.tree.depth),
                          (position, s.tree.position), (alen, s.alen), (anodes, s.anodes), (bonus, s.bonus)):
            assert torch.equal(got, want.cpu())
        assert (out.float() - s.out.cpu().float()).abs().max() <= ATT_TOL
    t.close()


@pytest.mark.parametrize("kind", ["random", "two_values", "plateau"])
@pytest.mark.parametrize("K", [33, 64, 65, 127])
def test_wide_lists(K, kind):
    """Lists past 32 keys: register merges of two lists a warp and of many, ties at the bound."""
    B, V, N, D = 2, 9001, 128, 3
    talon, t = _talon(B, V, N, 8, D, cand=K)
    gen = torch.Generator(device="cuda").manual_seed(K)
    draft = _rows(gen, B, N, V)
    if kind != "random":
        i = torch.arange(V, device="cuda")
        row = (i % 2).float() if kind == "two_values" else torch.where((i * 71) % 113 == 0, 3.0, -1.0 - (i % 97) * 1e-2)
        draft[:] = row
    root, plen = torch.zeros(B, dtype=torch.int32, device="cuda"), torch.zeros(B, dtype=torch.int32, device="cuda")
    tree = t.alloc_tree(B)
    t.reset(tree, root, plen)
    for _ in range(D):
        t.expand_layer(tree, draft)
    t.build_tree(tree)
    torch.cuda.synchronize()
    assert t.poll_status() == talon.OK
    for b in range(B):
        _check_tree(tree, b, draft[b].cpu().numpy(), 0, O.Params(N, 8, K, 0.03, D), f"{kind} K={K} [{b}]")
    t.close()


# a chunk is resident when every warp's slice fits its ring of three 512-element tiles: 8 x 1536 elements;
# the last shape is above the size from which the kernel asks L2 for rows ahead
@pytest.mark.parametrize("B,V", [(2, 511), (2, 513), (2, 4096), (2, 12287), (2, 12288), (2, 12289), (2, 24580), (30, 12292)])
@pytest.mark.parametrize("K,split", [(8, "1"), (16, "32"), (20, "3")])
def test_chunks_around_the_resident_size(B, V, K, split, monkeypatch):
    monkeypatch.setenv("TALON_EXPAND_MAX_SPLIT", split)               # read when the context is made
    from paper_2601_07353_b200.talon import ROWS_BY_NODE, ROWS_PACKED
    N, D = 2 * K + 3, 4
    talon, t = _talon(B, V, N, K, D)
    draft = _rows(torch.Generator(device="cuda").manual_seed(V + K), B, N, V)
    root, plen = torch.zeros(B, dtype=torch.int32, device="cuda"), torch.zeros(B, dtype=torch.int32, device="cuda")
    by_node, packed = t.alloc_tree(B), t.alloc_tree(B)
    t.reset(by_node, root, plen)
    for _ in range(D):
        t.expand_layer(by_node, draft, layout=ROWS_BY_NODE)
    t.build_tree(by_node)
    off = by_node.layer_off.cpu().numpy()
    t.reset(packed, root, plen)
    for d in range(D):
        rows = torch.zeros_like(draft)
        for b in range(B):
            lo, hi = off[b, d], off[b, d + 1]
            if hi > lo:
                rows[b, :hi - lo] = draft[b, lo:hi]
        pad = torch.full((B, N, (V + 3) // 4 * 4), float("nan"), device="cuda")
        pad[..., :V] = rows
        t.expand_layer(packed, pad[..., :V], rows_per_seq=N, layout=ROWS_PACKED)
    t.build_tree(packed)
    torch.cuda.synchronize()
    assert t.poll_status() == talon.OK
    for x, y in ((by_node.token, packed.token), (by_node.parent, packed.parent), (by_node.score, packed.score)):
        assert torch.equal(x, y)
    for b in range(min(B, 2)):
        _check_tree(by_node, b, draft[b].cpu().numpy(), 0, O.Params(N, K, K, 0.03, D), f"V={V} K={K} [{b}]")
    t.close()


# budgets of one, two and three query tiles of whole nodes; key ranges that divide, that do not, and more
# of them than there are key tiles (empty ranges)
@pytest.mark.parametrize("hq,hkv,N", [(8, 2, 30), (8, 2, 40), (8, 2, 70), (12, 2, 50), (14, 2, 40), (32, 1, 9)])
@pytest.mark.parametrize("tiles,splits", [("0", "0"), ("1", "1"), ("1", "2"), ("1", "3"), ("1", "4"), ("1", "7"), ("2", "1"),
                                          ("2", "2"), ("2", "5"), ("2", "8"), ("1", "9")])
def test_attention_query_tiles_and_key_ranges(hq, hkv, N, tiles, splits, monkeypatch):
    monkeypatch.setenv("TALON_ATTN_TILES", tiles)                     # read when the context is made
    monkeypatch.setenv("TALON_ATTN_SPLITS", splits)
    B, V, K, D, prefix = 3, 600, 6, 5, [700, 0, 385]
    talon, t = _talon(B, V, N, K, D, hq=hq, hkv=hkv)
    s = Step(t, B, V, N, D, hq, hkv, prefix, 3 + N)
    s.out.fill_(float("nan"))
    s.calls(t)
    torch.cuda.synchronize()
    assert t.poll_status() == talon.OK
    one = s.out.clone()
    s.step(t)                                                         # started on the prefix beside the growth
    torch.cuda.synchronize()
    assert t.poll_status() == talon.OK
    f32 = lambda x: x.float().cpu().numpy()
    at = 0
    for b in range(B):
        ref = _check_tree(s.tree, b, s.draft[b].cpu().numpy(), int(s.root[b]), O.Params(N, K, K, 0.03, D), f"[{b}]")
        L = prefix[b]
        want = O.tree_attention(f32(s.q[b]), f32(s.kp[at:at + L]), f32(s.vp[at:at + L]), f32(s.kt[b]), f32(s.vt[b]), ref, 1 / math.sqrt(DH))
        at += L
        for got in (one[b], s.out[b]):
            assert np.abs(f32(got) - want).max() <= ATT_TOL
            assert (got[ref.n_nodes:] == 0).all()
    t.close()
