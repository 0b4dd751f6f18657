"""What one call leaves behind for the next one, and what a call has to wait for."""
import math

import pytest
import torch

from tests.test_gpu_step_paths import ATT_TOL, DH, Step, _talon

pytestmark = pytest.mark.gpu


def _loop(t, s, n, **other):
    """The first n steps of s as one call; `other` replaces arguments."""
    a = dict(q=s.q, kp=s.kp, vp=s.vp, tokens=s.tokens, stride=s.hkv * DH, max_len=s.max_len, scale=1 / math.sqrt(DH))
    a.update(other)
    t.loop(s.tree, n, s.root, s.plen, s.draft, s.D, a["q"], a["kp"], a["vp"], s.kt, s.vt, s.start, s.limit, a["tokens"],
           a["stride"], DH, a["max_len"], a["scale"], s.out, s.target, s.tok, s.alen, s.anodes, s.bonus, s.counters)


def _results(s):
    return s.whole() + [s.plen, s.root, s.counters, s.kp, s.vp]


# what the attention refuses, and (no prefix, no cache) what only the commit refuses
REFUSALS = [dict(max_len=1 << 20), dict(scale=float("nan")), dict(stride=2 * DH + 1), dict(q="misaligned"),
            dict(kp=None, vp=None, max_len=0)]


def _other(s, refusal):
    r = dict(refusal)
    if r.get("q") == "misaligned":
        r["q"] = s.q.reshape(-1)[1:].as_strided(s.q.shape, s.q.stride())
    return r


@pytest.mark.parametrize("refusal", REFUSALS)
def test_a_refused_loop_enqueues_nothing_and_leaves_nothing(refusal):
    B, V, N, K, D, S = 2, 2003, 20, 5, 4, 6
    talon, t = _talon(B, V, N, K, D)
    shape = (t, B, V, N, D, 8, 2, [0, 0] if "kp" in refusal else [90, 33])
    s = Step(*shape, 3, steps=S)
    s.q = torch.cat([s.q.reshape(-1), s.q.new_zeros(8)])[:s.q.numel()].view(s.q.shape)     # (room for the shifted view)
    s.target += 50.0                                     # larger than any row of the loop that follows
    s.target[:, :, 1, 7] = float("nan")
    before, launches = [x.clone() for x in _results(s)], t.launch_count()
    with pytest.raises(talon.TalonError) as e:
        _loop(t, s, S, **_other(s, refusal))
    assert e.value.code == talon.ERR_INVALID_ARG
    assert t.launch_count() == launches
    torch.cuda.synchronize()
    for x, y in zip(before, _results(s)):
        assert torch.equal(x, y)
    good, ref = Step(*shape, 4, steps=S), Step(*shape, 4, steps=S)
    _loop(t, good, S)
    talon, fresh = _talon(B, V, N, K, D)
    _loop(fresh, ref, S)
    torch.cuda.synchronize()
    assert t.poll_status() == fresh.poll_status() == talon.OK
    for x, y in zip(_results(good), _results(ref)):
        assert torch.equal(x, y)
    t.close()
    fresh.close()


@pytest.mark.parametrize("refusal", REFUSALS[:4])
def test_a_refused_step_enqueues_nothing(refusal):
    B, V, N, K, D = 2, 2003, 20, 5, 4
    talon, t = _talon(B, V, N, K, D)
    s = Step(t, B, V, N, D, 8, 2, [90, 33], 3)
    s.q = torch.cat([s.q.reshape(-1), s.q.new_zeros(8)])[:s.q.numel()].view(s.q.shape)
    a = dict(q=s.q, tokens=s.tokens, stride=s.hkv * DH, max_len=s.max_len, scale=1 / math.sqrt(DH))
    a.update(_other(s, refusal))
    before, launches = s.whole(), t.launch_count()
    with pytest.raises(talon.TalonError) as e:
        t.step(s.tree, s.root, s.plen, s.draft, D, a["q"], s.kp, s.vp, s.kt, s.vt, s.start, a["tokens"], a["stride"], DH,
               a["max_len"], a["scale"], s.out, s.target, s.tok, s.alen, s.anodes, s.bonus)
    assert e.value.code == talon.ERR_INVALID_ARG
    assert t.launch_count() == launches
    torch.cuda.synchronize()
    for x, y in zip(before, s.whole()):
        assert torch.equal(x, y)
    t.close()


def test_a_loop_that_fails_after_its_first_launch_leaves_nothing():
    """A token stride that no tensor map can hold is only found when the attention is launched."""
    B, V, N, K, D, S = 2, 2003, 20, 5, 4, 6
    talon, t = _talon(B, V, N, K, D)
    shape = (t, B, V, N, D, 8, 2, [90, 33])
    s = Step(*shape, 3, steps=S)
    s.target += 50.0
    s.target[:, :, 1, 7] = float("nan")
    with pytest.raises(talon.TalonError) as e:
        _loop(t, s, S, stride=1 << 40)
    assert e.value.code == talon.ERR_CUDA
    good, ref = Step(*shape, 4, steps=S), Step(*shape, 4, steps=S)
    _loop(t, good, S)
    talon, fresh = _talon(B, V, N, K, D)
    _loop(fresh, ref, S)
    torch.cuda.synchronize()
    assert t.poll_status() == fresh.poll_status() == talon.OK
    for x, y in zip(_results(good), _results(ref)):
        assert torch.equal(x, y)
    t.close()
    fresh.close()


@pytest.mark.parametrize("own", [False, True])
def test_a_host_step_follows_what_its_stream_still_has_to_do(own):
    """The pinned inputs are filled by copies that are enqueued, behind 50 ms of other work, but not finished."""
    B, V, N, K, D = 2, 3000, 40, 8, 5
    talon, t = _talon(B, V, N, K, D)
    s = Step(t, B, V, N, D, 8, 2, [70, 120], 5)
    s.draft, s.target = s.draft.contiguous(), s.target.contiguous()
    s.calls(t)
    torch.cuda.synchronize()
    pinned = lambda x: torch.zeros(x.shape, dtype=x.dtype).pin_memory()
    names = ("draft", "target", "q", "kp", "vp", "kt", "vt")
    host = {n: pinned(getattr(s, n)) for n in names}
    res = [pinned(x) for x in (s.out, s.tree.n_nodes, s.tree.token, s.tree.parent, s.tree.depth, s.tree.position, s.alen,
                               s.anodes, s.bonus)]
    root, plen = s.root.cpu(), s.plen.cpu()
    call = lambda: t.step_host(root, plen, *(host[n] for n in names), 1 / math.sqrt(DH), *res)
    assert call() == talon.OK                            # (allocates the staging buffers, which synchronises)
    stream = torch.cuda.Stream() if own else torch.cuda.default_stream()
    with torch.cuda.stream(stream):
        torch.cuda._sleep(100_000_000)
        for n in names:
            host[n].copy_(getattr(s, n), non_blocking=True)
        assert call() == talon.OK
    for got, want in zip(res[1:], (s.tree.n_nodes, s.tree.token, s.tree.parent, s.tree.depth, s.tree.position, s.alen, s.anodes,
                                   s.bonus)):
        assert torch.equal(got, want.cpu())
    assert (res[0].float() - s.out.cpu().float()).abs().max() <= ATT_TOL
    t.close()


# (keys a row, budget, batch) of an older context and of a smaller one that uses the same kernels
@pytest.mark.parametrize("older,newer", [((8, 128, 40), (5, 66, 1)), ((32, 128, 40), (17, 65, 1)), ((60, 128, 40), (33, 40, 1))])
def test_a_smaller_context_does_not_stop_an_older_one(older, newer):
    (k, N, B), (k2, N2, B2), V, D = older, newer, 3001, 4
    talon, t = _talon(B, V, N, 8, D, cand=k)
    s = Step(t, B, V, N, D, 8, 2, [10] * B, 5)
    s.step(t)
    torch.cuda.synchronize()
    want = s.whole()
    talon, other = _talon(B2, V, N2, 8, D, cand=k2)
    for run in (s.step, s.calls):
        run(t)
        torch.cuda.synchronize()
        assert t.poll_status() == talon.OK
        for a, b in zip(want, s.whole()):
            assert torch.equal(a, b)
    other.close()
    t.close()


@pytest.mark.parametrize("where", ["draft", "target"])
@pytest.mark.parametrize("bad", [0, 3, 9, 10])
def test_the_status_after_a_loop_is_the_last_steps(bad, where):
    """Eleven steps, whose rows are prepared eight at a time; a NaN in one of them."""
    B, V, N, K, D, S = 2, 2003, 20, 5, 4, 11
    talon, t = _talon(B, V, N, K, D)
    s = Step(t, B, V, N, D, 8, 2, [90, 33], 3, steps=S)
    getattr(s, where)[bad, 1, 0, 17] = float("nan")
    _loop(t, s, S)
    torch.cuda.synchronize()
    assert t.poll_status() == (talon.ERR_NONFINITE if bad == S - 1 else talon.OK)
    t.close()


def test_a_host_step_whose_staging_does_not_fit_can_be_called_again():
    """Room for 1024 sequences of 16 rows of four million tokens, twice, is more than any device has."""
    V, N, D, B = 1 << 22, 16, 2, 1024
    talon, t = _talon(B, V, N, 4, D)
    row = torch.zeros(1, N, V)
    bf = lambda heads: torch.zeros(1, N, heads, DH, dtype=torch.bfloat16)
    i32 = lambda *shape: torch.zeros(*shape, dtype=torch.int32)
    for _ in range(2):
        assert t.step_host(i32(1), i32(1), row, row, bf(8), None, None, bf(2), bf(2), 0.1, bf(8), i32(1), i32(1, N), i32(1, N), i32(1, N),
                           i32(1, N), i32(1), i32(1, D + 1), i32(1)) == talon.ERR_CUDA
    torch.zeros(8, device="cuda").sum().item()           # nothing is left behind in the CUDA runtime either
    t.close()
