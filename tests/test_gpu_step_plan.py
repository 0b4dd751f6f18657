"""Whole steps over the sizes at which they go in one round, in two, or layer by layer: the same results as single calls."""
import pytest
import torch

from tests.test_gpu_step_paths import ATT_TOL, SCORE_TOL, Step, _talon

pytestmark = pytest.mark.gpu

V = 128256


# (sequences, budget, layers, launches of a step): one round is row pass, growth, attention; two are two of each before the
# attention, then the arg-max (and the walk, where the arg-max does not do it); by layers reset, a launch each, attention, arg-max
@pytest.mark.parametrize("B,N,D,launches", [(8, 60, 6, (3, 4)), (32, 60, 12, (6, 7)), (32, 60, 6, (9, 10)), (20, 128, 24, (3, 4)),
                                            (32, 128, 24, (6, 7))])
@pytest.mark.parametrize("spread", [0.5, 3.0])
def test_a_whole_step_equals_single_calls(B, N, D, launches, spread):
    talon, t = _talon(B, V, N, 8, D)
    s = Step(t, B, V, N, D, 8, 2, [130] * B, 9)
    s.draft *= spread / 4.0                              # flat rows give wide trees, steep ones narrow trees
    s.calls(t)
    torch.cuda.synchronize()
    want, score, out = s.whole(), s.tree.score.clone(), s.out.clone()
    for x in (s.tree.token, s.out, s.tok, s.alen, s.anodes):
        x.zero_()
    before = t.launch_count()
    s.step(t)
    assert t.launch_count() - before in launches
    torch.cuda.synchronize()
    assert t.poll_status() == talon.OK
    for a, g in zip(want, s.whole()):
        assert torch.equal(a, g)
    for b in range(B):
        n = int(want[0][b])
        assert (s.tree.score[b, :n] - score[b, :n]).abs().max() <= SCORE_TOL
    assert (s.out.float() - out.float()).abs().max() <= ATT_TOL
    t.close()
