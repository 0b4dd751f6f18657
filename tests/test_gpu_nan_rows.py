"""A NaN in a draft row is found wherever it sits: alone in a warp's slice, among masked (-inf) tokens, a whole tile of it."""
import pytest
import torch

from tests.test_gpu_step_paths import Step, _talon

pytestmark = pytest.mark.gpu

BLOCK = range(512, 1024)
# vocabulary, tokens that hold NaN, whether everything else but two tokens is masked; one chunk a row or many
ROWS = [(513, [512], False), (512, [0], True), (4096, [100], True), (4096, BLOCK, False), (24581, [24580], False),
        (24580, [20000], True), (24580, range(3073, 3585), False)]


@pytest.mark.parametrize("V,at,masked", ROWS)
@pytest.mark.parametrize("K,cand", [(4, 4), (12, 12), (20, 20), (4, 40)])
@pytest.mark.parametrize("split", ["1", "32"])
def test_a_nan_is_found_wherever_it_sits(V, at, masked, K, cand, split, monkeypatch):
    monkeypatch.setenv("TALON_EXPAND_MAX_SPLIT", split)               # read when the context is made
    B, N, D = 2, 50, 3
    talon, t = _talon(B, V, N, K, D, cand=cand)
    s = Step(t, B, V, N, D, 8, 2, [70, 120], 5)
    if masked:
        keep = s.draft[1, 0, 7:9].clone()
        s.draft[1, 0] = float("-inf")
        s.draft[1, 0, 7:9] = keep
    s.draft[1, 0, list(at)] = float("nan")
    for run in (s.calls, s.step):
        run(t)
        torch.cuda.synchronize()
        assert t.poll_status() == talon.ERR_NONFINITE
        assert s.tree.n_nodes.tolist()[1] == 1 and s.tree.n_nodes.tolist()[0] > 1
    t.close()
