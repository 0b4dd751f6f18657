"""Verification of a tree that the caller built, not the library."""
import pytest
import torch

from oracle import talon_oracle as O
from tests import parity_util as PU
from tests.test_gpu_step_paths import Step, _talon

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B", [1, 40])                   # the walk folded into the arg-max, and a kernel of its own
def test_the_first_of_several_siblings_with_the_same_token_is_accepted(B):
    V, N, D = 2000, 70, 4
    talon, t = _talon(B, V, N, 5, D)
    s = Step(t, B, V, N, D, 8, 2, [70] * B, 5)
    s.calls(t)                                           # (sets the batch; the tree is replaced)
    tr = s.tree
    choice = s.target.argmax(-1).int()
    # 66 children of the root that all carry the target's choice, then a child of the first and of the last of them
    tr.n_nodes[:] = 69
    tr.token[:, 1:67], tr.parent[:, 1:67], tr.depth[:, 1:67] = choice[:, :1], 0, 1
    for node, parent in ((67, 1), (68, 66)):
        tr.token[:, node], tr.parent[:, node], tr.depth[:, node] = choice[:, parent], parent, 2
    tr.layer_off[:] = torch.tensor([0, 1, 67, 69, 69, 69], dtype=torch.int32, device="cuda")
    t.accept(tr, s.target, s.alen, s.anodes, s.bonus, s.tok)
    torch.cuda.synchronize()
    for b in range(B):
        ref = PU.oracle_tree_from_arrays(PU.tree_to_host(tr, b), N, D)
        alen, path, bonus = O.accept(ref, O.target_argmax(s.target[b].cpu().numpy(), 69))
        assert path == [0, 1, 67]
        assert (int(s.alen[b]), s.anodes[b, :3].tolist(), int(s.bonus[b])) == (alen, path, bonus)
    t.close()
