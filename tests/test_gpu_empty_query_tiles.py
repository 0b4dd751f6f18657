"""Trees that leave whole query tiles of the attention without a node, at the edges of those tiles: the nodes' rows are right and every
other row is zero, with one range of keys, with ranges merged in a cluster and with ranges merged by the second kernel."""
import pytest
import torch

from tests.test_gpu_attention_precision import _error
from tests.test_gpu_step_paths import Step, _talon

pytestmark = pytest.mark.gpu


# 32 nodes a query tile at four query heads a kv head, 25 at five; (sequences, prefix): ranges in a cluster, one range, an
# attention long enough to wait for the trees
@pytest.mark.parametrize("B,L,cluster", [(1, 2000, "1"), (1, 2000, "0"), (20, 300, "1"), (3, 90000, "1")])
@pytest.mark.parametrize("N,hq,sizes", [(128, 32, (1, 31, 32, 33, 64, 65, 96, 97, 128)), (96, 32, (2, 33, 64, 95)), (60, 40, (1, 25, 26, 50, 51))])
def test_tiles_without_nodes(N, hq, sizes, B, L, cluster, monkeypatch):
    monkeypatch.setenv("TALON_ATTN_CLUSTER", cluster)
    V, D = 1000, 40
    talon, t = _talon(B, V, N, 8, D, hq=hq, hkv=8)
    s = Step(t, B, V, N, D, hq, 8, [L] * B, 31)
    for size in sizes:
        # a tree of that many nodes: as the library grows it, cut to its first nodes (parents come first)
        t.reset(s.tree, s.root, s.plen)
        for _ in range(D):
            t.expand_layer(s.tree, s.draft)
        assert int(s.tree.n_nodes.min()) >= min(size, N)
        s.tree.n_nodes.fill_(size)
        t.build_tree(s.tree)
        s.out.fill_(float("nan"))
        t.tree_attention(s.tree, s.q, s.kp, s.vp, s.kt, s.vt, s.start, s.tokens, 8 * 128, 128, s.max_len, 128 ** -0.5, s.out)
        torch.cuda.synchronize()
        assert (s.out[:, size:] == 0).all()
        if L < 10000:
            assert _error(s, hq, 8) <= 2.35e-3                # as test_gpu_attention_precision: 2.33e-3 with 2^8 of slack
    # whole steps: the same rows, whatever was known of the tree at the start
    s.calls(t)
    torch.cuda.synchronize()
    want, n = s.out.clone(), s.tree.n_nodes.clone()
    s.out.fill_(float("nan"))
    s.step(t)
    torch.cuda.synchronize()
    assert torch.equal(n, s.tree.n_nodes)
    assert (s.out.float() - want.float()).abs().max() <= 1e-2
    assert t.poll_status() == talon.OK
    t.close()
