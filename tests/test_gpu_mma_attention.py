"""The warp-MMA attention kernel, which takes what the tcgen05 one cannot: a scale of zero or less, kv heads that share
one prefix (a head stride of 0, which no tensor map can hold), more than 128 query heads a kv head; with key ranges merged by
the second kernel (few sequences) and without (many)."""
import numpy as np
import pytest
import torch

from oracle import talon_oracle as O
from tests.test_gpu_step_paths import ATT_TOL, DH, Step, _check_tree, _talon

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hq,hkv,scale,shared", [(8, 2, 0.0, False), (8, 2, -0.06, False), (10, 2, -0.05, False), (8, 2, 0.08, True),
                                                 (130, 1, 0.08, False)])
@pytest.mark.parametrize("B", [1, 2, 80])
def test_against_the_oracle(hq, hkv, scale, shared, B):
    V, N, K, D = 600, 34, 6, 4
    prefix = [300, 129][:B] if B < 3 else [70 + b for b in range(B)]
    talon, t = _talon(B, V, N, K, D, hq=hq, hkv=hkv)
    s = Step(t, B, V, N, D, hq, hkv, prefix, 8)
    if shared:
        s.kp, s.vp = s.kp[:, :1].contiguous(), s.vp[:, :1].contiguous()
    token, head = (DH, 0) if shared else (hkv * DH, DH)
    t.reset(s.tree, s.root, s.plen)
    for _ in range(D):
        t.expand_layer(s.tree, s.draft)
    t.build_tree(s.tree)
    s.out.fill_(float("nan"))
    before = t.launch_count()
    t.tree_attention(s.tree, s.q, s.kp, s.vp, s.kt, s.vt, s.start, s.tokens, token, head, s.max_len, scale, s.out)
    blocks = -(-hq // hkv * N // 128) * B * hkv
    assert t.launch_count() - before == (2 if blocks <= 74 else 1)     # 148 SMs: room for two ranges a block, or none
    torch.cuda.synchronize()
    assert t.poll_status() == talon.OK
    # the same arguments on pages are refused, since only the other kernel reads pages
    pages = torch.zeros(4 * talon.PAGE_TOKENS, hkv, DH, dtype=torch.bfloat16, device="cuda")
    table = torch.zeros(B, 4, dtype=torch.int32, device="cuda")
    with pytest.raises(talon.TalonError) as e:
        t.tree_attention_paged(s.tree, s.q, pages, pages, s.kt, s.vt, table, 4, token, head, s.max_len, scale, s.out.clone())
    assert e.value.code == talon.ERR_UNSUPPORTED
    f32 = lambda x: x.float().cpu().numpy()
    at = 0
    for b in range(B):
        L = prefix[b]
        if b < 3 or b == B - 1:
            ref = _check_tree(s.tree, b, s.draft[b].cpu().numpy(), int(s.root[b]), O.Params(N, K, K, 0.03, D), f"[{b}]")
            k, v = (f32(x[at:at + L].expand(L, hkv, DH)) for x in (s.kp, s.vp))
            want = O.tree_attention(f32(s.q[b]), k, v, f32(s.kt[b]), f32(s.vt[b]), ref, scale)
            assert np.abs(f32(s.out[b]) - want).max() <= ATT_TOL
            assert (s.out[b, ref.n_nodes:] == 0).all()
        at += L
    t.close()
