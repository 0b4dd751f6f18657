"""The attention with one query tile a CTA for every shape, as where the kernel for two cannot have its registers."""
import pytest
import torch

from tests.test_gpu_step_paths import ATT_TOL, Step, _talon

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,N,hq,hkv,L", [(1, 60, 32, 8, 700), (40, 60, 32, 8, 300), (24, 128, 16, 2, 5000), (3, 16, 8, 2, 0)])
def test_one_query_tile_a_cta_gives_what_two_give(B, N, hq, hkv, L, monkeypatch):
    outs = []
    for tiles in ("0", "1"):
        monkeypatch.setenv("TALON_ATTN_TILES", tiles)    # read when the context is made
        talon, t = _talon(B, 2000, N, 8, 5, hq=hq, hkv=hkv)
        s = Step(t, B, 2000, N, 5, hq, hkv, [L] * B, 4)
        s.out.fill_(float("nan"))
        s.step(t)
        torch.cuda.synchronize()
        assert t.poll_status() == talon.OK
        outs.append(s.out.float())
        t.close()
    assert (outs[0] - outs[1]).abs().max() <= ATT_TOL
