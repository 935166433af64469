"""A tile whose elements lie on both sides of a change of the stream position's high word (element 2^35 of a tensor, reached by a
shard of a larger tensor), directly before and behind it.  Blocks of 128 and 256: the sixteen-per-thread kernel computes what the
counters have in common once per tile, for the high word and for the one after; blocks of 2048 too, but a tile of theirs begins at
a multiple of its size and so never lies on both sides.  Blocks of 64, and bf16 parameters with modes that are read from the
arguments: every counter as it is, like the general kernel's."""
import pytest
import torch

pytestmark = pytest.mark.gpu

KEYS = ("codes_m", "codes_v", "scale_m", "scale_v", "alpha")


@pytest.mark.parametrize("hk", [dict(round_m=1), dict(param_dtype=1, param_round=1), dict(v_codebook=1, param_dtype=1, param_round=1),
                                dict(fixed_alpha=0.5, param_dtype=1, param_round=1), dict(belief=1)])
@pytest.mark.parametrize("bits_m,bits_v,block,before",       # `before`: elements before element 2^35
                         [(2, 3, 64, b) for b in (0, 64, 1024, 2048 + 192, 4096)] + [(8, 8, 64, b) for b in (0, 64, 1024, 2048 + 192, 4096)] +
                         [(2, 3, 128, b) for b in (0, 128, 1024, 2048 + 256, 4096)] + [(8, 8, 128, b) for b in (128, 4096 + 1920)] +
                         [(4, 4, 256, b) for b in (256, 1024, 2048 + 1792)] + [(4, 4, 2048, b) for b in (0, 2048, 4096)])
def test_high_word_of_the_stream_position(bits_m, bits_v, block, before, hk):
    from paper_2505_00347_b200 import binding as B
    n = 2048 * 5
    gen = torch.Generator().manual_seed(3)
    g = torch.randn(n, generator=gen).mul(1e-3).bfloat16().cuda()
    dt = torch.bfloat16 if hk.get("param_dtype") else torch.float32
    p0 = torch.randn(n, generator=gen).mul(0.02).to(dt)
    h = B.hyper(lr=1e-3, beta1=0.5, weight_decay=0.01, seed=11, **hk)
    got = []
    for policy in (1, 3):
        p = p0.cuda()
        state = B.State(n, bits_m, bits_v, block)
        state.set_origin([5], [2 ** 35 - before])
        B.set_kernel_policy(policy)
        try:
            for t in (1, 2):
                B.solo_step(p, g, state, h, t)
        finally:
            B.set_kernel_policy(0)
        got.append([state.raw_get(k) for k in KEYS] + ([p.view(torch.int16).cpu()] if dt == torch.bfloat16 else []))
        assert state.status() == 0
        state.destroy()
    for a, b in zip(*got):
        assert torch.equal(a, b)
