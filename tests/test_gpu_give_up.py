"""A copy that never completes costs the tiles of one CTA, not those of CTAs that have not started: more tiles than fit the
GPU at once, so that the CTA that gives up has others left to take over, in shares of one and of three tiles."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tiles,share,bits_m,bits_v,block", [(6000, 1, 2, 3, 128), (6000, 1, 8, 8, 2048), (30000, 3, 2, 3, 128)])
def test_only_the_giving_up_cta_loses_tiles(tiles, share, bits_m, bits_v, block):
    from paper_2505_00347_b200 import binding as B
    n = 2048 * tiles
    gen = torch.Generator(device="cuda").manual_seed(5)
    p0 = torch.empty(n, device="cuda").normal_(0.0, 0.02, generator=gen)
    g = torch.empty(n, device="cuda").normal_(0.0, 1e-3, generator=gen).bfloat16()
    h = B.hyper(lr=1e-3, beta1=0.5, weight_decay=0.01, seed=4)
    stalled = 3 * share + 1
    got = []
    for hit in (False, True):
        state = B.State(n, bits_m, bits_v, block)
        p = p0.clone()
        B.set_kernel_policy(3)
        try:
            if hit:
                B.debug_stall_copy(stalled)
            B.solo_step(p, g, state, h, 1)
            torch.cuda.synchronize()
        finally:
            B.set_kernel_policy(0)
        assert state.status() == (2 if hit else 0)
        got.append((p.view(tiles, 2048), state.raw_get("codes_m").view(tiles, -1), state.raw_get("codes_v").view(tiles, -1)))
        state.destroy()
    (p_ref, m_ref, v_ref), (p_hit, m_hit, v_hit) = got
    lost = (p_hit == p0.view(tiles, 2048)).all(dim=1)
    assert lost[stalled] and int(lost.sum()) <= 2 * share       # the rest of its share and one share it had asked for
    kept = ~lost
    assert torch.equal(p_hit[kept], p_ref[kept])
    kept, lost = kept.cpu(), lost.cpu()
    assert torch.equal(m_hit[kept], m_ref[kept]) and torch.equal(v_hit[kept], v_ref[kept])
    assert not m_hit[lost].any() and not v_hit[lost].any()      # the zero state they started from
