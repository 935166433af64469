"""The launch for the tiles that the sixteen-per-thread kernel leaves: every tensor's tail once, tensors that are not
16-byte aligned whole (dealt to one CTA up to sixteen tiles, shared by all beyond), more tensors than one group of
the walk, a descriptor mismatch reported.  Compared with the one-launch kernels on the same inputs, bit for bit."""
import pytest
import torch

from paper_2505_00347_b200 import synth

pytestmark = pytest.mark.gpu

KEYS = ("codes_m", "codes_v", "scale_m", "scale_v", "alpha")


def _views(sizes, offsets, dtype, make):
    out = []
    for i, (n, o) in enumerate(zip(sizes, offsets)):
        buf = torch.zeros(n + 16, dtype=dtype, device="cuda")
        buf[o:o + n] = make(i).cuda()
        out.append(buf[o:o + n])
    return out


@pytest.mark.parametrize("hk,one_launch", [(dict(), 2), (dict(round_m=1), 1), (dict(param_dtype=1, param_round=1), 2)])
@pytest.mark.parametrize("bits_m,bits_v,block", [(2, 3, 128), (8, 8, 64), (4, 4, 256)])
def test_every_remaining_tile_is_stepped_once(bits_m, bits_v, block, hk, one_launch):
    from paper_2505_00347_b200 import binding as B
    sizes = [2048 * 40 + 5, 2048 * 16, 2048 * 17, 3, 2048, 2049] + [100 + 7 * i for i in range(600)] + [2048 * 33, 2048 * 3 + 1]
    offsets = [1, 1, 0, 1, 0, 0] + [(i % 3 == 0) * 2 for i in range(600)] + [3, 0]
    w = synth.workload(3, sizes=tuple(sizes))
    dt = torch.bfloat16 if hk.get("param_dtype") else torch.float32
    grads = _views(sizes, offsets, torch.bfloat16, lambda i: synth.make_grad(w, i, 1))
    h = B.hyper(lr=1e-3, beta1=0.5, weight_decay=0.01, seed=3, **hk)
    got = {}
    for policy in (3, one_launch):
        params = _views(sizes, offsets, dt, lambda i: synth.make_param(w, i, dtype=dt))
        state = B.State(sizes, bits_m, bits_v, block)
        B.set_kernel_policy(policy)
        try:
            for t in (1, 2):
                B.solo_multi_step(B.TensorSet(params, grads, state), h, t)
            torch.cuda.synchronize()
        finally:
            B.set_kernel_policy(0)
        assert state.status() == 0
        got[policy] = [state.raw_get(k).clone() for k in KEYS] + [p.float().cpu() for p in params]
        state.destroy()
    for a, b in zip(got[3], got[one_launch]):
        if a.dtype == torch.float32 and one_launch == 1 and a.numel() in sizes:
            assert torch.allclose(a, b, rtol=1e-6, atol=1e-8)       # IEEE division in the general kernel: 3e-7 of lr
        else:
            assert torch.equal(a, b)


def test_mismatched_descriptor_is_reported_without_tails():
    """A list whose tensors all end on a tile has no tile left for the second launch, which still checks its sizes."""
    from paper_2505_00347_b200 import binding as B
    sizes = [2048 * 4, 2048 * 2]
    params = [torch.zeros(n, device="cuda") for n in sizes]
    grads = [torch.ones(n, device="cuda", dtype=torch.bfloat16) for n in sizes]
    state = B.State(sizes, 2, 3, 128)
    ts = B.TensorSet(params, grads, state)
    ts.numel[1] = 2048
    B.set_kernel_policy(3)
    try:
        B.solo_multi_step(ts, B.hyper(), 1)
        torch.cuda.synchronize()
    finally:
        B.set_kernel_policy(0)
    assert state.status() == 1
    assert bool((params[0] != 0).all()) and not bool(params[1].any())
    state.destroy()
