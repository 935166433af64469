"""bf16 parameters: the update that is taken by approximations and kept only where it rounds to the same pattern from both ends
of its error, against the general kernel's IEEE operations, bit for bit: rates that put many results next to a rounding boundary,
parameters of zero, from 2 up, infinite and NaN, rates of zero and near the smallest number; then first and second moments near
and below the smallest normal number under a small eps."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def _params(kind, n, gen):
    p = torch.randn(n, generator=gen) * 0.02
    if kind == "zero":
        p.zero_()
    elif kind == "large":
        p *= 200.0
    elif kind == "special":
        p[::7] = float("nan")
        p[3::11] = float("inf")
        p[5::13] = -float("inf")
        p[1::17] = 3.0e38
    elif kind == "tiny":
        p *= 2.0 ** -100
    return p.bfloat16()


@pytest.mark.parametrize("sr", [0, 1])
@pytest.mark.parametrize("lr,eps", [(2e-5, 1e-8), (1e-3, 1e-8), (0.3, 1e-8), (0.3, 1e-12), (0.0, 1e-8), (2.0 ** -120, 1e-8), (1e-3, 1.0)])
@pytest.mark.parametrize("kind", ["normal", "zero", "large", "special", "tiny"])
def test_patterns_are_the_ieee_updates(kind, lr, eps, sr):
    from paper_2505_00347_b200 import binding as B
    n = 2048 * 64
    for bits_m, bits_v, block, scale in ((2, 2, 128, 1e-3), (8, 8, 2048, 1e-3), (4, 3, 64, 2.0 ** -64)):
        gen = torch.Generator().manual_seed(21)
        p0 = _params(kind, n, gen)
        grads = [(torch.randn(n, generator=gen) * scale).bfloat16().cuda() for _ in range(3)]
        h = B.hyper(lr=lr, beta1=0.5, eps=eps, weight_decay=0.01, seed=2, param_dtype=1, param_round=sr)
        got = []
        for policy in (1, 3):
            p = p0.cuda()
            state = B.State(n, bits_m, bits_v, block)
            B.set_kernel_policy(policy)
            try:
                for t, g in enumerate(grads, 1):
                    B.solo_step(p, g, state, h, t)
            finally:
                B.set_kernel_policy(0)
            got.append(p.view(torch.int16).cpu())
            state.destroy()
        nan = [(x.int() & 0x7FFF) > 0x7F80 for x in got]
        assert torch.equal(nan[0], nan[1])
        assert torch.equal(got[0][~nan[0]], got[1][~nan[1]])


@pytest.mark.parametrize("kind", ["normal", "zero", "tiny"])
@pytest.mark.parametrize("lr", [1e-3, 0.3, 2.0 ** 18])
@pytest.mark.parametrize("exponent", [-59, -64, -126])
@pytest.mark.parametrize("bits_m,bits_v,block,round_m", [(2, 2, 128, 0), (8, 8, 2048, 0), (3, 3, 128, 1), (4, 2, 2048, 1)])
def test_patterns_where_moments_are_subnormal(bits_m, bits_v, block, round_m, exponent, lr, kind):
    """Blocks whose update is tried by approximations (128 and 2048; plain and Eq. 5).  Gradients of 2^-59: second moments around
    2^-128, whose root times 31.6, the first step's bias correction, is 2^-19 of eps = 1e-12, far more than the bracket is wide.
    2^-64: some 2^-138.  2^-126: first moments whose division leaves remainders below the smallest subnormal number; a rate of
    2^18 lifts the quotients to where they are not looked at again."""
    from paper_2505_00347_b200 import binding as B
    n = 2048 * 64
    gen = torch.Generator().manual_seed(22)
    p0 = _params(kind, n, gen)
    grads = [(torch.randn(n, generator=gen) * 2.0 ** exponent).bfloat16().cuda() for _ in range(3)]
    h = B.hyper(lr=lr, beta1=0.5, eps=1e-12, weight_decay=0.0, seed=2, param_dtype=1, param_round=1, round_m=round_m)
    got = []
    for policy in (1, 3):
        p = p0.cuda()
        state = B.State(n, bits_m, bits_v, block)
        B.set_kernel_policy(policy)
        try:
            for t, g in enumerate(grads, 1):
                B.solo_step(p, g, state, h, t)
        finally:
            B.set_kernel_policy(0)
        got.append([p.view(torch.int16).cpu()] + [state.raw_get(k) for k in ("codes_m", "codes_v", "scale_m", "scale_v", "alpha")])
        state.destroy()
    for a, b in zip(*got):
        assert torch.equal(a, b)


@pytest.mark.parametrize("sr", [0, 1])
@pytest.mark.parametrize("lr", [1e-3, -0.3, 0.0])
@pytest.mark.parametrize("bits_m,bits_v,block,hk", [(2, 2, 128, {}), (8, 8, 2048, {}), (3, 3, 128, dict(round_m=1)), (4, 2, 256, dict(belief=1)),
                                                    (4, 3, 64, dict(v_codebook=3))])
def test_zero_moments(bits_m, bits_v, block, hk, lr, sr):
    """Rows without gradient (padding, masked weights): their results are not looked at for being small.  Zeros of both signs among the
    gradients, the moments and the weights, weights of every size, whole warps of them, single threads and single elements."""
    from paper_2505_00347_b200 import binding as B
    n = 2048 * 32
    gen = torch.Generator().manual_seed(23)
    w = torch.randn(n, generator=gen) * torch.exp2(torch.randint(-148, 3, (n // 16,), generator=gen).float()).repeat_interleave(16)
    w[torch.rand(n, generator=gen) < 0.3] = 0.0
    w[2048 * 8:2048 * 16] = 0.0
    w[torch.rand(n, generator=gen) < 0.3] *= -1.0
    w[::4099] = float("inf")
    p0 = w.bfloat16()
    runs = torch.rand(n // 16, generator=gen).repeat_interleave(16) < torch.tensor([0.0, 0.5, 0.95, 0.0]).repeat_interleave(n // 4)
    grads = []
    for _ in range(3):
        g = torch.randn(n, generator=gen) * 1e-3
        g[~runs] = 0.0
        g[torch.rand(n, generator=gen) < 0.1] = 0.0
        grads.append(torch.where(torch.rand(n, generator=gen) < 0.5, g, -g).bfloat16().cuda())
    h = B.hyper(lr=lr, beta1=0.5, weight_decay=0.01, seed=2, param_dtype=1, param_round=sr, **hk)
    got = []
    for policy in (1, 3):
        p = p0.cuda()
        state = B.State(n, bits_m, bits_v, block)
        B.set_kernel_policy(policy)
        try:
            for t, g in enumerate(grads, 1):
                B.solo_step(p, g, state, h, t)
        finally:
            B.set_kernel_policy(0)
        got.append(p.view(torch.int16).cpu())
        state.destroy()
    assert torch.equal(*got)
