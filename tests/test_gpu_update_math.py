"""The square root and division of bf16 parameters' update are correctly rounded: every mantissa of two binades (the
square root of other numbers differs by a power of two), small and subnormal numbers, and both ends of the range."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lo,hi", [(0x3F800000, 0x407FFFFF),          # [1, 4): all mantissas, both parities of the exponent
                                   (0x00000000, 0x0000FFFF),          # zero and subnormal numbers
                                   (0x007F0000, 0x0080FFFF),          # around the smallest normal number
                                   (0x4CFF0000, 0x4CFFFFFF)])         # up to 2^27
def test_square_root_and_quotients_are_the_ieee_ones(lo, hi):
    from paper_2505_00347_b200 import binding as B
    assert B.debug_check_update_math(lo, hi) == 0


@pytest.mark.parametrize("tiny", [False, True])
@pytest.mark.parametrize("hk", [dict(param_dtype=1), dict(param_dtype=1, param_round=1), dict(param_dtype=1, adamw=0)])
@pytest.mark.parametrize("bits_m,bits_v,block", [(2, 2, 128), (4, 2, 64), (3, 3, 256), (8, 8, 2048)])
def test_parameters_are_those_of_the_general_kernel(bits_m, bits_v, block, hk, tiny):
    """`tiny`: quotients of a few units of the smallest subnormal number, which a large rate lifts to where their rounding
    to that grid shows."""
    from paper_2505_00347_b200 import binding as B
    n = 2048 * 8
    gen = torch.Generator().manual_seed(9)
    if tiny:
        g = torch.randint(-60, 61, (n,), generator=gen).float().mul(2.0 ** -133).bfloat16().cuda()
        p0 = torch.zeros(n)
        h = B.hyper(lr=2.0 ** 18, beta1=0.5, eps=3e4, weight_decay=0.0, bias_correction=0, seed=2, **hk)
    else:
        g = torch.randn(n, generator=gen).mul(1e-3).bfloat16().cuda()
        p0 = torch.randn(n, generator=gen).mul(0.02)
        h = B.hyper(lr=1e-3, beta1=0.5, weight_decay=0.01, seed=2, **hk)
    got = []
    for policy in (1, 3):
        p = p0.to(torch.bfloat16 if hk.get("param_dtype") else torch.float32).cuda()
        state = B.State(n, bits_m, bits_v, block)
        B.set_kernel_policy(policy)
        try:
            for t in (1, 2):
                B.solo_step(p, g, state, h, t)
        finally:
            B.set_kernel_policy(0)
        got.append(p.view(torch.int16 if hk.get("param_dtype") else torch.int32).cpu())
        state.destroy()
    assert got[0].any() and torch.equal(*got)
