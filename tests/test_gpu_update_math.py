"""The square root and division of bf16 parameters' update are correctly rounded: every mantissa of two binades (the
square root of other numbers differs by a power of two), small and subnormal numbers, and both ends of the range."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lo,hi", [(0x3F800000, 0x407FFFFF),          # [1, 4): all mantissas, both parities of the exponent
                                   (0x00000000, 0x0000FFFF),          # zero and subnormal numbers
                                   (0x007F0000, 0x0080FFFF),          # around the smallest normal number
                                   (0x4CFF0000, 0x4CFFFFFF)])         # up to 2^27
def test_square_root_and_quotients_are_the_ieee_ones(lo, hi):
    from paper_2505_00347_b200 import binding as B
    assert B.debug_check_update_math(lo, hi) == 0
