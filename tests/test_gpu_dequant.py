"""solo_dequant against the oracle, bit for bit (Eq. 2 is a fixed sequence of binary32 operations), where its
row split can go wrong: rows that end inside a tile, in the first or second block of 64 of a row, tensors whose
output starts off a 16-byte boundary, and tensors of one element."""
import numpy as np
import pytest
import torch

from parity import split_state, to_numpy_state, upload_state
from paper_2505_00347_b200 import synth

pytestmark = pytest.mark.gpu

SIZES = (2048 * 3, 1, 63, 64, 65, 127, 128, 129, 2048 + 4, 511, 512, 513, 2047, 4096 + 640)


@pytest.mark.parametrize("block", [64, 128, 256, 2048])
@pytest.mark.parametrize("bits", [2, 3, 4, 8])
def test_dequant_is_the_oracles_bit_for_bit(bits, block):
    import oracle
    from paper_2505_00347_b200 import binding as B
    sd = to_numpy_state(synth.make_state(SIZES, bits, bits, block, seed=31 * bits + block))
    state = B.State(list(SIZES), bits, bits, block)
    upload_state(state, sd)
    ostates = split_state(sd, SIZES, bits, bits, block)
    for which in (0, 1):
        got = B.solo_dequant(state, which).cpu().numpy()
        want = np.concatenate([oracle.dequant(s, which) for s in ostates])
        assert np.array_equal(got.view(np.uint32), want.astype(np.float32).view(np.uint32)), which
    torch.cuda.synchronize()
    state.destroy()
