"""Eq. 5 alone and a baseline codebook alone have instantiations of their own in the sixteen-per-thread kernel, any further mode
takes the one that reads them all: each against the oracle (codes, scales and bases bit for bit), and the routes on both
sides of each line of the choice."""
import pytest
import torch

from parity import run_lockstep
from paper_2505_00347_b200 import synth

pytestmark = pytest.mark.gpu

# The fp32 update term u is taken with an approximate square root (2^-23 relative, halved in the denominator's error when eps
# counts) and a quotient within 0.6 units of the last place: three roundings more than the oracle's, 1.8e-7 |u| in all.  The plain bar
# is relative to the parameter; a codebook that decodes a small second moment as zero makes |u| a multiple of it.
UPDATE_TOL = 3e-7
SIZES = (2048 * 2 + 700, 2048, 130)


@pytest.mark.parametrize("hk", [dict(round_m=1), dict(round_m=1, weight_decay=0.01), dict(round_m=1, adamw=0, weight_decay=0.01),
                                dict(round_m=1, belief=1), dict(round_m=1, fixed_alpha=0.5), dict(round_m=1, round_v=0),
                                dict(round_m=1, param_dtype=1, param_round=1), dict(v_codebook=1), dict(v_codebook=2, fixed_alpha=0.5),
                                dict(v_codebook=3, round_v=0), dict(v_codebook=1, param_dtype=1), dict(v_codebook=1, belief=1),
                                dict(v_codebook=3, round_m=1), dict(v_codebook=1, adamw=0, weight_decay=0.01)])
@pytest.mark.parametrize("bits_m,bits_v,block", [(4, 2, 128), (8, 8, 2048), (2, 8, 64), (3, 3, 256)])
def test_modes_alone_and_together(bits_m, bits_v, block, hk):
    hk = {"weight_decay": 0.0, **hk}
    w = synth.workload(3, sizes=SIZES)
    dt = torch.bfloat16 if hk.get("param_dtype") else torch.float32
    rep = run_lockstep(SIZES, bits_m, bits_v, block, dict(lr=1e-3, beta1=0.5, beta2=0.999, seed=9, **hk), steps=2,
                       grads_fn=lambda t: [synth.make_grad(w, i, t) for i in range(len(SIZES))],
                       params0=[synth.make_param(w, i, dtype=dt) for i in range(len(SIZES))], policies=(3,), update_tol=UPDATE_TOL)
    assert rep.exempt_v == 0 and rep.exempt_m == 0
