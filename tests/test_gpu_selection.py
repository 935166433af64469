"""The p-quantile of the sixteen-per-thread kernel (rank selection over a group of lanes) at any rank, on inputs
that are hard for it: keys that ascend with the element index (one lane holds all the smallest), equal keys,
blocks of zeros with a few values, and random states.  Blocks of 2048 span the CTA: histogram bins that hold few,
more than 512 or all of the keys.  The packed state, and with it the base that the quantile
decides, is compared with the oracle's bit for bit; parameters within the bar of every other parity test."""
import numpy as np
import pytest
import torch

from parity import run_lockstep
from paper_2505_00347_b200 import synth

pytestmark = pytest.mark.gpu

SIZES = (2048 * 3, 2048 + 700, 4096)


def _grads(kind, t, n, seed):
    g = torch.Generator().manual_seed(1000 * seed + t)
    i = torch.arange(n, dtype=torch.float32)
    if kind == "ascending":                                   # the smallest keys side by side
        x = 1e-3 * (1.0 + (i % 256) * (7 / 256))
    elif kind == "descending":
        x = 1e-3 * (8.0 - (i % 256) * (7 / 256))
    elif kind == "equal":
        x = torch.full((n,), 2.5e-4)
    elif kind == "clusters":                                  # most keys within one bin of the block's range, 2-bit levels apart
        x = 1e-3 * (1.0 + 1e-2 * torch.randn(n, generator=g)) * torch.where(torch.rand(n, generator=g) < 0.8, 1.0, 30.0)
    elif kind == "zeros":
        x = torch.randn(n, generator=g) * 1e-3
        x[torch.rand(n, generator=g) < 0.9] = 0.0
    else:
        x = torch.randn(n, generator=g) * 1e-3
    return x.to(torch.bfloat16)


@pytest.mark.parametrize("kind", ["ascending", "descending", "equal", "zeros", "clusters", "random"])
@pytest.mark.parametrize("block", [64, 128, 256, 2048])
def test_selection_at_any_rank(block, kind):
    w = synth.workload(3, sizes=SIZES)
    for p in (0.0, 0.05, 0.1, 0.2, 0.5, 0.99):
        rep = run_lockstep(SIZES, 2, 3, block, dict(lr=1e-3, beta1=0.5, beta2=0.999, weight_decay=0.0, seed=9, p_quantile=p),
                           steps=2, grads_fn=lambda t: [_grads(kind, t, n, i) for i, n in enumerate(SIZES)],
                           params0=[synth.make_param(w, i) for i in range(len(SIZES))], policies=(3,))
        assert rep.exempt_v == 0 and rep.exempt_m == 0
