"""8-bit states in the sixteen-per-thread kernel: cell look-ups of the fixed codebooks and the level tables of the
logarithmic one.  With both betas zero and a zero state the ratios that are quantized are the gradients and their
squares, so every bf16 value of [-1, 1] meets every cell, threshold and sign; random states cover the decoding.  The
packed state is compared with the oracle's bit for bit."""
import numpy as np
import pytest
import torch

from parity import run_lockstep
from paper_2505_00347_b200 import synth

pytestmark = pytest.mark.gpu

RANDOM_STATE_TOL = 3e-7
MODES = [dict(), dict(v_codebook=1), dict(v_codebook=2), dict(v_codebook=3), dict(round_m=1), dict(round_m=1, v_codebook=1),
         dict(fixed_alpha=0.97), dict(belief=1), dict(adamw=0, weight_decay=0.05), dict(round_v=0, p_quantile=0.3)]


def _all_bf16(block):
    """Every bf16 value of [-1, 1] with magnitude from 2^-26 on, and zeros, in a shuffled order; the first of each block is +-1."""
    bits = np.arange(0x3280, 0x3F81, dtype=np.uint16)
    vals = np.concatenate([bits, bits | 0x8000, np.zeros(64, np.uint16), np.full(64, 0x8000, np.uint16)])
    np.random.default_rng(3).shuffle(vals)
    vals = np.resize(vals, 4 * 2048 + 2048 * (-(-len(vals) // 2048)))
    vals[::block] = 0x3F80
    vals[block::2 * block] = 0xBF80
    return synth.bits_to_bf16(vals)


@pytest.mark.parametrize("mode", range(len(MODES)))
@pytest.mark.parametrize("bits_m,bits_v", [(8, 8), (8, 3), (4, 8)])
def test_every_cell_of_the_codebooks(bits_m, bits_v, mode):
    for block in (64, 128, 256, 2048):
        g = _all_bf16(block)
        n = g.numel()
        rep = run_lockstep((n,), bits_m, bits_v, block, dict(lr=1e-3, beta1=0.0, beta2=0.0, weight_decay=0.0, seed=21) | MODES[mode],
                           steps=1, grads_fn=lambda t: [g], params0=[torch.linspace(-1, 1, n)], policies=(3,), multi=True,
                           update_tol=RANDOM_STATE_TOL)
        assert rep.exempt_m == 0 and rep.exempt_v == 0


@pytest.mark.parametrize("mode", range(len(MODES)))
@pytest.mark.parametrize("bits_m,bits_v,block", [(8, 8, 64), (8, 8, 128), (8, 8, 256), (2, 8, 128), (3, 8, 64), (4, 8, 256), (8, 2, 128), (8, 4, 64),
                                                 (8, 8, 2048), (2, 3, 2048), (4, 2, 2048), (3, 8, 2048)])
def test_random_states(bits_m, bits_v, block, mode):
    sizes = (2048 * 3, 2048 * 2 + 77)
    w = synth.workload(3, sizes=sizes)
    bf16 = mode % 3 == 1
    hk = dict(lr=1e-3, beta1=0.9, beta2=0.99, weight_decay=0.01, seed=5, param_dtype=int(bf16), param_round=int(bf16)) | MODES[mode]
    rep = run_lockstep(sizes, bits_m, bits_v, block, hk, steps=2, grads_fn=lambda t: [synth.make_grad(w, i, t) for i in range(2)],
                       params0=[synth.make_param(w, i, dtype=torch.bfloat16 if bf16 else torch.float32) for i in range(2)],
                       state0=synth.make_state(sizes, bits_m, bits_v, block, seed=17), policies=(3,), update_tol=RANDOM_STATE_TOL)
    assert rep.exempt_m == 0 and rep.exempt_v == 0


def test_nan_and_infinite_blocks():
    sizes = (2048 * 2,)
    for mode in (dict(), dict(v_codebook=1), dict(round_m=1)):
        g = synth.make_grad(synth.workload(3, sizes=sizes), 0, 1)
        g[5], g[200], g[333], g[334] = float("nan"), float("inf"), -float("inf"), 0.0
        run_lockstep(sizes, 8, 8, 128, dict(lr=1e-3, beta1=0.9, beta2=0.99, weight_decay=0.0, seed=5) | mode, steps=1,
                     grads_fn=lambda t: [g], params0=[torch.zeros(sizes[0])], policies=(3,), multi=True,
                     state0=synth.make_state(sizes, 8, 8, 128, seed=2), update_tol=RANDOM_STATE_TOL)


@pytest.mark.parametrize("block", [64, 128, 256, 2048])
@pytest.mark.parametrize("bits_m,bits_v,bf16", [(8, 8, 0), (2, 8, 1), (8, 3, 0)])
def test_blocks_whose_largest_value_has_no_finite_reciprocal(bits_m, bits_v, bf16, block):
    """Scales between 0 and 2^-128, for the second moment (gradients of 1e-19) and for both (1e-39): a vanishing block."""
    sizes = (2048 * 6,)
    scale = torch.tensor([1e-19, 1.0, 1e-39, 1e-19, 0.0, 1e-3]).repeat_interleave(2048)
    for mode in (dict(), dict(v_codebook=1), dict(v_codebook=2), dict(round_m=1), dict(round_m=1, v_codebook=3)):
        g = (synth.make_grad(synth.workload(3, sizes=sizes), 0, 1).float() * 1e3).clamp(-1, 1).mul(scale).bfloat16()
        run_lockstep(sizes, bits_m, bits_v, block, dict(lr=1e-3, beta1=0.9, beta2=0.99, weight_decay=0.0, seed=5, param_dtype=bf16) | mode,
                     steps=2, grads_fn=lambda t: [g], params0=[torch.zeros(sizes[0], dtype=torch.bfloat16 if bf16 else torch.float32)],
                     policies=(3,), multi=True, update_tol=RANDOM_STATE_TOL)
