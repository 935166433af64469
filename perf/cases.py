"""Workloads whose time matters to a user of the fused low-bit optimizer step.

A case is one call that a training program makes over and over: `solo_step` on one tensor,
`solo_multi_step` on a model's tensor list, `solo_multi_step_static` with the caller's own state
buffers, `solo_multi_step_host` with gradients in page-locked host memory, or `solo_dequant`.
Shapes and value distributions are those of `synth.py`; they are drawn here from the seed alone and
as flat buffers (a tensor is a 256-byte aligned view of its buffer, as in a flattened parameter group).

Every program keeps two sets of gradients and steps with one after the other, so that the moments do
not settle on one gradient; the step count grows from pass to pass as in training.
"""
from __future__ import annotations

import math

import torch

from paper_2505_00347_b200 import binding as B
from paper_2505_00347_b200 import shard, synth

ALIGN = 128                     # elements between the starts of two views: 256 bytes of bf16
PARAMS = ("fp32", "bf16", "bf16_sr")
# what is varied of solo_hyper_t: the paper's step (AdamW, quantile base, dither), and its options
VARIANTS = {
    "adamw": {},
    "adam_l2": {"adamw": 0},                          # decay joins the gradient
    "adabelief": {"belief": 1},
    "fixed_base": {"fixed_alpha": 0.5},               # standard logarithmic quantizer, no quantile
    "stochastic_m": {"round_m": 1},                   # Eq. 5 for the first moment
    "de": {"v_codebook": 1},                          # baseline: unsigned dynamic exponent (8-bit Adam)
    "linear_nozero": {"v_codebook": 3},               # baseline: linear without zero (4-bit Adam)
    "p05": {"p_quantile": 0.05},
    "p20": {"p_quantile": 0.2},
}


def _case(call, shape, n, bits_m, bits_v, block, params="fp32", variant="adamw", grads="normal", name=None):
    c = {"call": call, "shape": shape, "n": n, "bits_m": bits_m, "bits_v": bits_v, "block": block,
         "params": params, "variant": variant, "grads": grads}
    return c if name is None else {"name": name, **c}


def listed():
    return [
        # one LoRA factor (4096 x 16) stepped by itself: launch and latency, nothing else
        _case("step", "single", 1 << 16, 4, 4, 128, name="lora_factor"),
        # one matrix of 2^20 elements, the first benchmark workload
        _case("step", "single", 1 << 20, 4, 4, 128, name="single_1Mi"),
        # a GPT-style model of 125M parameters, trained from scratch
        _case("multi", "gpt", 12, 3, 3, 128, grads="scaled", name="gpt125m"),
        # one of four ranks' share of the LLaMA-7B-shaped set, partitioned as under FSDP: the headline widths
        _case("multi", "llama7b_shard", 4, 2, 3, 128, grads="student", name="llama7b_quarter"),
        # 4096 tensors from 1 to 4M elements: odd sizes, tails, exact zeros
        _case("multi", "ragged", 4096, 2, 3, 128, grads="mixed", name="ragged4096"),
        # two points of the width / block sweep on one tensor of 2^28 elements
        _case("step", "single", 1 << 28, 4, 4, 256, name="sweep_4_4_b256"),
        _case("step", "single", 1 << 28, 8, 8, 2048, name="sweep_8_8_b2048"),
        # the 8-bit Adam baseline of the experiments: dynamic exponent for both moments
        _case("multi", "gpt", 12, 8, 8, 128, variant="de", grads="scaled", name="gpt125m_adam8"),
        # fine-tuning with bf16 weights and 2-bit Adam: one LLaMA layer, stochastically rounded weights
        _case("multi", "llama_layers", 1, 2, 2, 128, params="bf16_sr", grads="student", name="llama_layer_bf16"),
        # 4/2-bit Adam with the stochastic rounding that the variance bound assumes
        _case("multi", "llama_layers", 1, 4, 2, 128, variant="stochastic_m", grads="student", name="llama_layer_eq5"),
        # gradients arrive in host memory, updated weights go back there
        _case("host", "gpt", 12, 4, 2, 128, grads="scaled", name="gpt125m_host"),
        # reading the second moment back (inspection, export to another optimizer)
        _case("dequant_v", "gpt", 12, 3, 3, 128, grads="scaled", name="gpt125m_dequant"),
    ]


def draw(rng):
    call = rng.choice(("step", "step", "multi", "multi", "multi", "multi", "static", "host", "dequant_m", "dequant_v"))
    if call == "step":
        shape, n = "single", int(math.exp(rng.uniform(math.log(1000), math.log(1 << 28))))
        if rng.random() < 0.5:
            n = max(1024, n // 1024 * 1024)               # a matrix; otherwise whatever was drawn, odd sizes too
    elif call == "host":
        shape, n = rng.choice((("gpt", rng.randint(2, 12)), ("ragged", rng.randint(16, 400))))
    elif call == "static":
        shape, n = rng.choice((("gpt", rng.randint(2, 24)), ("ragged", rng.randint(16, 1024))))
    else:
        shape, n = rng.choice((("gpt", rng.randint(2, 24)), ("llama_layers", rng.randint(1, 4)),
                               ("ragged", int(math.exp(rng.uniform(math.log(32), math.log(4096)))))))
    bits_m, bits_v = rng.choice(((2, 2), (2, 3), (3, 3), (4, 2), (4, 4), (3, 4), (8, 8), (8, 4)))
    block = rng.choice((64, 128, 128, 128, 256, 2048))
    params = rng.choice(("fp32", "fp32", "fp32", "bf16", "bf16_sr"))
    variant = rng.choice(("adamw",) * 8 + tuple(v for v in VARIANTS if v != "adamw"))
    grads = {"single": "normal", "gpt": "scaled", "llama_layers": "student", "ragged": "mixed"}[shape]
    return _case(call, shape, n, bits_m, bits_v, block, params, variant, grads)


def _sizes(case):
    """Element counts of the case's tensors, and the pieces' place in their tensors (None: whole tensors)."""
    shape, n = case["shape"], case["n"]
    if shape == "single":
        return [n], None
    if shape == "gpt":                                    # `n` layers, d = 768, 4x MLP, vocabulary 50257, 1024 positions
        d = 768
        s = [50257 * d, 1024 * d]
        for _ in range(n):
            s += [d, d, d * 3 * d, 3 * d, d * d, d, d, d, d * 4 * d, 4 * d, 4 * d * d, d]
        return s + [d, d], None
    if shape == "llama_layers":                           # `n` layers, d = 4096, MLP 11008
        d, f = 4096, 11008
        return ([d * d] * 4 + [d * f, d * f, f * d, d, d]) * n, None
    if shape == "ragged":
        return list(synth.ragged_sizes(n)), None
    pieces = shard.partition(synth.llama7b_sizes(), case["block"], n)[1]
    return [p.numel for p in pieces], ([p.tensor for p in pieces], [p.elem_offset for p in pieces])


def _offsets(sizes):
    offs, at = [], 0
    for n in sizes:
        offs.append(at)
        at += -(-n // ALIGN) * ALIGN
    return offs, at


def _flat_grad(case, sizes, offs, total, gen):
    """Gradients of the whole list as one bf16 buffer (distributions of synth.make_grad)."""
    dev = "cuda"
    out = torch.empty(total, dtype=torch.bfloat16, device=dev)
    scales = torch.exp(torch.empty(len(sizes)).uniform_(math.log(1e-4), math.log(1e-2),
                                                        generator=torch.Generator().manual_seed(gen.initial_seed())))
    step = 1 << 26
    for lo in range(0, total, step):
        n = min(step, total - lo)
        x = torch.empty(n, device=dev).normal_(generator=gen)
        if case["grads"] == "student":                    # t(3), heavy tails
            chi = torch.empty(n, device=dev).normal_(generator=gen).square_()
            for _ in range(2):
                chi += torch.empty(n, device=dev).normal_(generator=gen).square_()
            x *= torch.rsqrt(chi / 3.0)
        elif case["grads"] == "mixed":                    # blocks of exact zeros (30 %), N(0, 1e-6), N(0, 1)
            kind = torch.rand(-(-n // 128), device=dev, generator=gen)
            sigma = torch.where(kind < 0.30, 0.0, torch.where(kind < 0.65, 1e-3, 1e3))
            x *= sigma.repeat_interleave(128)[:n]
        out[lo:lo + n] = x.mul_(1e-3)
    if case["grads"] == "scaled":
        for o, n, s in zip(offs, sizes, scales.tolist()):
            out[o:o + n] *= s
    return out


class _Raw:
    """A state's device buffer as a tensor without a copy; holds on to the state that owns it."""

    def __init__(self, owner, ptr, count, kind):
        self.owner = owner
        self.__cuda_array_interface__ = {"shape": (count,), "typestr": kind, "data": (ptr, False), "version": 3}


def _state_views(state):
    out = {}
    for key in ("codes_m", "codes_v", "scale_m", "scale_v", "alpha"):
        ptr, nbytes = state.raw_ptr(key)
        code = key.startswith("codes")
        out[key] = torch.as_tensor(_Raw(state, ptr, nbytes if code else nbytes // 4, "|u1" if code else "<f4"), device="cuda")
    return out


def prepare(case, seed):
    sizes, origin = _sizes(case)
    offs, total = _offsets(sizes)
    gen = torch.Generator(device="cuda").manual_seed(1_000_003 * seed + 17)
    pdt = torch.float32 if case["params"] == "fp32" else torch.bfloat16
    flat = torch.empty(total, dtype=pdt, device="cuda").normal_(0.0, 0.02, generator=gen)
    grads = [_flat_grad(case, sizes, offs, total, gen) for _ in range(2)]

    def views(buf):
        return [buf[o:o + n] for o, n in zip(offs, sizes)]

    scratch = case["shape"] in ("gpt", "ragged")
    kw = dict(lr=1e-3 if scratch else 2e-5, beta1=B.default_beta1(case["bits_m"], scratch) or 0.9, beta2=0.999,
              weight_decay=0.01 if scratch else 0.0, seed=seed, param_dtype=0 if case["params"] == "fp32" else 1,
              param_round=1 if case["params"] == "bf16_sr" else 0)
    kw.update(VARIANTS[case["variant"]])
    if case["variant"] == "adam_l2":
        kw["weight_decay"] = 0.01
    s = {"case": case, "hyper": B.hyper(**kw), "step": 0, "params": flat, "views": views(flat), "sizes": sizes,
         "grads": grads, "grad_views": [views(g) for g in grads]}
    bm, bv, block = case["bits_m"], case["bits_v"], case["block"]
    if case["call"] == "static":
        nb = sum(-(-n // block) for n in sizes)
        padded = -(-nb // 4) * 4
        s["buffers"] = {k: torch.zeros(nb * block * b // 8 + 16, dtype=torch.uint8, device="cuda")
                        for k, b in (("codes_m", bm), ("codes_v", bv))}
        s["buffers"] |= {k: torch.zeros(padded, device="cuda") for k in ("scale_m", "scale_v")}
        s["buffers"]["alpha"] = torch.full((padded,), 0.5, device="cuda")
        s["param_ptrs"] = torch.tensor([p.data_ptr() for p in s["views"]], dtype=torch.int64, device="cuda")
        s["grad_ptrs"] = [torch.tensor([g.data_ptr() for g in gv], dtype=torch.int64, device="cuda") for gv in s["grad_views"]]
        return s
    state = B.State(sizes[0] if case["call"] == "step" else sizes, bm, bv, block)
    if origin is not None:
        state.set_origin(*origin)
    s["state"] = state
    s["moments"] = _state_views(state)
    if case["call"] == "host":
        host = []
        for g in grads:
            host.append(torch.empty(total, dtype=torch.bfloat16, pin_memory=True))
            host[-1].copy_(g)
        s["grads"] = host
        s["grad_views"] = [views(h) for h in host]
        s["params_out"] = torch.zeros(total, dtype=pdt, pin_memory=True)
        s["out_views"] = views(s["params_out"])
    elif case["call"] != "step":
        s["sets"] = [B.TensorSet(s["views"], gv, state) for gv in s["grad_views"]]
    if case["call"].startswith("dequant"):
        for k in range(2):
            B.solo_multi_step(s["sets"][k], s["hyper"], k + 1)
    return s


def run(s):
    case = s["case"]
    call = case["call"]
    if call == "dequant_m":
        return B.solo_dequant(s["state"], 0)
    if call == "dequant_v":
        return B.solo_dequant(s["state"], 1)
    s["step"] += 1
    k = s["step"] & 1
    if call == "step":
        B.solo_step(s["views"][0], s["grad_views"][k][0], s["state"], s["hyper"], s["step"])
    elif call == "multi":
        B.solo_multi_step(s["sets"][k], s["hyper"], s["step"])
    elif call == "host":
        B.solo_multi_step_host(s["views"], s["grad_views"][k], s["out_views"], s["state"], s["hyper"], s["step"])
        return {"params_out": s["params_out"], "params": s["params"], **s["moments"]}
    else:
        B.solo_multi_step_static(s["views"], s["grad_views"][k], s["sizes"], s["buffers"], case["bits_m"], case["bits_v"],
                                 case["block"], s["hyper"], s["step"], s["param_ptrs"], s["grad_ptrs"][k])
        return {"params": s["params"], **s["buffers"]}
    return {"params": s["params"], **s["moments"]}


def work(case):
    sizes, _ = _sizes(case)
    n, block = sum(sizes), case["block"]
    nb = sum(-(-k // block) for k in sizes)
    if case["call"].startswith("dequant"):
        v = case["call"] == "dequant_v"
        bits = case["bits_v" if v else "bits_m"]
        base = v and case["variant"] not in ("de", "linear_nozero")
        return {"bytes": n * 4 + n * bits / 8 + nb * (8 if base else 4), "flops": 0}
    pb = 4 if case["params"] == "fp32" else 2
    bits = case["bits_m"] + case["bits_v"]
    return {"bytes": n * (2 * pb + 2) + 2 * n * bits / 8 + 24 * nb + (n * (2 + pb) if case["call"] == "host" else 0),
            "flops": 20 * n}


def tolerance(case):
    """Codes, scales and bases are the same bits for every correct implementation, bf16 weights too.
    fp32 weights may take the quotient of the update to an ulp or two instead of to half an ulp: two such
    implementations differed by 1.1e-8 (2-norm) and 2.8e-7 (largest) after three steps.  With the L2 term the
    weights feed back into the moments: one code in 4e7 then differed, and with it one weight by 2.3e-4."""
    if case["params"] == "fp32" and case["variant"] == "adam_l2":
        return {"rel": 1e-6, "max": 0.02, "differ": 1e-6}
    if case["params"] == "fp32" and not case["call"].startswith("dequant"):
        return {"rel": 1e-7, "max": 2e-6, "differ": 0.0}
    return {"rel": 1e-8, "max": 1e-7, "differ": 0.0}
