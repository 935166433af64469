"""A step reads nothing before the work ahead of it on the stream is complete and visible: every kernel that a step
launches waits for it first, in every CTA, and the kernel after a step finds all that both launches wrote."""
import re
from pathlib import Path

import pytest
import torch

from paper_2505_00347_b200 import synth

CSRC = Path(__file__).resolve().parent.parent / "paper_2505_00347_b200" / "csrc"


@pytest.mark.parametrize("name", ["solo_device.cuh", "solo_fast.cuh", "solo_fast16.cuh"])
def test_every_step_kernel_waits_before_it_touches_memory(name):
    text = re.sub(r"//[^\n]*", "", (CSRC / name).read_text())
    body = text[re.search(r"__global__[^;{]*\bsolo_step_\w*kernel\(", text).end():]
    body = body[: body.index("\n}")]
    lines = [ln.strip() for ln in body.splitlines()]
    at = lines.index("pdl_wait();")                         # a statement of its own: under no condition
    assert lines[at + 1] == "pdl_release();"
    assert body.count("pdl_wait(") == 1 and body.count("pdl_release(") == 1
    for ln in lines[:at]:                                   # only declarations come before it
        assert "a." not in ln and "if" not in ln.split("(")[0], ln


@pytest.mark.gpu
@pytest.mark.parametrize("hk", [dict(), dict(round_m=1), dict(param_dtype=1, param_round=1)])
def test_steps_queued_behind_writes_of_their_inputs(hk):
    """Gradients rewritten by a kernel or by a copy, and the lists of pointers by a copy, directly before each of many steps;
    against the same steps one by one."""
    from paper_2505_00347_b200 import binding as B
    sizes = [2048 * 9 + 5, 3, 2048 * 4, 4099] + [200 + 37 * i for i in range(120)] + [2048 * 30 + 2047]
    w = synth.workload(3, sizes=tuple(sizes))
    dt = torch.bfloat16 if hk.get("param_dtype") else torch.float32
    fresh = [[synth.make_grad(w, i, t).cuda() for i in range(len(sizes))] for t in range(4)]
    h = B.hyper(lr=1e-3, beta1=0.5, weight_decay=0.01, seed=3, **hk)
    got = []
    for one_by_one in (False, True):
        params = [synth.make_param(w, i, dtype=dt).cuda() for i in range(len(sizes))]
        grads = [[torch.zeros_like(g) for g in fresh[0]] for _ in range(2)]
        state = B.State(sizes, 2, 3, 128)
        ts = B.TensorSet(params, grads[0], state)
        lists = [torch.tensor([g.data_ptr() for g in gs], dtype=torch.int64, device="cuda") for gs in grads]
        B.set_kernel_policy(3)
        try:
            torch.cuda.synchronize()
            for t in range(1, 25):
                k = t & 1
                if t % 3:
                    torch._foreach_copy_(grads[k], fresh[t % 4])
                else:
                    torch._foreach_add_(grads[k], fresh[t % 4])
                ts.grad_ptrs.copy_(lists[k])
                if one_by_one:
                    torch.cuda.synchronize()
                B.solo_multi_step(ts, h, t)
                torch._foreach_zero_(grads[k ^ 1])           # of the step before: done with
                if one_by_one:
                    torch.cuda.synchronize()
            torch.cuda.synchronize()
        finally:
            B.set_kernel_policy(0)
        assert state.status() == 0
        got.append([state.raw_get(k) for k in ("codes_m", "codes_v", "scale_m", "scale_v", "alpha")] + [p.cpu() for p in params])
        state.destroy()
    for a, b in zip(*got):
        assert torch.equal(a, b)
