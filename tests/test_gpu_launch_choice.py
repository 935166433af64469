"""One launch or two: by the full tiles that the launch has, not by how many tensors or chunks the set is cut into; and a
chunk of a host-buffer call costs its own tensors."""
import time

import pytest
import torch

from paper_2505_00347_b200 import synth

pytestmark = pytest.mark.gpu

KEYS = ("codes_m", "codes_v", "scale_m", "scale_v", "alpha")


def _list(sizes):
    at = [0]
    for n in sizes:
        at.append(at[-1] + -(-n // 128) * 128)
    gen = torch.Generator(device="cuda").manual_seed(1)
    flat_p = torch.empty(at[-1], device="cuda").normal_(0.0, 0.02, generator=gen)
    flat_g = torch.empty(at[-1], device="cuda").normal_(0.0, 1e-3, generator=gen).bfloat16()
    return [flat_p[o:o + n] for o, n in zip(at, sizes)], [flat_g[o:o + n] for o, n in zip(at, sizes)]


@pytest.mark.parametrize("sizes,bits_m,bits_v,block,hk,launches", [
    ([768] * 4096, 2, 3, 128, dict(), 1),                        # no full tile at all
    ([768] * 4096, 4, 2, 128, dict(round_m=1), 1),
    ([3000] * 2000, 2, 3, 128, dict(), 1),                       # as many others as full ones
    ([2048 * 400 + 5] * 8, 2, 3, 128, dict(), 2),
    ([2048 * 400 + 5] * 8, 4, 2, 128, dict(round_m=1), 2),
    ([2048 * 400] * 4, 2, 3, 128, dict(), 1),
    ([2048 * 2 + 5] * 1200, 8, 8, 128, dict(), 1),
    ([2048 * 2 + 5] * 600, 8, 8, 2048, dict(), 2),
])
def test_second_launch_only_where_full_tiles_pay_for_it(sizes, bits_m, bits_v, block, hk, launches):
    from paper_2505_00347_b200 import binding as B
    params, grads = _list(sizes)
    state = B.State(sizes, bits_m, bits_v, block)
    ts = B.TensorSet(params, grads, state)
    before = B.launch_count()
    B.solo_multi_step(ts, B.hyper(lr=1e-3, beta1=0.5, **hk), 1)
    torch.cuda.synchronize()
    assert B.launch_count() - before == launches
    assert state.status() == 0
    state.destroy()


@pytest.mark.parametrize("policy,per_chunk", [(0, 1), (3, 2)])
def test_chunks_of_a_host_call_choose_and_walk_for_themselves(policy, per_chunk):
    """A large list in small chunks: one launch each, and with the two-launch form forced no walk over all the other chunks'
    tensors (nor a look at their gradient pointers, which were not uploaded)."""
    from paper_2505_00347_b200 import binding as B
    sizes = [2048 * 2 + 700, 2048, 900] * 500                    # 3 + 1 + 1 tiles
    chunk = 2048 * 5
    w = synth.workload(3, sizes=tuple(sizes[:3]))
    grads = [synth.make_grad(w, i, 1) for i in range(3)] * 500
    pinned = [g.pin_memory() for g in grads[:3]] * 500
    h = B.hyper(lr=1e-3, beta1=0.5, weight_decay=0.01, seed=6)
    got, seconds = {}, {}
    for which in (policy, 2):
        params = [torch.full((n,), 0.01, device="cuda") for n in sizes]
        state = B.State(sizes, 2, 3, 128)
        B.set_kernel_policy(which)
        try:
            for t in (1, 2):                                     # the first call creates the staging
                torch.cuda.synchronize()
                before, start = B.launch_count(), time.perf_counter()
                B.solo_multi_step_host(params, pinned, None, state, h, t, chunk_elems=chunk)
                torch.cuda.synchronize()
                seconds[which] = time.perf_counter() - start
                if which == policy:
                    assert B.launch_count() - before == 500 * per_chunk
        finally:
            B.set_kernel_policy(0)
        assert state.status() == 0
        got[which] = [state.raw_get(k) for k in KEYS] + [p.cpu() for p in params]
        state.destroy()
    for a, b in zip(got[policy], got[2]):
        assert torch.equal(a, b)
    assert seconds[policy] < 4 * seconds[2]                      # a walk over 1500 tensors per chunk: more than ten times
