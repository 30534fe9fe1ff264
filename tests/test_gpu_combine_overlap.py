"""Steps launched one behind the other: a merge whose blocks wait on the SMs while the attention pass ends (an SM for
each block, or several), and whose partial results the next step's pass writes over."""
import numpy as np
import pytest

from oracle.run import run_workload as oracle_run
from paper_2508_08895_b200 import binding as B, workloads as W
from parity_check import check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,d,heads,page", [("bf16", 128, (4, 1), 16), ("bf16", 64, (4, 1), 16), ("f32", 128, (4, 1), 16), ("f32", 64, (4, 2), 8)])
@pytest.mark.parametrize("more", [None, 0, 1])               # one block; a block per SM; one block more
def test_back_to_back_steps(dtype, d, heads, page, more):
    """Bit for bit what each step gives by itself, and the first within the oracle's tolerance."""
    import torch
    from paper_2508_08895_b200 import engine as E
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = 1 if more is None else sms + more                    # four query heads: a block of four warps per token
    q_lens = [n // 8 + (i < n % 8) for i in range(8)]
    wl = W.build_segment_workload("overlap", 90, *heads, d, dtype, 1e6, [900], [[3] * 8], [q_lens], page_size=page, serial_steps=0)
    ref = oracle_run(wl)
    run = E.WorkloadRun(wl, fused=True)
    last = [run.step(ph) for ph in wl.phases][-1]
    ph = wl.phases[-1]
    plan = B.Plan(run.shape, ph.desc, wl.n_pool_pages, ph.mode)
    assert plan.info.n_new == n and not plan.info.direct_output and not plan.info.single_launch
    q = E.to_device(ph.q, wl.dtype)
    qs = [q.roll(i, 0) * (1 + i) for i in range(12)]
    outs = [torch.full_like(q, float("nan")) for _ in qs]
    torch.cuda.synchronize()
    for x, o in zip(qs, outs):
        B.branch_attn(plan, x, run.cache.k, run.cache.v, o)
    torch.cuda.synchronize()
    for x, o in zip(qs, outs):
        alone = torch.full_like(q, float("nan"))
        B.branch_attn(plan, x, run.cache.k, run.cache.v, alone)
        torch.cuda.synchronize()
        assert torch.equal(o, alone)
    np.testing.assert_array_equal(last, E.to_host_f32(outs[0]))
    for g, r in zip(run.outputs, ref.outputs):
        check(g, r, wl.dtype, f"{dtype} {d} {n}")
