"""What aspd_attn_static takes: plans that are cut for speed into more items than its scratch has room for are made with
fewer and longer ones."""
import numpy as np
import pytest

from oracle.run import run_workload as oracle_run
from paper_2508_08895_b200 import binding as B, workloads as W
from parity_check import check

# dtype, head_dim, page size, heads, kernel, prefixes, tokens of the branches before, new tokens: 4 to 7.2 MiB of records with a
# share of the pages for every SM, 8.0 to 9.1 as the plans of the device are cut
CASES = [("f32", 128, 16, (28, 4), B.KERNEL_AUTO, [3000], [[5] * 8], [[2] * 8]),
         ("f32", 64, 16, (4, 1), B.KERNEL_AUTO, [200] * 24, [[30] * 4] * 24, [[40] * 4] * 24),
         ("f32", 128, 32, (8, 8), B.KERNEL_AUTO, [3000] * 2, [[0] * 2] * 2, [[30] * 2] * 2),
         ("bf16", 128, 16, (28, 4), B.KERNEL_GENERIC, [3000], [[5] * 8], [[2] * 8]),
         ("bf16", 64, 8, (64, 1), B.KERNEL_GENERIC, [400] * 20, [[5] * 6] * 20, [[2] * 6] * 20),
         ("bf16", 128, 32, (64, 1), B.KERNEL_AUTO, [800] * 4, [[60] * 4] * 4, [[7] * 4] * 4)]


def made(case, **kw):
    dtype, d, page, heads, kernel, prefix, prior, new = case
    wl = W.build_segment_workload("scratch", 97, *heads, d, dtype, 1e4, prefix, prior, new, serial_steps=0, page_size=page)
    ph = wl.phases[-1]
    shape = B.make_shape(*heads, d, page, dtype, 1e4, wl.sm_scale)
    return wl, ph, B.Plan(shape, ph.desc, wl.n_pool_pages, ph.mode, kernel=kernel, **kw)


@pytest.mark.parametrize("case", range(len(CASES)))
def test_host_only_plans_fit(case):
    _, ph, plan = made(CASES[case], host_only=True)
    (hq, hkv), d, i = CASES[case][3], CASES[case][1], plan.info
    records = i.n_partials * (hq // hkv) * (4 * d + 8)
    tables = 40 * i.n_items + 16 * i.n_ctas + 8 * i.n_stream_pages + i.n_new * (16 + 4 * d + 4 * hkv + 8) + 8 * 256
    assert records + tables <= B.STATIC_SCRATCH_BYTES - 256
    # every page of every stream is in one item still
    it = plan.items()
    for key in set(zip(it["row_block"].tolist(), it["kv_head"].tolist())):
        mine = it[(it["row_block"] == key[0]) & (it["kv_head"] == key[1])]
        assert (mine["part_slot"] == np.arange(len(mine))).all() and (mine["page0"][:-1] + mine["n_pages"][:-1] == mine["page0"][1:]).all()


@pytest.mark.gpu
@pytest.mark.parametrize("case", range(len(CASES)))
def test_the_call_takes_them(case):
    import torch
    from paper_2508_08895_b200 import engine as E
    wl, ph, plan = made(CASES[case], host_only=True)
    ref = oracle_run(wl)
    run = E.WorkloadRun(wl, kernel=CASES[case][4])
    for x in wl.phases:
        run.step(x)
    q = E.to_device(ph.q, wl.dtype)
    out = torch.full_like(q, float("nan"))
    B.attn_static(plan, q, run.cache.k, run.cache.v, out)
    check(E.to_host_f32(out), ref.outputs[-1], wl.dtype, f"case {case}")
    assert B.static_status() == 0
