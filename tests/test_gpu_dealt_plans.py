"""Streams dealt out whole: when a plan does so, the balance, new rows of a CTA in more than one batch, and updates that
keep the way a plan was made."""
import numpy as np
import pytest

from oracle.run import run_workload as oracle_run
from paper_2508_08895_b200 import binding as B, workloads as W
from parity_check import check

EVEN, SKEWED = [700, 710, 690], [1000, 950, 40]


def workload(prefix, n_new=1, n_br=2):
    return W.build_segment_workload("dealt", 55, 28, 4, 128, "bf16", 1e6, prefix, [[9] * n_br] * len(prefix), [[n_new] * n_br] * len(prefix),
                                    serial_steps=0)


def shape_of(wl):
    return B.make_shape(28, 4, 128, wl.page_size, "bf16", 1e6, 128 ** -0.5)


# prefixes, CTAs, dealt: twelve streams, whose split can be an even one or not
@pytest.mark.parametrize("prefix,n_ctas,dealt", [(EVEN, 6, 1), (EVEN, 7, 0), (SKEWED, 6, 0), (SKEWED, 3, 1), (EVEN, 5, 0)])
def test_rule_and_balance(prefix, n_ctas, dealt):
    wl = workload(prefix)
    plan = B.Plan(shape_of(wl), wl.phases[-1].desc, wl.n_pool_pages, wl.phases[-1].mode, n_ctas=n_ctas, host_only=True)
    assert plan.info.dealt == dealt
    items, at = plan.items(), plan.cta_ranges()
    pages = [int(items["n_pages"][at[c]:at[c + 1]].sum()) for c in range(n_ctas)]
    if dealt:                                                   # the greedy bound: no CTA above the mean by more than a stream
        assert len(items) == 12 and max(pages) <= np.mean(pages) + items["n_pages"].max() + 8 * 4


@pytest.mark.gpu
@pytest.mark.parametrize("prefix,n_ctas", [(EVEN, 6), (EVEN, 3), (SKEWED, 6), (SKEWED, 3), (EVEN, 2), (EVEN, 1)])
@pytest.mark.parametrize("n_new,n_br", [(1, 2), (2, 8)])        # (2, 8): 32 rows of every pair of streams
def test_steps(prefix, n_ctas, n_new, n_br):
    """Outputs against the oracle, and bit for bit against attention over the pools as the step left them."""
    import torch
    from paper_2508_08895_b200 import engine as E
    wl = workload(prefix, n_new, n_br)
    ref = oracle_run(wl)
    run = E.WorkloadRun(wl, fused=True, n_ctas=n_ctas, stable_cache=True)
    outs = [run.step(ph) for ph in wl.phases]
    ph = wl.phases[-1]
    plan = B.Plan(run.shape, ph.desc, wl.n_pool_pages, ph.mode, n_ctas=n_ctas)
    if n_ctas <= 3:
        assert plan.info.fused_append                           # 16 tiles and more: 64 to 192 rows of a CTA
    q = E.to_device(ph.q, wl.dtype)
    again = torch.full_like(q, float("nan"))
    B.branch_attn(plan, q, run.cache.k, run.cache.v, again)
    np.testing.assert_array_equal(outs[-1], E.to_host_f32(again))
    for g, r in zip(run.outputs, ref.outputs):
        check(g, r, wl.dtype, f"{prefix} {n_ctas}")
    assert run.cache.canaries_intact()


@pytest.mark.gpu
@pytest.mark.parametrize("first,then,n_ctas", [(EVEN, SKEWED, 6), (SKEWED, EVEN, 6), (EVEN, [690, 700, 640], 3)])
def test_an_update_keeps_the_way_of_its_plan(first, then, n_ctas):
    from paper_2508_08895_b200 import engine as E
    a, b = workload(first, 2, 8), workload(then, 2, 8)
    run = E.WorkloadRun(b, fused=True, n_ctas=n_ctas)
    for ph in b.phases[:-1]:
        run.step(ph)
    ph = b.phases[-1]
    n_pool = max(a.n_pool_pages, b.n_pool_pages)
    plan = B.Plan(run.shape, a.phases[-1].desc, n_pool, ph.mode, n_ctas=n_ctas, updatable=True)
    dealt, fused = plan.info.dealt, plan.info.fused_append
    plan.update(ph.desc)
    assert (plan.info.dealt, plan.info.fused_append) == (dealt, fused)
    q, k, v = (E.to_device(x, b.dtype) for x in (ph.q, ph.k_new, ph.v_new))
    out = q.clone()
    B.branch_step(plan, q, k, v, run.cache.k, run.cache.v, out)
    check(E.to_host_f32(out), oracle_run(b).outputs[-1], b.dtype, "updated")
    assert plan.status() == 0
