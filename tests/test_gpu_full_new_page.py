"""Pages of 32 tokens all of which are new in a step: the plan's page entries count to 31."""
import pytest

from oracle.run import run_workload as oracle_run
from paper_2508_08895_b200 import binding as B, workloads as W
from parity_check import check

pytestmark = pytest.mark.gpu


def two_requests(new):
    return W.build_segment_workload("full-page", 93, 4, 1, 64, "bf16", 1e6, [1000, 1000], [[0], [0]], [[n] for n in new], serial_steps=0, page_size=32)


@pytest.mark.parametrize("new", [[31, 1], [32, 0], [16, 16], [33, 31], [64, 5]])
def test_steps(new):
    from paper_2508_08895_b200 import engine as E
    wl = two_requests(new)
    ref = oracle_run(wl)
    for n_ctas in (0, 1, 2):
        run = E.run_workload(wl, fused=True, n_ctas=n_ctas, stable_cache=True)
        check(run.outputs[-1], ref.outputs[-1], wl.dtype, f"{new} {n_ctas}")


def test_an_update_to_such_a_page_is_refused_or_right():
    """A plan of 16 + 16 new tokens that writes them itself, updated to 32 tokens of one page."""
    from paper_2508_08895_b200 import engine as E
    a, b = two_requests([16, 16]), two_requests([32, 0])
    ref = oracle_run(b)
    run = E.WorkloadRun(b, fused=True)
    for ph in b.phases[:-1]:
        run.step(ph)
    ph = b.phases[-1]
    plan = B.Plan(run.shape, a.phases[-1].desc, max(a.n_pool_pages, b.n_pool_pages), ph.mode, n_ctas=2, updatable=True)
    assert plan.info.fused_append and plan.info.n_ctas == 2
    try:
        plan.update(ph.desc)
    except B.AspdError as e:
        assert e.status == -3                                   # ASPD_ERR_UNSUPPORTED: the caller makes a new plan
        return
    q, k, v = (E.to_device(x, b.dtype) for x in (ph.q, ph.k_new, ph.v_new))
    out = q.clone()
    B.branch_step(plan, q, k, v, run.cache.k, run.cache.v, out)
    check(E.to_host_f32(out), ref.outputs[-1], b.dtype, "updated")
