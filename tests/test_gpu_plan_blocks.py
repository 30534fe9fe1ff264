"""Device blocks of destroyed plans: the park follows the sizes a program uses now (GPU)."""
import pytest

from paper_2508_08895_b200 import binding as B, workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("earlier", [0, 7, 8, 20])
def test_a_plan_size_used_after_many_others_is_parked_too(earlier):
    """However many plans of other sizes came before, the block of a plan that is destroyed is kept
    and the next plan of that size takes it: free device memory is the same while it lives and after."""
    import torch
    B.release_cached_memory()
    for n in range(earlier):
        wl = W.build_segment_workload("p", 3, 28, 4, 128, "bf16", 1e6, [16 * (n + 1)], [[0]], [[2 ** (n % 10) + n]])
        B.Plan(_shape(wl), wl.phases[-1].desc, wl.n_pool_pages, B.MODE_BRANCH).destroy()
    wl = W.build_segment_workload("big", 3, 28, 4, 128, "bf16", 1e6, [64], [[0]], [[3000]])    # a block of tens of MB
    ph = wl.phases[-1]
    B.Plan(_shape(wl), ph.desc, wl.n_pool_pages, B.MODE_BRANCH).destroy()
    torch.cuda.synchronize()
    parked = torch.cuda.mem_get_info()[0]
    plan = B.Plan(_shape(wl), ph.desc, wl.n_pool_pages, B.MODE_BRANCH)
    assert torch.cuda.mem_get_info()[0] == parked
    assert plan.info.workspace_bytes > (4 << 20)          # it would show
    plan.destroy()
    torch.cuda.synchronize()
    assert torch.cuda.mem_get_info()[0] == parked
    B.release_cached_memory()
    assert torch.cuda.mem_get_info()[0] > parked


def _shape(wl):
    return B.make_shape(wl.Hq, wl.Hkv, wl.d, wl.page_size, wl.dtype, wl.theta, wl.sm_scale)
