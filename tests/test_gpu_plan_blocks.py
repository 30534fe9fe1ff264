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


@pytest.mark.parametrize("n_streams", [1, 3])
def test_blocks_that_change_streams_keep_the_plans_apart(n_streams):
    """Plans made and destroyed in turn on several streams, with different steps sharing one size of block: every
    result is its own step's, also for the plans whose block was last used on another stream."""
    import torch
    from paper_2508_08895_b200 import engine as E
    wls = [W.build_segment_workload("s", 60 + i, 28, 4, 128, "bf16", 1e6, [300 + 64 * i], [[20, 9 + i]], [[1, 1]]) for i in range(3)]
    runs, want, args = [], [], []
    for wl in wls:
        run = E.WorkloadRun(wl)
        for ph in wl.phases:
            run.step(ph)
        ph = wl.phases[-1]
        runs.append(run); want.append(run.outputs[-1])
        args.append([E.to_device(x, wl.dtype) for x in (ph.q, ph.k_new, ph.v_new)])
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in range(n_streams)]
    outs = []
    for i in range(40):
        wl, run, st, (q, k, v) = wls[i % 3], runs[i % 3], streams[(i * 7 // 3) % n_streams], args[i % 3]
        out = torch.full_like(q, float("nan"))
        st.wait_stream(torch.cuda.current_stream())
        plan = B.Plan(run.shape, wl.phases[-1].desc, wl.n_pool_pages, B.MODE_BRANCH, stream=st)
        B.branch_attn(plan, q, run.cache.k, run.cache.v, out, stream=st)
        plan.destroy()
        outs.append(out)
    torch.cuda.synchronize()
    for i, out in enumerate(outs):
        assert (E.to_host_f32(out) == want[i % 3]).all(), i


@pytest.mark.parametrize("tokens,least", [(80, 1 << 30), (160, 2 << 30)])
def test_a_plan_that_just_fits_is_made(tokens, least):
    """Blocks are rounded up to sizes that plans share; with less than that free, the plan's own size will do."""
    import torch
    wl = W.build_segment_workload("near", 3, 28, 4, 128, "bf16", 1e6, [15000], [[0] * 8], [[tokens // 8] * 8])
    ph = wl.phases[-1]
    make = lambda: B.Plan(_shape(wl), ph.desc, wl.n_pool_pages, B.MODE_BRANCH, chunk_tokens=16)   # noqa: E731
    plan = make()
    need = plan.info.workspace_bytes
    assert least < need < least + (least >> 4)                  # a 16th above a power of two: rounded up by up to a quarter of it
    plan.destroy()
    torch.cuda.synchronize()
    B.release_cached_memory()
    torch.cuda.empty_cache()
    spare = torch.cuda.mem_get_info()[0] - need - (96 << 20)
    held = torch.empty(spare, dtype=torch.uint8, device="cuda")
    plan = make()
    assert plan.status() == 0
    plan.destroy()
    del held
    torch.cuda.empty_cache()
    B.release_cached_memory()
