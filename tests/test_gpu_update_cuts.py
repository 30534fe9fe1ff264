"""Updates of plans cut by tiles (short steps, no number of CTAs given): lengths that change the cut, and steps that the plan
cannot take, which are refused and leave it and the captured step as they were."""
import numpy as np
import pytest

from oracle.run import run_workload as oracle_run
from paper_2508_08895_b200 import binding as B, workloads as W
from parity_check import check

pytestmark = pytest.mark.gpu


def serial(prefix, heads, d, page):
    return W.build_segment_workload("cuts", 78, *heads, d, "bf16", 1e6, prefix, [[0]] * len(prefix), [[1]] * len(prefix), serial_steps=1, page_size=page)


@pytest.mark.parametrize("heads,d,page,few,many", [((28, 4), 128, 16, [2056, 3976, 2741], [2412, 4665, 3216]),
                                                   ((32, 8), 64, 16, [363, 3401, 758, 3586], [395, 3709, 826, 3910]),
                                                   ((28, 4), 128, 32, [3759, 3805, 2123, 823, 2461], [2622, 4006, 877, 4055, 2262])])
def test_updates_that_change_the_cut(heads, d, page, few, many):
    import torch
    from paper_2508_08895_b200 import engine as E
    lens = [few, many, few[::-1], [n + 40 for n in many]]
    steps = [serial(x, heads, d, page) for x in lens]
    runs = [E.run_workload(wl) for wl in steps]
    big = max(runs, key=lambda r: r.cache.k.numel())
    pool_k, pool_v = torch.zeros_like(big.cache.k), torch.zeros_like(big.cache.v)
    q, k, v = (E.to_device(x, "bf16") for x in (steps[0].phases[-1].q, steps[0].phases[-1].k_new, steps[0].phases[-1].v_new))
    out = torch.zeros_like(q)
    n_pool, mode, stream = max(wl.n_pool_pages for wl in steps), steps[0].phases[-1].mode, torch.cuda.Stream()
    ppt, longest = 128 // page, []
    with torch.cuda.stream(stream):
        plan = B.Plan(runs[0].shape, steps[0].phases[-1].desc, n_pool, mode, updatable=True, stable_cache=True, stream=stream)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            B.serial_step(plan, q, k, v, pool_k, pool_v, out, stream=stream)

        def replayed(i):
            pool_k[:runs[i].cache.k.numel()] = runs[i].cache.k
            pool_v[:runs[i].cache.v.numel()] = runs[i].cache.v
            for dst, src in zip((q, k, v), (steps[i].phases[-1].q, steps[i].phases[-1].k_new, steps[i].phases[-1].v_new)):
                dst.copy_(E.to_device(src, "bf16"))
            graph.replay()
            stream.synchronize()
            assert plan.status(stream) == 0
            check(E.to_host_f32(out), runs[i].outputs[-1], "bf16", f"{heads} {lens[i]}")
            check(E.to_host_f32(out), oracle_run(steps[i]).outputs[-1], "bf16", f"{heads} {lens[i]}")

        for i, wl in enumerate(steps):
            if i:
                plan.update(wl.phases[-1].desc, stream=stream)
            longest.append(int((-(-plan.items()["n_pages"] // ppt)).max()))
            replayed(i)
        assert longest[0] == longest[2] < longest[1] == longest[3]
        n_ctas, items = plan.info.n_ctas, plan.items()
        assert len(items) <= n_ctas <= 148                     # cut by tiles: an item to a CTA
        # more streams than the plan has CTAs, more new tokens, fewer: another launch sequence
        for other in ([40] * 40, few + [10], few[1:]):
            with pytest.raises(B.AspdError) as e:
                plan.update(serial(other, heads, d, page).phases[-1].desc, stream=stream)
            assert e.value.status == -3                        # ASPD_ERR_UNSUPPORTED
        assert plan.info.n_ctas == n_ctas and np.array_equal(plan.items(), items)
        out.zero_()
        replayed(len(steps) - 1)
    plan.destroy()
