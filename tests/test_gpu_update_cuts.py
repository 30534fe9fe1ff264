"""Updates of plans cut by tiles (short steps, no number of CTAs given): lengths that change the cut, lengths that need more
room, and steps that the plan cannot take, which are refused and leave it and the captured step as they were."""
import numpy as np
import pytest

from oracle.run import run_workload as oracle_run
from paper_2508_08895_b200 import binding as B, workloads as W
from parity_check import check

pytestmark = pytest.mark.gpu


def serial(prefix, heads, d, page):
    return W.build_segment_workload("cuts", 78, *heads, d, "bf16", 1e6, prefix, [[0]] * len(prefix), [[1]] * len(prefix), serial_steps=1, page_size=page)


class Captured:
    """The first of some workloads' last steps, captured with an updatable plan over a pool for all of them."""

    def __init__(self, steps):
        import torch
        from paper_2508_08895_b200 import engine as E
        self.E, self.steps, self.runs = E, steps, [E.run_workload(wl) for wl in steps]
        big, ph = max(self.runs, key=lambda r: r.cache.k.numel()), steps[0].phases[-1]
        self.pools = torch.zeros_like(big.cache.k), torch.zeros_like(big.cache.v)
        self.new = [E.to_device(x, "bf16") for x in (ph.q, ph.k_new, ph.v_new)]
        self.out, self.stream = torch.zeros_like(self.new[0]), torch.cuda.Stream()
        step = B.serial_step if ph.mode == W.MODE_SERIAL else B.branch_step
        with torch.cuda.stream(self.stream):
            self.plan = B.Plan(self.runs[0].shape, ph.desc, max(wl.n_pool_pages for wl in steps), ph.mode, updatable=True, stable_cache=True,
                               stream=self.stream)
            self.graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(self.graph, stream=self.stream):
                step(self.plan, *self.new, *self.pools, self.out, stream=self.stream)

    def update(self, wl):
        self.plan.update(wl.phases[-1].desc, stream=self.stream)

    def replay(self, i):
        import torch
        E, run, ph = self.E, self.runs[i], self.steps[i].phases[-1]
        with torch.cuda.stream(self.stream):
            for dst, src in zip(self.pools, (run.cache.k, run.cache.v)):
                dst[:src.numel()] = src
            for dst, src in zip(self.new, (ph.q, ph.k_new, ph.v_new)):
                dst.copy_(E.to_device(src, "bf16"))
            self.out.zero_()
            self.graph.replay()
            self.stream.synchronize()
        assert self.plan.status(self.stream) == 0
        check(E.to_host_f32(self.out), run.outputs[-1], "bf16", f"workload {i}, a new plan")
        check(E.to_host_f32(self.out), oracle_run(self.steps[i]).outputs[-1], "bf16", f"workload {i}")


@pytest.mark.parametrize("heads,d,page,few,many", [((28, 4), 128, 16, [2056, 3976, 2741], [2412, 4665, 3216]),
                                                   ((32, 8), 64, 16, [363, 3401, 758, 3586], [395, 3709, 826, 3910]),
                                                   ((28, 4), 128, 32, [3759, 3805, 2123, 823, 2461], [2622, 4006, 877, 4055, 2262])])
def test_updates_that_change_the_cut(heads, d, page, few, many):
    steps = [serial(x, heads, d, page) for x in (few, many, few[::-1], [n + 40 for n in many])]
    cap, longest = Captured(steps), []
    for i, wl in enumerate(steps):
        if i:
            cap.update(wl)
        longest.append(int((-(-cap.plan.items()["n_pages"] // (128 // page))).max()))
        cap.replay(i)
    assert longest[0] == longest[2] < longest[1] == longest[3]
    n_ctas, items = cap.plan.info.n_ctas, cap.plan.items()
    assert len(items) <= n_ctas <= 148                         # cut by tiles: an item to a CTA
    # more streams than the plan has CTAs, more new tokens, fewer: another launch sequence
    for other in ([40] * 40, few + [10], few[1:]):
        with pytest.raises(B.AspdError) as e:
            cap.update(serial(other, heads, d, page))
        assert e.value.status == -3                            # ASPD_ERR_UNSUPPORTED
    assert cap.plan.info.n_ctas == n_ctas and np.array_equal(cap.plan.items(), items)
    cap.replay(len(steps) - 1)
    cap.plan.destroy()


RAGGED = [[26, 95, 115, 108, 147],
          [144, 91, 146, 99, 116, 40, 224, 38, 56, 162, 172, 119, 142, 208, 25, 49, 157, 108, 159, 53, 208, 66, 164]]


@pytest.mark.parametrize("heads,d,page,new,before,after", [
    ((28, 4), 128, 8, 1, ([95, 95], RAGGED), ([114, 114], RAGGED)),            # a few pages more, a third more records
    # by tiles the first plan would write its new rows itself, and the second would not
    ((14, 2), 64, 16, 12, ([25, 21, 35], [[71], [213, 212, 25], [52, 167]]), ([23, 30, 39], [[106, 25], [253], [35, 230, 161]]))])
def test_updates_that_the_cut_by_pages_takes(heads, d, page, new, before, after):
    steps = [W.build_segment_workload("room", 81, *heads, d, "bf16", 1e6, prefix, prior, [[new] * len(p) for p in prior], serial_steps=0, page_size=page)
             for prefix, prior in (before, after)]
    cap = Captured(steps)
    cap.replay(0)
    cap.update(steps[1])
    cap.replay(1)
    cap.plan.destroy()
