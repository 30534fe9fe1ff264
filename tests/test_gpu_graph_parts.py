"""A captured step keeps the merge kernel that it was recorded with; an update of its plan may cut a row into many more
parts than that kernel asks for at once."""
import numpy as np
import pytest

from oracle.run import run_workload as oracle_run
from paper_2508_08895_b200 import binding as B, workloads as W
from parity_check import check

pytestmark = pytest.mark.gpu


def serial(prefix, heads):
    return W.build_segment_workload("parts", 75, *heads, 128, "bf16", 1e6, prefix, [[0]] * len(prefix), [[1]] * len(prefix), serial_steps=1)


# heads, prefixes at capture and after the update, parts of a row then (148 CTAs: up to 8, 16, 24 and more at capture)
@pytest.mark.parametrize("heads,at_capture,updated,most", [
    ((8, 1), [1000] * 20, [17000] + [100] * 19, (8, 107)), ((8, 1), [1400] * 14, [17000] + [100] * 13, (12, 119)),
    ((8, 1), [2800] * 7, [18500] + [100] * 6, (22, 134)), ((8, 1), [2800] * 7, [8200] * 2 + [500] * 5, (22, 62)),
    ((16, 2), [2500] * 4, [9300] + [100] * 3, (20, 69)), ((8, 1), [5000] * 4, [18500] + [300] * 3, (38, 137))])
def test_updates_to_many_parts(heads, at_capture, updated, most):
    import torch
    from paper_2508_08895_b200 import engine as E
    before, after = serial(at_capture, heads), serial(updated, heads)
    ref = oracle_run(after).outputs[-1]
    run = E.run_workload(after)                     # fills the cache of the updated lengths
    ph = after.phases[-1]
    q, k, v = (E.to_device(x, "bf16") for x in (ph.q, ph.k_new, ph.v_new))
    out, want = torch.zeros_like(q), torch.zeros_like(q)
    stream = torch.cuda.Stream()
    make = lambda desc, **kw: B.Plan(run.shape, desc, max(before.n_pool_pages, after.n_pool_pages), ph.mode, n_ctas=148, stream=stream, **kw)  # noqa: E731
    with torch.cuda.stream(stream):
        plan = make(before.phases[-1].desc, updatable=True)
        parts = [int(plan.items()["n_parts"].max())]
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            B.serial_step(plan, q, k, v, run.cache.k, run.cache.v, out, stream=stream)
        plan.update(ph.desc, stream=stream)
        parts.append(int(plan.items()["n_parts"].max()))
        graph.replay()
        fresh = make(ph.desc)
        B.serial_step(fresh, q, k, v, run.cache.k, run.cache.v, want, stream=stream)
        stream.synchronize()
        assert plan.status(stream) == 0 and fresh.status(stream) == 0
    assert tuple(parts) == most
    check(E.to_host_f32(out), ref, "bf16", f"{heads} {parts}")
    np.testing.assert_array_equal(E.to_host_f32(out), E.to_host_f32(want))
    plan.destroy(), fresh.destroy()
