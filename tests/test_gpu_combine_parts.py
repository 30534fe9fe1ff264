"""The merge of rows cut into one part up to more than the 64 that share a maximum (a new plan each, so in the instance made
for that many; test_gpu_graph_parts.py has each instance take more)."""
import numpy as np
import pytest

from oracle.run import run_workload as oracle_run
from paper_2508_08895_b200 import binding as B, workloads as W
from parity_check import check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(28, 4, 128, "bf16"), (14, 2, 64, "bf16"), (4, 1, 64, "f32")])
@pytest.mark.parametrize("parts", [(1, 7), (8, 9), (16, 17), (24, 25), (31, 33), (64, 65), (2, 130)])
def test_rows_of_many_parts(shape, parts):
    from paper_2508_08895_b200 import engine as E
    hq, hkv, d, dtype = shape
    # a forced cut every 16 keys: as many parts as pages (the serial token's own page is one of them)
    wl = W.build_segment_workload("parts", 72, hq, hkv, d, dtype, 1e4, [max(0, 16 * (n - 1)) for n in parts], [[0], [0]], [[1], [1]])
    ref = oracle_run(wl)
    run = E.run_workload(wl, chunk_tokens=16)
    ph = wl.phases[-1]
    plan = B.Plan(run.shape, ph.desc, wl.n_pool_pages, ph.mode, chunk_tokens=16, host_only=True)
    assert sorted(set(int(x) for x in plan.items()["n_parts"])) == sorted(set(parts))
    plan.destroy()
    for g, r in zip(run.outputs, ref.outputs):
        check(g, r, wl.dtype, f"{shape} {parts}")
