"""The merge's rows, four to a block, for head counts that blocks and groups do not divide."""
import pytest

from oracle.run import run_workload as oracle_run
from paper_2508_08895_b200 import workloads as W
from parity_check import check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("heads", [(1, 1), (3, 3), (5, 1), (14, 2), (21, 7), (63, 1)])
@pytest.mark.parametrize("d,dtype", [(64, "bf16"), (128, "bf16"), (64, "f32")])
def test_rows(heads, d, dtype):
    from paper_2508_08895_b200 import engine as E
    wl = W.build_segment_workload("rows", 80, *heads, d, dtype, 1e4, [70, 0, 33], [[5, 0, 9], [40], [0, 20]], [[1, 2, 1], [3], [1, 1]], serial_steps=1)
    ref, run = oracle_run(wl), E.run_workload(wl, chunk_tokens=16)
    for g, r in zip(run.outputs, ref.outputs):
        check(g, r, dtype, f"{heads} {d} {dtype}")
