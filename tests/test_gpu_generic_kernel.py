"""The CUDA-core kernel at the edges of its chunks of 32 keys and of its rows per warp, in fp32 against the oracle."""
import pytest

from oracle.run import run_workload as oracle_run
from paper_2508_08895_b200 import binding as B, workloads as W
from parity_check import check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,page,heads", [(64, 16, (4, 1)), (64, 8, (8, 8)), (128, 32, (12, 4)), (128, 8, (28, 4)), (64, 32, (64, 1)), (128, 16, (34, 2))])
def test_chunk_and_row_edges(d, page, heads):
    from paper_2508_08895_b200 import engine as E
    wl = W.build_segment_workload("gen", 51, *heads, d, "f32", 1e4, [31, 32, 33, 0, 65, 250],
                                  [[30, 31, 32], [0], [63, 0, 1], [5, 0], [64], [8, 16, 9, 33, 1]],
                                  [[1, 1, 1], [1], [1, 0, 1], [2, 1], [9], [1] * 5], serial_steps=2, page_size=page)
    for mask in (B.MASK_BRANCH_INVISIBLE, B.MASK_SHARED):
        ref = oracle_run(wl, mask)
        for kw in (dict(), dict(n_ctas=1), dict(n_ctas=7, fused=True), dict(chunk_tokens=32)):
            run = E.run_workload(wl, mask=mask, **kw)
            assert len(run.outputs) == len(ref.outputs) == 3 and run.cache.canaries_intact()
            for g, r in zip(run.outputs, ref.outputs):
                check(g, r, "f32", f"{kw} mask {mask}")
