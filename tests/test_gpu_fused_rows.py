"""The fused step's new rows inside the attention pass: tiles that the producers patch (plans of at most two tiles per
CTA) and tiles copied after the append (longer plans)."""
import numpy as np
import pytest

from oracle.run import run_workload as oracle_run
from paper_2508_08895_b200 import binding as B, workloads as W
from parity_check import check

pytestmark = pytest.mark.gpu

CASES = [
    # prefix, tokens of every branch before the step, new tokens per branch, CTAs (0: automatic)
    ([0], [[1]], [[1]], 0),                                            # a single page, a single tile
    ([2048], [[128] * 4], [[1] * 4], 0),                               # one tile per CTA
    ([112], [[15, 0, 16, 31, 7, 0, 1, 2]], [[1] * 8], 4),              # a tile whose eight pages all get a row
    ([130], [[15, 0, 16, 31, 7, 0, 1, 2]], [[1] * 8], 4),              # two tiles, new rows in both slots
    ([40, 0, 17], [[14, 3], [0, 0], [9]], [[2, 2], [3, 1], [5]], 6),   # several rows of a page, several items per CTA
    ([40], [[0, 5, 16]], [[3, 3, 3]], 2),                              # eighteen rows of a CTA, of two KV heads (a fused step takes up to 20)
    ([700, 300], [[100, 30, 5], [60]], [[1, 1, 1], [1]], 3),           # many tiles per CTA: not patched
    ([16 * 24], [[255] * 8], [[1] * 8], 4),                            # many tiles, new rows in every second one
]


@pytest.mark.parametrize("stable", [False, True])
@pytest.mark.parametrize("case", range(len(CASES)))
def test_fused_rows_reach_the_scores_and_the_pools(case, stable):
    """Outputs against the oracle, and bit for bit against attention over the pools as the step left them: what the
    scores saw is what was stored."""
    import torch
    from paper_2508_08895_b200 import engine as E
    prefix, prior, q_lens, n_ctas = CASES[case]
    wl = W.build_segment_workload("fused", 70 + case, 28, 4, 128, "bf16", 1e6, prefix, prior, q_lens, serial_steps=1)
    ref = oracle_run(wl)
    run = E.WorkloadRun(wl, fused=True, n_ctas=n_ctas, stable_cache=stable)
    for i, ph in enumerate(wl.phases):
        out = run.step(ph)
        if not ph.compare:
            continue
        plan = B.Plan(run.shape, ph.desc, wl.n_pool_pages, ph.mode, n_ctas=n_ctas)
        assert plan.info.fused_append
        q = E.to_device(ph.q, wl.dtype)
        again = torch.full_like(q, float("nan"))
        (B.branch_attn if ph.mode == B.MODE_BRANCH else B.serial_attn)(plan, q, run.cache.k, run.cache.v, again)
        np.testing.assert_array_equal(out, E.to_host_f32(again))
    for g, r in zip(run.outputs, ref.outputs):
        check(g, r, wl.dtype, f"case {case}")
    assert run.cache.canaries_intact()
