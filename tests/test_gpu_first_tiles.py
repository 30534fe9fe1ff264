"""Logits so low or so high that a tile cannot be taken against the reference that its rows have: an item's first tile, and
rows that see their first key tiles later."""
import numpy as np
import pytest

from oracle.run import run_workload as oracle_run
from paper_2508_08895_b200 import workloads as W
from parity_check import check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_ctas", [0, 1])
@pytest.mark.parametrize("d,heads", [(128, (28, 4)), (128, (4, 4)), (64, (14, 2))])
@pytest.mark.parametrize("logit", [-32.0, -4.0, 5.0])
def test_equal_logits_far_from_zero(d, heads, n_ctas, logit):
    """Every logit near ``logit * 32 / sqrt(d)`` (keys and queries along the slowest rotary pair, which hardly turns): the
    softmax is close to uniform whatever the reference.  The second request has no prefix, so that with one CTA the rows
    of its second branch see nothing in the item's first two tiles."""
    from paper_2508_08895_b200 import engine as E
    wl = W.build_segment_workload("first", 71, *heads, d, "bf16", 1e6, [150, 0], [[7, 20], [300, 40]], [[1, 1], [1, 1]], serial_steps=1)
    for ph in wl.phases:
        ph.k_new[:] = 0.0
        ph.k_new[:, :, d // 2 - 1] = 32.0
        if ph.q is not None:
            ph.q[:] = 0.0
            ph.q[:, :, d // 2 - 1] = logit
    ref = oracle_run(wl)
    for fused in (False, True):
        run = E.run_workload(wl, n_ctas=n_ctas, fused=fused, stable_cache=fused)
        for g, r in zip(run.outputs, ref.outputs):
            assert np.isfinite(g).all()
            check(g, r, wl.dtype, f"{d} {heads} {n_ctas} {logit} {fused}")


@pytest.mark.parametrize("d,heads,page", [(128, (28, 4), 16), (128, (4, 4), 16), (128, (64, 1), 16), (64, (14, 2), 16), (128, (28, 4), 8)])
def test_the_largest_weight_is_one(d, heads, page):
    """Branches that begin a sequence: every token sees itself alone, and its output is its V to the bit.  The weights that
    meet V are bf16 and their sum is not, so that a weight of 2^x that bf16 does not hold would show."""
    from paper_2508_08895_b200 import engine as E
    prior = [[0], [0, 0, 0], [0] * 8]
    wl = W.build_segment_workload("lone", 76, *heads, d, "bf16", 1e6, [0, 0, 0], prior, [[1] * len(p) for p in prior], serial_steps=0, page_size=page)
    for fused in (False, True):
        run = E.run_workload(wl, fused=fused, stable_cache=fused)
        v = wl.phases[-1].v_new
        assert np.array_equal(run.outputs[-1], np.repeat(v, heads[0] // heads[1], axis=1))
