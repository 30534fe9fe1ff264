"""An item's first tile against a reference of 0, as the tensor-core kernels take it: logits so low or so high that the
tile has to be done again with the rows' own maxima, and rows that see their first key tiles later."""
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
