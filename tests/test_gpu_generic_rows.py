"""The CUDA-core kernel's step with its new rows written by the pass itself, against the same step with the append kernel:
the same cache to the bit and the same outputs, also with more rows than a CTA writes itself."""
import numpy as np
import pytest

from paper_2508_08895_b200 import binding as B, workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("page", [8, 16, 32])
@pytest.mark.parametrize("hq,hkv,d,dtype", [(4, 1, 64, "f32"), (8, 2, 128, "f32"), (14, 2, 64, "bf16"), (28, 4, 128, "bf16")])
@pytest.mark.parametrize("new", [1, 3, 24])
def test_rows_written_by_the_pass(page, hq, hkv, d, dtype, new):
    from paper_2508_08895_b200 import engine as E
    prior = [[31, 0, 7], [16], [15, 40]]
    wl = W.build_segment_workload("rows", 74, hq, hkv, d, dtype, 1e4, [100, 0, 33], prior, [[new] * len(p) for p in prior], serial_steps=1, page_size=page)
    sep, own = (E.run_workload(wl, kernel=B.KERNEL_GENERIC, fused=f, stable_cache=f) for f in (False, True))
    assert len(own.outputs) == len(sep.outputs) > 0 and own.cache.canaries_intact()
    # the separate route rotates at the caller's positions with its own sines: the same formula, so the same bits
    assert (own.cache.k == sep.cache.k).all() and (own.cache.v == sep.cache.v).all()
    for g, f in zip(own.outputs, sep.outputs):
        assert np.array_equal(g, f)
