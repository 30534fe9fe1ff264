"""The two-tile kernel with rows whose reference maximum moves at every half tile, so that the rows' sums are rescaled between
any two P.V: the wait for the one before, in both groups, over items of any length."""
import numpy as np
import pytest

from oracle.run import run_workload as oracle_run
from paper_2508_08895_b200 import engine as E, workloads as W
from parity_check import check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_ctas", [1, 3])
@pytest.mark.parametrize("prefix", [[700, 64, 1000], [576, 129, 65], [448, 0, 127]])
def test_reference_moves_at_every_half(prefix, n_ctas):
    """Logits rise by 49 in log2 units every 64 keys of the prefix for three heads of four (keys and queries along the slowest
    rotary pair, which hardly turns), and stay at 0 for the fourth."""
    wl = W.build_segment_workload("stairs", 79, 28, 4, 128, "bf16", 1e6, prefix, [[5, 0], [0], [70]], [[30, 7], [40], [19]], serial_steps=0)
    assert len(wl.phases) >= 2
    lens = [p for p in prefix if p > 0]
    fill, step = wl.phases[0], wl.phases[-1]
    for ph in wl.phases:
        ph.k_new[:] = 0.0
    at = np.concatenate([np.arange(p) for p in lens])
    assert len(at) == len(fill.k_new)
    fill.k_new[:, :, 63] = 12.0 * (at // 64)[:, None]
    step.q[:] = 0.0
    step.q[:, np.arange(28) % 4 != 0, 63] = 32.0
    ref = oracle_run(wl)
    run = E.run_workload(wl, n_ctas=n_ctas, wide_rows=256)
    for g, r in zip(run.outputs, ref.outputs):
        assert np.isfinite(g).all()
        check(g, r, wl.dtype, f"{prefix} {n_ctas}")
