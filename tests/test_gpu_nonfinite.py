"""Inf and NaN in one branch's values stay in that branch: to rows that do not see them they do not exist."""
import numpy as np
import pytest

from paper_2508_08895_b200 import binding as B, workloads as W

pytestmark = pytest.mark.gpu

# dtype, head_dim, page size, heads, kernel
SHAPES = [("f32", 64, 16, (4, 1), B.KERNEL_AUTO), ("f32", 128, 8, (28, 4), B.KERNEL_AUTO), ("f32", 64, 32, (64, 2), B.KERNEL_AUTO),
          ("bf16", 128, 16, (28, 4), B.KERNEL_GENERIC), ("bf16", 64, 16, (14, 2), B.KERNEL_GENERIC),
          ("bf16", 64, 16, (14, 2), B.KERNEL_AUTO), ("bf16", 128, 8, (28, 4), B.KERNEL_AUTO), ("bf16", 64, 32, (64, 1), B.KERNEL_AUTO),
          ("bf16", 128, 32, (16, 2), B.KERNEL_AUTO), ("bf16", 64, 8, (4, 4), B.KERNEL_AUTO)]


def run(dtype, d, page, heads, kernel, poison, fill=0, **kw):
    """Outputs of the parallel step (rows by token) and of the serial step after it.  poison: list of (phase label, token of
    the phase, KV head, element, value) put into the phase's values; fill: byte the pools hold before their first use."""
    from paper_2508_08895_b200 import engine as E
    wl = W.build_segment_workload("nf", 95, *heads, d, dtype, 1e4, [130, 20], [[40, 17, 3], [9, 30]], [[1, 2, 1], [1, 1]], serial_steps=1, page_size=page)
    for label, t, h, e, v in poison:
        next(ph for ph in wl.phases if ph.label == label).v_new[t, h, e] = v
    r = E.WorkloadRun(wl, kernel=kernel, **kw)
    r.cache.k.fill_(fill), r.cache.v.fill_(fill)
    for ph in wl.phases:
        r.step(ph)
    return r.outputs


def same(out, exp, shape):
    """Bit for bit; from the tensor-core kernel, which takes items with such values again on the CUDA cores, up to the rounding
    to bf16 of results that agree to about 1e-6: one value of some thousands, by one step (2^-8 of the value)."""
    if shape[0] == "f32" or shape[4] == B.KERNEL_GENERIC:
        return np.testing.assert_array_equal(out, exp)
    fin = np.isfinite(exp)
    np.testing.assert_array_equal(out[~fin], exp[~fin])
    assert np.isfinite(out[fin]).all() and np.linalg.norm(out[fin] - exp[fin]) <= 1e-3 * np.linalg.norm(exp[fin])
    assert (out[fin] != exp[fin]).mean() <= 0.02


@pytest.mark.parametrize("kw", [dict(), dict(n_ctas=1, fused=True), dict(n_ctas=3, fused=True, stable_cache=True)])
@pytest.mark.parametrize("shape", SHAPES)
def test_they_reach_the_rows_that_see_them_and_no_other(shape, kw):
    (dtype, d, page, heads, kernel), G = shape, shape[3][0] // shape[3][1]
    clean = run(*shape, [], **kw)
    last = heads[1] - 1
    # tokens of the fill phase: request 0's branches (40, 17, 3), request 1's (9, 30).  Request 0: Inf in its first branch, NaN
    # in its second; request 1: both signs of Inf in its second; in the step itself, Inf in request 1's first branch
    poison = [("fill-branches", 5, 0, 3, np.inf), ("fill-branches", 45, last, d - 1, np.nan), ("fill-branches", 70, 0, 7, np.inf),
              ("fill-branches", 72, 0, 7, -np.inf), ("fill-branches", 75, 0, 8, -np.inf), ("parallel-step", 4, last, 0, np.inf)]
    got = run(*shape, poison, **kw)
    # row of the step (tokens 0; 1 2; 3 | 4; 5) -> what its elements become
    want = [{(0, 3): np.inf}, {(last, d - 1): np.nan}, {(last, d - 1): np.nan}, {}, {(last, 0): np.inf}, {(0, 7): np.nan, (0, 8): -np.inf}]
    serial = [{**want[0], **want[1]}, {**want[4], **want[5]}]              # the main branch sees all of its request
    for out, ref, rows in ((got[0], clean[0], want), (got[1], clean[1], serial)):
        exp = ref.copy()
        for t, cells in enumerate(rows):
            for (h, e), v in cells.items():
                exp[t, h * G:(h + 1) * G, e] = v
        same(out, exp, shape)


@pytest.mark.parametrize("shape", SHAPES)
def test_rows_that_no_token_was_written_to_do_not_matter(shape):
    for a, b in zip(run(*shape, []), run(*shape, [], fill=255)):            # 0xff bytes: NaN in either type
        same(a, b, shape)
