"""The tensor-core kernel of the bf16 shapes with head_dim 64 or pages of 8 / 32 (aspd_attn_dec.cu) against
the oracle and against the CUDA-core kernel, whose fp32 queries and weights it has to equal."""
import numpy as np
import pytest

from oracle.run import run_workload as oracle_run
from paper_2508_08895_b200 import binding as B, workloads as W
from parity_check import check

pytestmark = pytest.mark.gpu

# head_dim, page size, heads (1, 4, 7, 8, 16 query heads to a KV head: row blocks of every padded size)
SHAPES = [(64, 16, (14, 2)), (64, 8, (4, 4)), (64, 32, (16, 4)), (128, 8, (28, 4)), (128, 32, (32, 4)), (64, 16, (64, 1)), (128, 32, (16, 1))]


def both(wl, tol=None, **kw):
    """Against the oracle; and against the CUDA-core kernel: two correct roundings to bf16 of results that agree to
    about 1e-6 differ in one value of some thousands, by one step (2^-8 of the value)."""
    from paper_2508_08895_b200 import engine as E
    ref = oracle_run(wl, kw.get("mask", 0))
    run, gen = E.run_workload(wl, **kw), E.run_workload(wl, kernel=B.KERNEL_GENERIC, **kw)
    assert len(run.outputs) == len(ref.outputs) > 0 and run.cache.canaries_intact()
    for g, f, r in zip(run.outputs, gen.outputs, ref.outputs):
        check(g, r, wl.dtype, f"{wl.name} {kw}", tol=tol)
        assert np.linalg.norm(g - f) <= 1e-3 * np.linalg.norm(f) and (g != f).mean() <= 0.02, (wl.name, kw, (g != f).mean())
    assert (run.cache.k == gen.cache.k).all() and (run.cache.v == gen.cache.v).all()
    return run


@pytest.mark.parametrize("d,page,heads", SHAPES)
def test_ragged_requests(d, page, heads):
    wl = W.build_segment_workload("dec", 41, *heads, d, "bf16", 1e6, [15, 16, 17, 0, 127, 129, 700],
                                  [[14, 15, 16], [0], [31, 0, 47, 1], [5, 0], [16], [127, 128, 1], [255, 99, 33]],
                                  [[1, 1, 1], [1], [1, 1, 0, 1], [1, 1], [1], [1, 1, 1], [1, 1, 1]], serial_steps=2, page_size=page)
    run = both(wl)
    plan = B.Plan(run.shape, wl.phases[-1].desc, wl.n_pool_pages, wl.phases[-1].mode, host_only=True)
    assert plan.info.kernel == B.KERNEL_MMA
    for n_ctas, fused in ((1, True), (3, False), (37, True)):
        both(wl, n_ctas=n_ctas, fused=fused, stable_cache=fused)
    both(wl, chunk_tokens=max(16, page), mask=B.MASK_SHARED)


@pytest.mark.parametrize("d,page,heads", SHAPES[:5])
def test_many_query_tokens(d, page, heads):
    """Whole branches as queries: cut streams with a separate append, and whole streams dealt to few CTAs."""
    wl = W.build_segment_workload("open", 42, *heads, d, "bf16", 1e6, [200, 33], [[0, 5, 0], [17]], [[24, 12, 7], [40]], serial_steps=1, page_size=page)
    both(wl, fused=True)
    both(wl, n_ctas=2, fused=True)


@pytest.mark.parametrize("d,page,heads", [SHAPES[0], SHAPES[3]])
def test_references_that_move(d, page, heads):
    """From slot 300 on logits 2^40 above the earlier ones: a later tile raises the references and O is rescaled; and
    keys that make every logit very negative (no reference below which weights vanish)."""
    wl = W.build_segment_workload("jump", 43, *heads, d, "bf16", 1e6, [600], [[20, 9]], [[1, 1]], page_size=page)
    for ph in wl.phases:
        if ph.label == "fill-prefix":
            ph.k_new[300:, :, d // 2 - 1] = 96.0
        if ph.q is not None:
            ph.q[:, :, d // 2 - 1] = 4.0
    both(wl, n_ctas=1, fused=True)
    for ph in wl.phases:
        ph.k_new[:, :, d // 2 - 1] = -96.0
    both(wl, n_ctas=1)


def test_plan_update_keeps_a_captured_graph_valid_with_heads_of_64():
    import torch
    from paper_2508_08895_b200 import engine as E
    wl = W.build_segment_workload("upd", 44, 14, 2, 64, "bf16", 1e6, [300, 40], [[30, 9], [50]], [[1, 1], [1]], serial_steps=6)
    run = E.WorkloadRun(wl, stable_cache=True)
    ref = oracle_run(wl)
    serial = [ph for ph in wl.phases if ph.label.startswith("serial")]
    for ph in wl.phases[:-len(serial)]:
        run.step(ph)
    q, k, v = (E.to_device(x, wl.dtype) for x in (serial[0].q, serial[0].k_new, serial[0].v_new))
    out = torch.empty_like(q)
    plan = B.Plan(run.shape, serial[0].desc, wl.n_pool_pages, B.MODE_SERIAL, updatable=True, stable_cache=True)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        B.serial_step(plan, q, k, v, run.cache.k, run.cache.v, out)
    for i, ph in enumerate(serial):
        plan.update(ph.desc)
        for t, x in zip((q, k, v), (ph.q, ph.k_new, ph.v_new)):
            t.copy_(E.to_device(x, wl.dtype))
        graph.replay()
        check(E.to_host_f32(out), ref.outputs[1 + i], wl.dtype, f"serial step {i}")
    assert plan.status() == 0
