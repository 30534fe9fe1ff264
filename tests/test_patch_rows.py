"""Plans whose fused step patches its tiles: the new rows of a CTA wait in shared memory, where twenty have a place."""
import random
from collections import Counter

import numpy as np
import pytest

from oracle.run import run_workload as oracle_run
from paper_2508_08895_b200 import binding as B, workloads as W
from parity_check import check

MOST = 20                 # new rows of a CTA that a patching launch has room for
# prefix, tokens of every branch before the step, new tokens per branch, KV heads, chunk_tokens, CTAs.  Forced cuts leave
# the last CTA with 24 to 96 rows in 16 to 361 tiles, while a CTA has two tiles or less on average.
PILED = [(200, [10] * 8, [1] * 8, 4, 16, 0), (200, [0, 9, 9], [5, 4, 4], 4, 48, 0), (200, [0, 9, 9], [5, 4, 4], 4, 16, 0),
         (600, [0, 9, 9], [5, 4, 4], 4, 80, 0), (1000, [0] * 4, [4] * 4, 8, 16, 0), (200, [10] * 8, [1] * 8, 4, 16, 11)]


def workload(prefix, prior, new, hkv=4):
    return W.build_segment_workload("patch", 91, 7 * hkv, hkv, 128, "bf16", 1e6, [prefix], [prior], [new], serial_steps=0)


def plan_of(wl, **kw):
    ph = wl.phases[-1]
    return B.Plan(B.make_shape(wl.Hq, wl.Hkv, 128, 16, "bf16", 1e6, 128 ** -0.5), ph.desc, wl.n_pool_pages, ph.mode, **kw)


def rows_and_tiles(plan, desc, mode):
    """(new rows, tiles) of every CTA."""
    _, slot, req = B.positions(desc, mode)
    new = Counter((desc["page_ids"][desc["page_begin"][req] + slot // 16]).tolist())
    per_page = np.array([new[p] for p in plan.stream_pages()[0].tolist()] + [0])
    it, at = plan.items(), plan.cta_ranges()
    rows = [sum(int(per_page[x["page0"]:x["page0"] + x["n_pages"]].sum()) for x in it[a:b]) for a, b in zip(at, at[1:])]
    return rows, [sum((int(x["n_pages"]) + 7) // 8 for x in it[a:b]) for a, b in zip(at, at[1:])]


def check_bound(plan, desc, mode):
    """A fused plan of at most two tiles per CTA on average patches, and then no CTA has more rows than have a place."""
    info = plan.info
    it = plan.items()
    few = not info.dealt and int(it["n_pages"].sum()) <= 16 * info.n_ctas
    rows, tiles = rows_and_tiles(plan, desc, mode)
    if info.fused_append and few:
        assert max(rows) <= MOST, (rows, tiles)
    assert info.patch_tiles == int(bool(info.fused_append and few))
    return rows, tiles


@pytest.mark.parametrize("prefix,prior,new,hkv,chunk,n_ctas", PILED)
def test_a_cta_with_more_rows_takes_the_append_kernel(prefix, prior, new, hkv, chunk, n_ctas):
    wl = workload(prefix, prior, new, hkv)
    plan = plan_of(wl, chunk_tokens=chunk, n_ctas=n_ctas, host_only=True)
    rows, tiles = check_bound(plan, wl.phases[-1].desc, B.MODE_BRANCH)
    assert max(rows) > MOST and tiles[int(np.argmax(rows))] >= 16 and not plan.info.fused_append


@pytest.mark.parametrize("rows,tiles", [(20, 1), (21, 1), (33, 1), (20, 16), (21, 16), (32, 16), (33, 16), (20, 17), (21, 17), (21, 21), (32, 32), (33, 32)])
def test_either_side_of_the_bound(rows, tiles):
    """One KV head, one CTA asked for: all rows of the step are its own."""
    n_br = tiles                                                # a branch a page; every page a tile of its own
    new = [rows // n_br + (b < rows % n_br) for b in range(n_br)]
    wl = W.build_segment_workload("edge", 92, 1, 1, 128, "bf16", 1e6, [0], [[0] * n_br], [new], serial_steps=0)
    plan = plan_of(wl, n_ctas=1, chunk_tokens=16 if tiles > 1 else 0, host_only=True)
    got = check_bound(plan, wl.phases[-1].desc, B.MODE_BRANCH)
    assert got[0] == [rows] and got[1] == [tiles]
    assert plan.info.fused_append == int(rows <= MOST or 16 < tiles >= rows)     # from 17 pages on over two tiles on average: not patched


def test_random_plans():
    rng = random.Random(5)
    fused = patched = 0
    for n in range(250):
        n_req = rng.choice([1, 1, 2, 5])
        prefix = [rng.choice([0, 16, 200, 600, rng.randint(1, 1500)]) for _ in range(n_req)]
        prior = [[rng.randint(0, 40) for _ in range(rng.randint(1, 8))] for _ in range(n_req)]
        new = [[rng.choice([1, 1, 2, 5]) for _ in p] for p in prior]
        hkv = rng.choice([1, 4, 8])
        wl = W.build_segment_workload("rnd", n, 7 * hkv, hkv, 128, "bf16", 1e6, prefix, prior, new, serial_steps=0)
        plan = plan_of(wl, chunk_tokens=rng.choice([0, 16, 48, 80, 128]), n_ctas=rng.choice([0, 0, 1, 3, 40]), host_only=True)
        check_bound(plan, wl.phases[-1].desc, B.MODE_BRANCH)
        fused += plan.info.fused_append
        patched += plan.info.patch_tiles
    assert 50 < patched < fused < 250


@pytest.mark.gpu
@pytest.mark.parametrize("prefix,prior,new,hkv,chunk,n_ctas", PILED)
def test_steps_of_such_plans(prefix, prior, new, hkv, chunk, n_ctas):
    from paper_2508_08895_b200 import engine as E
    wl = workload(prefix, prior, new, hkv)
    ref = oracle_run(wl)
    run = E.run_workload(wl, fused=True, chunk_tokens=chunk, n_ctas=n_ctas, stable_cache=True)
    for g, r in zip(run.outputs, ref.outputs):
        check(g, r, wl.dtype, f"{prefix} {chunk}")
    assert run.cache.canaries_intact()
