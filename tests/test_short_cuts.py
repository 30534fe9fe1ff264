"""How steps of a few tiles per CTA are cut (host integers only): every stream is covered, and no CTA has two tiles where
all tiles fit on CTAs of their own."""
import numpy as np
import pytest

from paper_2508_08895_b200 import binding as B, workloads as W

SMS = 148


@pytest.mark.parametrize("d,page", [(128, 16), (64, 16), (64, 8), (128, 32)])
@pytest.mark.parametrize("seed", range(6))
def test_tiles_of_short_steps(d, page, seed):
    rng = np.random.default_rng(seed)
    n_req = int(rng.integers(1, 8))
    prefix = [int(x) for x in rng.integers(0, 3000 // n_req + 40, size=n_req)]
    prior = [[int(x) for x in rng.integers(0, 200, size=int(rng.integers(1, 6)))] for _ in range(n_req)]
    wl = W.build_segment_workload("short", 73, 28, 4, d, "bf16", 1e6, prefix, prior, [[1] * len(p) for p in prior], serial_steps=1, page_size=page)
    shape = B.make_shape(wl.Hq, wl.Hkv, wl.d, wl.page_size, wl.dtype, wl.theta, wl.sm_scale)
    for ph in [x for x in wl.phases if x.q is not None]:
        plan = B.Plan(shape, ph.desc, wl.n_pool_pages, ph.mode, host_only=True)
        items, first = plan.items(), plan.cta_ranges()
        assert plan.info.n_ctas == len(first) - 1 <= SMS and first[-1] == len(items)
        ppt = 128 // page
        tiles = -(-items["n_pages"] // ppt)
        streams = {}
        for it in items:                             # in order, without a gap, from key 0 to the stream's end
            key = (int(it["request"]), int(it["row_block"]), int(it["kv_head"]))
            done, parts = streams.get(key, (0, 0))
            assert it["key0"] == done * page and it["part_slot"] == parts
            streams[key] = (done + int(it["n_pages"]), parts + 1)
        for it in items:
            key = (int(it["request"]), int(it["row_block"]), int(it["kv_head"]))
            assert it["n_parts"] == streams[key][1]
        assert sum(n for n, _ in streams.values()) == int(items["n_pages"].sum()) >= plan.info.n_stream_pages
        if sum(-(-n // ppt) for n, _ in streams.values()) <= SMS:
            assert max(int(tiles[first[c]:first[c + 1]].sum()) for c in range(len(first) - 1)) == 1
        plan.destroy()


@pytest.mark.parametrize("heads,d,page,n_req,prefix,seed", [((16, 2), 128, 16, 10, (500, 1600), 20), ((4, 1), 64, 8, 26, (470, 1420), 0),
                                                            ((4, 1), 64, 8, 26, (470, 1420), 30)])
def test_cuts_keep_the_pass_that_writes_the_new_rows(heads, d, page, n_req, prefix, seed):
    """Up to 24 branches of one token: by tiles a CTA would get more new rows than it writes itself, by pages none does."""
    rng = np.random.default_rng(seed)
    lens = [int(x) for x in rng.integers(*prefix, size=n_req)]
    prior = [[0] * int(rng.integers(1, 25)) for _ in range(n_req)]
    wl = W.build_segment_workload("rows", 73, *heads, d, "bf16", 1e6, lens, prior, [[1] * len(p) for p in prior], page_size=page)
    ph = wl.phases[-1]
    plan = B.Plan(B.make_shape(*heads, d, page, "bf16", 1e6, d ** -0.5), ph.desc, wl.n_pool_pages, ph.mode, host_only=True)
    assert plan.info.fused_append == 1
    plan.destroy()
