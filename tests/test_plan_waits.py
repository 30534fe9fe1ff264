"""The cuts of key streams among the CTAs: complete and in order, with fewer pages for CTAs that come to new rows at once."""
import numpy as np
import pytest

from paper_2508_08895_b200 import binding as B, workloads as W


@pytest.mark.parametrize("prefix,prior,n_ctas", [([4000], [[100] * 8], 36), ([4000], [[100] * 8], 37), ([700, 2500, 90], [[20, 0], [255, 3, 70], [1]], 20),
                                                 ([0, 1], [[2], [0]], 3), ([6000, 5000], [[0] * 8] * 2, 148)])
def test_cuts(prefix, prior, n_ctas):
    wl = W.build_segment_workload("cuts", 3, 28, 4, 128, "bf16", 1e6, prefix, prior, [[1] * len(p) for p in prior], serial_steps=0)
    ph = wl.phases[-1]
    plan = B.Plan(B.make_shape(28, 4, 128, wl.page_size, "bf16", 1e6, 128 ** -0.5), ph.desc, wl.n_pool_pages, ph.mode, n_ctas=n_ctas, host_only=True)
    it, at, vis = plan.items(), plan.cta_ranges(), plan.stream_pages()[0]
    assert at[0] == 0 and at[-1] == len(it) and (np.diff(at) >= 0).all() and len(at) == plan.info.n_ctas + 1
    streams = {}
    for x in it:
        streams.setdefault((int(x["request"]), int(x["q_tok0"]), int(x["kv_head"])), []).append(x)
    for parts in streams.values():
        assert [int(x["part_slot"]) for x in parts] == list(range(len(parts))) and all(int(x["n_parts"]) == len(parts) for x in parts)
        for a, b in zip(parts, parts[1:]):
            assert int(a["page0"]) + int(a["n_pages"]) == int(b["page0"])
    assert sum(int(x["n_pages"]) for x in it) == 4 * len(vis)
    pages = np.array([int(it["n_pages"][at[c]:at[c + 1]].sum()) for c in range(len(at) - 1)])
    if prefix == [4000]:                                        # page 250 + 7 b + 6 of the stream has branch b's new row
        new = {256 + 7 * b for b in range(8)}
        first = [next((i for i, p in enumerate(p for x in it[at[c]:at[c + 1]] for p in range(int(x["page0"]), int(x["page0"] + x["n_pages"])))
                       if p in new), 99) for c in range(len(pages) - 1)]
        # A CTA with a new row in its page f < 10 is charged 10 - f pages; cuts are rounded to tiles of 8, up to 4 pages off
        # either way, which evens out: less on average, and no CTA (but the last, which takes what is left) above the mean
        # by more than a tile and the charge of the others.
        at_once = np.array([f < 8 for f in first])
        assert at_once.sum() >= 4 and pages[:-1][at_once].mean() < pages[:-1][~at_once].mean() - 1 and pages.max() <= pages.mean() + 8 + 10
