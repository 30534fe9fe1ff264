"""How many new rows a fused step's CTAs write themselves: twenty, or a few to a tile where a CTA has many tiles."""
import random
from collections import Counter

import numpy as np
import pytest

from paper_2508_08895_b200 import binding as B


def descriptors(prefix, prior, new):
    up = lambda n: -(-n // 16) * 16   # noqa: E731
    d = {k: [] for k in ("prefix_len", "n_branches", "branch_begin", "page_begin", "n_pages", "tail_off", "tail_len", "br_kv_off", "br_kv_len", "br_q_len")}
    pages = 0
    for p, pr, nw in zip(prefix, prior, new):
        at = up(p)
        row = dict(prefix_len=p, n_branches=len(pr), branch_begin=len(d["br_kv_off"]), page_begin=pages, tail_len=0)
        for a, n in zip(pr, nw):
            for key, x in (("br_kv_off", at), ("br_kv_len", a + n), ("br_q_len", n)):
                d[key].append(x)
            at += up(max(1, a + n))
        for key, x in {**row, "tail_off": at, "n_pages": at // 16}.items():
            d[key].append(x)
        pages += at // 16
    out = {k: np.asarray(v, np.int32) for k, v in d.items()}
    out["page_ids"] = np.arange(pages, dtype=np.int32)
    return out, pages


def rows_per_tile(plan, desc):
    """Over the CTAs with more than twenty new rows: the fewest tiles, and the most rows to a tile; rows to a tile of the step."""
    _, slot, req = B.positions(desc, B.MODE_BRANCH)
    new = Counter((desc["page_ids"][desc["page_begin"][req] + slot // 16]).tolist())
    ids, valid = plan.stream_pages()
    at, it = plan.cta_ranges(), plan.items()
    before = np.concatenate([[0], np.cumsum([new[p] for p in ids.tolist()])])
    rows = [sum(int(before[x["page0"] + x["n_pages"]] - before[x["page0"]]) for x in it[a:b]) for a, b in zip(at, at[1:])]
    tiles = [sum((int(x["n_pages"]) + 7) // 8 for x in it[a:b]) for a, b in zip(at, at[1:])]
    many = [(t, r / t) for r, t in zip(rows, tiles) if r > 20]
    return (min(t for t, _ in many), max(q for _, q in many), sum(rows) / sum(tiles)) if many else None


def plan_of(desc, pages, **kw):
    return B.Plan(B.make_shape(28, 4, 128, 16, "bf16", 1e6, 128 ** -0.5), desc, pages, B.MODE_BRANCH, host_only=True, **kw)


# prefixes, tokens of the branches before, new tokens, dealt, fused: whole branches over a few requests; an opening step; eight
# branches decoding in twelve requests and in 32; a large batch with one token, and one with two, to a branch
@pytest.mark.parametrize("prefix,prior,new,dealt,fused", [
    ([6000, 2500, 1000], [[3, 40], [30], [8, 0, 0, 1]], [[90, 60], [133], [61, 80, 12, 50]], 0, 0),
    ([2000, 4100, 6000, 3300], [[0] * 6] * 4, [[12] * 6] * 4, 0, 0),
    ([8000] * 12, [[100] * 8] * 12, [[1] * 8] * 12, 0, 1),
    ([2000] * 148, [[20] * 8] * 148, [[1] * 8] * 148, 1, 1),
    ([1000] * 148, [[0] * 8] * 148, [[2] * 8] * 148, 1, 1),
    ([150] * 296, [[0] * 8] * 296, [[2] * 8] * 296, 1, 0)])
def test_either_side(prefix, prior, new, dealt, fused):
    desc, pages = descriptors(prefix, prior, new)
    plan = plan_of(desc, pages)
    assert (plan.info.dealt, plan.info.fused_append) == (dealt, fused)


def test_random_plans():
    rng = random.Random(8)
    long_fused = 0
    for _ in range(150):
        n_req = rng.choice([1, 2, 5, 12, 30, 100])
        br = [rng.randint(1, 8) for _ in range(n_req)]
        most = rng.choice([1, 1, 2, 6, 60])
        desc, pages = descriptors([rng.randint(1, 6000 if n_req < 40 else 1200) for _ in br], [[rng.randint(0, 60) for _ in range(b)] for b in br],
                                  [[rng.randint(1, most) for _ in range(b)] for b in br])
        plan = plan_of(desc, pages, n_ctas=rng.choice([0, 0, 20, 5]))
        if plan.info.fused_append:
            many = rows_per_tile(plan, desc)
            if many:
                tiles, worst, mean = many
                assert tiles >= 16 and (mean <= 2.5 if plan.info.dealt else worst <= 1.0)
                long_fused += 1
    assert long_fused >= 8
