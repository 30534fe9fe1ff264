"""The work a user has this library do, as timed cases: decoding steps, whole-branch steps, key
renumbering, through the public calls of ``paper_2508_08895_b200.binding``.

A case describes one decoding step of a model's attention layers: how many requests, the range their
prefix and branch lengths are drawn from (``lens`` seeds that draw, so that a case always has the same
lengths), the heads, the storage type, and how the program drives the library:

  plan      a new plan for the step, one ``branch_step`` / ``serial_step`` per layer, the plan destroyed
            (the loop of an engine that launches from the host)
  graph     the layers' steps captured once with an updatable plan; per step ``Plan.update`` and a replay
            (bf16, heads of 128, pages of 16: the shapes the library re-plans in place)
  host      the step's q / k_new / v_new in page-locked host memory, the outputs read back: plans and
            streams taken in turn by the layers (``step_host_async``)
  rerotate  a finished segment's keys moved to new position IDs in every layer's pool

Values are what the path meets: K (already rotated), V, Q ~ N(0, 1) in the storage type, logits scaled
by 1/sqrt(d), physical pages scattered over the pool.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_2508_08895_b200 import binding as B

_DTYPE = {"bf16": torch.bfloat16, "f32": torch.float32}
_ESIZE = {"bf16": 2, "f32": 4}


def _case(name, step, drive, layers, n_req, prefix, branches, prior, new, lens=1, heads=(28, 4), d=128, page=16, dtype="bf16", tail=0):
    c = {"step": step, "drive": drive, "layers": layers, "n_req": n_req, "prefix_lo": prefix[0], "prefix_hi": prefix[1],
         "branches_lo": branches[0], "branches_hi": branches[1], "prior_lo": prior[0], "prior_hi": prior[1], "new": new, "lens": lens,
         "hq": heads[0], "hkv": heads[1], "d": d, "page": page, "dtype": dtype, "tail": tail}
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest call: one fp32 layer of 4 heads, 3 short branches over 256 tokens -- all latency
        _case("tiny-f32", "branch", "plan", 1, 1, (256, 256), (3, 3), (9, 23), 1, heads=(4, 1), d=64, dtype="f32"),
        # one chat request decoding four branches of a parallel segment, launched layer by layer
        _case("one-request", "branch", "plan", 28, 1, (2048, 2048), (4, 4), (128, 128), 1),
        # the first step of a segment: six branches take their 12 forced header tokens at once
        _case("branch-open", "branch", "plan", 28, 1, (1024, 1024), (6, 6), (0, 0), 12),
        # serial decoding of the same request after the merge, halfway through 64 tokens, as a graph
        _case("serial-chain", "serial", "graph", 28, 1, (1024, 1024), (6, 6), (12, 12), 0, tail=32),
        # one retrieval-augmented request: a long shared context, eight ragged branches, as a graph
        _case("long-rag", "branch", "graph", 28, 1, (16384, 16384), (8, 8), (32, 256), 1),
        # a serving batch in mixed states: ragged prefixes, 1 to 8 branches each
        _case("serving-mix", "branch", "plan", 28, 32, (512, 8192), (1, 8), (1, 256), 1),
        # the same batch after its segments have closed: one token per request over the merged cache
        _case("serving-serial", "serial", "graph", 28, 32, (512, 8192), (1, 8), (1, 256), 0),
        # the largest serving batch
        _case("serving-large", "branch", "plan", 4, 160, (512, 8192), (1, 8), (1, 256), 1),
        # teacher forcing / masked prefill: every token of every branch is a query of one step
        _case("masked-prefill", "branch", "plan", 28, 32, (512, 8192), (1, 8), (0, 0), 256),
        # renumbering the keys of the batch's finished segments, all layers
        _case("rerotate", "rerotate", "rerotate", 28, 32, (512, 8192), (1, 8), (1, 256), 0),
        # a model with heads of 64 and two KV heads, a small serving batch
        _case("serving-d64", "branch", "plan", 24, 8, (512, 4096), (1, 8), (1, 256), 1, heads=(14, 2), d=64),
        # activations that live in host memory: the step from pinned buffers, outputs back to the host
        _case("host-step", "branch", "host", 28, 8, (512, 4096), (1, 8), (1, 256), 1),
    ]


def _log_int(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    """One more case of the ranges above."""
    kind = rng.choice(["decode", "decode", "decode", "serial", "open", "prefill", "rerotate", "d64", "page", "f32", "host"])
    lens, drive = rng.randrange(1, 1 << 20), rng.choice(["plan", "graph"])
    if kind == "f32":
        heads, d = rng.choice([((4, 1), 64), ((8, 2), 128), ((28, 4), 128)])
        lo = _log_int(rng, 32, 1024)
        return _case(None, rng.choice(["branch", "serial"]), "plan", rng.choice([1, 4]), rng.randint(1, 3), (lo, 2 * lo), (1, 6), (1, 64), 1, lens,
                     heads, d, rng.choice([8, 16, 32]), "f32", rng.randint(0, 9))
    if kind in ("open", "prefill"):
        n_req = 1 if kind == "open" else _log_int(rng, 1, 24)
        lo = _log_int(rng, 128, 4096)
        new = rng.randint(2, 24) if kind == "open" else rng.randint(25, 256)
        return _case(None, "branch", "plan", 28, n_req, (lo, min(8192, 2 * lo)), (1, 8), (0, rng.choice([0, 40])), new, lens)
    n_req = _log_int(rng, 1, 150)
    lo = _log_int(rng, 100, 8000 if n_req <= 16 else 1500)
    prefix, layers = (lo, min(16384, lo * rng.randint(1, 4))), 28 if n_req <= 32 else 4
    common = dict(lens=lens, tail=rng.randint(0, 64))
    if kind in ("d64", "page", "host"):
        n_req, layers = min(n_req, 12), 24 if kind == "d64" else 28
    if kind == "d64":
        return _case(None, rng.choice(["branch", "serial"]), "plan", layers, n_req, (lo, min(4096, 2 * lo)) if lo < 4096 else (2048, 4096), (1, 8),
                     (1, 256), 1, heads=rng.choice([(14, 2), (16, 8), (32, 4)]), d=64, **common)
    if kind == "page":
        return _case(None, rng.choice(["branch", "serial"]), "plan", layers, min(n_req, 4), (lo, min(4096, 2 * lo)) if lo < 4096 else (2048, 4096),
                     (1, 8), (1, 256), 1, page=rng.choice([8, 32]), **common)
    if kind == "host":
        return _case(None, rng.choice(["branch", "serial"]), "host", layers, n_req, prefix, (1, 8), (1, 256), 1, **common)
    if kind == "rerotate":
        return _case(None, "rerotate", "rerotate", layers, n_req, prefix, (2, 8), (1, 256), 0, **common)
    heads = rng.choice([(28, 4), (28, 4), (32, 8), (16, 2)]) if n_req <= 40 else (28, 4)
    return _case(None, "serial" if kind == "serial" else "branch", drive, layers, n_req, prefix, (1, 8), (1, 256), 1, heads=heads, **common)


# ------------------------------------------------------------------------------------ lengths and layout
def _lengths(case):
    """Per request: prefix length, tokens of every branch before the step, new tokens of every branch."""
    rng = random.Random(case["lens"])
    out = []
    for _ in range(case["n_req"]):
        prefix = _log_int(rng, case["prefix_lo"], case["prefix_hi"])
        n_br = rng.randint(case["branches_lo"], case["branches_hi"])
        prior = [rng.randint(case["prior_lo"], case["prior_hi"]) for _ in range(n_br)]
        # a decoding step adds one token per branch, an opening step the forced header, a teacher-forcing
        # step whole branches of up to `new` tokens
        new = [case["new"] if case["new"] <= 24 else rng.randint(1, case["new"]) for _ in range(n_br)]
        if case["step"] != "branch":
            new = [0] * n_br
        out.append((prefix, prior, new))
    return out


def _descriptors(case, seed):
    """Descriptor arrays of the step: page-aligned branch regions and tail, pages scattered by the seed."""
    ps, serial = case["page"], case["step"] == "serial"
    up = lambda n: -(-n // ps) * ps   # noqa: E731
    keys = ("prefix_len", "n_branches", "branch_begin", "page_begin", "n_pages", "tail_off", "tail_len", "br_kv_off", "br_kv_len", "br_q_len")
    d = {k: [] for k in keys}
    pages = 0
    for prefix, prior, new in _lengths(case):
        at = up(prefix)
        d["prefix_len"].append(prefix)
        d["n_branches"].append(len(prior))
        d["branch_begin"].append(len(d["br_kv_off"]))
        for p, n in zip(prior, new):
            d["br_kv_off"].append(at)
            d["br_kv_len"].append(p + n)
            d["br_q_len"].append(n)
            at += up(max(1, p + n))
        tail = case["tail"] + 1 if serial else 0
        d["tail_off"].append(at)
        d["tail_len"].append(tail)
        d["page_begin"].append(pages)
        d["n_pages"].append((at + up(tail)) // ps)
        pages += d["n_pages"][-1]
    desc = {k: np.asarray(v, dtype=np.int32) for k, v in d.items()}
    n_pool = pages + 3
    desc["page_ids"] = np.random.default_rng(seed).permutation(n_pool)[:pages].astype(np.int32)
    return desc, n_pool


# ------------------------------------------------------------------------------------------ the program
def prepare(case, seed):
    desc, n_pool = _descriptors(case, seed)
    mode = B.MODE_SERIAL if case["step"] == "serial" else B.MODE_BRANCH
    hq, hkv, d, L, dt = case["hq"], case["hkv"], case["d"], case["layers"], _DTYPE[case["dtype"]]
    shape = B.make_shape(hq, hkv, d, case["page"], case["dtype"], 1.0e6, d ** -0.5)
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    normal = lambda *size: torch.randn(*size, dtype=dt, device="cuda", generator=gen)   # noqa: E731
    elems = B.pool_bytes(shape, n_pool) // _ESIZE[case["dtype"]]
    s = {"case": case, "shape": shape, "desc": desc, "n_pool": n_pool, "mode": mode, "k": normal(L, elems)}
    s["k_layers"] = list(s["k"])
    if case["step"] == "rerotate":
        # sequential renumbering: every branch moves by the tokens of the branches listed before it
        ranges = []
        for r in range(case["n_req"]):
            moved, b0 = 0, int(desc["branch_begin"][r])
            for b in range(b0, b0 + int(desc["n_branches"][r])):
                if moved:
                    ranges.append((int(desc["page_begin"][r]), int(desc["br_kv_off"][b]), int(desc["br_kv_len"][b]), moved))
                moved += int(desc["br_kv_len"][b])
        s["ranges"] = np.asarray(ranges, dtype=np.int32).reshape(-1, 4)
        s["page_table"] = torch.from_numpy(desc["page_ids"]).cuda()
        return s
    n = B.count_new_tokens(desc, mode)
    s["v"] = normal(L, elems)
    s["v_layers"] = list(s["v"])
    q, k_new, v_new = normal(L, n, hq, d), normal(L, n, hkv, d), normal(L, n, hkv, d)
    if case["drive"] == "host":
        packed = torch.cat([x.reshape(L, -1) for x in (q, k_new, v_new)], dim=1).cpu().pin_memory()
        s["out"] = torch.zeros(L, n, hq, d, dtype=dt).pin_memory()
        nq, nk = n * hq * d, n * hkv * d
        s["layers"] = [(packed[l, :nq], packed[l, nq:nq + nk], packed[l, nq + nk:], s["k_layers"][l], s["v_layers"][l], s["out"][l]) for l in range(L)]
        s["streams"] = [torch.cuda.Stream() for _ in range(4)]
        return s
    s["out"] = torch.zeros(L, n, hq, d, dtype=dt, device="cuda")
    s["layers"] = [(q[l], k_new[l], v_new[l], s["k_layers"][l], s["v_layers"][l], s["out"][l]) for l in range(L)]
    if case["drive"] == "graph":
        s["plan"] = B.Plan(shape, desc, n_pool, mode, stable_cache=True, updatable=True)
        step = B.serial_step if mode == B.MODE_SERIAL else B.branch_step
        torch.cuda.synchronize()
        s["graph"] = torch.cuda.CUDAGraph()
        with torch.cuda.graph(s["graph"]):
            for x in s["layers"]:
                step(s["plan"], *x)
    return s


def run(s):
    case, desc = s["case"], s["desc"]
    if case["drive"] == "rerotate":
        B.k_rerotate_ranges_layers(s["shape"], s["k_layers"], s["page_table"], s["ranges"])
        return {"k": s["k"]}
    if case["drive"] == "host":
        pos, _, _ = B.positions(desc, s["mode"])
        plans = [B.Plan(s["shape"], desc, s["n_pool"], s["mode"], stable_cache=True, stream=st) for st in s["streams"]]
        for i, x in enumerate(s["layers"]):
            q, k_new, v_new, k_pool, v_pool, out = x
            B.step_host_async(plans[i % 4], q, k_new, v_new, pos, k_pool, v_pool, out, stream=s["streams"][i % 4])
        for p in plans:
            p.destroy()
    elif case["drive"] == "graph":
        s["plan"].update(desc)
        s["graph"].replay()
    else:
        step = B.serial_step if s["mode"] == B.MODE_SERIAL else B.branch_step
        plan = B.Plan(s["shape"], desc, s["n_pool"], s["mode"], stable_cache=True)
        for x in s["layers"]:
            step(plan, *x)
        plan.destroy()
    return {"out": s["out"], "k": s["k"], "v": s["v"]}


# --------------------------------------------------------------------------------- what a pass must move
def work(case):
    hq, hkv, d, es = case["hq"], case["hkv"], case["d"], _ESIZE[case["dtype"]]
    kv_read, pairs, n_new, moved = 0, 0, 0, 0
    for prefix, prior, new in _lengths(case):
        if case["step"] == "serial":
            cached = prefix + sum(prior) + case["tail"]
            kv_read += cached
            pairs += cached + 1
            n_new += 1
        else:
            kv_read += prefix + sum(prior)
            pairs += sum(n * (prefix + p) + n * (n + 1) // 2 for p, n in zip(prior, new))
            n_new += sum(new)
        moved += sum(prior[1:])
    if case["step"] == "rerotate":
        return {"bytes": case["layers"] * 2 * hkv * d * es * moved, "flops": case["layers"] * 3 * hkv * d * moved}
    # cached K and V once, the new rows in and into the cache, q in, out
    rows = 2 * hkv * d * es * (kv_read + 2 * n_new) + 2 * hq * d * es * n_new
    return {"bytes": case["layers"] * rows, "flops": case["layers"] * 4 * d * hq * pairs}


def tolerance(case):
    # against attention in 64 bits from the same stored inputs the outputs are off by 4e-7 (f32) and 2.9e-3 (bf16
    # queries, weights and outputs over fp32 sums; largest single value 0.03), appended keys by 1.7e-3
    if case["dtype"] == "f32":
        return {"rel": 2e-6, "max": 1e-4}
    if case["step"] == "rerotate":
        return {"rel": 4e-3, "max": 0.02}   # one rounding of a rotated key to bf16
    return {"rel": 1e-2, "max": 0.12}
