"""Plan blocks and threads: a plan that waits for its block's last copy does not hold up the plans of another thread."""
import threading
import time

import pytest

from paper_2508_08895_b200 import binding as B, workloads as W

pytestmark = pytest.mark.gpu


def maker(tokens):
    wl = W.build_segment_workload("thr", 98, 28, 4, 128, "bf16", 1e6, [64], [[0]], [[tokens]])
    ph = wl.phases[-1]
    shape = B.make_shape(28, 4, 128, 16, "bf16", 1e6, 128 ** -0.5)
    return lambda stream: B.Plan(shape, ph.desc, wl.n_pool_pages, ph.mode, stream=stream)


def test_a_wait_for_one_size_leaves_the_others_alone():
    import torch
    small, large = maker(1), maker(3000)                        # blocks of 4 MB and of tens of MB: neither fits the other's plans
    busy, free = torch.cuda.Stream(), torch.cuda.Stream()
    B.release_cached_memory()
    plans = [small(busy), small(busy)]                          # two small blocks and one large one, parked and idle
    for p in plans:
        p.destroy()
    large(free).destroy()
    torch.cuda.synchronize()
    with torch.cuda.stream(busy):
        torch.cuda._sleep(800_000_000)                          # some 0.4 s on this stream
    for p in [small(busy), small(busy)]:                        # their copies queue behind it
        p.destroy()
    times = {}

    def timed(name, make, stream):
        t = time.perf_counter()
        make(stream).destroy()
        times[name] = time.perf_counter() - t

    waits = threading.Thread(target=timed, args=("small", small, busy))
    waits.start()
    time.sleep(0.05)
    timed("large", large, free)
    waits.join()
    torch.cuda.synchronize()
    assert times["small"] > 0.15 and times["large"] < 0.1, times
    B.release_cached_memory()
