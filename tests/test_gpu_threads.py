"""The library called from several host threads: what one thread has asked of the device must hold whatever the others
ask, and calls on streams of their own do not disturb each other."""
from concurrent.futures import ThreadPoolExecutor

import numpy as np
import pytest
import torch

from oracle import reference as ref
from paper_2510_07651_b200 import api

pytestmark = pytest.mark.gpu


def _scores(heads, n, seed):
    return np.random.default_rng(seed).random((1, heads, n), dtype=np.float32)


def test_selections_of_different_sizes_from_two_threads():
    """The selection kernel takes shared memory by the length of a head, and what a launch may use is set per process: a
    short head selected by a thread that has selected nothing yet must not take from another thread what it was given."""
    jobs = []
    for heads, n, budget in ((8, 32768, 2048), (1, 1024, 256), (3, 70000, 900)):
        s = _scores(heads, n, n)
        dev = torch.from_numpy(s).cuda()
        want = ref.select_pipeline(s, [n], [budget], 0, 32, "max", 7, budget)
        want_ad, _ = ref.select_adaptive_pipeline(s, [n], [budget], 0, 32, "max", 7, 0.2, 2 * budget)
        jobs.append((dev, budget, want, want_ad))

    def run(job):
        dev, budget, want, want_ad = job
        kw = dict(budget=budget, n_recent=32, pool="max", pool_kernel=7)
        idx = api.obc_select(dev, **kw)
        idx_ad, _ = api.obc_select_adaptive(dev, idx_stride=2 * budget, **kw)
        torch.cuda.synchronize()
        return np.array_equal(idx.cpu().numpy(), want) and np.array_equal(idx_ad.cpu().numpy(), want_ad)

    with ThreadPoolExecutor(1) as a, ThreadPoolExecutor(1) as b, ThreadPoolExecutor(1) as c:
        for _ in range(2):                                     # strictly in turn: long, short, long by the first thread again, ...
            for thread, job in ((a, 0), (b, 1), (a, 0), (c, 2), (a, 0), (b, 1), (b, 0), (a, 2)):
                assert thread.submit(run, jobs[job]).result()


def test_threads_with_streams_of_their_own():
    """Score, select and compact by four threads at once, each with its own stream, inputs and sizes: the same as one after another."""
    shapes = [(1, 8, 2, 16, 3000), (1, 4, 4, 10, 700), (2, 14, 2, 64, 1500), (1, 1, 1, 16, 1024)]
    inputs = []
    for i, (B, Hq, H, W, N) in enumerate(shapes):
        g = torch.Generator(device="cuda").manual_seed(i)
        dt = torch.float32 if i == 3 else torch.bfloat16
        inputs.append([torch.randn((B, h, t, 128), generator=g, device="cuda").to(dt) for h, t in ((Hq, W), (H, N), (H, N))])

    def run(i):
        q, k, v = inputs[i]
        return api.evict_prefill(q, k, v, budget=k.shape[2] // 4, n_recent=16, pool="max", pool_kernel=7)

    def repeat(i):
        with torch.cuda.stream(torch.cuda.Stream()):
            got = [run(i) for _ in range(20)]
            torch.cuda.current_stream().synchronize()
        return got

    alone = [run(i) for i in range(len(shapes))]
    torch.cuda.synchronize()
    with ThreadPoolExecutor(len(shapes)) as pool:
        for i, results in enumerate(pool.map(repeat, range(len(shapes)))):
            for got in results:
                assert all(torch.equal(x, y) for x, y in zip(got, alone[i])), shapes[i]
