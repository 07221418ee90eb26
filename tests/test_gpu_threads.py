"""Contexts on different host threads: each thread has its own context,
stream, points and workspace, and what one does leaves the other's calls
alone."""
import threading

import pytest
import torch

from paper_2104_07526_gb300 import build, pcr, scenes

pytestmark = pytest.mark.gpu

SEED = 7


def _reorders(source, expect, mode, rounds, calls, start, failures):
    """`rounds` times: `calls` reorders on end of a copy of `source`, which
    give `expect`."""
    n = source.shape[0]
    try:
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream), pcr.Context(0, stream=stream) as c:
            points = torch.empty_like(source)
            ws = torch.empty(pcr.pcr_reorder_workspace_size(n), dtype=torch.uint8, device="cuda")
            wrong = torch.zeros((), dtype=torch.int64, device="cuda")
            start.wait()
            for _ in range(rounds):
                points.copy_(source)
                for _ in range(calls):
                    pcr.pcr_reorder_morton_shuffle128(c.handle, points, n, SEED, mode, ws)
                wrong += (points != expect).sum()
            stream.synchronize()
        if int(wrong):
            failures.append(f"{n} points: {int(wrong)} words differ")
    except Exception as e:  # would end the thread unseen
        failures.append(f"{n} points: {e!r}")


# sorts of records in few buckets and in many, and sorts of 128-point batches
@pytest.mark.parametrize("mode,sizes,rounds,calls", [
    (pcr.PCR_ORDER_SHUFFLE, (2_001, 100_003), 100, 50),
    (pcr.PCR_ORDER_SHUFFLE, (9_001, 2048 * 1984), 20, 50),
    (pcr.PCR_ORDER_MORTON_SHUFFLE128, (300_001, 2_000_003), 1000, 1)])
def test_two_threads_reorder_clouds_of_different_sizes(oracle, mode, sizes, rounds, calls):
    build.build()
    sources, expects = [], []
    for n in sizes:
        cloud = scenes.random_cloud(n, seed=n % 89).numpy()
        sources.append(torch.from_numpy(cloud).cuda())
        perm = oracle.reorder(cloud, SEED, mode)  # the shuffle's is the same for whatever the call before left
        for _ in range(calls):
            cloud = oracle.gather(cloud, perm)
        expects.append(torch.from_numpy(cloud).cuda())
    torch.cuda.synchronize()
    failures, start = [], threading.Barrier(len(sizes))
    threads = [threading.Thread(target=_reorders, args=(s, e, mode, rounds, calls, start, failures))
               for s, e in zip(sources, expects)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not failures, failures
