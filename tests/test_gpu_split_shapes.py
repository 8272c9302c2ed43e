"""The class split and the worker lists where their chunks, threads and launches change (few numbers added up by every CTA, or by a scan)."""
import numpy as np
import pytest

import test_gpu_cluster as cluster
from test_gpu_parity import check_exact, rcd, orc  # noqa: F401  (fixtures)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [1, 31, 256, 257, 40960, 40961, 147456, 147457, 1310720, 2359296, 2359297])
@pytest.mark.parametrize("W", [1, 2, 31, 113, 114, 1024, 1025])
def test_lists(rcd, N, W):
    """Against numpy's stable sort; one worker without a sample, and twice on one context (what a launch leaves for the next)."""
    import torch
    rng = np.random.default_rng(N + W)
    a = rng.integers(0, W, size=N).astype(np.int32)
    if W > 2:
        a[a == 1] = 2
    with rcd.Context(0) as ctx:
        for _ in range(2):
            offsets, indices = rcd.rcd_worker_lists(ctx, torch.from_numpy(a).cuda(), W)
        ctx.sync_status()
        assert np.array_equal(offsets.cpu().numpy(), np.concatenate([[0], np.cumsum(np.bincount(a, minlength=W))]))
        assert np.array_equal(indices.cpu().numpy(), np.argsort(a, kind="stable"))


@pytest.mark.parametrize("N,W", [(2048, 1024), (2049, 1024), (4096, 512), (4097, 512), (8192, 256), (8200, 257), (45056, 372), (45057, 372), (300, 6000), (5000, 2048)])
def test_lists_of_many_workers(rcd, N, W):
    """On either side of 8192 numbers of small chunks, of 16384 of large ones, and of 1024 workers."""
    test_lists(rcd, N, W)


@pytest.mark.parametrize("N,W,at", [(300, 4, 299), (50000, 64, 0), (1000000, 64, 123456)])
def test_lists_bad_entry(rcd, N, W, at):
    """An entry out of range is refused, and the next call is not disturbed."""
    import torch
    a = torch.arange(N, dtype=torch.int32, device="cuda") % W
    bad = a.clone()
    bad[at] = W
    with rcd.Context(0) as ctx:
        with pytest.raises(rcd.RcdError):
            rcd.rcd_worker_lists(ctx, bad, W)
        offsets, indices = rcd.rcd_worker_lists(ctx, a, W)
        ctx.sync_status()
        assert bool((a[indices.long()][1:] >= a[indices.long()][:-1]).all()) and int(offsets[-1]) == N


@pytest.mark.parametrize("sizes", [[1], [128, 128], [129, 128], [64] * 127 + [63], [64] * 128, [128] * 32, [128] * 64 + [1], [20] * 170])
def test_partition_split(rcd, orc, sizes):
    """On either side of 32 chunks, and of 4096 numbers of chunks and labels."""
    check_exact(rcd, orc, cluster.workload(sizes, 24, 3, len(sizes)))


def test_partition_bad_label(rcd):
    import torch
    X, y = torch.zeros((500, 16), dtype=torch.int8, device="cuda"), torch.zeros(500, dtype=torch.int32, device="cuda")
    bad = y.clone()
    bad[300] = -1
    with rcd.Context(0) as ctx:
        with pytest.raises(rcd.RcdError):
            ctx.rcd_partition(X, bad, [1.0, 2.0], 1)
        a, o, v = ctx.rcd_partition(X, y, [1.0, 1.0], 1)
        ctx.sync_status()
        assert np.bincount(a.cpu().numpy()).tolist() == [250, 250]


def test_threads_with_lists_of_very_different_shared_memory(rcd):
    """Two threads, a context and a stream each: one's counters take 131 KB of shared memory, the other's 51 KB."""
    import threading
    import torch
    bad = []

    def work(W):
        try:
            a = np.random.default_rng(W).integers(0, W, size=50000).astype(np.int32)
            want = np.argsort(a, kind="stable")
            st = torch.cuda.Stream()
            with torch.cuda.stream(st), rcd.Context(0) as ctx:
                t = torch.from_numpy(a).cuda()
                for _ in range(2000):
                    offsets, indices = rcd.rcd_worker_lists(ctx, t, W)
                ctx.sync_status()
                if not np.array_equal(indices.cpu().numpy(), want):
                    bad.append(W)
        except Exception as e:      # noqa: BLE001
            bad.append(repr(e))

    threads = [threading.Thread(target=work, args=(W,)) for W in (1024, 400)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad
