"""The greedy loop of small classes (similarities in one SM's shared memory) at the edges of its warps, lists and shared memory,
against the oracle."""
import numpy as np
import pytest

import test_gpu_cluster as cluster
from test_gpu_parity import check_exact, check_float, rcd, orc, run_partition  # noqa: F401  (fixtures)

pytestmark = pytest.mark.gpu


def form(rcd, wl, **cfg):
    import torch
    with rcd.Context(0, **cfg) as ctx:
        ctx.rcd_partition(rcd.features_to_torch(wl.features, device="cuda"), torch.from_numpy(wl.labels).cuda(), wl.capacities, wl.L,
                          M_max=int(np.bincount(wl.labels).max()))
        ctx.sync_status()
        return ctx.profile()["greedy_form"]


@pytest.mark.parametrize("sizes,d,W", [
    ([1], 16, 1), ([1, 0, 2, 3], 17, 5),          # a sample, none, fewer samples than blocks
    ([31, 32, 33, 64, 65], 64, 3),                # edges of a warp
    ([224, 217, 7], 40, 4),                       # nearly all of the shared memory; classes of one warp beside it
    ([220], 64, 1),                               # one block takes everything
    ([160] * 3, 128, 33), ([96, 90], 32, 65), ([193, 161], 48, 20), ([60] * 5, 32, 128),       # two and four blocks per lane
    ([50] * 700, 24, 9),                          # several CTAs per SM, several turns
])
@pytest.mark.parametrize("copies", [0, 20])
def test_int8_exact(rcd, orc, sizes, d, W, copies):
    wl = cluster.workload(sizes, d, W, W + copies, copies=copies)
    check_exact(rcd, orc, wl)
    assert form(rcd, wl) == rcd.RCD_FORM_SMALL


def test_int8_sums_beyond_32_bits(rcd, orc):
    """Gains of up to 160 x 16384 x 127^2, and rows that raise every column."""
    wl = cluster.workload([160], 16384, 6, 7)
    wl.features = np.random.default_rng(7).integers(60, 128, size=wl.features.shape).astype(np.int8)
    check_exact(rcd, orc, wl)
    assert form(rcd, wl) == rcd.RCD_FORM_SMALL


@pytest.mark.parametrize("M,W", [(224, 4), (233, 4), (144, 60), (168, 60)])
def test_where_shared_memory_ends(rcd, orc, M, W):
    """One class that fits with all its blocks, and one that does not (the cluster form)."""
    wl = cluster.workload([M, 20], 32, W, M)
    check_exact(rcd, orc, wl)
    assert form(rcd, wl) == (rcd.RCD_FORM_SMALL if (M, W) in ((224, 4), (144, 60)) else rcd.RCD_FORM_CLUSTER)


@pytest.mark.parametrize("similarity", ["gaussian", "dot"])
@pytest.mark.parametrize("sizes,W", [([128, 1, 77], 5), ([200, 33], 12), ([65] * 4, 90)])
def test_float_is_exact_in_fixed_point(rcd, orc, similarity, sizes, W):
    cluster.test_float_is_exact_in_fixed_point(rcd, orc, similarity, sizes, W)
    kind = rcd.RCD_SIM_GAUSSIAN if similarity == "gaussian" else rcd.RCD_SIM_DOT
    assert form(rcd, cluster.workload(sizes, 64, W, 5 * W, dtype="bf16"), similarity_kind=kind) == rcd.RCD_FORM_SMALL


def test_float_norms_far_apart(rcd, orc):
    """Classes left in floating point beside one that is not."""
    wl = cluster.workload([200, 120, 64], 64, 6, 3, dtype="bf16", scale=lambda rng, M: 10.0 ** rng.uniform(-1.5 if M != 120 else 0.0, 1.5 if M != 120 else 0.1, M))
    check_float(rcd, orc, wl)
    assert form(rcd, wl) == rcd.RCD_FORM_SMALL


@pytest.mark.parametrize("sizes,W,copies", [([1, 2, 0, 33], 5, 0), ([224, 100], 3, 40), ([90] * 150, 20, 0), ([100, 64], 40, 10), ([70] * 3, 100, 0)])
def test_graph_cut_int8_exact(rcd, orc, sizes, W, copies):
    wl = cluster.workload(sizes, 48, W, W, copies=copies)
    a, o, v = run_partition(rcd, wl, objective=rcd.RCD_OBJ_GRAPH_CUT)
    ref = orc.partition(wl.features, wl.labels, wl.capacities, wl.L, variant="incremental", objective="cut")
    assert np.array_equal(a, ref.assignment) and np.array_equal(o, ref.order) and np.array_equal(v, ref.part_values)
    assert form(rcd, wl, objective=rcd.RCD_OBJ_GRAPH_CUT) == rcd.RCD_FORM_SMALL


@pytest.mark.parametrize("M,W", [(155, 1), (233, 1), (9, 1), (33, 1), (97, 2), (129, 2), (217, 3)])
def test_graph_cut_few_blocks_after_the_similarities(rcd, orc, M, W):
    """Class sizes far below the next multiple of eight, with few blocks: threads beyond the class read no row beyond it (nothing that
    large follows the similarities in shared memory)."""
    test_graph_cut_int8_exact(rcd, orc, [M, M - 1], W, 0)


def test_threads_with_contexts_of_their_own(rcd):
    """Four threads, each with a context and a stream, problems of very different shared memory at a time: each gets its own results."""
    import threading
    import torch
    wls = [cluster.workload([n], 64, w, n) for n, w in ((210, 4), (60, 3), (140, 40), (100, 9))]
    want = [run_partition(rcd, wl, greedy_path=4) for wl in wls]
    bad = []

    def work(wl, ref):
        try:
            st = torch.cuda.Stream()
            with torch.cuda.stream(st), rcd.Context(0) as ctx:
                X, y = rcd.features_to_torch(wl.features, device="cuda"), torch.from_numpy(wl.labels).cuda()
                for _ in range(20):
                    got = ctx.rcd_partition(X, y, wl.capacities, wl.L)
                    ctx.sync_status()
                    if not all(np.array_equal(g.cpu().numpy(), r) for g, r in zip(got, ref)):
                        bad.append(len(wl.labels))
        except Exception as e:      # noqa: BLE001
            bad.append(repr(e))

    threads = [threading.Thread(target=work, args=p) for p in zip(wls, want)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad
