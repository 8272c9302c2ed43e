"""The graph cut in step (integers, several blocks) at the edges of its columns per thread and of its clusters, against the oracle."""
import numpy as np
import pytest

import test_gpu_cluster as cluster
from test_gpu_parity import rcd, orc, run_partition  # noqa: F401  (fixtures)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes,W,copies", [
    ([257, 31], 6, 0), ([300, 0, 1, 250], 9, 40),          # one or two columns per thread; an empty class, one of a sample, ties
    ([513], 33, 0), ([770, 5], 65, 30),                    # two and four blocks per lane; a class that leaves most CTAs without columns
    ([1300, 1281], 8, 60), ([2600], 50, 0),                # clusters
    ([260] * 160, 2, 0), ([250] * 70, 5, 20),              # more classes than SMs, few blocks
])
def test_exact(rcd, orc, sizes, W, copies):
    import torch
    wl = cluster.workload(sizes, 32, W, W + len(sizes), copies=copies)
    a, o, v = run_partition(rcd, wl, objective=rcd.RCD_OBJ_GRAPH_CUT)
    ref = orc.partition(wl.features, wl.labels, wl.capacities, wl.L, variant="incremental", objective="cut")
    assert np.array_equal(a, ref.assignment) and np.array_equal(o, ref.order) and np.array_equal(v, ref.part_values)
    with rcd.Context(0, objective=rcd.RCD_OBJ_GRAPH_CUT) as ctx:
        ctx.rcd_partition(rcd.features_to_torch(wl.features, device="cuda"), torch.from_numpy(wl.labels).cuda(), wl.capacities, wl.L)
        ctx.sync_status()
        assert ctx.profile()["greedy_form"] == rcd.RCD_FORM_CUT_STEPS


def test_like_the_chain(rcd):
    """A class over clusters of 16, one and two columns per thread, against one CTA with everything in global memory (more than 128 blocks)."""
    import torch
    for M, W in ((6000, 12), (3000, 100)):
        wl = cluster.workload([M, 300], 48, W, W)
        X, y = rcd.features_to_torch(wl.features, device="cuda"), torch.from_numpy(wl.labels).cuda()
        out = []
        for caps in (list(wl.capacities), list(wl.capacities) + [1e-9] * (129 - W)):       # (blocks that get nothing)
            with rcd.Context(0, objective=rcd.RCD_OBJ_GRAPH_CUT) as ctx:
                r = ctx.rcd_partition(X, y, caps, wl.L)
                ctx.sync_status()
                out.append((r[0].cpu().numpy(), r[1].cpu().numpy(), r[2].cpu().numpy()[:, :W], ctx.profile()["greedy_form"]))
        assert out[0][3] == rcd.RCD_FORM_CUT_STEPS and out[1][3] == rcd.RCD_FORM_CUT_CHAIN
        for got, want in zip(out[0][:3], out[1][:3]):
            assert np.array_equal(got, want)


# number and size of classes, blocks, and what the plan makes of them on 148 SMs (test_dispatch_rules.py): CTAs per class, columns per thread
SHAPES = [
    (200, 700, 8, 1, 3), (300, 900, 7, 1, 4), (160, 1100, 6, 1, 8),          # a CTA each; the last one's columns end before its threads' do
    (2, 1300, 8, 8, 1), (10, 5000, 8, 8, 3), (40, 4000, 8, 2, 8), (75, 2100, 6, 4, 3),
    (1, 16000, 6, 16, 4), (1, 17000, 4, 16, 8),
]


@pytest.mark.parametrize("L,M,W,C,K", SHAPES)
def test_columns_per_thread(rcd, L, M, W, C, K):
    """One to eight columns per thread, alone and in clusters, against the chain as above, with a smaller class beside the others."""
    import torch
    wl = cluster.workload([M] * L + [min(M - 1, 300)], 16, W, W, copies=20)
    X, y = rcd.features_to_torch(wl.features, device="cuda"), torch.from_numpy(wl.labels).cuda()
    out = []
    for caps in (list(wl.capacities), list(wl.capacities) + [1e-9] * (129 - W)):       # (blocks that get nothing)
        with rcd.Context(0, objective=rcd.RCD_OBJ_GRAPH_CUT) as ctx:
            r = ctx.rcd_partition(X, y, caps, wl.L, M_max=M)
            ctx.sync_status()
            out.append((r[0].cpu().numpy(), r[1].cpu().numpy(), r[2].cpu().numpy()[:, :W], ctx.profile()["greedy_form"]))
    assert out[0][3] == rcd.RCD_FORM_CUT_STEPS and out[1][3] == rcd.RCD_FORM_CUT_CHAIN
    for got, want in zip(out[0][:3], out[1][:3]):
        assert np.array_equal(got, want)


def test_only_where_the_library_chooses(rcd, orc):
    """An option of the pass-based forms keeps the chain, as before."""
    import torch
    wl = cluster.workload([300, 250], 32, 8, 3)
    with rcd.Context(0, objective=rcd.RCD_OBJ_GRAPH_CUT, greedy_path=3) as ctx:
        a, o, v = ctx.rcd_partition(rcd.features_to_torch(wl.features, device="cuda"), torch.from_numpy(wl.labels).cuda(), wl.capacities, wl.L)
        ctx.sync_status()
        assert ctx.profile()["greedy_form"] == rcd.RCD_FORM_CUT_CHAIN
    ref = orc.partition(wl.features, wl.labels, wl.capacities, wl.L, variant="incremental", objective="cut")
    assert np.array_equal(a.cpu().numpy(), ref.assignment) and np.array_equal(v.cpu().numpy(), ref.part_values)


@pytest.mark.parametrize("M,d", [(8400, 64), (14400, 131071)])
def test_values_beyond_the_packed_word(rcd, M, d):
    """Equal samples into two blocks: picks in index order, the blocks in turn, f = (M / 2)^2 x S.  The second class passes 3 x 2^55."""
    import torch
    X, y = torch.full((M, d), 127, dtype=torch.int8, device="cuda"), torch.zeros(M, dtype=torch.int32, device="cuda")
    with rcd.Context(0, objective=rcd.RCD_OBJ_GRAPH_CUT) as ctx:
        a, o, v = ctx.rcd_partition(X, y, [1.0, 1.0], 1, M_max=M)
        ctx.sync_status()
        assert ctx.profile()["greedy_form"] == (rcd.RCD_FORM_CUT_STEPS if d == 64 else rcd.RCD_FORM_CUT_CHAIN)
    assert np.array_equal(o.cpu().numpy(), np.arange(M)) and np.array_equal(a.cpu().numpy(), np.arange(M) % 2)
    assert v.cpu().numpy().tolist() == [[(M // 2) ** 2 * 127 * 127 * d] * 2]


def test_no_outputs_where_the_loop_stops_early(rcd):
    """A class whose quotas end before its samples: the loop in step and the cluster form stop, say so, and leave the outputs alone
    (the self-test fails with its own status where they do not)."""
    with rcd.Context(0, objective=rcd.RCD_OBJ_GRAPH_CUT) as ctx:
        ctx.selftest_bounded_wait()
        with pytest.raises(rcd.RcdError) as e:
            ctx.sync_status()
        assert e.value.status == 5          # RCD_ERR_TIMEOUT, of the waits that follow


def test_profile(rcd):
    """Steps executed, and picks that corrected stored gains: all but the last of each block that gets samples, by their own row only."""
    import torch
    wl = cluster.workload([400, 390], 16, 8, 1)
    for caps, blocks in (([1.0] * 8, 8), ([1.0] * 8 + [1e-9] * 3, 8)):
        with rcd.Context(0, objective=rcd.RCD_OBJ_GRAPH_CUT, profile=1) as ctx:
            ctx.rcd_partition(rcd.features_to_torch(wl.features, device="cuda"), torch.from_numpy(wl.labels).cuda(), caps, wl.L)
            ctx.sync_status()
            p = ctx.profile()
        assert p["greedy_form"] == rcd.RCD_FORM_CUT_STEPS and p["steps"] == 400
        assert p["incremental_updates"] == 400 + 390 - 2 * blocks and p["incremental_rows"] == 0
    with rcd.Context(0, objective=rcd.RCD_OBJ_GRAPH_CUT, greedy_path=3) as ctx:
        ctx.rcd_partition(rcd.features_to_torch(wl.features, device="cuda"), torch.from_numpy(wl.labels).cuda(), caps, wl.L)
        ctx.sync_status()
        assert ctx.profile()["steps"] == 400


@pytest.mark.parametrize("L,M,W,form", [(67, 609, 6, "RCD_FORM_CLUSTER"), (118, 1138, 126, "RCD_FORM_CUT_CHAIN"), (3, 700, 126, "RCD_FORM_CUT_STEPS")])
def test_where_another_form_is_faster(rcd, L, M, W, form):
    import torch
    X = torch.randint(-9, 10, (L * M, 16), dtype=torch.int8, device="cuda")
    y = torch.arange(L * M, dtype=torch.int32, device="cuda") % L
    with rcd.Context(0, objective=rcd.RCD_OBJ_GRAPH_CUT) as ctx:
        ctx.rcd_partition(X, y, [1.0] * W, L, M_max=M)
        ctx.sync_status()
        assert ctx.profile()["greedy_form"] == getattr(rcd, form)
