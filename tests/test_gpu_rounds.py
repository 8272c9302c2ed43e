"""The greedy loop in rounds (taken where classes of about one size fill the SMs one by one and blocks are many) at the edges of its
tiles, batches, lists and shared memory, against the oracle or the pass-based form."""
import numpy as np
import pytest

import test_gpu_cluster as cluster
from test_gpu_parity import check_exact, check_float, rcd, orc  # noqa: F401  (fixtures)

pytestmark = pytest.mark.gpu


def ran_in_rounds(rcd, wl, lists=None, tiles=None, **cfg):
    """Whether the library takes the problem in rounds, and whether it corrects by lists and by tiles (None: either will do)."""
    import torch
    with rcd.Context(0, profile=1, **cfg) as ctx:
        ctx.rcd_partition(rcd.features_to_torch(wl.features, device="cuda"), torch.from_numpy(wl.labels).cuda(), wl.capacities, wl.L,
                          M_max=int(np.bincount(wl.labels).max()))
        ctx.sync_status()
        prof = ctx.profile()
    print("form %d, lists %d, tiles %d" % (prof["greedy_form"], prof["round_lists"], prof["round_tiles"]))
    assert prof["greedy_form"] == rcd.RCD_FORM_ROUNDS
    assert lists is None or (prof["round_lists"] > 0) == lists
    assert tiles is None or (prof["round_tiles"] > 0) == tiles


@pytest.mark.parametrize("sizes,d,W", [
    ([37] * 97, 16, 64),                          # fewer samples than blocks; batches of fewer blocks than wait (narrow features)
    ([129, 128, 127, 126] * 25, 40, 64),          # edges of 128 columns
    ([129, 128, 127, 126] * 25, 40, 48),          # (as many blocks as the cluster form is still faster with)
    ([257] * 60, 75, 100),                        # more than 64 blocks: two batches a round
    ([64] * 450, 24, 56),                         # two CTAs per SM
    ([90] * 60 + [0, 1, 0], 16, 128),             # the most blocks; empty classes and one of a sample
    ([333] * 98, 520, 61),                        # a last group of three columns, a number of blocks that is no multiple of four
])
@pytest.mark.parametrize("copies", [0, 30])
def test_int8_exact(rcd, orc, sizes, d, W, copies):
    wl = cluster.workload(sizes, d, W, W + copies, copies=copies)
    check_exact(rcd, orc, wl)
    if W != 48:
        ran_in_rounds(rcd, wl)


def test_int8_sums_beyond_32_bits(rcd, orc):
    """The losses of a column add up to more than 2^32 (300 rows, each of up to 2048 x 127^2): they are widened on the way."""
    wl = cluster.workload([300] * 98, 2048, 60, 7)
    wl.features = np.random.default_rng(7).integers(90, 128, size=wl.features.shape).astype(np.int8)
    check_exact(rcd, orc, wl)
    ran_in_rounds(rcd, wl, tiles=True)


@pytest.mark.parametrize("sizes,d,W", [([1000] * 148, 32, 16), ([1003] * 148, 256, 40), ([1610] * 140, 64, 49)])
def test_int8_like_the_passes(rcd, sizes, d, W):
    import torch
    wl = cluster.workload(sizes, d, W, W)
    X, y = rcd.features_to_torch(wl.features, device="cuda"), torch.from_numpy(wl.labels).cuda()
    results = []
    for path in (0, 4):
        with rcd.Context(0, greedy_path=path) as ctx:
            results.append(ctx.rcd_partition(X, y, wl.capacities, wl.L, M_max=max(sizes)))
            ctx.sync_status()
    for got, want in zip(*results):
        assert torch.equal(got, want)
    ran_in_rounds(rcd, wl, lists=True, tiles=True)


@pytest.mark.parametrize("similarity", ["gaussian", "dot"])
@pytest.mark.parametrize("sizes,W", [([101] * 98, 57), ([66] * 60, 100), ([66] * 60, 70)])
def test_float_is_exact_in_fixed_point(rcd, orc, similarity, sizes, W):
    cluster.test_float_is_exact_in_fixed_point(rcd, orc, similarity, sizes, W)
    if W != 70:                                       # (where the cluster form is still faster)
        ran_in_rounds(rcd, cluster.workload(sizes, 64, W, 5 * W, dtype="bf16"),
                      similarity_kind=rcd.RCD_SIM_GAUSSIAN if similarity == "gaussian" else rcd.RCD_SIM_DOT)


def test_float_norms_far_apart(rcd, orc):
    """A class left in floating point beside those that run in rounds."""
    wl = cluster.workload([141] + [140] * 99, 32, 60, 1, dtype="bf16", scale=lambda rng, M: 10.0 ** rng.uniform(-1.5 if M == 141 else 0.0, 1.5 if M == 141 else 0.1, M))
    check_float(rcd, orc, wl)
    ran_in_rounds(rcd, wl)


def test_copies_that_never_arrive(rcd, orc):
    """The wait for a step's copies runs out for half of the threads only: all of them leave at that step (another status than the
    timeout's where they do not), and the context goes on."""
    wl = cluster.workload([37] * 97, 16, 64, 64)
    with rcd.Context(0) as ctx:
        ctx.selftest_bounded_wait()
        with pytest.raises(rcd.RcdError) as e:
            ctx.sync_status()
        assert e.value.status == 5          # RCD_ERR_TIMEOUT
    check_exact(rcd, orc, wl)
    ran_in_rounds(rcd, wl)


@pytest.mark.parametrize("L,M,W,dtype,rounds", [
    (148, 1000, 24, "int8", False),        # two CTAs per class and full rows: the cluster form is faster
    (148, 1030, 24, "int8", True),         # rows of three steps
    (148, 1000, 16, "int8", True),         # one CTA per class
    (200, 400, 64, "int8", False),         # two turns of rounds, the second a third full, against three of the cluster form
    (296, 200, 48, "int8", False), (296, 200, 64, "int8", True),          # one CTA per class either way, two turns
    (60, 500, 80, "int8", False), (60, 500, 128, "int8", True),
    (100, 1300, 64, "int8", False), (100, 1300, 128, "int8", True),
    (60, 500, 65, "bf16", False), (300, 500, 64, "bf16", True), (300, 700, 64, "bf16", False), (444, 1300, 56, "bf16", False),
])
def test_form(rcd, L, M, W, dtype, rounds):
    """Which form the library takes, on either side of where the two were measured to change places (on 148 SMs)."""
    import torch
    if torch.cuda.get_device_properties(0).multi_processor_count != 148:
        pytest.skip("measured on 148 SMs")
    g = torch.Generator(device="cuda").manual_seed(M)
    X = torch.randint(-9, 10, (L * M, 16), generator=g, device="cuda").to(torch.int8)
    if dtype == "bf16":
        X = (X / X.float().norm(dim=1, keepdim=True).clamp_min(1)).to(torch.bfloat16)
    y = torch.arange(L, dtype=torch.int32, device="cuda").repeat(M)
    with rcd.Context(0) as ctx:
        a, o, v = ctx.rcd_partition(X, y, [1.0 + j % 4 for j in range(W)], L, M_max=M)
        ctx.sync_status()
        assert ctx.profile()["greedy_form"] == (rcd.RCD_FORM_ROUNDS if rounds else rcd.RCD_FORM_CLUSTER)
    assert bool((o.sort()[0] == torch.arange(L * M, device="cuda")).all())
