"""The cluster form of the greedy loop (the library's own choice) against the oracle, at the sizes where its layout changes:
one or several blocks per team, one to seven 16-byte pieces per thread, lists of raised columns longer than their room, blocks
in shared or in global memory; and the class split, the objective and the fixed-point scale at their own edges."""
import numpy as np
import pytest

from test_gpu_parity import check_exact, check_float, rcd, orc, run_partition  # noqa: F401  (fixtures)

pytestmark = pytest.mark.gpu


def workload(sizes, d, W, seed, dtype="int8", scale=None, copies=0):
    from paper_2211_00839_b200.workloads import Workload, make_mixture, fp32_to_bf16_bits
    rng = np.random.default_rng(seed)
    feats, labels = [], []
    for l, M in enumerate(sizes):
        x = make_mixture(rng, M, d, 4, "dirichlet", "gauss", 4.0) if M else np.zeros((0, d), np.float32)
        if copies and M > copies:
            x[rng.choice(M, copies, replace=False)] = x[0]                   # equal gains: the lowest index wins
        if dtype == "int8":
            x = np.clip(np.rint(x), -127, 127).astype(np.int8)
        else:
            x = x / np.maximum(np.sqrt((x ** 2).sum(1, keepdims=True)), 1e-30)
            x = fp32_to_bf16_bits(x if scale is None else x * scale(rng, M)[:, None])
        feats.append(x)
        labels.append(np.full(M, l, np.int32))
    feats, labels = np.concatenate(feats), np.concatenate(labels)
    perm = rng.permutation(len(labels))
    caps = np.exp(rng.uniform(0, np.log(8.0), size=W))
    return Workload("edges", dtype, np.ascontiguousarray(feats[perm]), np.ascontiguousarray(labels[perm]), caps, len(sizes), W)


@pytest.mark.parametrize("sizes,d,W", [
    ([1, 2, 3, 0, 33], 17, 1),            # one block; classes of a few samples
    ([127, 128, 129], 64, 2),             # edges of a warp's columns
    ([500], 32, 3),                       # one class over a whole cluster
    ([1921, 60], 96, 5),                  # more columns than one piece per thread of 15 warps; a tiny class beside
    ([700, 300, 5], 64, 16),              # one block per CTA of the largest cluster
    ([900] * 9, 48, 20),                  # several blocks per CTA
    ([130] * 160, 24, 33),                # more classes than SMs: all blocks of a class in one CTA
    ([40] * 20, 16, 128),                 # the most blocks the form takes; more blocks than samples
    ([40] * 3, 16, 129),                  # one more: the pass-based forms
])
def test_int8_exact(rcd, orc, sizes, d, W):
    check_exact(rcd, orc, workload(sizes, d, W, 7 + len(sizes) + W))


@pytest.mark.parametrize("sizes,d,W", [
    ([3841], 40, 2),                      # three pieces per thread
    ([13441, 14500], 32, 5),              # the most pieces the registers take, and one class beyond: gains in shared memory
    ([2300] * 20, 64, 40),                # teams of 16 warps with several blocks
    ([5000] * 10, 48, 100),               # two blocks of one team each per CTA
])
def test_int8_like_the_passes(rcd, sizes, d, W):
    """Sizes that would hold the oracle up: the pass-based form, itself checked against it, is the reference."""
    wl = workload(sizes, d, W, W)
    for got, want in zip(run_partition(rcd, wl), run_partition(rcd, wl, greedy_path=3)):
        assert np.array_equal(got, want)


@pytest.mark.parametrize("W", [3, 24])
def test_int8_ties_exact(rcd, orc, W):
    check_exact(rcd, orc, workload([600, 90], 32, W, W, copies=80))


@pytest.mark.parametrize("sizes,W", [([130] * 160, 33), ([900] * 9, 100), ([300] * 40, 128)])
def test_lists_under_contention(rcd, sizes, W):
    """Many blocks that compete for the same samples: teams of one, two and eight warps hand stored gains to the listing warps,
    and those hand lists to the leader, thousands of times over.  Results do not depend on the timing of any of it: twenty calls
    give the first one's, which is the pass-based form's."""
    import torch
    wl = workload(sizes, 24, W, W, copies=16)
    X, y = rcd.features_to_torch(wl.features, device="cuda"), torch.from_numpy(wl.labels).cuda()
    with rcd.Context(0) as ctx:
        first = [t.clone() for t in ctx.rcd_partition(X, y, wl.capacities, wl.L)]
        for _ in range(20):
            assert all(torch.equal(a, b) for a, b in zip(first, ctx.rcd_partition(X, y, wl.capacities, wl.L)))
        ctx.sync_status()
    for got, want in zip(first, run_partition(rcd, wl, greedy_path=4)):
        assert np.array_equal(got.cpu().numpy(), want)


@pytest.mark.parametrize("sizes,W", [([257, 31], 4), ([800] * 3, 24)])
def test_float(rcd, orc, sizes, W):
    check_float(rcd, orc, workload(sizes, 96, W, W, dtype="bf16"))


def test_float_norms_far_apart(rcd, orc):
    """Classes whose norms span three orders of magnitude stay in floating point, beside classes that do not."""
    wl = workload([300, 220, 64], 64, 6, 3, dtype="bf16", scale=lambda rng, M: 10.0 ** rng.uniform(-1.5 if M != 220 else 0.0, 1.5 if M != 220 else 0.1, M))
    check_float(rcd, orc, wl)


def test_float_class_beyond_the_passes_is_refused(rcd):
    """Bf16 classes that the forms with passes cannot hold are refused whatever their norms, although the cluster form could run
    one whose norms lie close together (zero rows here)."""
    import torch
    X = torch.zeros((51976, 64), dtype=torch.bfloat16, device="cuda")
    y = torch.zeros(51976, dtype=torch.int32, device="cuda")
    with rcd.Context(0) as ctx:
        with pytest.raises(rcd.RcdError, match="coverage vector"):
            ctx.rcd_partition(X, y, [1.0, 2.0], 1)


@pytest.mark.parametrize("sizes,W,apart", [([900, 700], 6, 2), ([1200, 33, 700], 24, 3), ([600, 300, 1, 500], 100, 2)])
def test_float_norms_far_apart_on_all_sms(rcd, orc, sizes, W, apart):
    """Few classes left in floating point are swept by every SM, as they are when the asynchronous form is asked for; the first
    `apart` classes are such.  Once a few long rows cover all that is left every gain is zero, so most picks are ties."""
    import torch
    spread = set(sizes[:apart])
    wl = workload(sizes, 64, W, W, dtype="bf16", scale=lambda rng, M: 10.0 ** rng.uniform(-1.5 if M in spread else 0.0, 1.5 if M in spread else 0.1, M))
    X, y = rcd.features_to_torch(wl.features, device="cuda"), torch.from_numpy(wl.labels).cuda()
    with rcd.Context(0, profile=1) as ctx:
        ctx.rcd_partition(X, y, wl.capacities, wl.L)
        ctx.sync_status()
        assert ctx.profile()["async_visits"] > 0
    check_float(rcd, orc, wl)


@pytest.mark.parametrize("sizes,W,apart", [([800, 500, 300], 100, 1), ([140] * 12 + [130] * 148, 33, 12)])
def test_float_norms_far_apart_with_lists(rcd, orc, sizes, W, apart):
    """The largest classes, which clusters draw first, stay in floating point; the next ones use lists of candidates (several
    blocks per team).  Twice on one context: shared memory then holds what the first call left."""
    import torch
    M0 = sizes[apart - 1]
    wl = workload(sizes, 32, W, W, dtype="bf16", scale=lambda rng, M: 10.0 ** rng.uniform(-1.5 if M == M0 else 0.0, 1.5 if M == M0 else 0.1, M))
    X, y = rcd.features_to_torch(wl.features, device="cuda"), torch.from_numpy(wl.labels).cuda()
    with rcd.Context(0) as ctx:
        first = [t.clone() for t in ctx.rcd_partition(X, y, wl.capacities, wl.L)]
        again = ctx.rcd_partition(X, y, wl.capacities, wl.L)
        ctx.sync_status()
    assert all(torch.equal(a, b) for a, b in zip(first, again))
    check_float(rcd, orc, wl)


@pytest.mark.parametrize("similarity", ["gaussian", "dot"])
@pytest.mark.parametrize("sizes,W", [([128, 1, 77], 5), ([120] * 6, 48)])
def test_float_is_exact_in_fixed_point(rcd, orc, similarity, sizes, W):
    """Floating-point similarities become integers once, and from there on nothing is rounded: picks and values are those of the
    oracle's integer arithmetic on those integers, bit for bit.  And where no two candidates lie closer than the similarities'
    own rounding, the picks are the fp64 oracle's with no tolerance (asserted on the first set of classes)."""
    wl = workload(sizes, 64, W, 5 * W, dtype="bf16")
    kind = rcd.RCD_SIM_GAUSSIAN if similarity == "gaussian" else rcd.RCD_SIM_DOT
    a, o, v = run_partition(rcd, wl, similarity_kind=kind)
    off = 0
    for l, ids in enumerate(orc.split_by_label(wl.labels, wl.L)):
        M = len(ids)
        with rcd.Context(0) as ctx:
            X = rcd.features_to_torch(wl.features[ids], device="cuda").view(1, M, -1)
            S = ctx.rcd_similarity_gaussian(X)[0] if similarity == "gaussian" else ctx.rcd_similarity(X)
            ctx.sync_status()
            S = S.cpu().numpy()[0, :, :M].astype(np.float64)
        # the largest value lands in [2^29, 2^30); the Gaussian kernel's is 1
        e = 29 if similarity == "gaussian" else 30 - int(np.frexp(np.float32(S.diagonal().max()))[1])
        F = np.clip(np.rint(S * 2.0 ** e), 1 - 2 ** 30, 2 ** 30 - 1).astype(np.int64)
        q = orc.quotas(M, wl.capacities)
        want, oj, ov, fv = orc.partition_class(F, q, "incremental")
        assert np.array_equal(o[off:off + M], ids[ov]) and np.array_equal(a[ids], want)
        assert np.array_equal(v[l], np.ldexp(fv.astype(np.float64), -e))
        if len(sizes) == 3:
            exact = orc.class_similarity(wl.features[ids], similarity)
            assert orc.replay_class(exact, q, oj, ov, 0.0)[0] == -1
        off += M


@pytest.mark.parametrize("sizes,W", [([400, 3], 5), ([600] * 4, 24), ([90] * 150, 20)])
def test_graph_cut_int8_exact(rcd, orc, sizes, W):
    wl = workload(sizes, 48, W, W)
    a, o, v = run_partition(rcd, wl, objective=rcd.RCD_OBJ_GRAPH_CUT)
    ref = orc.partition(wl.features, wl.labels, wl.capacities, wl.L, variant="incremental", objective="cut")
    assert np.array_equal(a, ref.assignment) and np.array_equal(o, ref.order) and np.array_equal(v, ref.part_values)


@pytest.mark.parametrize("L", [255, 6000, 6001])
def test_class_split_many_labels(rcd, orc, L):
    """Chunk counters in shared memory up to 6000 labels, in global memory beyond."""
    rng = np.random.default_rng(L)
    wl = workload([3, 2], 32, 2, L)
    wl.labels = np.sort(rng.integers(0, L, 3000).astype(np.int32))[rng.permutation(3000)]
    wl.features = rng.integers(-9, 10, size=(3000, 32)).astype(np.int8)
    wl.L = L
    check_exact(rcd, orc, wl)


@pytest.mark.parametrize("dtype", ["int8", "bf16"])
def test_objective_samples_in_no_block(rcd, orc, dtype):
    """Rows in units of 128, columns in units of 512; entries below zero belong to no block, one block is empty."""
    import torch
    wl = workload([129, 513, 1], 96, 4, 11, dtype=dtype)
    rng = np.random.default_rng(5)
    a = rng.integers(-1, 3, size=len(wl.labels)).astype(np.int32)
    with rcd.Context(0) as ctx:
        X = rcd.features_to_torch(wl.features, device="cuda")
        vals, total = ctx.rcd_objective(X, torch.from_numpy(wl.labels).cuda(), torch.from_numpy(a).cuda(), wl.W, wl.L)
        ctx.sync_status()
        vals, total = vals.cpu().numpy(), total.cpu().numpy()
    want = np.zeros((wl.L, wl.W))
    for l, ids in enumerate(orc.split_by_label(wl.labels, wl.L)):
        S = np.asarray(orc.similarity(wl.features[ids]), dtype=np.float64)
        for p in range(wl.W):
            m = a[ids] == p
            if m.any():
                want[l, p] = np.maximum(S[:, m].max(1), 0).sum()
    if dtype == "int8":
        assert np.array_equal(vals, want.astype(np.int64)) and total[0] == vals.sum()
    else:
        assert np.allclose(vals, want, rtol=1e-5, atol=1e-5) and np.isclose(total[0], want.sum(), rtol=1e-5)


@pytest.mark.parametrize("M", [1, 2, 64, 65, 127, 130, 1027])
def test_gaussian_edges(rcd, orc, M):
    """Row groups of 64, column groups of 128 and, from 1025 on, a warp's second group."""
    wl = workload([M, M], 40, 1, M, dtype="bf16")
    x = np.concatenate([wl.features[wl.labels == l] for l in (0, 1)])
    with rcd.Context(0) as ctx:
        S, sigma = ctx.rcd_similarity_gaussian(rcd.features_to_torch(x, device="cuda").view(2, M, 40))
        ctx.sync_status()
        S, sigma = S.cpu().numpy(), sigma.cpu().numpy()
    for b in range(2):
        want, sg = orc.similarity_gaussian(x[b * M:(b + 1) * M])
        assert sigma[b] == pytest.approx(sg, rel=2e-6)
        assert np.allclose(S[b, :, :M], want, rtol=2e-5, atol=1e-7) and np.all(S[b, :, M:] == 0)


@pytest.mark.parametrize("M,batch,d,dtype", [(129, 1, 1024, "int8"), (256, 3, 1040, "int8"), (257, 2, 512, "bf16"), (500, 80, 520, "bf16"),
                                             (1000, 9, 1024, "int8"), (1024, 1, 1024, "int8")])
def test_similarity_long_rows(rcd, orc, M, batch, d, dtype):
    """Pairs of SMs: one and several row blocks, whole rounds of tiles and rounds cut into strips; two calls overlap on two streams."""
    import torch
    g = torch.Generator().manual_seed(M)
    X = torch.randint(-128, 128, (batch, M, d), generator=g).to(torch.int8) if dtype == "int8" else torch.randn(batch, M, d, generator=g).to(torch.bfloat16)
    X = X.cuda()
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    torch.cuda.synchronize()
    with rcd.Context(0) as ctx:
        got = []
        for st in streams:
            with torch.cuda.stream(st):
                got.append(ctx.rcd_similarity(X))
        torch.cuda.synchronize()
        ctx.sync_status()
    w = X.double()
    want = torch.matmul(w, w.transpose(1, 2))
    for S in got:
        assert bool((S[:, :, M:] == 0).all()) and torch.equal(S[:, :, :M], S[:, :, :M].transpose(1, 2))
        err = (S[:, :, :M].double() - want).abs().max().item()
        assert err == 0 if dtype == "int8" else err <= 2e-5 * want.abs().max().item()
