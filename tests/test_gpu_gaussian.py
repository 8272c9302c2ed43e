"""Gaussian-kernel similarity (Section 4 item 2) on the GPU against the oracle.

The kernel values are fp32 on the GPU and double in the oracle; for int8 features the squared
distances are exact integers on both sides, so the only differences are the fp32 bandwidth factor
and expf (relative 1e-6); for bf16 features the fp32 dot products add about 1e-6 absolute to the
exponent.  Partitions are compared with the same teacher-forced rule as the cosine configurations.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

OBJ_RTOL = 1e-4
PICK_RTOL = 1e-3


@pytest.fixture(scope="module")
def rcd():
    from paper_2211_00839_b200 import binding
    return binding


@pytest.fixture(scope="module")
def orc():
    from oracle import rcd_oracle
    return rcd_oracle


@pytest.mark.parametrize("name,M,d,batch", [("C1", 200, 64, 2), ("C2", 333, 512, 1), ("C4", 257, 256, 2), ("C3", 130, 37, 1)])
def test_gaussian_similarity_matches_oracle(rcd, orc, name, M, d, batch):
    import torch
    from paper_2211_00839_b200.workloads import make_workload
    wl = make_workload(name, L=batch, M=M, d=d, shuffle=False)
    with rcd.Context(0) as ctx:
        X = rcd.features_to_torch(wl.features, device=torch.device("cuda", 0)).view(batch, M, d)
        S, sigma = ctx.rcd_similarity_gaussian(X)
        ctx.sync_status()
        S, sigma = S.cpu().numpy(), sigma.cpu().numpy()
    for b in range(batch):
        want, sg = orc.similarity_gaussian(wl.features[b * M:(b + 1) * M])
        assert sigma[b] == pytest.approx(sg, rel=2e-6)
        assert np.allclose(S[b, :, :M], want, rtol=2e-5, atol=1e-7)
        assert np.all(np.diag(S[b, :, :M]) == 1.0)
        assert np.array_equal(S[b, :, :M], S[b, :, :M].T)
        assert np.all(S[b, :, M:] == 0)


def test_gaussian_similarity_of_coincident_points(rcd):
    import torch
    X = torch.full((1, 40, 128), 3, dtype=torch.int8, device="cuda")
    with rcd.Context(0) as ctx:
        S, sigma = ctx.rcd_similarity_gaussian(X)
        ctx.sync_status()
        assert float(sigma[0]) == 0.0 and bool((S[0, :, :40] == 1).all())


def test_call_after_one_that_was_given_up_under_way(rcd):
    """More classes than the Gaussian kernel takes are refused once the class sizes are known, with copies out of the context's
    pinned memory under way: the next call, on another stream, must not write into that memory before they are done."""
    import torch
    rng = np.random.default_rng(1)
    X = torch.from_numpy(rng.integers(-9, 10, size=(70000, 128)).astype(np.int8)).cuda()
    many = (torch.arange(70000, device="cuda") % 66000).to(torch.int32)
    few = (torch.arange(70000, device="cuda") % 200).to(torch.int32)
    with rcd.Context(0, similarity_kind=rcd.RCD_SIM_GAUSSIAN) as ctx:
        want = [t.clone() for t in ctx.rcd_partition(X, few, [1.0, 2.0], 200)]
        torch.cuda.synchronize()
        for _ in range(3):
            with pytest.raises(rcd.RcdError):
                ctx.rcd_partition(X, many, [1.0, 2.0], 66000, M_max=2)
            still_used, ctx._ws = ctx._ws, None                          # (streams that overlap need a workspace each)
            with torch.cuda.stream(torch.cuda.Stream()):
                got = ctx.rcd_partition(X, few, [1.0, 2.0], 200)
                ctx.sync_status()
            assert all(torch.equal(a, b) for a, b in zip(want, got))


def test_distance_roots_to_one_unit_in_the_last_place(rcd):
    """Distances are rooted by two of Heron's steps from a 22-bit reciprocal root: 2^-65 of the root is left after them, so the
    last rounding leaves half a unit in the last place of fp64 and next to nothing more; one unit is allowed.  Classes of two
    samples, the second zero: the class's sum of distances, an fp64 word of the scratch buffer, is twice the first one's norm.
    Squared norms n 2^2k, n < 2^24 a sum of squares of whole numbers: exact in fp32."""
    import torch
    rng = np.random.default_rng(3)
    d, cases = 1024, []
    for k in (-74, -70, -63, -40, -1, 0, 1, 30, 52):
        for n in (1, 2, 3, 40):
            cases.append((rng.integers(1, 256, size=n), k))
    most = np.concatenate([np.full(258, 255), [27, 6]])                  # 2^24 - 1: the largest fp32 at k = 52
    cases += [(np.zeros(1, np.int64), 0), (most, 52), (most, -74), (np.ones(1, np.int64), 64)]       # (the last: infinity)
    x = np.zeros((len(cases), 2, d), np.float32)
    square = np.zeros(len(cases))
    for i, (n, k) in enumerate(cases):
        x[i, 0, :len(n)] = n * np.float32(2.0) ** k
        square[i] = float((n.astype(np.int64) ** 2).sum()) * 2.0 ** (2 * k)
    square[square >= 2.0 ** 128] = np.inf
    assert np.array_equal(square.astype(np.float32).astype(np.float64), square)
    with rcd.Context(0) as ctx:
        X = torch.from_numpy(x).to(torch.bfloat16).cuda()
        assert np.array_equal(X.float().cpu().numpy(), x)
        ctx.rcd_similarity_gaussian(X)
        ctx.sync_status()
        at = (2 * len(cases) * 4 + 255) // 256 * 256                     # behind the norms of the rows
        got = ctx.workspace(at + 8 * len(cases))[at:at + 8 * len(cases)].cpu().numpy().view(np.float64)
    want = np.sqrt(square)
    fin = np.isfinite(want)
    assert np.array_equal(got[~fin], want[~fin])
    assert np.all(np.abs(got[fin] / 2 - want[fin]) <= np.spacing(want[fin]) * (want[fin] > 0))


@pytest.mark.parametrize("name,L,M,d,path", [("C1", 2, 200, 64, 0), ("C2", 2, 700, 128, 0), ("C4", 3, 400, 256, 1)])
def test_partition_with_gaussian_similarity(rcd, orc, name, L, M, d, path):
    import torch
    from paper_2211_00839_b200.workloads import make_workload
    wl = make_workload(name, L=L, M=M, d=d)
    dev = torch.device("cuda", 0)
    with rcd.Context(0, similarity_kind=rcd.RCD_SIM_GAUSSIAN, greedy_path=path) as ctx:
        X = rcd.features_to_torch(wl.features, device=dev)
        y = torch.from_numpy(wl.labels).to(dev)
        a, o, v = ctx.rcd_partition(X, y, wl.capacities, wl.L)
        vals, total = ctx.rcd_objective(X, y, a, wl.W, wl.L)
        ctx.sync_status()
        assert v.dtype == torch.float64 and vals.dtype == torch.float64
        a, o, v, vals = a.cpu().numpy(), o.cpu().numpy(), v.cpu().numpy(), vals.cpu().numpy()
    assert np.allclose(v, vals, rtol=OBJ_RTOL)
    groups = orc.split_by_label(wl.labels, wl.L)
    off = 0
    for l, ids in enumerate(groups):
        Ml = len(ids)
        q = orc.quotas(Ml, wl.capacities)
        assert np.array_equal(np.bincount(a[ids], minlength=wl.W), q)
        picked = o[off:off + Ml]
        off += Ml
        local = np.searchsorted(ids, picked).astype(np.int32)
        S, _ = orc.similarity_gaussian(wl.features[ids])
        bad, stats, fv = orc.replay_class(S, q, a[picked], local, PICK_RTOL)
        assert bad == -1, (l, bad, stats)
        assert np.allclose(v[l], fv, rtol=OBJ_RTOL, atol=1e-9)
    want = orc.objective(wl.features, wl.labels, a, wl.W, wl.L, similarity_kind="gaussian")
    assert np.allclose(vals, want, rtol=1e-5, atol=1e-7)
