"""The objective of an assignment where the blocks' maxima are taken from the accumulator tiles: runs of columns and rows of one block
from one sample to more than a tile, edges of tiles, samples in no block, rows of any alignment."""
import numpy as np
import pytest

import test_gpu_cluster as cluster
from test_gpu_parity import rcd, orc  # noqa: F401  (fixtures)

pytestmark = pytest.mark.gpu


def objective(rcd, wl, X, a, **cfg):
    import torch
    with rcd.Context(0, **cfg) as ctx:
        vals, total = ctx.rcd_objective(X, torch.from_numpy(wl.labels).cuda(), torch.from_numpy(a).cuda(), wl.W, wl.L)
        ctx.sync_status()
        return vals.cpu().numpy(), total.cpu().numpy()


def maxima(S, blocks, W):
    """f of every block from a class's similarities (a NaN is above nothing)."""
    S = np.where(S > 0, S, 0.0)
    return [S[:, blocks == p].max(1).sum() if (blocks == p).any() else 0.0 for p in range(W)]


@pytest.mark.parametrize("dtype", ["int8", "bf16"])
@pytest.mark.parametrize("sizes,d,W", [
    ([31, 32, 33, 0, 1], 75, 3),          # within a column block; rows that are no multiple of 16 bytes
    ([127, 128, 129, 255, 257], 96, 2),   # edges of both sides of a tile; runs longer than a row block
    ([300, 40], 64, 150),                 # runs of one or two samples, blocks without any
    ([520, 700], 144, 20),                # two to four runs in 32 rows
    ([520, 700], 72, 95),                 # five to eight: about as many as are gone through by themselves
    ([900], 200, 1024),                   # the most blocks
    ([65, 130], 520, 3),                  # rows of more than 512 bytes
])
def test_objective_by_tiles(rcd, orc, sizes, d, W, dtype):
    wl = cluster.workload(sizes, d, W, 3 + W, dtype=dtype)
    a = np.random.default_rng(W).integers(-2, W + 1, size=len(wl.labels)).astype(np.int32)       # (outside [0, W): in no block)
    vals, total = objective(rcd, wl, rcd.features_to_torch(wl.features, device="cuda"), a)
    want = np.array([maxima(np.asarray(orc.similarity(wl.features[ids]), np.float64), a[ids], W) if len(ids) else [0.0] * W
                     for ids in orc.split_by_label(wl.labels, wl.L)])
    if dtype == "int8":
        assert np.array_equal(vals, want.astype(np.int64)) and total[0] == vals.sum()
    else:
        # fp32 sums of 200 products of unit rows: 200 x 2^-24 of the largest similarity at most per entry
        assert np.allclose(vals, want, rtol=1e-5, atol=1e-5) and np.isclose(total[0], want.sum(), rtol=1e-5)


def test_objective_not_a_number(rcd, orc):
    """Similarities with a sample whose features are not numbers are above nothing; the other blocks' values stay."""
    wl = cluster.workload([200], 64, 5, 9, dtype="bf16")
    X = rcd.features_to_torch(wl.features, device="cuda")
    X[17] = float("nan")
    a = (np.arange(200) % 5).astype(np.int32)
    S = (X.double() @ X.double().T).cpu().numpy()
    vals, total = objective(rcd, wl, X, a)
    assert np.allclose(vals[0], maxima(S, a, 5), rtol=1e-5, atol=1e-5) and np.isclose(total[0], vals.sum(), rtol=1e-5)


def test_objective_infinite(rcd):
    """Infinite similarities of either sign: those above zero make their blocks' values infinite, the others change nothing."""
    wl = cluster.workload([200, 150], 64, 5, 9, dtype="bf16")
    X = rcd.features_to_torch(wl.features, device="cuda")
    ids = np.nonzero(wl.labels == 0)[0]
    a = np.zeros(350, np.int32)
    for l in (0, 1):
        a[wl.labels == l] = np.arange((wl.labels == l).sum()) % 5
    X[:, 7] = X[:, 7].abs().clamp_min(0.01)
    for i in ids[a[ids] != 3]:
        X[i, 7] *= -1                                         # (sample 17 of the class, in block 2: -inf to all but block 3 and itself)
    X[ids[17], 7] = float("inf")
    vals, total = objective(rcd, wl, X, a)
    Xd = X.double().cpu()
    for l in (0, 1):
        x = Xd[wl.labels == l]
        want = np.array(maxima((x @ x.T).numpy(), a[wl.labels == l], 5))
        assert np.isinf(want).tolist() == [False, False, l == 0, l == 0, False]
        assert np.allclose(vals[l], want, rtol=1e-5, atol=1e-5)
    assert np.isposinf(total[0])


def test_objective_many_samples_per_warp(rcd, orc):
    """More samples of a class than the sorting warps keep in registers (1024 blocks leave room for the counters of eleven warps)."""
    wl = cluster.workload([3000, 70], 64, 1024, 4)
    a = np.random.default_rng(4).integers(-1, 1024, size=len(wl.labels)).astype(np.int32)
    vals, total = objective(rcd, wl, rcd.features_to_torch(wl.features, device="cuda"), a)
    want = [maxima(np.asarray(orc.similarity(wl.features[ids]), np.float64), a[ids], 1024) for ids in orc.split_by_label(wl.labels, wl.L)]
    assert np.array_equal(vals, np.array(want).astype(np.int64)) and total[0] == vals.sum()


@pytest.mark.parametrize("sizes,W", [([129, 513, 1], 4), ([127, 128, 700, 0], 150)])
@pytest.mark.parametrize("dtype,similarity", [("int8", "dot"), ("bf16", "dot"), ("int8", "gaussian"), ("bf16", "gaussian")])
def test_objective_through_s(rcd, orc, sizes, W, dtype, similarity):
    """The maxima taken from S (generic similarity kernel, Gaussian kernel): units of 128 rows and 512 columns, samples in no block."""
    cfg = dict(similarity_path=2) if similarity == "dot" else dict(similarity_kind=rcd.RCD_SIM_GAUSSIAN)
    wl = cluster.workload(sizes, 96, W, W, dtype=dtype)
    a = np.random.default_rng(W).integers(-2, W + 1, size=len(wl.labels)).astype(np.int32)
    vals, total = objective(rcd, wl, rcd.features_to_torch(wl.features, device="cuda"), a, **cfg)
    sim = orc.similarity if similarity == "dot" else lambda x: orc.similarity_gaussian(x)[0]
    want = np.array([maxima(np.asarray(sim(wl.features[ids]), np.float64), a[ids], W) if len(ids) else [0.0] * W
                     for ids in orc.split_by_label(wl.labels, wl.L)])
    if vals.dtype == np.int64:
        assert np.array_equal(vals, want.astype(np.int64)) and total[0] == vals.sum()
    else:
        # dot products as above; the Gaussian kernel's entries lie within 2e-5 of the oracle's (test_gaussian_edges)
        rtol = 1e-5 if similarity == "dot" else 2e-5
        assert np.allclose(vals, want, rtol=rtol, atol=1e-5) and np.isclose(total[0], want.sum(), rtol=rtol)
