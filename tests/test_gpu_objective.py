"""The objective of an assignment where the blocks' maxima are taken from the accumulator tiles: runs of columns and rows of one block
from one sample to more than a tile, edges of tiles, samples in no block, rows of any alignment."""
import numpy as np
import pytest

import test_gpu_cluster as cluster
from test_gpu_parity import rcd, orc  # noqa: F401  (fixtures)

pytestmark = pytest.mark.gpu


def objective(rcd, wl, X, a):
    import torch
    with rcd.Context(0) as ctx:
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
    import torch
    wl = cluster.workload([200], 64, 5, 9, dtype="bf16")
    X = rcd.features_to_torch(wl.features, device="cuda")
    X[17] = float("nan")
    a = (np.arange(200) % 5).astype(np.int32)
    S = (X.double() @ X.double().T).cpu().numpy()
    vals, _ = objective(rcd, wl, X, a)
    assert np.allclose(vals[0], maxima(S, a, 5), rtol=1e-5, atol=1e-5)
    assert torch.isnan(X[17]).all()
