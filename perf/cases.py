"""Cases of the partition path, for measuring it through the package's public entry points.

A case names one use of the library: ``op`` is the entry point that a program calls, the other keys are its
sizes and options.

  partition     ``Context.rcd_partition``: device tensors in, device tensors out (Algorithm 1 on every class)
  host          ``Context.rcd_partition_host``: the same with pinned host tensors, copies inside the call
  objective     ``Context.rcd_objective``: f(A_j^l) of a given assignment from the plain definition
  similarity    ``Context.rcd_similarity``: the similarity matrices alone
  lists         ``rcd_worker_lists``: an assignment turned into one index list per worker

Inputs follow the law of the package's own synthetic workloads (``workloads.py``): every class is a mixture of ``K``
Gaussian components with Dirichlet weights, samples arrive with their labels interleaved; int8 features are rounded
and clipped, bf16 features are rows normalised in fp32 (``law`` "relu": absolute values first, as after a rectifier).
They are drawn on the device, from the seed alone.

What is compared.  int8 features with dot products are exact arithmetic end to end: assignment, pick order and the
int64 block values are returned and have to be identical.  With floating-point similarities Algorithm 1 takes an
argmax over sums of thousands of fp32 values, so two correct implementations part ways at the first pair of
candidates closer than the rounding of those sums, and from there on the two assignments are different, equally good
partitions: such cases return the block values f(A_j^l) and the worker lists' boundaries (how many samples every
worker got, which the quotas fix exactly).
"""
import numpy as np
import torch

from paper_2211_00839_b200 import binding as rcd

_CAPS = {
    # a small cluster with one fast and one faster machine, and the same mix on eight workers
    "list4": [1, 1, 2, 4],
    "list8": [1, 1, 1, 1, 2, 2, 4, 4],
}


def listed():
    return [
        # The smallest call: two classes of 200 samples on four workers (400 picks: launches and latency).
        dict(name="int8_2x200", op="partition", dtype="int8", sim="dot", obj="facility", L=2, M=200, tail=1, d=64, W=4,
             K=3, law="gauss", caps="list4"),
        # The default benchmark: a ten-class data set of 50 000 samples, exact int8 features, eight workers.
        dict(name="int8_10x5000", op="partition", dtype="int8", sim="dot", obj="facility", L=10, M=5000, tail=1, d=512,
             W=8, K=8, law="gauss", caps="list8"),
        # The same data set with normalised bf16 features (cosine similarity), sixteen workers.
        dict(name="bf16_10x5000", op="partition", dtype="bf16", sim="dot", obj="facility", L=10, M=5000, tail=1, d=512,
             W=16, K=8, law="gauss", caps="half"),
        # A hundred classes of 500 rectified bf16 features of width 2048, 32 workers of very different speed.
        dict(name="bf16_100x500", op="partition", dtype="bf16", sim="dot", obj="facility", L=100, M=500, tail=1, d=2048,
             W=32, K=4, law="relu", caps="loguniform"),
        # The largest: a thousand classes, 1.3 million samples, 64 workers in four tiers.
        dict(name="int8_1000x1300", op="partition", dtype="int8", sim="dot", obj="facility", L=1000, M=1300, tail=1,
             d=2048, W=64, K=16, law="gauss", caps="tiers"),
        # Long-tailed classes (sizes falling from 2500 to 50) with a feature width that is no multiple of 16 bytes.
        dict(name="int8_longtail", op="partition", dtype="int8", sim="dot", obj="facility", L=20, M=2500, tail=50, d=200,
             W=10, K=8, law="gauss", caps="half"),
        # The Gaussian kernel in place of the dot product (the paper's own experiments used it).
        dict(name="gauss_10x5000", op="partition", dtype="int8", sim="gaussian", obj="facility", L=10, M=5000, tail=1,
             d=512, W=8, K=8, law="gauss", caps="list8"),
        # The graph-cut objective in place of facility location.
        dict(name="cut_10x5000", op="partition", dtype="int8", sim="dot", obj="cut", L=10, M=5000, tail=1, d=512, W=8,
             K=8, law="gauss", caps="list8"),
        # End to end from host memory: features up, assignment, order and values back.
        dict(name="host_100x500", op="host", dtype="int8", sim="dot", obj="facility", L=100, M=500, tail=1, d=512, W=8,
             K=4, law="gauss", caps="list8"),
        # The value of a given assignment (how a user compares a partition with a random one).
        dict(name="objective_10x5000", op="objective", dtype="int8", sim="dot", obj="facility", L=10, M=5000, tail=1,
             d=512, W=8, K=8, law="gauss", caps="list8"),
        # Similarity matrices alone, wide features.
        dict(name="similarity_100x500", op="similarity", dtype="bf16", sim="dot", obj="facility", L=100, M=500, tail=1,
             d=2048, W=1, K=4, law="relu", caps="half"),
        # Index lists for 64 workers from an assignment of 1.3 million samples.
        dict(name="lists_1300000", op="lists", dtype="int8", sim="dot", obj="facility", L=1000, M=1300, tail=1, d=16,
             W=64, K=1, law="gauss", caps="tiers"),
    ]


def _log(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    op = rng.choice(["partition"] * 8 + ["host", "objective", "similarity", "lists"])
    dtype = rng.choice(["int8", "bf16"])
    L = _log(rng, 1, 1000)
    if op == "lists":
        return dict(op=op, dtype="int8", sim="dot", obj="facility", L=L, M=max(1, _log(rng, 500, 1300000) // L), tail=1,
                    d=16, W=_log(rng, 2, 64), K=1, law="gauss", caps="half")
    # at most as many samples and similarity entries as the largest listed case has; a class has at least 16 samples
    M = _log(rng, 16, min(5000, int((1.0e9 / L) ** 0.5), 1000000 // L))
    tail = rng.choice([1, 1, _log(rng, 2, 100)]) if M >= 200 and L > 1 and op != "similarity" else 1
    # widths with rows of whole 16-byte pieces (the usual ones) and any others
    d = _log(rng, 64, min(2048, max(64, int(2.0e9 / (L * M)))))
    if rng.random() < 0.75:
        d = max(64, d // 64 * 64)
    return dict(op=op, dtype=dtype, sim=rng.choice(["dot", "dot", "dot", "gaussian"]) if op == "partition" else "dot",
                obj=rng.choice(["facility"] * 5 + ["cut"]) if op == "partition" else "facility",
                L=L, M=M, tail=tail, d=d, W=_log(rng, 2, 64), K=rng.choice([3, 4, 8, 16]),
                law=rng.choice(["gauss", "gauss", "relu"]), caps=rng.choice(["half", "loguniform"]))


def _sizes(case):
    """Class sizes: all M, or falling geometrically from M to M / tail."""
    L, M, tail = case["L"], case["M"], case["tail"]
    if tail == 1 or L == 1:
        return [M] * L
    return [max(1, int(round(M * float(tail) ** (-l / (L - 1))))) for l in range(L)]


def _capacities(case, seed):
    W, kind = case["W"], case["caps"]
    if kind in _CAPS:
        return np.asarray(_CAPS[kind], dtype=np.float64)
    if kind == "tiers":          # equal tiers of speed 1:2:4:8
        return np.asarray([2.0 ** (4 * j // W) for j in range(W)], dtype=np.float64)
    rng = np.random.default_rng(seed)
    if kind == "half":           # uniform on [1, 4] in steps of one half
        return np.round(rng.uniform(1.0, 4.0, size=W) * 2.0) / 2.0
    return np.exp(rng.uniform(0.0, 1.0, size=W) * np.log(8.0))      # "loguniform" over [1, 8]


def _features(case, labels, gen):
    L, K, d, dev = case["L"], case["K"], case["d"], labels.device
    N = labels.numel()
    std = 1.0 if case["law"] == "relu" else 4.0
    mu = torch.randn((L, K, d), generator=gen, device=dev) * std
    w = -torch.log(torch.rand((L, K), generator=gen, device=dev).clamp_min(1e-12))     # Dirichlet(1) after division
    w = w / w.sum(1, keepdim=True)
    out = torch.empty((N, d), dtype=torch.int8 if case["dtype"] == "int8" else torch.bfloat16, device=dev)
    step = max(1, (1 << 27) // d)
    for a in range(0, N, step):
        lab = labels[a:a + step].long()
        u = torch.rand((lab.numel(), 1), generator=gen, device=dev)
        comp = (u > w[lab].cumsum(1)).sum(1).clamp_max(K - 1)
        x = torch.randn((lab.numel(), d), generator=gen, device=dev)
        x += mu[lab, comp]
        if case["law"] == "relu":
            x.abs_()
        if case["dtype"] == "int8":
            out[a:a + step] = x.round_().clamp_(-127, 127).to(torch.int8)
        else:
            x /= x.norm(dim=1, keepdim=True).clamp_min(1e-30)
            out[a:a + step] = x.to(torch.bfloat16)
    return out


def prepare(case, seed):
    dev = torch.device("cuda", 0)
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed)
    op, sizes = case["op"], _sizes(case)
    s = {"op": op, "case": case, "L": case["L"], "W": case["W"], "M_max": max(sizes),
         "exact": case["dtype"] == "int8" and case["sim"] == "dot"}
    s["ctx"] = rcd.Context(device=0, similarity_kind=rcd.RCD_SIM_GAUSSIAN if case["sim"] == "gaussian" else rcd.RCD_SIM_DOT,
                           objective=rcd.RCD_OBJ_GRAPH_CUT if case["obj"] == "cut" else rcd.RCD_OBJ_FACILITY)
    N = sum(sizes)
    if op in ("objective", "lists"):
        # every sample on a worker drawn with probability proportional to the worker's capacity
        edges = torch.from_numpy(np.cumsum(_capacities(case, seed))).to(dev)
        u = torch.rand(N, generator=gen, device=dev, dtype=torch.float64) * edges[-1]
        s["assignment"] = torch.searchsorted(edges, u, right=True).clamp_max(case["W"] - 1).to(torch.int32)
        if op == "lists":
            return s
    labels = torch.repeat_interleave(torch.arange(case["L"], device=dev), torch.tensor(sizes, device=dev))
    if op == "similarity":
        s["X"] = _features(case, labels, gen).view(case["L"], case["M"], case["d"])
        return s
    s["labels"] = labels[torch.randperm(N, generator=gen, device=dev)].to(torch.int32)
    s["features"] = _features(case, s["labels"], gen)
    s["capacities"] = _capacities(case, seed)
    if op == "host":
        s["features"] = s["features"].cpu().pin_memory()
        s["labels"] = s["labels"].cpu().pin_memory()
        # the buffers a program that partitions again and again keeps for the results
        s["out"] = (torch.empty(N, dtype=torch.int32).pin_memory(), torch.empty(N, dtype=torch.int32).pin_memory(),
                    torch.empty((case["L"], case["W"]), dtype=torch.int64 if s["exact"] else torch.float64).pin_memory())
    return s


def run(s):
    op, ctx = s["op"], s["ctx"]
    if op == "partition":
        assignment, order, values = ctx.rcd_partition(s["features"], s["labels"], s["capacities"], s["L"], M_max=s["M_max"])
        if s["exact"]:
            return {"assignment": assignment, "order": order, "values": values}
        offsets, _ = rcd.rcd_worker_lists(ctx, assignment, s["W"])
        return {"values": values, "offsets": offsets}
    if op == "host":
        assignment, order, values = ctx.rcd_partition_host(s["features"], s["labels"], s["capacities"], s["L"],
                                                           M_max=s["M_max"], out=s["out"])
        if s["exact"]:
            return {"assignment": assignment, "order": order, "values": values}
        return {"values": values}
    if op == "objective":
        values, total = ctx.rcd_objective(s["features"], s["labels"], s["assignment"], s["W"], s["L"], M_max=s["M_max"])
        return {"values": values, "total": total}
    if op == "similarity":
        return ctx.rcd_similarity(s["X"])
    offsets, indices = rcd.rcd_worker_lists(ctx, s["assignment"], s["W"])
    return {"offsets": offsets, "indices": indices}


def work(case):
    """Inputs read once, outputs written once; the distinct products of the symmetric similarity matrices, and for the
    partition and the objective one comparison and one addition per entry of them (the gains of the first pick of a
    class, the maxima of the plain definition): what any exact method evaluates at least once."""
    sizes, op, d, L, W = _sizes(case), case["op"], case["d"], case["L"], case["W"]
    eb = 1 if case["dtype"] == "int8" else 2
    if op == "lists":
        N = sum(sizes)
        return {"bytes": 8 * N + 8 * (W + 1), "flops": 0}
    if op == "similarity":
        M = case["M"]
        return {"bytes": L * M * (d * eb + 4 * M), "flops": L * M * (M + 1) * d}
    N = sum(sizes)
    flops = sum(m * (m + 1) * d + 2 * m * m for m in sizes)
    if op == "objective":
        return {"bytes": N * d * eb + 8 * N + 8 * L * W + 8, "flops": flops}
    lists = case["dtype"] != "int8" or case["sim"] != "dot"
    return {"bytes": N * d * eb + 4 * N + 8 * N + 8 * L * W + ((8 * N + 8 * (W + 1)) if lists and op == "partition" else 0),
            "flops": flops}


def tolerance(case):
    """int8 dot products, and everything made from them, are whole numbers.  A similarity of bf16 rows is an fp32 sum
    of up to 2048 products, and the plain-definition objective a double sum of those.  Block values of a floating-point
    partition differ by 1e-6 to 2e-4 (one block by up to 3e-3) between this library's own two similarity kernels, whose
    products are added in different orders (up to a fifth of the samples then sit on another worker)."""
    if case["op"] == "lists" or (case["dtype"] == "int8" and case["sim"] == "dot"):
        return "exact"
    if case["op"] in ("similarity", "objective"):
        return {"rel": 1e-5, "max": 1e-4}
    return {"rel": 1e-3, "max": 1e-2}
