"""Performance cases: the calls a user of the k-d tree builder makes, with
inputs of the workloads that the build is exercised on.

A case is a dict of plain values.  ``op`` names the public entry point:

  build    build_tree (kd_presort + kd_build) of one cloud on the device
  batch    kd_build_batch_packed: many uneven clouds in one call
  serve    kd_submit / kd_wait: a burst of requests in host memory
  select   kd_build_select: the median-selection build
  presort  kd_presort_noalloc: a small presort into the caller's buffers
  knn      kd_knn: nearest neighbours of given query points
  knn_all  kd_knn_all: nearest neighbours of every tuple of a tree
  region   kd_region: the tuples inside given boxes

and ``dist`` the coordinates: "int" (uniform in [0, 2^bits), int32 or int64),
"gmm" (float32, 64-component isotropic Gaussian mixture) or "cube" (float32
uniform in the unit cube).  ``dup`` is the share of tuples that are exact
copies of another one.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1410_5420_gb300 import api

DEVICE = "cuda"
TORCH_TYPE = {"i32": torch.int32, "i64": torch.int64, "f32": torch.float32}
WORD = {"i32": 4, "i64": 8, "f32": 4}
TREE = ("node_tuple", "left", "right", "dim")  # 13 bytes per node in all


def listed() -> list:
    return [
        # the smallest clouds a request stream brings: launches and host round trips count, not work
        dict(name="build_256_k2_i32", op="build", n=256, k=2, dtype="i32", dist="int", bits=24, dup=0.0),
        # the small parity configuration: 1% exact duplicates, 64-bit keys
        dict(name="build_16384_k3_i64", op="build", n=16384, k=3, dtype="i64", dist="int", bits=20, dup=0.01),
        # a ragged cloud of the middle of the served range, four dimensions
        dict(name="build_300007_k4_f32", op="build", n=300007, k=4, dtype="f32", dist="gmm", bits=0, dup=0.0),
        # the end of the dimension sweep: six dimensions of 64-bit keys
        dict(name="build_4194304_k6_i64", op="build", n=1 << 22, k=6, dtype="i64", dist="int", bits=40, dup=0.0),
        # the headline workload: 2^26 three-dimensional points
        dict(name="build_67108864_k3_f32", op="build", n=1 << 26, k=3, dtype="f32", dist="gmm", bits=0, dup=0.0),
        # thousands of uneven clouds built together
        dict(name="batch_4096_k3_f32", op="batch", count=4096, lo=6, hi=16, k=3, dtype="f32", dist="cube", bits=0,
             dup=0.005),
        # a burst of requests to the serving loop, mixed dimensions and types, host memory in and out
        dict(name="serve_48", op="serve", count=48, lo=8, hi=20),
        # the comparison algorithm on the dimension sweep's three-dimensional cloud
        dict(name="select_4194304_k3_i64", op="select", n=1 << 22, k=3, dtype="i64", dist="int", bits=40, dup=0.0),
        # the allocation-free presort at its largest size
        dict(name="presort_16384_k3_f32", op="presort", n=16384, k=3, dtype="f32", dist="cube", bits=0, dup=0.005),
        # nearest neighbours of fresh query points among clustered points
        dict(name="knn_100003_of_1000000", op="knn", n=1000000, nq=100003, kn=5, k=3, dtype="f32", dist="gmm", bits=0,
             dup=0.0),
        # the neighbours workload: eight nearest of every tuple, and boxes around tuples that hold a few each
        dict(name="knn_all_4194304_k3_i64", op="knn_all", n=1 << 22, kn=8, k=3, dtype="i64", dist="int", bits=40,
             dup=0.0),
        dict(name="region_1048576_of_4194304", op="region", n=1 << 22, nq=1 << 20, k=3, dtype="i64", dist="int",
             bits=40, dup=0.0),
    ]


def _size(rng, lo: float, hi: float) -> int:
    """floor(2^U(lo, hi))."""
    return int(2.0 ** rng.uniform(lo, hi))


def _coordinates(rng, case: dict, sparse: bool = False) -> dict:
    """A type and a distribution; sparse: of coordinates that hardly ever coincide by chance."""
    dist = rng.choice(["int32", "int64", "cube"] if sparse else ["int32", "int64", "gmm", "cube"])
    if dist == "int32":
        case.update(dtype="i32", dist="int", bits=30 if sparse else rng.choice([20, 24, 30]))
    elif dist == "int64":
        case.update(dtype="i64", dist="int", bits=rng.choice([40, 56] if sparse else [20, 40, 56]))
    else:
        case.update(dtype="f32", dist=dist, bits=0)
    case["dup"] = rng.choice([0.0, 0.005, 0.01])
    return case


def draw(rng) -> dict:
    op = rng.choice(["build", "build", "build", "build", "batch", "serve", "select", "presort", "knn", "knn_all",
                     "region"])
    if op == "build":
        n = _size(rng, 6.0, 24.5)
        return _coordinates(rng, dict(op=op, n=n, k=rng.randint(2, 6 if n <= 1 << 22 else 4)))
    if op == "batch":
        lo = rng.randint(5, 8)
        return _coordinates(rng, dict(op=op, count=_size(rng, 4.0, 12.0), lo=lo, hi=lo + rng.randint(3, 8),
                                      k=rng.randint(3, 4)), sparse=True)
    if op == "serve":
        lo = rng.randint(6, 10)
        return dict(op=op, count=_size(rng, 2.0, 5.6), lo=lo, hi=lo + rng.randint(4, 10))
    if op == "select":
        return _coordinates(rng, dict(op=op, n=_size(rng, 8.0, 22.0), k=rng.randint(2, 6)))
    if op == "presort":
        return _coordinates(rng, dict(op=op, n=_size(rng, 5.0, 14.0), k=rng.randint(1, 6)))
    if op == "knn":
        return _coordinates(rng, dict(op=op, n=_size(rng, 8.0, 21.0), nq=_size(rng, 6.0, 17.5),
                                      kn=rng.choice([1, 2, 4, 5, 8, 16, 32]), k=rng.randint(2, 4)))
    if op == "knn_all":
        return _coordinates(rng, dict(op=op, n=_size(rng, 8.0, 20.0), kn=rng.choice([1, 4, 8, 10, 16]),
                                      k=rng.randint(3, 4)), sparse=True)
    return _coordinates(rng, dict(op=op, n=_size(rng, 8.0, 22.0), nq=_size(rng, 6.0, 20.0), k=rng.randint(2, 4)),
                        sparse=True)


def work(case: dict) -> dict:
    """Coordinates and queries read once, results written once; for the
    searches also the distances of the neighbours returned."""
    op = case["op"]
    if op == "serve":
        tuples = case["count"] * _mean_size(case)
        return {"bytes": tuples * (3 * 4 + 4), "flops": 0}
    k, w = case["k"], WORD[case["dtype"]]
    if op == "batch":
        return {"bytes": case["count"] * _mean_size(case) * (k * w + 13), "flops": 0}
    n = case["n"]
    if op in ("build", "select"):
        return {"bytes": n * (k * w + 13), "flops": 0}
    if op == "presort":
        return {"bytes": n * (k * w + 4 * k), "flops": 0}
    points = n * (k * w + 4)
    if op == "region":
        return {"bytes": points + case["nq"] * (2 * k * w + 8 + 3 * 4), "flops": 0}
    nq = n if op == "knn_all" else case["nq"]
    return {"bytes": points + nq * (case["kn"] * 12 + (k * w if op == "knn" else 0)), "flops": nq * case["kn"] * 3 * k}


def _mean_size(case: dict) -> float:
    return (2.0 ** case["hi"] - 2.0 ** case["lo"]) / ((case["hi"] - case["lo"]) * math.log(2.0))


# ------------------------------------------------------------------ inputs
def _generator(seed: int, purpose: int) -> torch.Generator:
    return torch.Generator(device=DEVICE).manual_seed((seed * 1000003 + purpose * 7919) & ((1 << 62) - 1))


def _points(case: dict, n: int, seed: int, purpose: int = 0) -> torch.Tensor:
    """n points of the case's distribution."""
    g, k = _generator(seed, purpose), case["k"]
    if case["dist"] == "int":
        return torch.randint(0, 1 << case["bits"], (n, k), generator=g, device=DEVICE, dtype=TORCH_TYPE[case["dtype"]])
    if case["dist"] == "cube":
        return torch.rand((n, k), generator=g, device=DEVICE, dtype=torch.float32)
    shape = _generator(seed, 99)  # the mixture is the seed's; queries come from the same one
    means = torch.rand((64, k), generator=shape, device=DEVICE) * 2000.0 - 1000.0
    sigma = torch.exp(torch.rand(64, generator=shape, device=DEVICE) * math.log(100.0) + math.log(0.1))
    comp = torch.randint(0, 64, (n,), generator=g, device=DEVICE)
    z = torch.randn((n, k), generator=g, device=DEVICE, dtype=torch.float32)
    return z.mul_(sigma[comp, None]).add_(means[comp])


def _cloud(case: dict, seed: int) -> torch.Tensor:
    """The case's cloud: its points, a share of them overwritten by copies of others."""
    n = case["n"]
    x = _points(case, n, seed)
    copies = int(case["dup"] * n)
    if copies:
        g = _generator(seed, 1)
        order = torch.randperm(n, generator=g, device=DEVICE)
        source = torch.randint(copies, n, (copies,), generator=g, device=DEVICE)
        x[order[:copies]] = x[order[source]]
    return x


def _sizes(case: dict) -> np.ndarray:
    """Log-uniform sizes in [2^lo, 2^hi), one from each of ``count`` equal strata, in random order (the same
    sizes for every seed: the outputs keep their shapes)."""
    count = case["count"]
    r = np.random.default_rng(count)
    u = (np.arange(count) + r.random(count)) / count
    return r.permutation(np.floor(2.0 ** (case["lo"] + (case["hi"] - case["lo"]) * u)).astype(np.int64))


def _packed(case: dict, seed: int):
    """Clouds back to back, their sizes, and the output slots past each cloud's distinct tuples."""
    sizes = _sizes(case)
    copies = (case["dup"] * sizes).astype(np.int64)
    ends = np.cumsum(sizes)
    x = _points(case, int(ends[-1]), seed)
    spare = np.repeat(ends - copies, copies) + np.arange(copies.sum()) - np.repeat(np.cumsum(copies) - copies, copies)
    slots = torch.from_numpy(spare).to(DEVICE)
    if len(spare):
        g = _generator(seed, 1)
        first = torch.from_numpy(np.repeat(ends - sizes, copies)).to(DEVICE)
        distinct = torch.from_numpy(np.repeat(sizes - copies, copies)).to(DEVICE)
        u = torch.rand(len(spare), generator=g, device=DEVICE, dtype=torch.float64)
        x[slots] = x[first + (u * distinct).long()]
        cloud = torch.repeat_interleave(torch.from_numpy(sizes).to(DEVICE)).double()
        x = x[torch.argsort(cloud + torch.rand(len(cloud), generator=g, device=DEVICE, dtype=torch.float64))]
    return x.contiguous(), sizes, slots


# ------------------------------------------------------------------- state
_shared: dict = {}


def _stream() -> torch.cuda.Stream:
    if "stream" not in _shared:
        _shared["stream"] = torch.cuda.Stream()
    return _shared["stream"]


def _context(serving: bool = False):
    """The context a program keeps for all its builds, on its own stream (serving: with a memory budget)."""
    key = "serving" if serving else "plain"
    if key not in _shared:
        _shared[key] = api.kd_create(0, mem_budget_bytes=64 << 30) if serving else api.kd_create(0, stream=_stream())
    return _shared[key]


class _Index:
    """A search index that goes with the state holding it."""

    def __init__(self, ctx, coords):
        tree = api.build_tree(ctx, coords)
        self.ctx, self.m, self.index = ctx, tree["m"], api.kd_index_create(ctx, coords, tree)

    def __del__(self):
        api.kd_index_destroy(self.ctx, self.index)


def prepare(case: dict, seed: int) -> dict:
    op = case["op"]
    state = {"case": case}
    if op == "serve":
        state["ctx"] = _context(serving=True)
        r = np.random.default_rng(case["count"] + 1)
        clouds = []
        for i, n in enumerate(_sizes(case)):
            one = dict(dtype="i32", dist="int", bits=24) if r.random() < 0.5 else dict(dtype="f32", dist="gmm", bits=0)
            clouds.append(_points(dict(one, k=int(r.integers(2, 5))), int(n), seed, 100 + i).cpu().numpy())
        state["clouds"] = clouds
        return state
    state["ctx"] = _context()
    with torch.cuda.stream(_stream()):
        if op == "batch":
            state["coords"], state["sizes"], state["spare"] = _packed(case, seed)
            return state
        coords = state["coords"] = _cloud(case, seed)
        if op == "presort":
            n, k = coords.shape
            state["arrays"] = torch.zeros((k, n), dtype=torch.int32, device=DEVICE)
            state["m"] = torch.zeros(1, dtype=torch.int32, device=DEVICE)
        elif op in ("knn", "knn_all", "region"):
            state["index"] = _Index(state["ctx"], coords)
            if op == "knn":
                state["queries"] = _points(case, case["nq"], seed, 2)
            elif op == "region":
                state["lo"], state["hi"] = _boxes(case, coords, seed)
                state["found"] = torch.zeros(8 * case["nq"] + 4096, dtype=torch.int32, device=DEVICE)
    torch.cuda.synchronize()
    return state


def _boxes(case: dict, coords: torch.Tensor, seed: int):
    """Boxes around tuples; their half widths are uniform up to about (1/n)^(1/k) of the data's extent."""
    g = _generator(seed, 3)
    nq, k = case["nq"], case["k"]
    centre = coords[torch.randint(0, case["n"], (nq,), generator=g, device=DEVICE)]
    reach = (1.0 / case["n"]) ** (1.0 / k) * 1.25
    u = torch.rand((nq, k), generator=g, device=DEVICE, dtype=torch.float64) * reach
    if case["dist"] == "int":
        half = (u * float(1 << case["bits"])).to(coords.dtype)
    else:
        half = (u * (1.0 if case["dist"] == "cube" else 200.0)).to(coords.dtype)
    return (centre - half).contiguous(), (centre + half).contiguous()


def _nodes(tree: dict, case: dict) -> dict:
    """The tree with one entry per tuple that prepare() made distinct: where a few more coincide by chance, the
    entries past the last node (each buffer has room for every tuple) are zeroed."""
    m, count = tree["m"], case["n"] - int(case["dup"] * case["n"])
    if m < count:
        for name in TREE:
            tree[name] = tree[name].as_strided((count,), (1,))
            tree[name][m:].zero_()
    return tree


def _nodes_host(a: np.ndarray, count: int) -> np.ndarray:
    return a if len(a) == count else np.concatenate([a, np.zeros(count - len(a), dtype=a.dtype)])


def run(state: dict):
    case, ctx = state["case"], state["ctx"]
    op = case["op"]
    if op == "serve":
        tickets = [api.kd_submit(ctx, c, children=False) for c in state["clouds"]]
        trees = [api.kd_wait(ctx, t) for t in tickets]
        return {"m": np.array([t["m"] for t in trees]),
                "node_tuple": [_nodes_host(t["node_tuple"], len(c)) for t, c in zip(trees, state["clouds"])]}
    with torch.cuda.stream(_stream()):
        if op == "build":
            return _nodes(api.build_tree(ctx, state["coords"]), case)
        if op == "select":
            return _nodes(api.kd_build_select(ctx, state["coords"]), case)
        if op == "batch":
            trees = api.kd_build_batch_packed(ctx, state["coords"], state["sizes"])
            for name in TREE:  # slots past a cloud's last node hold nothing: marked as such
                trees.arrays[name].index_fill_(0, state["spare"], 0)
            return dict(trees.arrays, m=trees.m, root=trees.root)
        if op == "presort":
            arrays, m = api.kd_presort_noalloc(ctx, state["coords"], state["arrays"], state["m"])
            return {"arrays": arrays, "m": m}
        if op == "knn":
            idx, dist = api.kd_knn(ctx, state["index"].index, state["queries"], case["kn"])
            return {"idx": idx, "dist": dist}
        if op == "knn_all":
            idx, dist = api.kd_knn_all(ctx, state["index"].index, state["index"].m, case["kn"])
            return {"idx": idx, "dist": dist}
        offsets, idx = api.kd_region(ctx, state["index"].index, state["lo"], state["hi"])
        found = state["found"]  # the boxes' tuples in a buffer of the program's own, zero past the last
        found[:len(idx)].copy_(idx)
        found[len(idx):].zero_()
        return {"offsets": offsets, "idx": found}


def exact(case: dict, seed: int):
    """Squared distances of the nearest neighbours by comparing every query
    with every distinct tuple in 64 bits; the other calls return whole numbers."""
    if case["op"] != "knn" or case["n"] * case["nq"] > 1.5e11:
        return None
    points = torch.unique(_cloud(case, seed), dim=0)
    queries = _points(case, case["nq"], seed, 2)
    if case["dist"] != "int":
        points, queries = points.double(), queries.double()
    kn = min(case["kn"], len(points))
    dist = torch.full((case["nq"], case["kn"]), math.inf, dtype=torch.float64, device=DEVICE)
    step = max(1, (1 << 28) // len(points))
    for q in range(0, case["nq"], step):
        d2 = 0.0
        for d in range(case["k"]):
            u = (queries[q:q + step, d, None].long() if case["dist"] == "int" else queries[q:q + step, d, None]) \
                - points[None, :, d]
            d2 = d2 + u.double() ** 2
        dist[q:q + step, :kn] = torch.topk(d2, kn, dim=1, largest=False, sorted=True).values
    return {"idx": None, "dist": dist.cpu()}
