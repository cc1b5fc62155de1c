"""Nearest neighbours and region search at the sizes where the box tree and
the offsets' scan can go wrong, against the brute-force search oracle:
whole and partial blocks of 32, one more level, every neighbour count class,
ties beyond the candidate list, coordinates at the ends of their types, and
an index without boxes.  Distances are exact, so every compare is equality.
GPU only."""
import numpy as np
import pytest

import kdgen
import oracle

pytestmark = pytest.mark.gpu


def _index(lib, ctx, coords):
    import torch
    x = torch.from_numpy(coords).cuda()
    tree = lib.build_tree(ctx, x)
    return lib.kd_index_create(ctx, x, tree), tree


def _check(lib, ctx, coords, queries, kn):
    import torch
    ix, tree = _index(lib, ctx, coords)
    gi, gd = lib.kd_knn(ctx, ix, torch.from_numpy(queries).cuda(), kn)
    ri, rd = oracle.knn(coords, queries, kn)
    np.testing.assert_array_equal(gi.cpu().numpy(), ri)
    np.testing.assert_array_equal(gd.cpu().numpy(), rd)
    lib.kd_index_destroy(ctx, ix)


@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 63, 1023, 1024, 1025, 32767, 32769])
@pytest.mark.parametrize("kn", [1, 5, 32])
def test_block_and_level_edges(cuda_lib, n, kn):
    ctx = cuda_lib.kd_create(0)
    try:
        coords = kdgen.cloud_int_uniform(n, 3, 40, 100 + n, np.int64)
        q = kdgen.cloud_int_uniform(70, 3, 40, 7, np.int64)
        _check(cuda_lib, ctx, coords, q, kn)
    finally:
        ctx.close()


@pytest.mark.parametrize("k", [1, 2, 4, 5, 8])
@pytest.mark.parametrize("kind", ["int32 lattice", "float32", "int64 ends"])
def test_dimensions_ties_and_type_ends(cuda_lib, k, kind):
    """int32 lattice: hundreds of tuples at equal distances, more than the
    candidate list holds.  int64 ends: differences up to 2^64 - 1."""
    rng = np.random.default_rng(k)
    if kind == "int32 lattice":
        coords = rng.integers(-4, 5, (3000, k)).astype(np.int32)
        coords[0], coords[1] = 2**31 - 1, -2**31
    elif kind == "float32":
        coords = np.concatenate([rng.normal(0, 1, (1500, k)), rng.normal(3e37, 1e30, (40, k)),
                                 rng.normal(0, 1e-30, (1500, k))]).astype(np.float32)
    else:
        ends = np.array([-2**63, -2**63 + 1, -1, 0, 1, 2**62, 2**63 - 2, 2**63 - 1], dtype=np.int64)
        coords = rng.choice(ends, (2000, k))
    q = coords[rng.integers(0, len(coords), 150)]
    ctx = cuda_lib.kd_create(0)
    try:
        for kn in (3, 16, 32):
            _check(cuda_lib, ctx, coords, q, kn)
    finally:
        ctx.close()


@pytest.mark.parametrize("kn", [2, 8, 9, 31])
def test_several_queries_per_warp(cuda_lib, kn):
    """Enough queries that a warp answers several; each block's last queries
    run past the end, and lattice ties make some candidate sets too wide."""
    import torch
    rng = np.random.default_rng(kn)
    coords = np.concatenate([rng.integers(0, 1 << 20, (20000, 3)), rng.integers(0, 12, (1700, 3))]).astype(np.int32)
    q = coords[rng.integers(0, len(coords), 200003)]
    ctx = cuda_lib.kd_create(0)
    try:
        ix, tree = _index(cuda_lib, ctx, coords)
        gi, gd = (t.cpu().numpy() for t in cuda_lib.kd_knn(ctx, ix, torch.from_numpy(q).cuda(), kn))
        pick = np.concatenate([rng.integers(0, len(q), 300), np.arange(len(q) - 40, len(q))])
        ri, rd = oracle.knn(coords, q[pick], kn)
        np.testing.assert_array_equal(gi[pick], ri)
        np.testing.assert_array_equal(gd[pick], rd)
        cuda_lib.kd_index_destroy(ctx, ix)
    finally:
        ctx.close()


def test_index_without_boxes_and_infinite_coordinates(cuda_lib):
    """A budget that holds the planes but not the boxes: the same answers,
    also where infinite coordinates leave tuples without a distance."""
    import torch
    coords = kdgen.cloud_gmm(5000, 3, 8)
    coords[::97, 1] = np.inf
    coords[5::193, 2] = -np.inf
    q = coords[::3].copy()
    q[1::2] += np.float32(0.5)
    ctx = cuda_lib.kd_create(0)
    small = cuda_lib.kd_create(0, mem_budget_bytes=60160 + 20224 + 256 + 1024)  # planes, tuples, status: no boxes
    try:
        ix, tree = _index(cuda_lib, ctx, coords)
        torch.cuda.synchronize()
        iw = cuda_lib.kd_index_create(small, torch.from_numpy(coords).cuda(), tree)
        qd = torch.from_numpy(q).cuda()
        for kn in (1, 7, 32):
            for a, b in zip(cuda_lib.kd_knn(ctx, ix, qd, kn), cuda_lib.kd_knn(small, iw, qd, kn)):
                np.testing.assert_array_equal(a.cpu().numpy(), b.cpu().numpy())
        cuda_lib.kd_index_destroy(ctx, ix)
        cuda_lib.kd_index_destroy(small, iw)
    finally:
        ctx.close()
        small.close()


@pytest.mark.parametrize("nq", [1, 2047, 2048, 2049, 70001])
def test_region_offsets_over_chunks(cuda_lib, nq):
    """The offsets' scan at its chunk edges, and boxes of every size."""
    import torch
    rng = np.random.default_rng(nq)
    coords = kdgen.cloud_int_uniform(3001, 2, 12, 5, np.int32, dup_frac=0.02)
    centre = rng.integers(0, 1 << 12, (nq, 2)).astype(np.int32)
    half = (2.0 ** rng.uniform(0, 9, (nq, 2))).astype(np.int32)
    lo, hi = centre - half, centre + half
    ctx = cuda_lib.kd_create(0)
    try:
        ix, _ = _index(cuda_lib, ctx, coords)
        offs, idx = (t.cpu().numpy() for t in cuda_lib.kd_region(ctx, ix, torch.from_numpy(lo).cuda(),
                                                                 torch.from_numpy(hi).cuda()))
        pick = np.unique(np.concatenate([rng.integers(0, nq, 200), [0, nq - 1]]))
        ref = oracle.region(coords, lo[pick], hi[pick])
        assert offs[0] == 0 and (np.diff(offs) >= 0).all() and offs[-1] == len(idx)
        for i, r in zip(pick, ref):
            np.testing.assert_array_equal(np.sort(idx[offs[i]:offs[i + 1]]), r)
        cuda_lib.kd_index_destroy(ctx, ix)
    finally:
        ctx.close()


@pytest.mark.parametrize("nq", [(1 << 17) - 1, 1 << 17, (1 << 19) + 3])
def test_region_of_many_boxes(cuda_lib, nq):
    """Boxes taken cell by cell, and boxes kept by the counting walk: none, up
    to 16 and more than 16 tuples, and inverted boxes."""
    import torch
    rng = np.random.default_rng(nq)
    coords = kdgen.cloud_gmm(70000, 3, 17)
    centre = coords[rng.integers(0, len(coords), nq)]
    half = (10.0 ** rng.uniform(-3, 0.7, (nq, 3))).astype(np.float32)
    lo, hi = centre - half, centre + half
    lo[::50], hi[::50] = hi[::50].copy(), lo[::50].copy()
    ctx = cuda_lib.kd_create(0)
    try:
        ix, _ = _index(cuda_lib, ctx, coords)
        L, H = torch.from_numpy(lo).cuda(), torch.from_numpy(hi).cuda()
        offs, idx = (t.cpu().numpy() for t in cuda_lib.kd_region(ctx, ix, L, H))
        pick = np.unique(np.concatenate([rng.integers(0, nq, 300), [0, nq - 1], np.argsort(np.diff(offs))[-20:]]))
        ref = oracle.region(coords, lo[pick], hi[pick])
        assert offs[-1] == len(idx) and max(len(r) for r in ref) > 16
        for i, r in zip(pick, ref):
            np.testing.assert_array_equal(np.sort(idx[offs[i]:offs[i + 1]]), r)
        L[5, 1] = float("nan")
        with pytest.raises(cuda_lib.KdError) as e:
            cuda_lib.kd_region(ctx, ix, L, H)
        assert e.value.code == -6
        cuda_lib.kd_index_destroy(ctx, ix)
    finally:
        ctx.close()
