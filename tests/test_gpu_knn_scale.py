"""Neighbours among coordinates whose squared differences leave the range of
32-bit floats (GPU only): the oracle's answers, and no walk of the whole
index."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


def _index(lib, ctx, coords):
    import torch
    x = torch.from_numpy(coords).cuda()
    tree = lib.build_tree(ctx, x)
    return lib.kd_index_create(ctx, x, tree), tree


def _scaled(scale):
    return (np.random.default_rng(3).normal(0, 1, (1 << 17, 3)) * scale).astype(np.float32)


@pytest.mark.parametrize("scale", [1e-42, 1e-30, 1e-20, 1e-18, 1e18, 1e20, 1e30, 1e37])
def test_neighbours_of_clouds_of_any_scale(cuda_lib, scale):
    import torch
    coords = _scaled(scale)
    ctx = cuda_lib.kd_create(0)
    try:
        ix, tree = _index(cuda_lib, ctx, coords)
        q = np.concatenate([coords[::20000], coords[:5] * np.float32(2), np.zeros((1, 3), np.float32)])
        gi, gd = cuda_lib.kd_knn(ctx, ix, torch.from_numpy(q).cuda(), 9)
        ri, rd = oracle.knn(coords, q, 9)
        np.testing.assert_array_equal(gi.cpu().numpy(), ri)
        np.testing.assert_array_equal(gd.cpu().numpy(), rd)
        hi, hd = cuda_lib.kd_knn(ctx, ix, q, 9)  # host in and out
        np.testing.assert_array_equal(hi, ri)
        np.testing.assert_array_equal(hd, rd)
        cuda_lib.kd_index_destroy(ctx, ix)
    finally:
        ctx.close()


@pytest.mark.parametrize("scale", [1e-30, 1e-20, 1e22])
def test_scale_does_not_make_the_search_visit_everything(cuda_lib, scale):
    """The walk in 64-bit distances visits the boxes that the walk in 32-bit
    ones visits at the scale of 1; its FP64 instructions run at 1/64 of the
    FP32 rate and are less than half of the walk's, so 32 times the time
    bounds it.  A walk of all 4096 blocks a query takes over 100 times."""
    import torch
    ctx = cuda_lib.kd_create(0)
    try:
        ms = []
        for s in (1.0, scale):
            ix, tree = _index(cuda_lib, ctx, _scaled(s))
            best = 1e9
            for _ in range(3):
                a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                torch.cuda.synchronize()
                a.record()
                cuda_lib.kd_knn_all(ctx, ix, tree["m"], 8)
                b.record()
                b.synchronize()
                best = min(best, a.elapsed_time(b))
            ms.append(best)
            cuda_lib.kd_index_destroy(ctx, ix)
        assert ms[1] <= 32 * ms[0], ms
    finally:
        ctx.close()


def test_reverse_neighbours_of_a_lattice(cuda_lib):
    """More ties than the candidate list holds, through the reverse search."""
    g = np.stack(np.meshgrid(*[np.arange(13)] * 3, indexing="ij"), -1).reshape(-1, 3).astype(np.int32)
    ctx = cuda_lib.kd_create(0)
    try:
        ix, tree = _index(cuda_lib, ctx, g)
        node = tree["node_tuple"].cpu().numpy()
        offs, rev = (t.cpu().numpy() for t in cuda_lib.kd_reverse_knn(ctx, ix, len(g), 30))
        ri, _ = oracle.knn(g, g, 31)
        lists = [[] for _ in range(len(g))]
        for t, row in enumerate(ri):
            for u in [u for u in row if u != t][:30]:
                lists[u].append(t)
        for a, t in enumerate(node):
            np.testing.assert_array_equal(np.sort(rev[offs[a]:offs[a + 1]]), np.sort(lists[t]))
        cuda_lib.kd_index_destroy(ctx, ix)
    finally:
        ctx.close()
