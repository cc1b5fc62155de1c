"""Region search under a budget that holds what it needs and nothing beside it
(GPU only)."""
import numpy as np
import pytest

import kdgen

pytestmark = pytest.mark.gpu


def _r256(n):
    return (n + 255) // 256 * 256


def _index(lib, ctx, coords):
    import torch
    x = torch.from_numpy(coords).cuda()
    tree = lib.build_tree(ctx, x)
    return lib.kd_index_create(ctx, x, tree), tree


def test_region_fits_a_budget_without_room_for_its_order(cuda_lib):
    """Host boxes under a budget that holds the index, the boxes, the offsets
    and the indices found, but not the boxes' order and kept tuples beside
    them."""
    import torch
    rng = np.random.default_rng(2)
    nq = (1 << 19) + 3
    coords = kdgen.cloud_int_uniform(70000, 2, 15, 5, np.int32)
    lo = rng.integers(0, 1 << 15, (nq, 2)).astype(np.int32)
    hi = lo + rng.integers(100, 1100, (nq, 2)).astype(np.int32)
    ctx = cuda_lib.kd_create(0)
    try:
        ix, tree = _index(cuda_lib, ctx, coords)
        offs, idx = cuda_lib.kd_region(ctx, ix, lo, hi)
        total, m = len(idx), tree["m"]
        assert total > 20 * nq
        boxes = sum(-(-(-(-m // 32 ** (lev + 1))) // 32) * 4 * 32 * 4 for lev in range(3))
        need = (_r256(8 * m) + _r256(4 * m) + _r256(boxes)
                + 2 * _r256(8 * nq) + _r256((nq + 2047) // 2048 * 8 + 4 * nq) + _r256(8 * (nq + 1)) + 256
                + _r256(4 * total))
        tight = cuda_lib.kd_create(0, mem_budget_bytes=need)
        try:
            x = torch.from_numpy(coords).cuda()
            it = cuda_lib.kd_index_create(tight, x, tree)
            offs2, idx2 = cuda_lib.kd_region(tight, it, lo, hi)
            np.testing.assert_array_equal(offs2, offs)
            for i in rng.integers(0, nq, 200):
                np.testing.assert_array_equal(np.sort(idx2[offs2[i]:offs2[i + 1]]), np.sort(idx[offs[i]:offs[i + 1]]))
            cuda_lib.kd_index_destroy(tight, it)
        finally:
            tight.close()
        cuda_lib.kd_index_destroy(ctx, ix)
    finally:
        ctx.close()
