"""More queries than one grid of the search without boxes holds (GPU only):
every row is written."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _r256(n):
    return (n + 255) // 256 * 256


def test_walk_of_more_queries_than_a_grid_holds(cuda_lib):
    """An index without boxes and 2^27 + 1000 queries (a grid of 2^20 blocks
    answers 2^27 at a time): every row is written, the last ones too."""
    import torch
    coords = np.arange(0, 3000, 3, dtype=np.int32)[:, None]
    n, nq = len(coords), (1 << 27) + 1000
    ctx = cuda_lib.kd_create(0)
    small = cuda_lib.kd_create(0, mem_budget_bytes=_r256(4 * n) * 2 + 256)  # planes, tuples, status: no boxes
    try:
        x = torch.from_numpy(coords).cuda()
        tree = cuda_lib.build_tree(ctx, x)
        torch.cuda.synchronize()
        ix = cuda_lib.kd_index_create(small, x, tree)
        which = torch.arange(nq, device="cuda", dtype=torch.int32) % n
        idx, _ = cuda_lib.kd_knn(small, ix, (which * 3)[:, None], 1, with_dist=False)
        assert torch.equal(idx[:, 0], which)
        cuda_lib.kd_index_destroy(small, ix)
    finally:
        ctx.close()
        small.close()
