"""Searches of few neighbours that are answered by one thread each (GPU only):
both sides of the rule's sizes, over one dimension and over planes more and
less filled, against the oracle."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,nq", [(70000, (1 << 16) - 1), (70000, 1 << 16), (900, 1 << 16)])
@pytest.mark.parametrize("k,span,dtype", [(1, 140000, np.int32), (1, 1 << 40, np.int64), (1, 1000, np.float32),
                                          (2, 370, np.int32), (2, 520, np.int64), (2, 540, np.int32), (3, 48, np.int32)])
def test_few_neighbours(cuda_lib, n, nq, k, span, dtype):
    """Planes of 370^2, 520^2 and 540^2 points under 70000 draws: half filled,
    just above and just below a quarter (of the distinct tuples)."""
    import torch
    rng = np.random.default_rng(n + k)
    lo = 0 if dtype == np.float32 else -span // 2
    coords, q = ((rng.integers(0, span, (c, k)) + lo).astype(dtype) for c in (n, nq))
    if dtype == np.float32:
        coords /= 7
        q /= 7
    ctx = cuda_lib.kd_create(0)
    try:
        x = torch.from_numpy(coords).cuda()
        tree = cuda_lib.build_tree(ctx, x)
        ix = cuda_lib.kd_index_create(ctx, x, tree)
        pick = rng.integers(0, nq, 150)
        for kn in (1, 2, 3, 4, 5):
            gi, gd = (t.cpu().numpy()[pick] for t in cuda_lib.kd_knn(ctx, ix, torch.from_numpy(q).cuda(), kn))
            ri, rd = oracle.knn(coords, q[pick], kn)
            np.testing.assert_array_equal(gi, ri)
            np.testing.assert_array_equal(gd, rd)
        node = tree["node_tuple"].cpu().numpy()
        gi = cuda_lib.kd_knn_all(ctx, ix, tree["m"], 2)[0].cpu().numpy()
        at = rng.integers(0, tree["m"], 100)
        ri, _ = oracle.knn(coords, coords[node[at]], 3)
        for a, row in zip(at, ri):
            np.testing.assert_array_equal(gi[a], [u for u in row if u != node[a]][:2])
        cuda_lib.kd_index_destroy(ctx, ix)
    finally:
        ctx.close()
