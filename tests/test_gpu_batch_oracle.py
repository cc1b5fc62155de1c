"""Large batches whose cloud ids come from the clouds' starts, and from a
gather where the clouds are too many for the table (GPU only): clouds from all
over the batch against the oracle."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu
FIELDS = ("node_tuple", "left", "right", "dim")


@pytest.mark.parametrize("sizes", [[2100] * 4000, [1025] * 8192, [1025] * 8193], ids=["starts", "most", "gather"])
def test_clouds_of_a_large_batch(cuda_lib, sizes):
    import torch
    rng = np.random.default_rng(len(sizes))
    sizes = np.maximum(np.array(sizes) + rng.integers(-20, 20, len(sizes)), 1)
    sizes[[0, len(sizes) // 2, -1]] += 30000
    ends = np.cumsum(sizes)
    assert ends[-1] >= 1 << 23
    coords = rng.integers(0, 1 << 9, (int(ends[-1]), 3)).astype(np.int32)
    ctx = cuda_lib.kd_create(0)
    try:
        got = cuda_lib.kd_build_batch_packed(ctx, torch.from_numpy(coords).cuda(), sizes)
        last = len(sizes) - 1
        for j in np.unique(np.concatenate([[0, 1, last // 2, last // 2 + 1, last - 1, last], rng.integers(0, last, 150)])):
            ref, tree = oracle.build_tree(coords[ends[j] - sizes[j]:ends[j]]), got[int(j)]
            assert tree["m"] == ref["m"]
            for f in FIELDS:
                np.testing.assert_array_equal(tree[f].cpu().numpy(), ref[f])
    finally:
        ctx.close()
