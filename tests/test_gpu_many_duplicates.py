"""Clouds and batches of mostly duplicate tuples above the block sorts' sizes
(GPU only): runs of equal tuples within a row of 32 positions, across rows and
tiles, whole rows of duplicates, against the oracle."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu
FIELDS = ("node_tuple", "left", "right", "dim")


def _same(got, ref):
    assert got["m"] == ref["m"]
    for f in FIELDS:
        np.testing.assert_array_equal(got[f].cpu().numpy(), ref[f])


def _copies(counts, k, dtype, seed):
    """Distinct random tuples, the i-th `counts[i]` times, shuffled."""
    rng = np.random.default_rng(seed)
    base = rng.integers(0, 1 << 20, (len(counts), k))
    base[:, 0] = np.arange(len(counts)) * 3 - 1000
    return np.ascontiguousarray(rng.permutation(np.repeat(base, counts, axis=0)).astype(dtype))


COUNTS = {"pairs": [2] * 150000, "rows": [1, 31, 32, 33, 64, 2, 95] * 900, "tiles": [5000, 1, 2047, 2048, 2049] * 20,
          "one": [200001]}


@pytest.mark.parametrize("name", list(COUNTS))
@pytest.mark.parametrize("k,dtype", [(1, np.int32), (2, np.int64), (3, np.float32), (6, np.int64)])
def test_cloud(cuda_lib, name, k, dtype):
    import torch
    coords = _copies(COUNTS[name], k, dtype, len(name))
    ctx = cuda_lib.kd_create(0)
    try:
        _same(cuda_lib.build_tree(ctx, torch.from_numpy(coords).cuda()), oracle.build_tree(coords))
    finally:
        ctx.close()


def test_batch(cuda_lib):
    """Equal tuples in neighbouring clouds are kept apart."""
    import torch
    clouds = [_copies(c, 3, np.int32, 7) for c in ([40] * 30, [40] * 30, [1000], [1000], [1], [3, 3, 3], COUNTS["rows"])]
    ctx = cuda_lib.kd_create(0)
    try:
        for c, got in zip(clouds, cuda_lib.kd_build_batch(ctx, [torch.from_numpy(c).cuda() for c in clouds])):
            _same(got, oracle.build_tree(c))
    finally:
        ctx.close()
