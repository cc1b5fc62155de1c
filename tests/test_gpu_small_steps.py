"""Builds whose sort passes and level steps are one launch each, against the
oracle: the edges of their tiles (1024 and 2048 positions), several segments
per tile, every dimension count, batches whose clouds start anywhere in a
tile, and the sizes at which the rules change.  GPU only."""
import numpy as np
import pytest

import kdgen
import oracle

pytestmark = pytest.mark.gpu
FIELDS = ("node_tuple", "left", "right", "dim")


def _same(got, ref):
    assert got["m"] == ref["m"]
    for f in FIELDS:
        np.testing.assert_array_equal(got[f].cpu().numpy(), ref[f])


def _build(lib, coords, **cfg):
    import torch
    ctx = lib.kd_create(0, **cfg)
    try:
        return lib.build_tree(ctx, torch.from_numpy(coords).cuda())
    finally:
        ctx.close()


@pytest.mark.parametrize("n", [1025, 2049, 4097, 20480, 196609, 198656, 198657, 204799])
@pytest.mark.parametrize("k", [2, 3, 4, 5, 8])
def test_tile_edges(cuda_lib, n, k):
    coords = kdgen.cloud_int_uniform(n, k, 9, n + k, np.int64, dup_frac=0.01) if k % 2 else kdgen.cloud_gmm(n, k, n)
    _same(_build(cuda_lib, coords), oracle.build_tree(coords))


@pytest.mark.parametrize("schedule", [1, 2])
def test_schedules(cuda_lib, schedule):
    coords = kdgen.cloud_int_uniform(30001, 4, 12, 3, np.int32, dup_frac=0.01)
    _same(_build(cuda_lib, coords, schedule=schedule), oracle.build_tree(coords))


def test_batch_of_uneven_clouds(cuda_lib):
    import torch
    clouds = [kdgen.cloud_unit_cube(n, 3, n, 0.01) for n in (5000, 1, 1027, 33000, 2, 2049, 70001, 1024, 3)]
    ctx = cuda_lib.kd_create(0)
    try:
        trees = cuda_lib.kd_build_batch(ctx, [torch.from_numpy(c).cuda() for c in clouds])
        for got, c in zip(trees, clouds):
            _same(got, oracle.build_tree(c))
    finally:
        ctx.close()


@pytest.mark.parametrize("n", [3 << 19, (3 << 19) + 1, 1 << 21, (1 << 21) + 1])
def test_sizes_where_the_rules_change(cuda_lib, n):
    coords = kdgen.cloud_unit_cube(n, 2, n)
    ref = oracle.build_tree(coords)
    got = _build(cuda_lib, coords)
    _same(got, ref)
