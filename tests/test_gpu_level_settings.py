"""The level step's settings on builds of every size (GPU only): a level tile
that the configuration fixes is the one that runs, under every schedule, and
the steps of one launch and of four give the oracle's tree."""
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


def _dev(x):
    import torch
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


def _launches(lib, x, **cfg):
    ctx = lib.kd_create(0, **cfg)
    try:
        h = lib.kd_presort(ctx, x)
        before = lib.kd_launch_count(ctx)
        tree = lib.kd_build(ctx, h)
        return lib.kd_launch_count(ctx) - before, tree
    finally:
        ctx.close()


@pytest.mark.parametrize("k", [2, 3, 4, 6])
@pytest.mark.parametrize("schedule", [0, 1, 2])
def test_a_fixed_tile_runs_on_small_builds(cuda_lib, k, schedule):
    """The level steps of a fixed tile are four launches each, those of a
    small build without one are one."""
    coords = kdgen.cloud_int_uniform(60001, k, 24, 70 + k, np.int64, dup_frac=0.01)
    ref, x = oracle.build_tree(coords), _dev(coords)
    one, tree = _launches(cuda_lib, x, schedule=schedule)
    _same(tree, ref)
    for tile in (1024, 2048):
        four, tree = _launches(cuda_lib, x, schedule=schedule, level_tile=tile)
        _same(tree, ref)
        # (top nodes and finisher beside the steps; same steps unless the tile changes their number)
        assert four - 2 == 4 * (one - 2), (tile, one, four)


def test_a_fixed_tile_runs_on_batches(cuda_lib):
    clouds = kdgen.batch_clouds(count=30, seed=9, lo_log2=6.0, hi_log2=14.0)
    for tile in (1024, 2048):
        ctx = cuda_lib.kd_create(0, level_tile=tile)
        try:
            for c, got in zip(clouds, cuda_lib.kd_build_batch(ctx, [_dev(c) for c in clouds])):
                _same(got, oracle.build_tree(c))
        finally:
            ctx.close()


def test_autotune_on_a_small_size_keeps_builds_of_one_launch_a_step(cuda_lib):
    """A tuned pair does not take the one-launch steps from a small build."""
    coords = kdgen.cloud_gmm(100003, 3, 5)
    x, ref = _dev(coords), oracle.build_tree(coords)
    ctx = cuda_lib.kd_create(0)
    try:
        h = cuda_lib.kd_presort(ctx, x)
        cuda_lib.kd_autotune(ctx, 3, "float32", 100003, reps=2)
        before = cuda_lib.kd_launch_count(ctx)
        tree = cuda_lib.kd_build(ctx, h)
        tuned = cuda_lib.kd_launch_count(ctx) - before
        pair = cuda_lib.kd_tuning_get(ctx, 3, "float32", 100003)
    finally:
        ctx.close()
    _same(tree, ref)
    plain, _ = _launches(cuda_lib, x, switch_threshold=pair["switch_threshold"])
    assert tuned == plain
