"""Chains by words with values that a share of the tuples too small for the
sample has in common (GPU only): runs longer than the compares take, which
the sort has left in order already, are not sorted once more by whole keys."""
import numpy as np
import pytest

import kdgen
import oracle

pytestmark = pytest.mark.gpu
FIELDS = ("node_tuple", "left", "right", "dim")
N = (1 << 20) + 77


@pytest.mark.parametrize("count", [65, 400, 5000])
def test_a_value_held_by_many_costs_no_second_sort(cuda_lib, count):
    import torch
    rng = np.random.default_rng(count)
    plain = kdgen.cloud_int_uniform(N, 3, 40, 21, np.int64)
    heavy = plain.copy()
    heavy[rng.choice(N, count, replace=False), 1] = 7 << 36
    heavy[rng.choice(N, count, replace=False), 2] = 0
    launches = []
    ctx = cuda_lib.kd_create(0)
    try:
        for coords in (plain, heavy):
            x = torch.from_numpy(coords).cuda()
            before = cuda_lib.kd_launch_count(ctx)
            got = cuda_lib.build_tree(ctx, x)
            launches.append(cuda_lib.kd_launch_count(ctx) - before)
        ref = oracle.build_tree(heavy)
        assert got["m"] == ref["m"]
        for f in FIELDS:
            np.testing.assert_array_equal(got[f].cpu().numpy(), ref[f])
    finally:
        ctx.close()
    assert launches[1] == launches[0], launches
