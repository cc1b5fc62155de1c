"""The missing rank planes of the presorted arrays on both sides of the size up
to which they are scattered without grouping, by the tree they lead to against
the one that is built without presorting.  GPU only."""
import pytest

import kdgen

pytestmark = pytest.mark.gpu
FIELDS = ("node_tuple", "left", "right", "dim")


@pytest.mark.parametrize("n,k", [(3428571, 8), (3428572 + 28, 8), (196609, 8), (24000000, 2), (24000001, 2)])
def test_rank_planes(cuda_lib, n, k):
    import torch
    ctx = cuda_lib.kd_create(0)
    try:
        coords = torch.from_numpy(kdgen.cloud_int_uniform(n, k, 24, 5, dup_frac=0.001)).cuda()
        want = cuda_lib.kd_build_select(ctx, coords)
        got = cuda_lib.build_tree(ctx, coords)
        assert got["m"] == want["m"] and got["root"] == want["root"]
        for f in FIELDS:
            assert torch.equal(got[f], want[f]), f
    finally:
        ctx.close()
