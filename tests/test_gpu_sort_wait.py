"""The bounded waits of the sort passes made to run out (GPU only, debug bit
8): in the passes of one launch and in the scan of the larger ones, also for a
cloud that is otherwise presorted in blocks, which has no such wait."""
import numpy as np
import pytest

import kdgen
import oracle

pytestmark = pytest.mark.gpu
FIELDS = ("node_tuple", "left", "right", "dim")
KD_ETIMEOUT = -4


def _same(got, ref):
    assert got["m"] == ref["m"]
    for f in FIELDS:
        np.testing.assert_array_equal(got[f].cpu().numpy(), ref[f])


def _dev(x):
    import torch
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


@pytest.mark.parametrize("n", [5000, 300000, (3 << 19) + 5])
def test_withheld_flag_of_a_sort_pass(cuda_lib, n):
    """5000 and 300000: passes of one launch (tiles of 2048), a cloud of the
    first size otherwise presorted in blocks; above 3 * 2^19: the scan over
    chunks of 64 tiles."""
    ctx = cuda_lib.kd_create(0, debug=8)
    try:
        coords = kdgen.cloud_gmm(n, 3, 12)
        x = _dev(coords)
        with pytest.raises(cuda_lib.KdError) as e:
            cuda_lib.build_tree(ctx, x)
        assert e.value.code == KD_ETIMEOUT
        _same(cuda_lib.build_tree(ctx, x), oracle.build_tree(coords))
    finally:
        ctx.close()
