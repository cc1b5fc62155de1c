"""The bounded waits of the level steps made to run out (GPU only): in the steps
of one launch and in the scan of the steps of four."""
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


@pytest.mark.parametrize("n,k", [(20000, 3), (300000, 2), (300000, 6)])
def test_withheld_status_of_a_level_step(cuda_lib, n, k):
    """debug bit 16: the first tile of the next build's first one-launch level
    step withholds its counts.  The waits that run out store nothing; the call
    reports them and the context then builds the oracle's tree."""
    ctx = cuda_lib.kd_create(0, debug=16)
    try:
        coords = kdgen.cloud_gmm(n, k, 13)
        x = _dev(coords)
        h = cuda_lib.kd_presort(ctx, x)
        with pytest.raises(cuda_lib.KdError) as e:
            cuda_lib.kd_build(ctx, h)
        assert e.value.code == KD_ETIMEOUT
        assert "wait" in str(e.value)
        _same(cuda_lib.build_tree(ctx, x), oracle.build_tree(coords))
    finally:
        ctx.close()


def test_withheld_status_of_a_scan(cuda_lib):
    """Steps of four launches: the scan has a second chunk, whose wait runs
    out, above 4096 tiles of 1024 positions.  (The same context's next build is
    compared with another's.)"""
    n = (1 << 22) + 5000
    x = _dev(kdgen.cloud_int_uniform(n, 2, 40, 3, np.int64))
    plain = cuda_lib.kd_create(0)
    ctx = cuda_lib.kd_create(0, debug=16, level_tile=1024)
    try:
        h = cuda_lib.kd_presort(ctx, x)
        with pytest.raises(cuda_lib.KdError) as e:
            cuda_lib.kd_build(ctx, h)
        assert e.value.code == KD_ETIMEOUT
        ref = {f: v.cpu().numpy() if hasattr(v, "cpu") else v for f, v in cuda_lib.build_tree(plain, x).items()}
        _same(cuda_lib.build_tree(ctx, x), ref)
    finally:
        ctx.close()
        plain.close()
