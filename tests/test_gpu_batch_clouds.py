"""Cloud ids of a batch's tuples looked up from the clouds' starts (large
batches) and gathered (small ones, and batches of too many clouds for the
table): the same trees as from small batches.  GPU only."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes", [
    [1, 0, 2] * 2000 + [4300, 1, 0, 4090] * 500 + [4200000],   # 8001 clouds, many to a cell of the table
    [8192 - i % 3 for i in range(1025)],                       # just past the size the table serves from
    [1025] * 8193 + [3],                                       # more clouds than the table holds
])
def test_large_batch_equals_small_ones(cuda_lib, sizes):
    import torch
    sizes = np.array(sizes)
    ctx = cuda_lib.kd_create(0)
    try:
        gen = torch.Generator(device="cuda").manual_seed(3)
        coords = torch.randint(0, 1 << 10, (int(sizes.sum()), 2), dtype=torch.int32, device="cuda", generator=gen)
        got = cuda_lib.kd_build_batch_packed(ctx, coords, sizes)
        part = np.minimum(np.cumsum(sizes) // 5000000, 8)  # batches below 2^23 tuples
        for p in np.unique(part):
            at = np.flatnonzero(part == p)
            lo = int(sizes[:at[0]].sum())
            want = cuda_lib.kd_build_batch_packed(ctx, coords[lo:lo + int(sizes[at].sum())].contiguous(), sizes[at])
            for j in np.unique(np.concatenate([at[:3], at[-3:], at[::97]])):
                a, b = got[int(j)], want[int(j - at[0])]
                assert a["m"] == b["m"]
                for f in ("node_tuple", "left", "right", "dim"):
                    assert torch.equal(a[f], b[f]), (j, f)
    finally:
        ctx.close()
