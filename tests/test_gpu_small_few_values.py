"""Clouds near the largest that are presorted in blocks, of few values per
coordinate (GPU only): left to the digit passes where the merge of the chunks
would compare coordinates at most of its steps, with the same arrays and trees
as the oracle, from device and host memory, and without the time that took."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu
FIELDS = ("node_tuple", "left", "right", "dim")


def _host(x):
    return x.cpu().numpy() if hasattr(x, "cpu") else np.asarray(x)


def _values(n, k, values, dtype, seed, few=None):
    rng = np.random.default_rng(seed)
    c = rng.integers(0, 1 << 22, (n, k))
    few = range(k) if few is None else few
    for d in few:
        c[:, d] = rng.integers(0, values, n)
    return np.ascontiguousarray(c.astype(dtype))


# (k, n, values, coordinates of few values): both sides of 350000 coordinates,
# of 150000 tuples with half of the coordinates and of 1100000 coordinates with
# short runs
CASES = [(2, 196608, 3, None), (3, 116666, 2, None), (3, 116667, 2, None), (4, 100000, 64, [0]), (4, 100000, 64, [0, 2, 3]),
         (4, 150000, 64, [0, 2]), (4, 150001, 64, [0, 2]), (5, 180000, 5, [1, 2]), (5, 180000, 5, [1, 2, 4]),
         (6, 65536, 1, None), (6, 183333, 1000, None), (6, 183334, 1000, None), (8, 196608, 2, None)]


@pytest.mark.parametrize("k,n,values,few", CASES)
@pytest.mark.parametrize("dtype", [np.int32, np.int64, np.float32], ids=["i32", "i64", "f32"])
def test_equals_the_oracle(cuda_lib, k, n, values, few, dtype):
    import torch
    coords = _values(n, k, values, dtype, n + k, few)
    ref = oracle.build_tree(coords)
    ctx = cuda_lib.kd_create(0)
    try:
        h = cuda_lib.kd_presort(ctx, torch.from_numpy(coords).cuda())
        np.testing.assert_array_equal(cuda_lib.kd_handle_arrays(ctx, h), oracle.presort(coords))
        for got in (cuda_lib.kd_build(ctx, h), cuda_lib.build_tree(ctx, coords)):
            assert got["m"] == ref["m"]
            for f in FIELDS:
                np.testing.assert_array_equal(_host(got[f]), ref[f])
    finally:
        ctx.close()


def test_nan_among_few_values(cuda_lib):
    import torch
    coords = _values(150000, 4, 3, np.float32, 1)
    coords[149999, 3] = np.nan
    ctx = cuda_lib.kd_create(0)
    try:
        with pytest.raises(cuda_lib.KdError) as e:
            cuda_lib.kd_presort(ctx, torch.from_numpy(coords).cuda())
        assert e.value.code == -6
    finally:
        ctx.close()


def _ms(lib, ctx, x):
    import torch
    best = 1e9
    for _ in range(6):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        a.record()
        lib.build_tree(ctx, x)
        b.record()
        b.synchronize()
        best = min(best, a.elapsed_time(b))
    return best


@pytest.mark.parametrize("values", [1, 2, 16])
def test_few_values_take_no_multiple_of_the_time(cuda_lib, values):
    """Eight int64 dimensions: the digit passes skip constant bytes, so that few
    values sort in less time than many by them; twice the time of many values
    in blocks leaves room for the block sorts before them."""
    import torch
    ctx = cuda_lib.kd_create(0)
    try:
        many, few = (torch.from_numpy(_values(196000, 8, v, np.int64, 5)).cuda() for v in (1 << 20, values))
        a, b = _ms(cuda_lib, ctx, many), _ms(cuda_lib, ctx, few)
        assert b <= 2 * a, (a, b)
    finally:
        ctx.close()
