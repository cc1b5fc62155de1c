"""The presort of small clouds (one block per super key and chunk) through
every entry point that uses it, against the oracle: the edges of its block
and chunk sizes, runs of equal coordinates below and above the length ordered
by compares, every type and dimension count, and outputs that overlap the
coordinates.  GPU only."""
import numpy as np
import pytest

import kdgen
import oracle

pytestmark = pytest.mark.gpu
FIELDS = ("node_tuple", "left", "right", "dim")
SIZES = [1, 2, 31, 255, 256, 257, 1023, 1024, 1025, 2048, 2049, 4096, 4097, 8192, 8193, 16383, 16384, 16385]


def _host(x):
    return x.cpu().numpy() if hasattr(x, "cpu") else np.asarray(x)


def _same(got, ref):
    assert got["m"] == ref["m"]
    for f in FIELDS:
        np.testing.assert_array_equal(_host(got[f]), ref[f])


def _check(lib, coords):
    import torch
    ctx = lib.kd_create(0)
    try:
        x = torch.from_numpy(coords).cuda()
        ref = oracle.build_tree(coords)
        h = lib.kd_presort(ctx, x)
        np.testing.assert_array_equal(lib.kd_handle_arrays(ctx, h), oracle.presort(coords))
        _same(lib.kd_build(ctx, h), ref)
        _same(lib.build_tree(ctx, coords), ref)  # host in and out
        _same(lib.kd_build_select(ctx, x), ref)
        if len(coords) <= 16384:
            arrays, m = lib.kd_presort_noalloc(ctx, x)
            torch.cuda.synchronize()
            assert int(m.item()) == ref["m"]
            np.testing.assert_array_equal(arrays.cpu().numpy()[:, :ref["m"]], oracle.presort(coords))
    finally:
        ctx.close()


@pytest.mark.parametrize("n", SIZES)
def test_block_size_edges(cuda_lib, n):
    _check(cuda_lib, kdgen.cloud_int_uniform(n, 3, 40, n, np.int64, dup_frac=0.01))
    _check(cuda_lib, kdgen.cloud_gmm(n, 2, n + 1))


@pytest.mark.parametrize("n", [65536, 65537, 81921, 196608, 196609])
def test_chunk_size_edges(cuda_lib, n):
    _check(cuda_lib, kdgen.cloud_int_uniform(n, 3, 34, n, np.int64, dup_frac=0.01))
    _check(cuda_lib, kdgen.cloud_gmm(n, 2, n + 1))


@pytest.mark.parametrize("k", [1, 2, 4, 5, 8])
@pytest.mark.parametrize("values", [1, 2, 40, 300, 3000])
def test_runs_of_equal_coordinates(cuda_lib, k, values):
    """5000 tuples over few values per coordinate: runs of 5000, 2500, about
    125 (the whole super key is sorted), 17 and 2 (ordered by compares), with
    many duplicates for small k, and equal tuples in different chunks; each
    type."""
    rng = np.random.default_rng(k * 10000 + values)
    coords = rng.integers(0, values, (5000, k))
    _check(cuda_lib, (coords - values // 2).astype(np.int32))
    _check(cuda_lib, (coords * ((1 << 33) + 1) - (1 << 40)).astype(np.int64))  # both key words differ
    f = ((coords - values // 2) / 8).astype(np.float32)
    f[f == 0] *= rng.choice([-1.0, 1.0], int((f == 0).sum())).astype(np.float32)  # -0.0 equals +0.0
    _check(cuda_lib, f)


def test_runs_at_the_compare_limit(cuda_lib):
    rng = np.random.default_rng(1)
    for run in (31, 32, 33):
        x = np.repeat(np.arange(3000 // run, dtype=np.int32), run)
        _check(cuda_lib, np.stack([rng.permutation(x), rng.integers(0, 4, len(x)), rng.permutation(x)], 1).astype(np.int32))


def test_noalloc_outputs_over_the_coordinates(cuda_lib):
    import torch
    coords = kdgen.cloud_unit_cube(16384, 3, 9, 0.01)
    ref = oracle.presort(coords)
    ctx = cuda_lib.kd_create(0)
    try:
        x = torch.from_numpy(coords).cuda()
        rows = x.view(torch.int32).view(3, 16384)  # the coordinates' own memory
        arrays, m = cuda_lib.kd_presort_noalloc(ctx, x, rows)
        torch.cuda.synchronize()
        assert int(m.item()) == ref.shape[1]
        np.testing.assert_array_equal(arrays.cpu().numpy()[:, :ref.shape[1]], ref)
    finally:
        ctx.close()


def test_nan_and_sizes_of_a_budget(cuda_lib):
    import torch
    bad = kdgen.cloud_gmm(9000, 3, 5)
    bad[8999, 2] = np.nan
    ctx = cuda_lib.kd_create(0)
    try:
        for call in (cuda_lib.kd_presort, cuda_lib.kd_build_select):
            with pytest.raises(cuda_lib.KdError) as e:
                call(ctx, torch.from_numpy(bad).cuda())
            assert e.value.code == -6
        ok = kdgen.cloud_gmm(9000, 3, 6)
        _same(cuda_lib.build_tree(ctx, torch.from_numpy(ok).cuda()), oracle.build_tree(ok))
    finally:
        ctx.close()
