"""The chain's sorts by 32-bit words, against the oracle: words that hold the
whole difference (exact), words of the three leading bytes whose runs are put
right afterwards, runs too long that the sample does not show (sorted once
more by whole keys), inputs whose sample keeps whole keys, and 32-bit keys of
many dimensions.  GPU only."""
import numpy as np
import pytest

import kdgen
import oracle

pytestmark = pytest.mark.gpu
FIELDS = ("node_tuple", "left", "right", "dim")
N = (1 << 20) + 77


def _check(lib, coords):
    import torch
    ctx = lib.kd_create(0)
    try:
        ref = oracle.build_tree(coords)
        got = lib.build_tree(ctx, torch.from_numpy(coords).cuda())
        assert got["m"] == ref["m"]
        for f in FIELDS:
            np.testing.assert_array_equal(got[f].cpu().numpy(), ref[f])
    finally:
        ctx.close()


@pytest.mark.parametrize("kind", ["exact", "leading bytes", "hidden long run", "outliers", "constant"])
def test_int64_words(cuda_lib, kind):
    coords = kdgen.cloud_int_uniform(N, 3, 30 if kind == "exact" else 52, 11, np.int64, dup_frac=0.01)
    rng = np.random.default_rng(4)
    if kind == "leading bytes":
        coords[:, 1] >>= 9  # 43 bits: 2^19 values of the leading three bytes, so runs of about two
        coords[5000:5040, 2] = coords[77, 2]  # a run of equal x_2
    elif kind == "hidden long run":
        at = rng.integers(0, N, 300)
        coords[at, 2] = (123 << 44) + rng.integers(0, 1 << 20, 300)
    elif kind == "outliers":
        coords &= (1 << 20) - 1
        coords[rng.integers(0, N, 3)] = 1 << 60
    elif kind == "constant":
        coords[:, 2] = -5
    _check(cuda_lib, coords)


def test_many_dimensions_of_32_bits(cuda_lib):
    _check(cuda_lib, kdgen.cloud_int_uniform((1 << 21) + 5, 5, 20, 3, np.int32))


def test_five_dimensions_of_64_bits(cuda_lib):
    _check(cuda_lib, kdgen.cloud_int_uniform(400001, 5, 40, 9, np.int64))
