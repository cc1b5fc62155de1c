"""Array 0's runs of equal x_0 in single clouds above the sizes that are
presorted in blocks (GPU only): runs of every length class ordered on chip,
runs that begin, end and cross at tile edges, and the lengths above which the
whole key is sorted, against the oracle."""
import numpy as np
import pytest

from test_gpu_ties import EDGES, check, runs_cloud

pytestmark = pytest.mark.gpu

# mean cost below 128 compares per tuple, so that the runs are ordered on
# chip: 900 x (33^2 + 34^2 + 100^2) + 600^2 + 2047^2 + 2048^2 over 221595
MIXED = [1, 2, 3, 5, 31, 32, 33, 34, 100] * 900 + [600, 2047, 2048]


@pytest.fixture(scope="module")
def ctx(cuda_lib):
    c = cuda_lib.kd_create(0)
    yield c
    c.close()


@pytest.mark.parametrize("dtype", [np.int32, np.int64, np.float32], ids=["i32", "i64", "f32"])
@pytest.mark.parametrize("k", [2, 3, 5, 8])
def test_runs_ordered_on_chip(cuda_lib, ctx, dtype, k):
    check(cuda_lib, ctx, runs_cloud(MIXED, k, dtype, 800 + k))


@pytest.mark.parametrize("dtype", [np.int32, np.int64], ids=["i32", "i64"])
@pytest.mark.parametrize("k", [2, 3])
def test_runs_at_tile_edges(cuda_lib, ctx, dtype, k):
    # (the runs of 20 keep the mean cost below the line)
    check(cuda_lib, ctx, runs_cloud(EDGES + [20] * 25000, k, dtype, 820 + k, other_bits=7))


@pytest.mark.parametrize("dtype", [np.int32, np.int64, np.float32], ids=["i32", "i64", "f32"])
@pytest.mark.parametrize("lengths", [[100] * 2200, [300] * 750, MIXED + [5000], [200000]],
                         ids=["below the cost", "above the cost", "long run", "one value"])
def test_lines_of_the_whole_key_sort(cuda_lib, ctx, dtype, lengths):
    check(cuda_lib, ctx, runs_cloud(lengths, 3, dtype, 840 + len(lengths), other_bits=9))
