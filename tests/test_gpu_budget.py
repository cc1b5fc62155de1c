"""The memory budget against what the device gives up (GPU only): small blocks
that are held or kept for reuse stay within it, and give way to a call that
needs the whole of it."""
import numpy as np
import pytest

import kdgen
import oracle

pytestmark = pytest.mark.gpu
MIB = 1 << 20


def _free():
    import torch
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def test_held_and_kept_blocks_stay_within_the_budget(cuda_lib):
    """Handles whose blocks are just above powers of two, held until the budget
    is used up: the device gives up the budget and the rounding of the two pools
    (32 MiB each), not the power of two above every block."""
    import torch
    budget = 256 * MIB
    x = torch.from_numpy(kdgen.cloud_int_uniform(8200, 2, 30, 1, np.int32)).cuda()
    warm = cuda_lib.kd_create(0)
    cuda_lib.build_tree(warm, x)  # kernels loaded, the caller's allocator warm
    warm.close()
    before = _free()
    ctx = cuda_lib.kd_create(0, mem_budget_bytes=budget)
    try:
        handles = []
        with pytest.raises(cuda_lib.KdError) as e:
            for _ in range(4000):
                handles.append(cuda_lib.kd_presort(ctx, x))
        assert e.value.code == -2
        assert len(handles) > 1000
        used = before - _free()
        assert used <= budget + 64 * MIB, used / MIB
        for h in handles:
            cuda_lib.kd_release(ctx, h)
        assert before - _free() <= budget + 64 * MIB
    finally:
        ctx.close()


@pytest.mark.parametrize("budget", [24 * MIB, 2048 * MIB])
def test_kept_blocks_give_way(cuda_lib, budget):
    """After many small builds of different sizes, the largest cloud that a new
    context builds under the same budget is built."""
    import torch
    def largest(ctx, lo, hi):  # a power of two of tuples that fits; KD_ENOMEM above
        n = lo
        while n < hi:
            try:
                cuda_lib.build_tree(ctx, cloud[:2 * n])
            except cuda_lib.KdError as e:
                assert e.code == -2
                return n
            n *= 2
        return n
    coords = kdgen.cloud_unit_cube(1 << 23, 3, 5)
    cloud = torch.from_numpy(coords).cuda()
    fresh = cuda_lib.kd_create(0, mem_budget_bytes=budget)
    ctx = cuda_lib.kd_create(0, mem_budget_bytes=budget)
    try:
        n = largest(fresh, 1 << 14, 1 << 22)
        for m in range(200, 20000, 331):
            cuda_lib.build_tree(ctx, cloud[:m])
        got = cuda_lib.build_tree(ctx, cloud[:n])
        if n <= 1 << 18:
            np.testing.assert_array_equal(got["node_tuple"].cpu().numpy(), oracle.build_tree(coords[:n])["node_tuple"])
        assert largest(ctx, n, 1 << 22) == n
    finally:
        fresh.close()
        ctx.close()
