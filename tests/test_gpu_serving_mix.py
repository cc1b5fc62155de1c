"""Served bursts while the caller's thread builds on contexts of its own (GPU
only): the fused steps of many small builds on three streams at a time, every
result against the oracle, round after round."""
import numpy as np
import pytest

import kdgen
import oracle

pytestmark = pytest.mark.gpu
ROUNDS = 25


def _cloud(i):
    n = int(2.0 ** np.random.default_rng(i).uniform(6, 15)) + (200000 if i % 11 == 0 else 0)
    k = 2 + i % 3
    return kdgen.cloud_gmm(n, k, i) if i % 2 else kdgen.cloud_int_uniform(n, k, 24, i, np.int32, dup_frac=0.01)


def test_bursts_beside_builds(cuda_lib):
    import torch
    clouds = [_cloud(i) for i in range(44)]
    refs = [oracle.build_tree(c)["node_tuple"] for c in clouds]
    devs = [torch.from_numpy(c).cuda() for c in clouds]
    torch.cuda.synchronize()
    serving = cuda_lib.kd_create(0, mem_budget_bytes=8 << 30)
    ctx = cuda_lib.kd_create(0, stream=torch.cuda.Stream())
    try:
        for r in range(ROUNDS):
            order = np.random.default_rng(r).permutation(len(clouds))
            tickets = [(i, cuda_lib.kd_submit(serving, clouds[i], children=False)) for i in order]
            for i in order[::5]:
                got = cuda_lib.build_tree(ctx, devs[i], children=False)["node_tuple"].cpu().numpy()
                np.testing.assert_array_equal(got, refs[i], err_msg=f"round {r} built {i}")
            for i, t in tickets:
                got = cuda_lib.kd_wait(serving, t)["node_tuple"]
                np.testing.assert_array_equal(got, refs[i], err_msg=f"round {r} served {i}")
    finally:
        serving.close()
        ctx.close()
