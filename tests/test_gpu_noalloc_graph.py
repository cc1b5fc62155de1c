"""kd_presort_noalloc recorded into a graph after one call of another size and
type (GPU only).  In a process of its own: kernels that an earlier test has
loaded would hide one that the set-up leaves to be loaded while recording."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SCRIPT = """
import sys
sys.path.insert(0, {root!r})
import numpy as np
import torch
import kdgen
import oracle
from paper_1410_5420_gb300 import api
s = torch.cuda.Stream()
ctx = api.kd_create(0, stream=s)
with torch.cuda.stream(s):
    api.kd_presort_noalloc(ctx, torch.zeros((200, 2), dtype=torch.int32, device="cuda"))
torch.cuda.synchronize()
cases = []
for n, k, dt in ((16384, 3, np.float32), (9000, 5, np.int64), (2048, 4, np.int64), (700, 2, np.float32), (3000, 1, np.int32)):
    coords = kdgen.cloud_gmm(n, k, n) if dt == np.float32 else kdgen.cloud_int_uniform(n, k, 14, n, dt, 0.01)
    x = torch.zeros(coords.shape, dtype=torch.from_numpy(coords).dtype, device="cuda")
    rows, m = torch.zeros((k, n), dtype=torch.int32, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        api.kd_presort_noalloc(ctx, x, rows, m)
    cases.append((coords, x, rows, m, g))
for coords, x, rows, m, g in cases:
    x.copy_(torch.from_numpy(coords))
    g.replay()
    torch.cuda.synchronize()
    ref = oracle.presort(coords)
    assert int(m.item()) == ref.shape[1], (coords.shape, int(m.item()))
    np.testing.assert_array_equal(rows.cpu().numpy()[:, :ref.shape[1]], ref)
ctx.close()
print("recorded")
"""


def test_recorded_after_one_call(cuda_lib):
    r = subprocess.run([sys.executable, "-c", SCRIPT.format(root=ROOT)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "recorded" in r.stdout, r.stderr[-2000:]
