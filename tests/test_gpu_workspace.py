"""Device memory that a call for one location takes: in proportion to it."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

CODE = """
import torch
import paper_1310_5182_gb300 as L
g = torch.Generator().manual_seed(1)
X, Y = torch.rand(500, 3, generator=g, dtype=torch.float64).cuda(), torch.rand(500, generator=g, dtype=torch.float64).cuda()
sel = torch.arange(128, dtype=torch.int32).reshape(1, 128).cuda()
call = {calls}
call(2)  # (loads the kernels and their local memory)
torch.cuda.synchronize()
before = torch.cuda.mem_get_info()[0]
r = call({n})
torch.cuda.synchronize()
assert int(r["status"][0]) == 0
print("MB", (before - torch.cuda.mem_get_info()[0]) / 2 ** 20)
"""
PREDICT = "lambda n: L.lagp_predict(X, Y, X[:1].contiguous(), sel[:, :n].contiguous(), n, 1.0, 1e-3)"
MLE = "lambda n: L.lagp_mle_step(X, Y, sel[:, :n].contiguous(), n, 1.0, 1e-2, 1e-3, 20.0, 3)"


@pytest.mark.parametrize("calls,n", [(PREDICT, 128), (MLE, 60)])
def test_one_location_takes_little_workspace(calls, n):
    """The FP64 kernel's matrices for one location are under 1 MB; the allocator
    hands out 2 MB at a time."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", CODE.format(calls=calls, n=n)], cwd=root, capture_output=True, text=True,
                       timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    assert float(r.stdout.split("MB")[1]) <= 8.0
