"""Sizes whose dynamic shared memory comes within the kernel's static arrays of
the device's limit: the launchers have to count both."""
import numpy as np
import pytest
import torch

import workloads as W
from test_gpu_parity import L, dev  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,p,Np,M", [(128, 8, 2500, 200), (128, 8, 2500, 20), (127, 8, 4096, 20), (128, 5, 2200, 200),
                                      (116, 60, 200, 20), (118, 58, 256, 20)])
def test_f32bulk_batches_next_to_the_limit(L, n, p, Np, M):
    """The automatic re-score batch, clamped to what fits, against batches of 4
    (which change no result)."""
    rng = np.random.default_rng(17)
    X, Xr = rng.uniform(size=(6_000, p)), rng.uniform(size=(M, p))
    idx, _ = L.lagp_knn(dev(X), dev(Xr), Np)
    run = lambda: L.lagp_alc_select(dev(X), dev(Xr), idx, 6, n, p / 4.0, 1e-2, prec="f32bulk", want_alc=True)
    got = run()
    L.set_tuning(rescore_max=4)
    try:
        ref = run()
    finally:
        L.set_tuning(rescore_max=0)
    assert (ref["status"] == 0).all()
    for k in ("sel", "alc", "status"):
        assert torch.equal(torch.nan_to_num(got[k]), torch.nan_to_num(ref[k])), k
