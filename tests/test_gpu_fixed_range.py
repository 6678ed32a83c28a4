"""The fixed-point kernels (csrc/fx59.cuh, fx_chol.cuh and what uses them) where
values leave their range, or are so small that an absolute 2^-59 is not enough.
References: the FP64 oracle, or the same formulas in extended precision
(numpy.longdouble: 64-bit mantissas on x86, 113 bits on Arm)."""
import numpy as np
import pytest
import torch

import workloads as W
from test_gpu_fixed import check_mle
from test_gpu_parity import L, O, check_pred, dev  # noqa: F401  (fixtures)

pytestmark = pytest.mark.gpu


def test_responses_out_of_range_in_an_uneven_batch(L, O):
    """Noise responses with a small nugget: |z| = |L^{-1} Y| leaves the range at
    many locations, at different columns of the factorisation, and the next
    evaluation follows at once (every thread of the CTA has to take the same
    way).  Repeated: the same bits."""
    rng = np.random.default_rng(91)
    n_arr = rng.integers(2, 101, 600).astype(np.int32)
    g, d = 1e-6, 2.0
    w = W.borehole(seed=91, N=4_000, M=600, n=100, Np=200, g=g)
    sel = O.knn(w.X, w.Xref, 100).astype(np.int32)
    Y = rng.normal(size=w.N)
    d0 = np.full(w.M, d)
    runs = [L.lagp_mle_step(dev(w.X), dev(Y), dev(sel), n_arr, d0, g, 1e-3, 20.0, 2) for _ in range(20)]
    for r in runs[1:]:
        for k in ("d", "llik", "dllik", "d2llik", "iters", "status"):
            assert torch.equal(torch.nan_to_num(r[k]), torch.nan_to_num(runs[0][k])), k
    check_mle(L.lagp_mle_step(dev(w.X), dev(Y), dev(sel), n_arr, d0, g, 1e-3, 20.0, 1),
              O.mle(w.X, Y, sel, n_arr, d0, g, 1e-3, 20.0, 1))
    ref = O.predict(w.X, Y, w.Xref, sel, n_arr, d, g)
    out = L.lagp_predict(dev(w.X), dev(Y), dev(w.Xref), dev(sel), n_arr, d, g)
    assert (out["status"].cpu().numpy() == 0).all()
    check_pred(out["mean"].cpu().numpy(), out["s2"].cpu().numpy(), ref, w.X, Y, w.Xref, sel, n_arr, d, g)
