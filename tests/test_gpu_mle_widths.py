"""The MLE's CTA widths and size classes (csrc/gp_fixed.cu) on both sides of
their lines, one size a call and all in one uneven call, with test_gpu_fixed's
bars against the FP64 oracle."""
import numpy as np
import pytest

import workloads as W
from test_gpu_fixed import check_mle, designs
from test_gpu_parity import L, O, dev  # noqa: F401  (fixtures)

pytestmark = pytest.mark.gpu

EDGES = [64, 65, 76, 77, 94, 95, 128]


@pytest.mark.parametrize("sizes", [[n] * 4 for n in EDGES] + [EDGES * 2], ids=str)
def test_mle_at_width_edges(L, O, sizes):
    g, n_arr = 1e-3, np.array(sizes, np.int32)
    w, sel = designs(O, 37, g, n_arr)
    n = n_arr if len(set(sizes)) > 1 else sizes[0]
    d0 = np.full(w.M, 1.5)
    check_mle(L.lagp_mle_step(dev(w.X), dev(w.Y), dev(sel), n, d0, g, 1e-3, 20.0, 2),
              O.mle(w.X, w.Y, sel, n, d0, g, 1e-3, 20.0, 2))


@pytest.mark.parametrize("d0,max_iter", [(1.85, 3), (2e-3, 3), (1.85, 12)])
def test_nearly_diagonal_covariances(L, O, d0, max_iter):
    """Small designs whose estimate runs to the lower bound, where all
    correlations (and l') are tiny and the sign of l' decides the step."""
    M = 1_500
    n = np.random.default_rng(41).integers(5, 13, M).astype(np.int32)
    w = W.borehole(seed=41, N=20_000, M=M, n=12, Np=200, g=1e-2, dtype=np.float32)
    sel = O.knn(w.X, w.Xref, 12).astype(np.int32)
    start = np.full(M, d0)
    out = L.lagp_mle_step(dev(w.X), dev(w.Y), dev(sel), n, start, 1e-2, 1e-3, 20.0, max_iter)
    ref = O.mle(w.X, w.Y, sel, n, start, 1e-2, 1e-3, 20.0, max_iter)
    assert np.array_equal(out["status"].cpu().numpy(), ref["status"])
    # (a location that turns on the rounding of l or l'' in the oracle itself: under 1%)
    off = np.abs(out["d"].cpu().numpy() - ref["d"]) > 1e-6 * ref["d"]
    assert off.mean() < 0.01
    low = ref["d"] <= 0.02
    assert low.sum() >= 3 and not off[low].any()
