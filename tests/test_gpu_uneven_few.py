"""Locations of different sizes: prediction and MLE in one fixed-point launch for
few of them, in one a size class for many."""
import numpy as np
import pytest
import torch

import workloads as W
from test_gpu_fixed import check_mle
from test_gpu_parity import L, O, check_pred, dev  # noqa: F401  (fixtures)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M", [1, 26, 152])
def test_few_uneven_locations_take_one_launch(L, O, M):
    """Size classes would only queue one after the other (launches: the
    fixed-point kernel and the FP64 one behind it)."""
    rng = np.random.default_rng(41)
    n_arr = rng.integers(1, 101, M).astype(np.int32)
    n_arr[0] = 100
    g, d = 1e-3, 1.5
    w = W.borehole(seed=41, N=4_000, M=M, n=100, Np=200, g=g)
    sel = O.knn(w.X, w.Xref, 100).astype(np.int32)
    X, Y, Xr, s, n = dev(w.X), dev(w.Y), dev(w.Xref), dev(sel), dev(n_arr)
    before = L.launch_count()
    out = L.lagp_predict(X, Y, Xr, s, n, d, g)
    assert L.launch_count() - before == 2
    ref = O.predict(w.X, w.Y, w.Xref, sel, n_arr, d, g)
    assert (out["status"].cpu().numpy() == 0).all()
    check_pred(out["mean"].cpu().numpy(), out["s2"].cpu().numpy(), ref, w.X, w.Y, w.Xref, sel, n_arr, d, g)
    d0 = np.full(M, d)
    before = L.launch_count()
    out = L.lagp_mle_step(X, Y, s, n, dev(d0), g, 1e-3, 20.0, 2)
    assert L.launch_count() - before == 2
    check_mle(out, O.mle(w.X, w.Y, sel, n_arr, d0, g, 1e-3, 20.0, 2))


@pytest.mark.parametrize("M", [2432, 2433, 20_000])
def test_one_launch_and_size_classes_give_the_same_bits(L, M):
    """Both sides of the MLE's line (16 locations a resident CTA, 152 SMs) and
    both entry points beyond it: a location's results do not depend on the
    other locations of the call."""
    rng = np.random.default_rng(42)
    g, d = 1e-2, 1.5
    w = W.borehole(seed=42, N=4_000, M=M, n=100, Np=200, g=g)
    n_arr = rng.integers(1, 101, M).astype(np.int32)
    n_arr[:2] = 100, 41
    X, Y, Xr, n = dev(w.X), dev(w.Y), dev(w.Xref), dev(n_arr)
    sel = L.lagp_knn(X, Xr, 100)[0]
    few = slice(0, 100)
    p = L.lagp_predict(X, Y, Xr, sel, n, d, g)
    q = L.lagp_predict(X, Y, Xr[few].contiguous(), sel[few].contiguous(), n[few].contiguous(), d, g)
    for k in ("mean", "s2", "df", "status"):
        assert torch.equal(p[k][few], q[k]), k
    p = L.lagp_mle_step(X, Y, sel, n, d, g, 1e-3, 20.0, 2)
    q = L.lagp_mle_step(X, Y, sel[few].contiguous(), n[few].contiguous(), d, g, 1e-3, 20.0, 2)
    for k in ("d", "llik", "iters", "status"):
        assert torch.equal(p[k][few], q[k]), k
    for k in ("dllik", "d2llik"):
        torch.testing.assert_close(p[k][few], q[k], rtol=1e-12, atol=0, equal_nan=True)
