"""The autotuner's samples: what a small one can tell, and what is tried."""
import numpy as np
import pytest
import torch

import workloads as W
from test_gpu_parity import L, dev  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


def problem(L, M, Np=400):
    w = W.borehole(seed=81, N=20_000, M=M, n=30, Np=Np, g=1e-3)
    X, Xr = dev(w.X), dev(w.Xref)
    return w, X, Xr, L.lagp_knn(X, Xr, Np)[0]


@pytest.mark.parametrize("prec", ["f32bulk", "f32bulk_f64", "f64schur", "f64"])
def test_few_locations_time_only_the_grids_that_differ(L, prec):
    """Up to a location an SM every count of CTAs is the same grid: one count is
    timed (the best of ties would be noise); results stay the same."""
    w, X, Xr, idx = problem(L, 100)
    for n in (10, 20, 25, 30):
        before = L.lagp_alc_select(X, Xr, idx, 6, n, w.d, w.g, prec=prec)["sel"]
        best = L.lagp_autotune(X, Xr, idx, 6, n, w.d, w.g, prec=prec)
        assert best["ctas_per_sm"] == 1
        assert torch.equal(L.lagp_alc_select(X, Xr, idx, 6, n, w.d, w.g, prec=prec)["sel"], before)


def test_schur_form_tries_its_default(L):
    """Four CTAs an SM, the fixed-point state's default, is 10% faster than three
    here: tuned, the search keeps it."""
    w, X, Xr, idx = problem(L, 2432, 1000)
    best = [L.lagp_autotune(X, Xr, idx, 6, 50, w.d, w.g, prec="f64schur")["ctas_per_sm"] for _ in range(3)]
    assert 4 in best
