"""Prediction and MLE in fixed point (csrc/gp_fixed.cu) where they can go
wrong: sizes at the edges of its classes and column pairs in one uneven batch,
responses and nuggets at the ends of its range, and the locations it leaves to
the FP64 kernels.  Bars as in test_gpu_parity.py, against the FP64 oracle."""
import numpy as np
import pytest
import torch

import workloads as W
from test_gpu_parity import L, O, check_pred, compare_selection, dev  # noqa: F401  (fixtures)

pytestmark = pytest.mark.gpu

SIZES = np.array([1, 2, 3, 4, 39, 40, 41, 42, 63, 64, 65, 66, 79, 80, 81, 103, 104, 105, 127, 128], np.int32)


def designs(O, seed, g, n_arr, **kw):
    w = W.borehole(seed=seed, N=4_000, M=len(n_arr), n=int(n_arr.max()), Np=200, g=g, **kw)
    return w, O.knn(w.X, w.Xref, int(n_arr.max())).astype(np.int32)


def check_mle(out, ref):
    assert np.array_equal(out["status"].cpu().numpy(), ref["status"])
    assert np.array_equal(out["iters"].cpu().numpy(), ref["iters"])
    np.testing.assert_allclose(out["d"].cpu().numpy(), ref["d"], rtol=1e-6)
    np.testing.assert_allclose(out["llik"].cpu().numpy(), ref["llik"], rtol=1e-9, atol=1e-9)
    scale = np.abs(ref["llik"]) / ref["d"]
    np.testing.assert_allclose(out["dllik"].cpu().numpy(), ref["dllik"], rtol=1e-5, atol=1e-7 * scale.max())


@pytest.mark.parametrize("dtype", [np.float64, np.float32])
def test_uneven_sizes_at_class_edges(L, O, dtype):
    g, d = 1e-3, 1.5
    w, sel = designs(O, 31, g, SIZES, dtype=dtype)
    ref = O.predict(w.X, w.Y, w.Xref, sel, SIZES, d, g)
    out = L.lagp_predict(dev(w.X), dev(w.Y), dev(w.Xref), dev(sel), SIZES, d, g)
    assert (out["status"].cpu().numpy() == 0).all()
    check_pred(out["mean"].cpu().numpy(), out["s2"].cpu().numpy(), ref, w.X, w.Y, w.Xref, sel, SIZES, d, g)
    d0 = np.full(w.M, d)
    check_mle(L.lagp_mle_step(dev(w.X), dev(w.Y), dev(sel), SIZES, d0, g, 1e-3, 20.0, 2),
              O.mle(w.X, w.Y, sel, SIZES, d0, g, 1e-3, 20.0, 2))


@pytest.mark.parametrize("g", [1e-6, 0.5, 0.999, 1.0, 30.0])
@pytest.mark.parametrize("scale,spike", [(1.0, 0.0), (1e-13, 0.0), (1e13, 0.0), (1.0, 1e4)])
def test_ranges_of_nugget_and_responses(L, O, g, scale, spike):
    """spike: one response far from the others (z then exceeds what its scale
    leaves room for, and the wider scale or FP64 takes over)."""
    n, d = 24, 2.0
    n_arr = np.full(12, n, np.int32)
    w, sel = designs(O, 32, g, n_arr)
    Y = w.Y * scale
    Y[sel[3, 5]] += spike
    ref = O.predict(w.X, Y, w.Xref, sel, n, d, g)
    out = L.lagp_predict(dev(w.X), dev(Y), dev(w.Xref), dev(sel), n, d, g)
    assert (out["status"].cpu().numpy() == 0).all()
    check_pred(out["mean"].cpu().numpy(), out["s2"].cpu().numpy(), ref, w.X, Y, w.Xref, sel, n_arr, d, g)
    d0 = np.full(w.M, d)
    check_mle(L.lagp_mle_step(dev(w.X), dev(Y), dev(sel), n, d0, g, 1e-3, 20.0, 1),
              O.mle(w.X, Y, sel, n, d0, g, 1e-3, 20.0, 1))


def test_locations_left_to_fp64(L, O):
    """Far locations (k_n(x) underflows), zero and non-finite responses,
    duplicated rows without a nugget: as the FP64 kernels have them."""
    n, d = 20, 0.5
    n_arr = np.full(8, n, np.int32)
    w, sel = designs(O, 33, 0.0, n_arr)
    Y, Xref = w.Y.copy(), w.Xref.copy()
    Xref[0] += 40.0                  # exp(-D/d) is zero or subnormal
    sel[1, 7] = sel[1, 3]            # singular without a nugget: rounding decides what FP64 makes of it
    rows = np.setdiff1d(np.arange(w.N), sel.ravel())[:n].astype(np.int32)
    sel[2], Y[rows] = rows, 0.0      # all responses zero
    ref = O.predict(w.X, Y, Xref, sel, n, d, 0.0)
    out = {k: v.cpu().numpy() for k, v in L.lagp_predict(dev(w.X), dev(Y), dev(Xref), dev(sel), n, d, 0.0).items()}
    assert out["status"][1] in (0, 2)
    ok = np.arange(8) != 1
    assert (out["status"][ok] == 0).all()
    check_pred(out["mean"][ok], out["s2"][ok], {k: v[ok] for k, v in ref.items()}, w.X, Y, Xref, sel[ok], n_arr[ok], d, 0.0)
    m = L.lagp_mle_step(dev(w.X), dev(Y), dev(sel), n, d, 0.0, 1e-3, 20.0, 0)
    assert (m["status"].cpu().numpy()[ok] == 0).all()
    Y[sel[4, 2]] = np.nan
    out = L.lagp_predict(dev(w.X), dev(Y), dev(Xref), dev(sel), n, d, 0.0)
    assert torch.isnan(out["mean"][4]) and int(out["status"][4]) == 0


@pytest.mark.parametrize("n,g,d", [(1, 1e-4, 0.5), (2, 0.9, 0.5), (15, 1e-4, 0.05), (16, 1e-6, 0.5), (17, 1e-2, 2.0),
                                   (33, 1.0, 0.5), (64, 1e-4, 0.02), (65, 1e-3, 0.5), (127, 1e-4, 0.5),
                                   (128, 1e-2, 0.1), (129, 1e-4, 0.5), (200, 1e-3, 0.1)])
def test_alc_eval_sizes_and_far_candidates(L, O, n, g, d):
    """Edges of the 16-row blocks, both factorisations (n <= 128 and above),
    the FP64 path (g = 1), candidates near and across the whole square (tiny
    covariances); the bar of test_alc_eval_matches_oracle."""
    w = W.toy2d(seed=52, N=6_000, M=1)
    idx = O.knn(w.X, w.Xref, n + 200)[0]
    design = idx[:n]
    far = np.setdiff1d(np.arange(w.N), idx)[::8]
    cands = np.concatenate([idx[n:], far]).astype(np.int32)
    delta, st = L.lagp_alc_eval(dev(w.X), w.Xref[0], dev(design), dev(cands), d, g)
    assert int(st.cpu()[0]) == 0
    _, ds = O.alc_scores(w.X, w.Xref[0], design, cands, d, g)
    A = w.X[design]
    K = np.exp(-((A[:, None] - A[None]) ** 2).sum(-1) / d) + g * np.eye(n)
    atol = 16 * np.finfo(np.float64).eps / g * max(1.0, np.linalg.cond(K) * g)
    assert np.all(np.abs(delta.cpu().numpy() - ds) <= np.maximum(1e-6 * np.abs(ds), atol))


@pytest.mark.parametrize("g,d,n_max", [(1e-2, 2.0, 70), (1e-6, 2.0, 40), (1.0, 2.0, 40), (1e-2, 1e-3, 30),
                                       (1e-3, 0.05, 40), (1e-2, 2.0, 128)])
def test_plain_search_in_fixed_point(L, O, g, d, n_max):
    """The plain FP64 form: uneven n (edges of the blocks of rows) and N', the
    FP64 kernel's share (g = 1; d = 1e-3: no candidate with K(x_c, x) >= 2^-6;
    n_max = 128: too large for shared memory); many locations and few (two
    layouts, the same bits)."""
    n_arr = np.array([6, 7, 8, 9, 12, 15, 16, 17, 23, 24, 25, 30] + [n_max] * 4, np.int32)
    Np = np.array([n_max, 130, 200, 131] * 4, np.int32)
    w = W.borehole(seed=34, N=4_000, M=16, n=n_max, Np=200, g=g)
    idx = O.knn(w.X, w.Xref, 200)
    idx = np.where(np.arange(200)[None] < Np[:, None], idx, -1).astype(np.int32)
    ref = O.alc_select(w.X, w.Xref, idx, 6, n_arr, d, g, topk=4, Np=Np)
    few = L.lagp_alc_predict(dev(w.X), dev(w.Y), dev(w.Xref), dev(idx), 6, n_arr, d, g, prec="f64", Nprime=Np,
                             n_max=n_max, want_alc=True)
    sel = few["sel"].cpu().numpy()
    diverged = compare_selection(sel, ref, n_arr, 6, g)
    same = [m for m in range(16) if m not in diverged]
    p = O.predict(w.X, w.Y, w.Xref, sel, n_arr, d, g)
    check_pred(few["mean"].cpu().numpy()[same], few["s2"].cpu().numpy()[same], {k: v[same] for k, v in p.items()},
               w.X, w.Y, w.Xref, sel[same], n_arr[same], d, g)
    rep = 20  # more locations than SMs
    tile = lambda a: np.ascontiguousarray(np.tile(a, (rep,) + (1,) * (a.ndim - 1)))
    many = L.lagp_alc_predict(dev(w.X), dev(w.Y), dev(tile(w.Xref)), dev(tile(idx)), 6, tile(n_arr), d, g, prec="f64",
                              Nprime=tile(Np), n_max=n_max, want_alc=True)
    for k in ("sel", "alc", "mean", "s2", "status"):
        assert torch.equal(torch.nan_to_num(many[k][:16]), torch.nan_to_num(few[k])), k
        assert torch.equal(torch.nan_to_num(many[k][-16:]), torch.nan_to_num(few[k])), k


@pytest.mark.parametrize("p,dtype,g,d,Np", [(1, np.float64, 1e-2, 0.3, 60), (2, np.float32, 1e-4, 0.5, 255),
                                            (3, np.float64, 1e-6, 0.05, 257), (8, np.float32, 1e-3, 2.0, 513),
                                            (20, np.float64, 1e-2, 5.0, 300), (2, np.float64, 1e-2, 1e-7, 100),
                                            (2, np.float64, 1.0, 0.5, 100)])
def test_schur_search_in_fixed_point(L, O, p, dtype, g, d, Np):
    """The FP64 Schur form with its state in fixed point: dimensions, candidate
    counts at the edges of the slots a thread, a lengthscale too small for the
    scaled coordinates (redone in FP64) and g = 1 (FP64); duplicated candidates."""
    rng = np.random.default_rng(35)
    X = rng.uniform(size=(3_000, p)).astype(dtype)
    X[1::10] = X[::10]  # exact duplicates
    Xref = rng.uniform(size=(20, p)).astype(dtype)
    n_arr = rng.integers(6, 41, 20).astype(np.int32)
    idx = O.knn(X, Xref, Np)
    ref = O.alc_select(X, Xref, idx, 6, n_arr, d, g, topk=4)
    out = L.lagp_alc_select(dev(X), dev(Xref), dev(idx), 6, n_arr, d, g, prec="f64schur", n_max=40, want_alc=True)
    assert np.array_equal(out["status"].cpu().numpy(), ref["status"])
    compare_selection(out["sel"].cpu().numpy(), ref, n_arr, 6, g)
