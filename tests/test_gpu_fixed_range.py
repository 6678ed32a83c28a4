"""The fixed-point kernels (csrc/fx59.cuh, fx_chol.cuh and what uses them) where
values leave their range, or are so small that an absolute 2^-59 is not enough.
References: the FP64 oracle, or the same formulas in extended precision
(numpy.longdouble: 64-bit mantissas on x86, 113 bits on Arm)."""
import numpy as np
import pytest
import torch

import workloads as W
from test_gpu_fixed import check_mle
from test_gpu_parity import L, O, alc_atol, check_pred, compare_selection, dev  # noqa: F401  (fixtures)

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


def exact_eval(X, x, design, cands, d, g):
    """Eq. (dxy), simplified, in extended precision."""
    LD = np.longdouble
    A, C, q = X[design].astype(LD), X[cands].astype(LD), np.asarray(x).astype(LD)
    n = len(design)
    k = lambda U, V: np.exp(-((U[:, None] - V[None]) ** 2).sum(-1) / LD(d))
    L = k(A, A) + LD(g) * np.eye(n)
    B = np.concatenate([k(A, q[None]), k(A, C)], axis=1)
    for c in range(n):  # L L^T in place, and L^{-1} B beside it
        L[c:, c] -= L[c:, :c] @ L[c, :c]
        L[c, c] = np.sqrt(L[c, c])
        L[c + 1:, c] /= L[c, c]
        B[c] = (B[c] - L[c, :c] @ B[:c]) / L[c, c]
    u, z = B[:, 1:], B[:, 0]
    r = k(C, q[None])[:, 0] - z @ u
    return r * r / (1 + LD(g) - (u * u).sum(0))


@pytest.mark.parametrize("n", [60, 128, 129, 200])
@pytest.mark.parametrize("shift", [0.0, 2.0, 3.5, 6.0])
def test_alc_eval_with_the_location_away_from_the_design(L, O, n, shift):
    """The location moved off the design and its candidates (largest covariance
    with the design down to 1e-30).  Bar: cond(K) 2^-53 is 2e-11 here, the root
    of a criterion value of 1e-6 of the best is 1e-3 of the best's, and ten
    times the quotient of the two is 2e-7: a relative 1e-6."""
    g, d = 1e-3, 0.5
    w = W.toy2d(seed=52, N=6_000, M=1)
    idx = O.knn(w.X, w.Xref, n + 800)[0]
    design, cands = idx[:n], idx[n:][::4]
    x = w.Xref[0] + np.array([shift, 0.0])
    delta, st = L.lagp_alc_eval(dev(w.X), x, dev(design), dev(cands), d, g)
    assert int(st.cpu()[0]) == 0
    ref = exact_eval(w.X, x, design, cands, d, g).astype(np.float64)
    top = ref >= 1e-6 * ref.max()
    np.testing.assert_allclose(delta.cpu().numpy()[top], ref[top], rtol=1e-6)


def wide_candidates(p, seed):
    """Candidate sets that reach many lengthscales from the location: the 300
    nearest rows, with d such that all but a few have tiny covariances."""
    w = W.toy2d(seed=seed, N=20_000, M=60) if p == 2 else W.borehole(seed=seed, N=4_000, M=60, n=40, Np=300, g=1e-2)
    idx = np.argsort(((w.X[None] - w.Xref[:, None]) ** 2).sum(-1), axis=1, kind="stable")[:, :300].astype(np.int32)
    return w, idx


def check_search(out, O, w, idx, n, d, g):
    ref = O.alc_select(w.X, w.Xref, idx, 6, n, d, g, topk=4)
    assert np.array_equal(out["status"].cpu().numpy(), ref["status"])
    sel, alc = out["sel"].cpu().numpy(), out["alc"].cpu().numpy()
    diverged = compare_selection(sel, ref, np.full(w.M, n, np.int32), 6, g)
    assert len(diverged) <= 2  # (near ties are rare)
    same = [m for m in range(w.M) if m not in diverged]
    # the criterion of the rows taken, where it is a normal number (and the
    # square of one): cond(K) is below 1e3 in these cases, ten times cond 2^-53 is 1e-12
    a, r = alc[same, 6:], ref["alc"][same, 6:]
    ok = r > 1e-280
    np.testing.assert_allclose(a[ok], r[ok], rtol=1e-9)


@pytest.mark.parametrize("p,d", [(2, 1e-5), (2, 1e-4), (2, 3e-4), (8, 0.003), (8, 0.01), (8, 0.03)])
def test_plain_search_many_lengthscales_away(L, O, p, d):
    w, idx = wide_candidates(p, 3)
    g, n = 1e-2, 40
    out = L.lagp_alc_select(dev(w.X), dev(w.Xref), dev(idx), 6, n, d, g, prec="f64", want_alc=True)
    check_search(out, O, w, idx, n, d, g)


@pytest.mark.parametrize("p,d", [(2, 1e-4), (2, 3e-4), (8, 0.01), (8, 0.03)])
def test_schur_search_many_lengthscales_away(L, O, p, d):
    """(Scores are r^2 / v in FP32: with still smaller d they underflow to zero,
    in the FP64 state as well, and the lowest rows are taken.)"""
    w, idx = wide_candidates(p, 3)
    g, n = 1e-2, 40
    out = L.lagp_alc_select(dev(w.X), dev(w.Xref), dev(idx), 6, n, d, g, prec="f64schur", want_alc=True)
    check_search(out, O, w, idx, n, d, g)


@pytest.mark.parametrize("n", [2, 8, 60])
@pytest.mark.parametrize("responses", ["smooth", "noise"])
def test_likelihood_derivatives_at_nearly_diagonal_k(L, n, responses):
    """l' and l'' where the correlations of the design are small (lengthscales
    from 0.002 of the box on), against extended precision.  Bar: (n^2 + t) 2^-50 of
    the sum of the terms' magnitudes: sums of n^2 products, eight roundings each,
    and exp(-t) of the nearest pair, t = D / d rounded."""
    LD = np.longdouble
    w = W.borehole(seed=31, N=4_000, M=40, n=60, Np=200, g=1e-3)
    sel = np.argsort(((w.X[None] - w.Xref[:, None]) ** 2).sum(-1), axis=1, kind="stable")[:, :n].astype(np.int32)
    Y = w.Y if responses == "smooth" else np.random.default_rng(7).normal(size=w.N)
    g = 1e-3
    for d in (0.002, 0.004, 0.01, 0.03, 0.1, 0.3):
        out = L.lagp_mle_step(dev(w.X), dev(Y), dev(sel), n, d, g, 1e-300, 1e300, 0)
        assert (out["status"].cpu().numpy() == 0).all()
        for m in range(w.M):
            A, y = w.X[sel[m]].astype(LD), Y[sel[m]].astype(LD)
            D = ((A[:, None] - A[None]) ** 2).sum(-1)
            E = np.exp(-D / LD(d))
            t0 = float(D[np.triu_indices(n, 1)].min() / d)
            K1, K2 = D / LD(d) ** 2 * E, (D * D / LD(d) ** 4 - 2 * D / LD(d) ** 3) * E
            Ki = np.eye(n, dtype=LD)  # by Gauss-Jordan (K is nearly diagonal)
            K = E + LD(g) * np.eye(n)
            for c in range(n):
                Ki[c], K[c] = Ki[c] / K[c, c], K[c] / K[c, c]
                f = K[:, c].copy()
                f[c] = 0
                Ki, K = Ki - f[:, None] * Ki[c], K - f[:, None] * K[c]
            a = Ki @ y
            psi, t, B = y @ a, K1 @ a, Ki @ K1
            phi = a @ t
            one = [-np.trace(B) / 2, LD(n) / 2 * phi / psi]
            two = [(B * B.T).sum() / 2, -(Ki * K2).sum() / 2,
                   LD(n) / 2 * (a @ K2 @ a) / psi, -LD(n) * (t @ Ki @ t) / psi, LD(n) / 2 * (phi / psi) ** 2]
            for k, terms in (("dllik", one), ("d2llik", two)):
                err = abs(LD(out[k][m].item()) - sum(terms))
                assert err <= (n * n + t0) * 2.0 ** -50 * sum(abs(v) for v in terms), (k, d, m, float(err))


@pytest.mark.parametrize("d", [0.01, 0.1, 0.5])
def test_mean_of_small_responses_beside_large_ones(L, d):
    """Responses over twelve decades and a nearly diagonal K: the mean is a small
    response times its covariance, far below the largest response.  Bar: 2^-40
    relative (the covariances' exponents are rounded at t 2^-53, t up to 100), or
    64 times FP64's rounding of the terms, cond(K) n 2^-53 |w| |z|."""
    LD = np.longdouble
    g, n = 1e-3, 40
    w = W.borehole(seed=31, N=4_000, M=60, n=n, Np=200, g=g)
    sel = np.argsort(((w.X[None] - w.Xref[:, None]) ** 2).sum(-1), axis=1, kind="stable")[:, :n].astype(np.int32)
    rng = np.random.default_rng(7)
    Y = rng.normal(size=w.N) * 10.0 ** rng.uniform(-6, 6, size=w.N)
    out = L.lagp_predict(dev(w.X), dev(Y), dev(w.Xref), dev(sel), n, d, g)
    assert (out["status"].cpu().numpy() == 0).all()
    for m in range(w.M):
        A, q = w.X[sel[m]].astype(LD), w.Xref[m].astype(LD)
        K = np.exp(-((A[:, None] - A[None]) ** 2).sum(-1) / LD(d)) + LD(g) * np.eye(n)
        cond = np.linalg.cond(K.astype(np.float64))
        v = np.stack([np.exp(-((A - q) ** 2).sum(-1) / LD(d)), Y[sel[m]].astype(LD)], 1)
        for c in range(n):  # K = L L^T in place, L^{-1} v beside it
            K[c:, c] -= K[c:, :c] @ K[c, :c]
            K[c, c] = np.sqrt(K[c, c])
            K[c + 1:, c] /= K[c, c]
            v[c] = (v[c] - K[c, :c] @ v[:c]) / K[c, c]
        mean, mag = v[:, 0] @ v[:, 1], abs(v[:, 0]) @ abs(v[:, 1])
        err = abs(LD(out["mean"][m].item()) - mean)
        assert err <= max(2.0 ** -40 * abs(mean), 64 * cond * n * 2.0 ** -53 * mag), (m, float(err / abs(mean)))


def test_alc_eval_status_and_values_agree(L):
    """Singular to rounding (no nugget, smooth kernel): the fixed-point factor
    may succeed where the FP64 one fails.  A candidate that is a design row leaves
    the range (1 - s = 0), and then FP64 decides for the call: ENOTPD and NaN
    for every candidate, or OK and the others' values."""
    rng = np.random.default_rng(5)
    both = 0
    for trial in range(1500):
        n = int(rng.integers(8, 26))
        X = rng.uniform(-2, 2, size=(200, 1 + trial % 2))
        d = 10.0 ** rng.uniform(-0.5, 2.0)
        cands = np.concatenate([np.arange(n, 200), [3]]).astype(np.int32)
        delta, st = L.lagp_alc_eval(dev(X), X[n], dev(np.arange(n, dtype=np.int32)), dev(cands), d, 0.0)
        delta, st = delta.cpu().numpy(), int(st.cpu()[0])
        assert st in (0, 2)
        if st == 2:
            assert np.isnan(delta).all(), (trial, n, d)
        both |= 1 << st
    assert both == 5


def test_zero_responses_cost_what_fp64_costs(L):
    """All responses zero: nothing to scale, every location goes to the FP64
    kernel, before any of the fixed-point work is done (g = 1 goes there by the
    launcher's rule; the same arithmetic)."""
    w = W.borehole(seed=1, N=4_000, M=2_000, n=60, Np=200)
    X, Xr, Y = dev(w.X), dev(w.Xref), dev(np.zeros(w.N))
    sel = L.lagp_knn(X, Xr, 100)[0]

    def ms(g):
        out = []
        for _ in range(20):
            e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            e[0].record()
            r = L.lagp_predict(X, Y, Xr, sel, 100, 2.0, g)
            e[1].record()
            torch.cuda.synchronize()
            out.append(e[0].elapsed_time(e[1]))
        assert (r["status"] == 0).all() and (r["mean"] == 0).all() and (r["s2"] == 0).all()
        return min(out)
    assert ms(1e-4) <= 1.15 * ms(1.0)  # 1.02; 1.28 when found after the covariances


def test_sums_of_the_factorisation_are_not_biased(L):
    """s2 = |z|^2 (1 + g - |w|^2) / n with K nearly diagonal and responses of one
    sign, where every inner product is rounded alike.  The mean of the relative
    errors over the locations: 60 rounded sums each, of either sign, so that a
    mean beyond 4 2^-53 is a bias (it was 12 with every share of a sum rounded
    down)."""
    LD = np.longdouble
    g, n, d = 1e-3, 60, 0.01
    w = W.borehole(seed=31, N=4_000, M=100, n=n, Np=200, g=g)
    sel = np.argsort(((w.X[None] - w.Xref[:, None]) ** 2).sum(-1), axis=1, kind="stable")[:, :n].astype(np.int32)
    Y = 2.0 + 0.1 * w.Y
    out = L.lagp_predict(dev(w.X), dev(Y), dev(w.Xref), dev(sel), n, d, g)
    rel = []
    for m in range(w.M):
        A, q = w.X[sel[m]].astype(LD), w.Xref[m].astype(LD)
        K = np.exp(-((A[:, None] - A[None]) ** 2).sum(-1) / LD(d)) + LD(g) * np.eye(n)
        v = np.stack([np.exp(-((A - q) ** 2).sum(-1) / LD(d)), Y[sel[m]].astype(LD)], 1)
        for c in range(n):  # K = L L^T in place, L^{-1} v beside it
            K[c:, c] -= K[c:, :c] @ K[c, :c]
            K[c, c] = np.sqrt(K[c, c])
            K[c + 1:, c] /= K[c, c]
            v[c] = (v[c] - K[c, :c] @ v[:c]) / K[c, c]
        s2 = (v[:, 1] ** 2).sum() * (1 + LD(g) - (v[:, 0] ** 2).sum()) / n
        rel.append(float((LD(out["s2"][m].item()) - s2) / s2))
    assert abs(np.mean(rel)) <= 4 * 2.0 ** -53


@pytest.mark.parametrize("M", [4, 200])  # both layouts
def test_plain_search_with_equidistant_rows(L, O, M):
    """A regular simplex as the seeds: K^{-1} has one value off its diagonal, a
    candidate above the centre one covariance with all rows, and the middle
    limbs' sums of 56 equal products are the largest there can be: for some of
    the candidates above 2^63, for others, further up, not.  Lengthscales in
    small steps, so that the low limb takes all values."""
    p, n0, n, g = 60, 56, 60, 1e-2
    rng = np.random.default_rng(23)
    C = 1.0 / n0 * (np.arange(p) < n0) + 1e-2 * rng.normal(size=(100, p))
    C[:, 57] += np.sqrt(rng.uniform(0, 3, size=100)) * rng.choice([-1, 1], 100)
    X = np.concatenate([np.eye(p)[:n0], C])
    Xref = np.tile(1.0 / n0 * (np.arange(p) < n0) + 0.3 * (np.arange(p) == 57), (M, 1))
    idx = np.tile(np.arange(len(X), dtype=np.int32), (M, 1))
    d = 20.0 + 0.37 * np.arange(M) if M > 100 else np.array([20.0, 31.7, 47.3, 66.1])
    out = L.lagp_alc_select(dev(X), dev(Xref), dev(idx), n0, n, d, g, prec="f64", want_alc=True)
    ref = O.alc_select(X, Xref, idx, n0, n, d, g, topk=4)
    assert (out["status"].cpu().numpy() == 0).all()
    diverged = compare_selection(out["sel"].cpu().numpy(), ref, np.full(M, n, np.int32), n0, g)
    same = [m for m in range(M) if m not in diverged]
    assert len(same) >= 0.9 * M
    np.testing.assert_allclose(out["alc"].cpu().numpy()[same, n0:], ref["alc"][same, n0:n], rtol=1e-6, atol=alc_atol(g))


@pytest.mark.parametrize("n,p,d", [(300, 2, 3.0), (600, 3, 2.0), (128, 2, 1.0)])
def test_alc_eval_of_candidates_beyond_a_dense_design(L, O, n, p, d):
    """Candidates outside a dense design with a tiny nugget: |L^{-1} k|^2, scaled
    by its largest covariance, passes through every size up to far above 32,
    where the fixed-point sum has wrapped once round, with all entries in range.
    Bar: 3 cond(K) 2^-53 of max(delta, K^2)."""
    rng = np.random.default_rng(29)
    g = 1e-8
    A = rng.uniform(size=(n, p))
    C = np.full((240, p), 0.5)
    C[:, 0] = np.linspace(1 + 2.7 * np.sqrt(d), 1 + 3.2 * np.sqrt(d), 240)
    X = np.concatenate([A, C])
    x = np.array([1.0 + 2 * np.sqrt(d)] + [0.45] * (p - 1))
    design, cands = np.arange(n, dtype=np.int32), np.arange(n, n + 240, dtype=np.int32)
    delta, st = L.lagp_alc_eval(dev(X), x, dev(design), dev(cands), d, g)
    assert int(st.cpu()[0]) == 0
    ref = exact_eval(X, x, design, cands, d, g).astype(np.float64)
    kap2 = np.exp(-2 * ((C - x) ** 2).sum(-1) / d)
    assert np.all(np.abs(delta.cpu().numpy() - ref) <= 3 * n / g * 2.0 ** -53 * np.maximum(ref, kap2))


@pytest.mark.parametrize("n", [20, 60])
def test_estimates_that_run_into_nearly_diagonal_k(L, O, n):
    """Noise responses: steps towards the lower bound, begun in fixed point and
    finished by the FP64 kernel from the last point that holds.  As the oracle's;
    all iterations count, and all evaluations."""
    g, M = 1e-2, 200
    w = W.borehole(seed=92, N=4_000, M=M, n=n, Np=200, g=g)
    sel = O.knn(w.X, w.Xref, n).astype(np.int32)
    Y = np.random.default_rng(92).normal(size=w.N)
    n_arr, d0 = np.full(M, n, np.int32), np.full(M, 0.5)
    for max_iter in (0, 1, 2, 3, 30):
        L.mle_work(torch.device("cuda", 0))
        out = L.lagp_mle_step(dev(w.X), dev(Y), dev(sel), n, d0, g, 1e-2, 20.0, max_iter)
        work = L.mle_work(torch.device("cuda", 0))
        ref = O.mle(w.X, Y, sel, n_arr, d0, g, 1e-2, 20.0, max_iter)
        it = out["iters"].cpu().numpy()
        assert (out["status"].cpu().numpy() == 0).all()
        same = it == ref["iters"]  # (the last step may differ where the likelihood is flat to rounding)
        assert same.mean() >= (0.95 if max_iter == 30 else 1.0)
        np.testing.assert_allclose(out["d"].cpu().numpy()[same], ref["d"][same], rtol=1e-6)
        np.testing.assert_allclose(out["llik"].cpu().numpy(), ref["llik"], rtol=1e-9, atol=1e-9)
        assert work["llik_n3"] >= (it.sum() + M) * n ** 3
    assert (out["d"].cpu().numpy() <= 0.05).mean() > 0.2  # (the case that is meant does occur)
