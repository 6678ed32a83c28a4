"""Sizes whose dynamic shared memory comes within the kernel's static arrays of
the device's limit: the launchers have to count both."""
import numpy as np
import pytest
import torch

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


@pytest.mark.parametrize("n,p,M", [(116, 6, 4), (117, 4, 160), (112, 27, 4), (115, 6, 4)])
def test_plain_search_next_to_the_limit(L, n, p, M):
    """The plain FP64 search where its fixed-point kernel just fits or just does
    not: the designs of the FP64 Schur form (no near ties at these sizes)."""
    rng = np.random.default_rng(18)
    X, Xr = rng.uniform(size=(3_000, p)), rng.uniform(size=(M, p))
    idx, _ = L.lagp_knn(dev(X), dev(Xr), 200)
    got, ref = (L.lagp_alc_select(dev(X), dev(Xr), idx, 6, n, p / 4.0, 1e-2, prec=prec, want_alc=True)
                for prec in ("f64", "f64schur"))
    assert (got["status"] == 0).all() and torch.equal(got["sel"], ref["sel"])
    torch.testing.assert_close(got["alc"][:, 6:], ref["alc"][:, 6:], rtol=1e-6, atol=16 * 2.0 ** -52 / 1e-2)


@pytest.mark.parametrize("n,p", [(228, 64), (403, 40), (973, 18), (974, 18), (403, 39)])
def test_alc_eval_next_to_the_limit(L, n, p):
    from test_gpu_fixed_range import exact_eval
    rng = np.random.default_rng(19)
    X = rng.uniform(size=(2_000, p))
    design, cands = np.arange(n, dtype=np.int32), np.arange(n, n + 100, dtype=np.int32)
    x = X[-1] + 0.01
    delta, st = L.lagp_alc_eval(dev(X), x, dev(design), dev(cands), p / 4.0, 1e-2)
    assert int(st.cpu()[0]) == 0
    ref = exact_eval(X, x, design, cands, p / 4.0, 1e-2).astype(np.float64)
    np.testing.assert_allclose(delta.cpu().numpy(), ref, rtol=1e-6, atol=1e-6 * ref.max())
