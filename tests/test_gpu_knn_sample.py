"""The sampled thresholds of the kNN's tensor-core collection (knn_sample in
csrc/knn.cu) against the CUDA-core path, which samples by other code:
bit-identical neighbour sets and statuses for every split of the warps, with
and without a first sweep, and where the list of values must overflow."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1310_5182_gb300 as lib
    return lib


def design(kind, N, M, p, rng):
    X, Q = rng.uniform(size=(N, p)), rng.uniform(size=(M, p))
    if kind == "lattice":    # a handful of distinct distances: whole bins of ties
        X, Q = np.floor(X * 3), np.floor(Q * 3)
    elif kind == "equal":    # every row the same: any list overflows
        X[:] = 0.5
    elif kind == "outlier":  # distances spread over many octaves
        X[7] = 1e6
        X[: N // 2] = 1e-3 * X[: N // 2] + 0.5
    elif kind == "sorted":   # a sample in the design's order would start in a corner
        X = X[np.argsort(X[:, 0])]
    elif kind == "nonfinite":
        X[::50, 0], X[1::50, p - 1], Q[0, 0] = np.nan, np.inf, np.nan
    return X, Q


@pytest.mark.parametrize("kind,N,M,p,Np", [
    ("uniform", 3_000, 5, 2, 300),       # stride 1: histograms of the whole design
    ("uniform", 60_000, 5, 3, 100),      # one query a CTA, listed values
    ("uniform", 60_001, 701, 8, 100),    # four queries a CTA
    ("uniform", 20_000, 5_003, 5, 64),   # sixteen, ragged, run-time p
    ("uniform", 9_000, 5_003, 8, 560),   # stride 2: the rank is too large for the list
    ("lattice", 40_000, 701, 2, 64), ("equal", 30_000, 33, 3, 32), ("outlier", 40_000, 701, 3, 200),
    ("sorted", 50_000, 5_003, 2, 128), ("nonfinite", 30_000, 701, 4, 50), ("uniform", 33, 7, 1, 33)])
@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
def test_sample_equals_cuda_core_path(L, kind, N, M, p, Np, dtype):
    rng = np.random.default_rng(47)
    X, Q = (torch.from_numpy(a).to(dtype).cuda() for a in design(kind, N, M, p, rng))
    sizes = torch.from_numpy(rng.integers(1, Np + 1, M).astype(np.int32)).cuda()
    sizes[3] = 0  # refused for this location only
    got = L.lagp_knn(X, Q, Np, Nprime=sizes)
    L.set_tuning(knn_path=1)
    try:
        ref = L.lagp_knn(X, Q, Np, Nprime=sizes)
    finally:
        L.set_tuning(knn_path=0)
    assert torch.equal(got[1], ref[1])
    assert torch.equal(got[0], ref[0])
