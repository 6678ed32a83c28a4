"""The kNN's spatial order and rank (csrc/knn.cu) against the CUDA-core path,
which uses neither: bit-identical neighbour sets and statuses on designs where
cells, boxes or buckets could go wrong."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

N, M = 33_000, 33_000  # above the order's thresholds (2^15 rows, 2^30 pairs)


@pytest.fixture(scope="module")
def L():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1310_5182_gb300 as lib
    return lib


def design(kind, p, rng):
    X, Q = rng.uniform(size=(N, p)), rng.uniform(size=(M, p))
    if kind == "lattice":      # exact ties and duplicates
        X, Q = np.floor(X * 12), np.floor(Q * 12)
    elif kind == "outlier":    # one far row: every other row in one cell
        X[7] = 1e6
    elif kind == "constant":   # a coordinate without extent
        X[:, 0] = Q[:, 0] = 0.25
    elif kind == "clusters":   # empty cells, boxes of very different sizes
        c = rng.uniform(size=(40, p))
        X = c[rng.integers(0, 40, N)] + 1e-3 * rng.normal(size=(N, p))
        Q[: M // 2] = X[rng.integers(0, N, M // 2)]
    elif kind == "nonfinite":
        X[11, 0], X[12, p - 1], Q[5, 0] = np.nan, np.inf, np.nan
    return X, Q


@pytest.mark.parametrize("kind,p,dtype,Np", [
    ("uniform", 1, torch.float64, 40), ("uniform", 2, torch.float32, 300), ("uniform", 3, torch.float64, 1100),
    ("uniform", 8, torch.float32, 64), ("uniform", 17, torch.float32, 33), ("uniform", 20, torch.float64, 20),
    ("lattice", 2, torch.float32, 50), ("lattice", 3, torch.float64, 90), ("outlier", 4, torch.float64, 64),
    ("constant", 3, torch.float32, 64), ("clusters", 2, torch.float64, 128), ("clusters", 6, torch.float32, 128),
    ("nonfinite", 3, torch.float64, 32)])
def test_order_equals_cuda_core_path(L, kind, p, dtype, Np):
    rng = np.random.default_rng(41)
    X, Q = (torch.from_numpy(a).to(dtype).cuda() for a in design(kind, p, rng))
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
