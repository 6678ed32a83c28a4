"""Candidate capacity of the kNN with few neighbours of many rows."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1310_5182_gb300 as lib
    return lib


@pytest.mark.parametrize("p,N,Np", [(2, 1_400_000, 88), (6, 1_100_000, 63), (3, 400_000, 300)])
def test_few_neighbours_of_many_rows_need_no_retry(L, p, N, Np):
    """Uniform rows: the threshold, from every 64th row, collects some 1,200 to
    1,900 of them, give or take 20%.  None of 400 queries overflows the buffer, and
    the neighbours are the CUDA-core path's."""
    g = torch.Generator(device="cuda").manual_seed(p)
    X = torch.rand(N, p, device="cuda", generator=g, dtype=torch.float64) * 4 - 2
    Q = torch.rand(400, p, device="cuda", generator=g, dtype=torch.float64) * 4 - 2
    got = L.lagp_knn(X, Q, Np)
    assert L.knn_stats() == {"retried": 0, "tc_failed": 0}
    L.set_tuning(knn_path=1)
    try:
        ref = L.lagp_knn(X, Q, Np)
    finally:
        L.set_tuning(knn_path=0)
    assert torch.equal(got[0], ref[0]) and torch.equal(got[1], ref[1])
