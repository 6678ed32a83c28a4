"""The kNN's check that the rows collected on the tensor cores hold the exact
neighbours (csrc/knn.cu), for queries that its rank leaves to the general sort
because many rows lie at nearly the same distance."""
import math

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


def widened(tau, p, K, B):
    """The collection's threshold for a sampled threshold (knn_common.cuh)."""
    u = 2.0 ** -24 * (1 + 2.0 ** -27)
    S, gp, e2 = 2.0 ** math.frexp(B)[1], p * u / (1 - p * u), 2 * u * B * math.sqrt(p)
    E = S * S * (4 * p * 2.0 ** -21 + 2 * (gp * p + 2.0 ** -22 * p + 2.0 ** -25) + 4 * p * 1.5 * 2.0 ** -22 + 2.0 ** -25 +
                 64 * (K // 16) * 2.0 ** -24 * 8 * p * (1 + 2.0 ** -9))
    r_col = math.sqrt(tau + 2 * E + E) + 2 * e2
    return r_col * r_col + E


@pytest.mark.parametrize("p", [3, 8])
def test_sampled_threshold_falls_short_with_many_rows_at_one_distance(L, p):
    """Every 25th row is the sample.  Around each of 24 locations lie the 22
    sampled rows that set its threshold, 38 further rows and a shell of 400 rows
    at one distance, 1e-9 apart, so close to the widened threshold that rounding
    on the tensor cores collects a part of them: the 100 nearest are then not
    all among the rows collected, although there are enough of them.  The shells
    of the locations step through the threshold; the CUDA-core path uses none of
    this."""
    rng = np.random.default_rng(71 + p)
    N, M, k, stride, r0, K = 20_000, 24, 100, 25, 0.05, -(-(3 * p + 4) // 16) * 16
    B = 0.999
    unit = lambda m: (v := rng.normal(size=(m, p))) / np.linalg.norm(v, axis=1)[:, None]
    X = rng.choice([-1.0, 1.0], size=(N, p)) * rng.uniform(0.9, B, size=(N, p))  # corners: far from every location
    X[1], X[2] = B, -B  # centre 0, half-width B
    Q = rng.uniform(-0.4, 0.4, size=(M, p))
    while True:  # locations apart
        D = np.linalg.norm(Q[:, None] - Q[None], axis=2) + 9 * np.eye(M)
        bad = np.flatnonzero(D.min(1) < 4 * r0)
        if not len(bad):
            break
        Q[bad[0]] = rng.uniform(-0.4, 0.4, size=p)
    # r0^2 in the middle of a bin of the threshold's bits [30:11]
    bits = np.float32(r0 * r0).view(np.uint32) >> 11
    mid, top = (np.uint32(bits << 11 | low).view(np.float32) for low in (1024, 2047))
    tau2 = widened(float(top), p, K, B * (1 + 2.0 ** -50))
    sampled = rng.permutation(np.arange(0, N, stride))[:M * 22].reshape(M, 22)
    other = rng.permutation(np.setdiff1d(np.arange(3, N), np.arange(0, N, stride)))[:M * 438].reshape(M, 438)
    for m in range(M):
        rad = np.sqrt(float(mid)) * np.append(rng.uniform(0.3, 0.9, 21), 1.0)
        X[sampled[m]] = Q[m] + rad[:, None] * unit(22)
        X[other[m, :38]] = Q[m] + r0 * rng.uniform(0.3, 0.9, (38, 1)) * unit(38)
        shell = math.sqrt(tau2 + (m - M // 2) * 6e-8) + 1e-9 * np.arange(400) / 400
        X[other[m, 38:]] = Q[m] + shell[:, None] * unit(400)
    Xd, Qd = torch.from_numpy(X).cuda(), torch.from_numpy(Q).cuda()
    got = L.lagp_knn(Xd, Qd, k)
    L.set_tuning(knn_path=1)
    try:
        ref = L.lagp_knn(Xd, Qd, k)
    finally:
        L.set_tuning(knn_path=0)
    exact = np.argsort(((X[None] - Q[:, None]) ** 2).sum(-1), axis=1, kind="stable")[:, :k]
    assert np.array_equal(np.sort(ref[0].cpu().numpy(), 1), np.sort(exact, 1))
    assert torch.equal(got[1], ref[1])
    assert torch.equal(got[0], ref[0])
