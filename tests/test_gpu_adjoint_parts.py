"""The parts of the adjoint and of the MLE step that the autograd functions
ask for alone, against the full calls."""
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


def case(n, M=37, p=3, N=500):
    rng = np.random.default_rng(53)
    X = torch.from_numpy(rng.uniform(size=(N, p))).cuda()
    Y = torch.sin(3.0 * X).sum(1)
    Q = torch.from_numpy(rng.uniform(size=(M, p))).cuda()
    sel = torch.from_numpy(np.stack([rng.permutation(N)[:n] for _ in range(M)]).astype(np.int32)).cuda()
    sizes = torch.from_numpy(rng.integers(2, n + 1, M).astype(np.int32)).cuda()
    return X, Y, Q, sel, sizes


@pytest.mark.parametrize("n", [2, 33, 50, 129])
def test_parts_equal_the_full_adjoint(L, n):
    X, Y, Q, sel, sizes = case(n)
    full = L.lagp_predict_grad(X, Y, Q, sel, sizes, 0.7, 1e-2)
    for keys in (L.lagp._GRADS[:4], L.lagp._GRADS[4:], L.lagp._GRADS[1:2]):
        part = L.lagp._predict_grad(X, Y, Q, sel, sizes, 0.7, 1e-2, keys)
        assert torch.equal(part["status"], full["status"])
        for k in keys:
            # two FP64 solutions with K (condition below n / g): n cond(K) 2^-53 < 2e-10 of the largest
            assert (part[k] - full[k]).abs().max() <= 2e-10 * full[k].abs().max().clamp_min(1e-300), k


@pytest.mark.parametrize("n", [2, 40, 41, 100, 129])
def test_value_alone_equals_the_mle_step(L, n):
    X, Y, Q, sel, sizes = case(n)
    full = L.lagp_mle_step(X, Y, sel, sizes, 0.7, 1e-2, 1e-3, 10.0, 0)
    part = L.lagp._mle_step(X, Y, sel, sizes, 0.7, 1e-2, 1e-3, 10.0, 0, ("llik",))
    assert torch.equal(part["status"], full["status"])
    assert torch.equal(part["llik"], full["llik"])  # the same factor, the same sums
