"""FP32-bulk search in steps with a single contender, where its two warp groups
run side by side between two barriers: repeated searches give the same bits,
and the designs are those of the FP64 form."""
import numpy as np
import pytest
import torch

import workloads as W
from test_gpu_parity import L, O, compare_selection, dev  # noqa: F401  (fixtures)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M", [40, 1300])  # a CTA an SM with the wide group; four CTAs an SM
def test_single_contender_steps_repeat(L, O, M):
    n, g = 40, 1e-4
    w = W.borehole(seed=61, N=20_000, M=M, n=n, Np=600, g=g)
    idx = O.knn(w.X, w.Xref, 600).astype(np.int32)
    X, Y, Xr, ix = dev(w.X), dev(w.Y), dev(w.Xref), dev(idx)
    L.alc_work(X.device)
    runs = [L.lagp_alc_predict(X, Y, Xr, ix, 6, n, w.d, g, prec="f32bulk", want_alc=True) for _ in range(30)]
    work = L.alc_work(X.device)
    assert work["rescored"] < 2 * work["locations"] * n  # (single contenders are the rule)
    for r in runs[1:]:
        for k in ("sel", "alc", "mean", "s2", "status"):
            assert torch.equal(torch.nan_to_num(r[k]), torch.nan_to_num(runs[0][k])), k
    first = slice(0, 40)
    ref = O.alc_select(w.X, w.Xref[first], idx[first], 6, n, w.d, g, topk=4)
    assert (runs[0]["status"] == 0).all()
    compare_selection(runs[0]["sel"][first].cpu().numpy(), ref, np.full(40, n, np.int32), 6, g)
