"""The candidate chunks of the FP32-bulk and FP64 Schur searches
(csrc/alc_bulk32.cu, csrc/alc_schur64.cu): sets that end
at the edges of the chunks and half chunks of the widest layout, against the
same location alone with its set as the largest (another layout, the same
arithmetic a candidate: the same bits), and against the FP64 oracle."""
import numpy as np
import pytest
import torch

import workloads as W
from test_gpu_parity import L, O, compare_selection, dev  # noqa: F401  (fixtures)

pytestmark = pytest.mark.gpu

NP = np.array([60, 127, 511, 512, 513, 1023, 1024, 1025, 1535, 1536, 1537, 2047, 2048], np.int32)


@pytest.mark.parametrize("prec,rep", [("f32bulk", 1), ("f32bulk", 13), ("f64schur", 1)])  # 13: two CTAs an SM
def test_sets_ending_at_chunk_edges(L, O, prec, rep):
    g, d, n = 1e-4, 2.0, 14
    w = W.borehole(seed=39, N=6_000, M=len(NP), n=n, Np=int(NP.max()), g=g)
    idx = O.knn(w.X, w.Xref, int(NP.max()))
    idx = np.where(np.arange(NP.max())[None] < NP[:, None], idx, -1).astype(np.int32)
    tile = lambda a: np.ascontiguousarray(np.tile(a, (rep,) + (1,) * (a.ndim - 1)))
    run = lambda Q, i, Np: L.lagp_alc_predict(dev(w.X), dev(w.Y), dev(Q), dev(i), 6, n, d, g, prec=prec,
                                              Nprime=Np, want_alc=True)
    out = run(tile(w.Xref), tile(idx), tile(NP))
    keys = ("sel", "alc", "mean", "s2", "status")
    for m, k in enumerate(NP):
        one = run(w.Xref[m:m + 1].copy(), idx[m:m + 1, :k].copy(), NP[m:m + 1])
        for key in keys:
            assert torch.equal(torch.nan_to_num(out[key][m::len(NP)]),
                               torch.nan_to_num(one[key]).expand_as(out[key][m::len(NP)])), (key, k)
    n_arr = np.full(len(NP), n, np.int32)
    ref = O.alc_select(w.X, w.Xref, idx, 6, n_arr, d, g, topk=4, Np=NP)
    compare_selection(out["sel"].cpu().numpy()[:len(NP)], ref, n_arr, 6, g)
