"""The MLE's CTA widths and size classes (csrc/gp_fixed.cu) on both sides of
their lines, one size a call and all in one uneven call, with test_gpu_fixed's
bars against the FP64 oracle."""
import numpy as np
import pytest

from test_gpu_fixed import check_mle, designs
from test_gpu_parity import L, O, dev  # noqa: F401  (fixtures)

pytestmark = pytest.mark.gpu

EDGES = [64, 65, 76, 77, 94, 95, 128]


@pytest.mark.parametrize("sizes", [[n] * 4 for n in EDGES] + [EDGES * 2], ids=str)
def test_mle_at_width_edges(L, O, sizes):
    g, n_arr = 1e-3, np.array(sizes, np.int32)
    w, sel = designs(O, 37, g, n_arr)
    n = n_arr if len(set(sizes)) > 1 else sizes[0]
    d0 = np.full(w.M, 1.5)
    check_mle(L.lagp_mle_step(dev(w.X), dev(w.Y), dev(sel), n, d0, g, 1e-3, 20.0, 2),
              O.mle(w.X, w.Y, sel, n, d0, g, 1e-3, 20.0, 2))
