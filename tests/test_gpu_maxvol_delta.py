"""maxvol with a delta below what FP32 pairs resolve, on matrices too large for the FP64 swap kernel's size rule.  Rows
and swaps are the oracle's."""
import numpy as np
import pytest

import test_gpu_maxvol_slices as M
from oracle import cross as X

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
W = M.W


@pytest.mark.parametrize("delta", [0.0, 1e-14, 1e-13, 1e-10])
@pytest.mark.parametrize("n,r", [(3000, 64), (9000, 10), (14000, 24)])
def test_small_delta(W, n, r, delta):
    A = M.matrix(n, r, n + r)
    h = W.weno_init()
    (idx, B, swaps), = W.weno_maxvol(h, [torch.from_numpy(A).cuda()], delta=delta, max_iters=400)
    W.weno_destroy(h)
    Io, _, so = X.maxvol(A, delta=max(delta, 1e-13), max_iters=400)
    assert so < 400 and np.array_equal(np.sort(idx.cpu().numpy()), np.sort(Io))
    assert delta == 0.0 or swaps == so
    B = B.cpu().numpy()
    assert np.abs(B).max() <= 1 + max(delta, 1e-13)


@pytest.mark.parametrize("n", [32767, 16383, 16384])
def test_longest_slices(W, n):
    """A rank-1 matrix beside one of rank 64: slices of up to 8192 rows, all that a CTA's row mask holds."""
    M.check(W, [M.matrix(n, 1, 2), M.matrix(64, 64, 3)])
