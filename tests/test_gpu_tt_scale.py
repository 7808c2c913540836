"""TT-rounding of sums so small that the squares of their smaller singular values leave the FP64 range.  Tolerances and
their derivation are those of test_gpu_tt_trees.py: the sum to eps and the cores' orthonormality do not depend on the
scale (the QRs square entries too: below a norm of 1e-150 those lose bits)."""
import numpy as np
import pytest

import test_gpu_tt_trees as T

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
W = T.W


@pytest.mark.parametrize("scale", [1e-149, 1e-148, 1e-145, 1e-120, 2e-148, 1e120, 1e150])
@pytest.mark.parametrize("eps", [1e-9, 1e-4])
def test_small_and_large_sums(W, scale, eps):
    rng = np.random.default_rng(6)
    n = (33, 24, 40)
    x, y = T.tt(rng, n, (12, 10), 3.0, scale), T.tt(rng, n, (5, 4), 1.0, scale)
    one = T.tt(rng, n, (12, 10), 3.0, 1.0)
    (G, _), (H, _) = T.check(W, [[(1.0, x), (0.5, y), (1.0, x)], [(1.0, one)]], eps)
    assert (G[0].shape[2], G[1].shape[2]) == (17, 14) or eps > 1e-9
