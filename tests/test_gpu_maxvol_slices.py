"""maxvol at the sizes where the split of a matrix over the cluster's CTAs and over shared memory can go wrong: square
matrices, slices without rows, slices that fit in shared memory and ones that do not, the largest rank, batches whose
CTAs share an SM; with rows swapped after the elimination (FP32-pair updates, then one FP64 product) and none.
Tolerances: the rows and the number of swaps are the oracle's; B = A A[I]^{-1} within 1e-11 of its largest entry (the
matrices' submatrices have condition numbers below 1e3, FP64 products of at most 64 terms)."""
import numpy as np
import pytest

from oracle import cross as X

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def W():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2405_12301_gb300 import build, weno
    build.build()
    weno.lib()
    return weno


def matrix(n, r, seed):
    return np.random.default_rng(seed).normal(size=(n, r))


def check(W, mats, max_iters=200):
    h = W.weno_init()
    outs = W.weno_maxvol(h, [torch.from_numpy(A).cuda() for A in mats], delta=1e-2, max_iters=max_iters)
    swapped = 0
    for A, (idx, B, swaps) in zip(mats, outs):
        Io, Bo, so = X.maxvol(A, delta=1e-2, max_iters=max_iters)
        assert swaps == so and np.array_equal(idx.cpu().numpy(), Io)
        B = B.cpu().numpy()
        assert np.array_equal(B[Io], np.eye(A.shape[1]))
        want = np.linalg.solve(A[Io].T, A.T).T
        assert np.abs(B - want).max() <= 1e-11 * np.abs(want).max()
        swapped += so
    W.weno_destroy(h)
    return swapped


@pytest.mark.parametrize("n,r", [(1, 1), (5, 5), (7, 3), (64, 64), (65, 64), (513, 1), (4097, 48), (3000, 64), (20000, 7), (1365, 48), (1366, 48), (900, 18),
                                 (65536, 8)])
def test_single_matrix(W, n, r):
    check(W, [matrix(n, r, n + r)])


def test_no_swaps_leave_the_elimination_result(W):
    assert check(W, [matrix(300, 6, 1)], max_iters=0) == 0


def test_batch_that_shares_the_sms(W):
    rng = np.random.default_rng(4)
    mats = [matrix(int(rng.integers(40, 6000)), int(rng.integers(2, 40)), k) for k in range(48)]
    assert check(W, mats) > 48
