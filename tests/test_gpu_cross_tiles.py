"""weno_cross_eval at the edges of how k_cross cuts its work: contracted rows of 1 to 32 entries (their pitch and the
columns that fit), one and few fixed indices, fibers shorter than a chunk, of one chunk and of several.  The oracle and
tolerances (with their derivation) are those of test_gpu_cross.py."""
import numpy as np
import pytest

import oracle as O
import test_gpu_cross as X

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
W = X.W


@pytest.mark.parametrize("fp64", [True, False])
@pytest.mark.parametrize("n,r", [([3, 3, 3], [1, 1]), ([5, 40, 6], [1, 9]), ([14, 20, 11], [4, 8]), ([9, 33, 10], [8, 5]),
                                 ([16, 12, 14], [12, 13]), ([24, 10, 37], [17, 32]), ([150, 7, 9], [5, 3]),
                                 ([40, 70, 33], [32, 20]), ([6, 261, 5], [3, 2])])
def test_ranks_and_chunks(W, n, r, fp64):
    inst = X.make_instance(7 + sum(n) + r[0], n, r, (O.TRANSMISSIVE, O.REFLECTIVE))
    h = W.weno_init(None, precision=W.FP64)
    sets, refs = X.make_sets(inst, 0, 60, fp64)
    W.weno_cross_eval(h, [X.dev_instance(inst)], sets, fp64_check=fp64)
    W.weno_sync(h)
    for s, (mode, fd, left, right) in zip(sets, refs):
        ref = X.oracle_out(inst, mode, fd, left, right)
        err = np.abs(s["out"].double().cpu().numpy() - ref)
        tol = X.tol_fp64(ref, inst) if fp64 else X.tol_fp32(inst)
        assert (err <= tol).all(), (mode, fd, float((err / tol).max()))
    W.weno_destroy(h)
