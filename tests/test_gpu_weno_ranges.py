"""The FP64 WENO5 value at the edges of the FP32 pairs' range: a smoothness parameter beyond what an FP32 number's square
holds, and fields far below sqrt(eps), where the weights are the linear ones.  The reference and the tolerance are those
of test_gpu_weno_pairs.py, without its allowance for terms below 2^-30 sqrt(4 eps)."""
import numpy as np
import pytest

import test_gpu_weno_pairs as P

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
W = P.W


def check(W, u, eps):
    n = len(u)
    s = W.Solver(1, (n,), (0.0,), (1.0,), model=W.MODEL_ADVECT, eps_weno=eps)
    U = torch.from_numpy(u.reshape(1, 1, 1, n)).cuda()
    R = torch.empty_like(U)
    s.rhs(U, R)
    s.sync()
    got = R.cpu().numpy().reshape(n)
    s.close()
    v = np.concatenate([u[-3:], u, u[:3]])
    M = np.max([np.abs(v[k:k + n]) for k in range(7)], axis=0)
    err, tol = np.abs(got - P.reference(u, eps)), 2 * 16 * 2.0 ** -53 * M * n
    assert np.all(err <= tol), float((err / tol).max())


@pytest.mark.parametrize("kind", ["wave", "front", "shock", "noise"])
@pytest.mark.parametrize("eps", [1e17, 1e18, 5e18, 1e19, 1e22, 1e30, 1e50])
@pytest.mark.parametrize("over", [0.1, 1.0, 30.0])
def test_large_eps(W, kind, eps, over):
    n = 300
    check(W, P.field(kind, n, np.random.default_rng(n)) * over * np.sqrt(eps), eps)


@pytest.mark.parametrize("kind", ["wave", "zero mean", "front", "shock", "jumps", "noise", "wide range"])
@pytest.mark.parametrize("eps", [1e-6, 1.0, 1e6, 1e-30])
@pytest.mark.parametrize("below", [2.0 ** -25, 2.0 ** -28, 2.0 ** -29, 2.0 ** -30, 2.0 ** -31, 2.0 ** -32, 2.0 ** -34, 2.0 ** -50])
def test_fields_below_sqrt_eps(W, kind, eps, below):
    n = 301
    check(W, P.field(kind, n, np.random.default_rng(n)) * below * np.sqrt(eps), eps)
