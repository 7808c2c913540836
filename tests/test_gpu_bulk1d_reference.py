"""L(U) of long 1D FP32-bulk grids: their rounding errors grow with a point's distance from its tile's reference state, so
a tile may not reach further from it than 122-cell tiles with the reference in their first cell do (124 cells).  The
yardstick is that form's own arithmetic in numpy, rounded to FP32 operation by operation: the GPU's errors against FP64,
their root mean square and their largest, stay within 1.25 times those of the yardstick (fused multiply-adds and the
approximate reciprocals move single roundings, about a tenth of the sum; a reach of twice the length doubles it)."""
import numpy as np
import pytest

import oracle as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
f4 = np.float32
GM1 = 0.4


def weno5(a, b, c, d, e, eps):
    t = a.dtype.type
    D1, D2, D3, D4 = b - a, c - b, d - c, e - d
    t0, t1, t2 = D4 - D3, D3 - D2, D2 - D1
    s0, s1, s2 = D4 - t(3) * D3, D2 + D3, t(3) * D2 - D1
    g = [(t(13 / 12) * x * x + (t(0.25) * y * y + t(eps))) ** 2 for x, y in ((t0, s0), (t1, s1), (t2, s2))]
    w0, w1, w2 = t(0.3) * (g[1] * g[2]), t(0.6) * (g[0] * g[2]), t(0.1) * (g[0] * g[1])
    sw = w0 + w1 + w2
    return c + (w0 * (t1 - t0) - t(2) * w2 * (t1 - t2) + (t(2) * D3 + D2) * sw) / (t(6) * sw)


def yardstick(U, alpha, n, eps, S=122, at=0):
    """L(U) in FP32 on differences from cell `at` of every tile of S cells (periodic)."""
    nt = -(-n // S)
    R = np.empty((3, nt * S), f4)
    idx = np.arange(nt)[:, None] * S + np.arange(-3, S + 3)[None]
    ref = U[:, np.minimum(np.arange(nt) * S + at, n - 1)][:, :, None]
    q, al, gm1 = (U[:, idx % n] - ref).astype(f4), f4(alpha), f4(GM1)
    rho0, m0, E0 = (ref[k].astype(f4) for k in range(3))
    u0 = m0 / rho0
    H0 = E0 + gm1 * (E0 - f4(0.5) * (m0 * u0))
    du = (q[1] - u0 * q[0]) / (rho0 + q[0])
    u = u0 + du
    dp = gm1 * (q[2] - f4(0.5) * (q[1] * u + m0 * du))
    dH = q[2] + dp
    F = [q[1], q[1] * u + m0 * du + dp, du * (H0 + dH) + u0 * dH]
    for f in range(3):
        fp, fm = f4(0.5) * (F[f] + al * q[f]), f4(0.5) * (F[f] - al * q[f])
        face = weno5(*[fp[:, k:k + S + 1] for k in range(5)], eps) + weno5(*[fm[:, k:k + S + 1] for k in (5, 4, 3, 2, 1)], eps)
        R[f] = (-(face[:, 1:] - face[:, :-1]) * f4(n)).reshape(-1)
    return R[:, :n].astype(np.float64)


def test_errors_of_a_long_grid():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2405_12301_gb300 import build, weno as W
    build.build()
    n, eps = 200000, 1e-6
    x = (np.arange(n) + 0.5) / n
    rho, u, p = 1 + 0.2 * np.sin(2 * np.pi * x + 1), 0.7 + 0.2 * np.sin(4 * np.pi * x), 1 + 0.3 * np.cos(2 * np.pi * x)
    U = np.stack([rho, rho * u, p / GM1 + 0.5 * rho * u * u])
    want, alpha = O.residual(O.Cfg(dim=1, n=(n,), eps=eps), U.reshape(3, 1, 1, n))
    want = want.reshape(3, n)
    s = W.Solver(1, (n,), (0.0,), (1.0,), eps_weno=eps, precision=W.FP32_BULK)
    Ud = torch.from_numpy(U.reshape(3, 1, 1, n)).cuda()
    R = torch.empty_like(Ud)
    s.rhs(Ud, R)
    s.sync()
    got = R.cpu().numpy().reshape(3, n)
    s.close()
    ref = yardstick(U, alpha[0], n, eps)
    for f in range(3):
        e, y = got[f] - want[f], ref[f] - want[f]
        assert np.sqrt((e * e).mean()) <= 1.25 * np.sqrt((y * y).mean()) and np.abs(e).max() <= 1.25 * np.abs(y).max()
