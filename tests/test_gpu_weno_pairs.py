"""The FP64 WENO5 value whose weights are formed in FP32 pairs (weno5_slide_pair), through the public API: linear
advection splits with alpha = 1, so f(+) = u, f(-) = 0 and L(u) = -(v_{i+1/2} - v_{i-1/2}) / h with v the WENO5 value
of the cell values themselves.  The reference is the paper's formula in long double.

Tolerance, per cell: v is c plus a combination of differences of at most 2 M each (M the largest magnitude of the
window's points) whose weights sum to at most 2; each of the formula's roundings on the way to v moves it by at most
2^-53 times a term of that size, and fewer than 16 of them do: |error of v| <= 16 2^-53 M, two values per cell.  Terms
below 2^-30 sqrt(4 eps) may carry the pairs' 2^-46 instead; 2^-75 sqrt(4 eps) per value covers them."""
import numpy as np
import pytest

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


def reference(u, eps):
    v = np.concatenate([u[-3:], u, u[:3]]).astype(np.longdouble)
    n = len(u)
    a, b, c, d, e = (v[k:k + n + 1] for k in range(5))  # face j (before cell j): cells j-3 .. j+1
    L = np.longdouble
    b0 = L(13) / 12 * (c - 2 * d + e) ** 2 + L(1) / 4 * (3 * c - 4 * d + e) ** 2
    b1 = L(13) / 12 * (b - 2 * c + d) ** 2 + L(1) / 4 * (b - d) ** 2
    b2 = L(13) / 12 * (a - 2 * b + c) ** 2 + L(1) / 4 * (a - 4 * b + 3 * c) ** 2
    g0, g1, g2 = (x + L(eps) for x in (b0, b1, b2))
    m = np.minimum(np.minimum(g0, g1), g2)
    w0, w1, w2 = 3 * (m / g0) ** 2, 6 * (m / g1) ** 2, (m / g2) ** 2
    x = (w0 * (2 * c + 5 * d - e) + w1 * (-b + 5 * c + 2 * d) + w2 * (2 * a - 7 * b + 11 * c)) / (6 * (w0 + w1 + w2))
    return -(x[1:] - x[:-1]) * n


def field(kind, n, rng):
    x = (np.arange(n) + 0.5) / n
    s = np.sin(2 * np.pi * x + rng.uniform(0, 6))
    return {
        "wave": 1.0 + 0.2 * s,
        "zero mean": 0.3 * s,
        "front": 1.0 + np.tanh((x - 0.4) * n / 4) - np.tanh((x - 0.8) * n / 4),
        "shock": 1.3 + np.tanh((x - 0.4) * n / 0.75) - np.tanh((x - 0.8) * n / 0.75) + 0.1 * s,
        "jumps": np.where(x < 0.3, 1.0, np.where(x < 0.7, 0.0, 1e-3)) + 0.0,
        "noise": rng.uniform(-1, 1, n),
        "round-off": 1.0 + 1e-15 * rng.uniform(-1, 1, n),
        "wide range": 10.0 ** rng.uniform(-12, 12, n),
        "constant": np.full(n, 0.7),
    }[kind]


@pytest.mark.parametrize("scale", [1.0, 1e-30, 1e-9, 1e8, 1e17, 1e25])
@pytest.mark.parametrize("kind", ["wave", "zero mean", "front", "shock", "jumps", "noise", "round-off", "wide range",
                                  "constant"])
@pytest.mark.parametrize("n,eps", [(3, 1e-6), (122, 1e-6), (123, 1e-40), (500, 1e-6), (257, 1e6)])
def test_values_match_long_double(W, n, eps, kind, scale):
    if kind == "wide range" and scale > 1e17:
        pytest.skip("values to 1e37: products of eight differences overflow FP64 in the formula itself")
    rng = np.random.default_rng(n + len(kind))
    u = field(kind, n, rng) * scale
    s = W.Solver(1, (n,), (0.0,), (1.0,), model=W.MODEL_ADVECT, eps_weno=eps)
    U = torch.from_numpy(u.reshape(1, 1, 1, n)).cuda()
    R = torch.empty_like(U)
    s.rhs(U, R)
    s.sync()
    got = R.cpu().numpy().reshape(n)
    s.close()
    want = reference(u, eps)
    v = np.concatenate([u[-3:], u, u[:3]])
    M = np.max([np.abs(v[k:k + n]) for k in range(7)], axis=0)
    assert np.all(np.abs(got - want) <= 2 * (16 * 2.0 ** -53 * M + 2.0 ** -75 * np.sqrt(4 * eps)) * n)
