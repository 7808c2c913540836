"""alpha where the FP32 estimates that pick the cells whose FP64 speeds are formed could mislead: gases with gamma near 1,
where gamma - 1 has few bits in FP32 once 1 has been taken from an FP32 gamma, and states whose speeds are so small that
their squares leave the FP32 range.  Fast cold cells and slow hot cells of nearly the same speed compete for the
maximum; alpha is the oracle's, bit for bit, of the state given and (through dt) of the one a step leaves.  FP32-bulk:
within 2^-18 (its speeds are sums of FP32 roundings of a few ulp)."""
import numpy as np
import pytest

import oracle as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
SHAPES = [(2100,), (61,), (40, 33), (14, 11, 12)]


@pytest.fixture(scope="module")
def W():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2405_12301_gb300 import build, weno
    build.build()
    weno.lib()
    return weno


def state(rng, n, gamma, rho0=1.0, speed=1.0):
    """Cells of |u| + a = 1.3 speed: at rest relative to their sound, or cold and fast; one of each stands out by up to
    2^-10, in either order."""
    dim, m = len(n), int(np.prod(n))
    hot = rng.random(m) < 0.5
    hot[:2] = True, False
    a, v = np.where(hot, 1.0, 0.3), np.where(hot, 0.3, 1.0)
    f = np.full(m, 1.0 - 2.0 ** -9)
    f[:2] = 1.0, 1.0 + rng.choice([-1, 1]) * 2.0 ** rng.uniform(-18, -10)
    a, v = a * f * speed, v * f * speed
    p = rng.permutation(m)
    a, v = a[p], v[p]
    d = rng.normal(size=(dim, m))
    u = v * d / np.sqrt((d * d).sum(0))
    rho = rho0 * rng.uniform(0.8, 1.2, m)
    E = rho * a * a / (gamma * (gamma - 1.0)) + 0.5 * rho * (u * u).sum(0)
    return np.ascontiguousarray(np.concatenate([rho[None], rho * u, E[None]]).reshape((dim + 2,) + (1,) * (3 - dim) + n[::-1]))


def alpha_of(s, U):
    out = torch.empty(1, dtype=torch.float64, device="cuda")
    s.alpha(torch.from_numpy(U).cuda(), out)
    s.sync()
    return float(out.cpu()[0])


def solver(W, n, gamma, **kw):
    return W.Solver(len(n), n, (0.0,) * len(n), (1.0,) * len(n), gamma=gamma, **kw)


@pytest.mark.parametrize("gamma", [1.4, 1.01, 1.001, 1.0001, 1.00001, 1 + 1e-8])
@pytest.mark.parametrize("n", SHAPES)
def test_gamma_near_one(W, n, gamma):
    rng = np.random.default_rng(len(n))
    cfg = O.Cfg(dim=len(n), n=n, gamma=gamma)
    s = solver(W, n, gamma)
    for _ in range(24):
        U = state(rng, n, gamma)
        assert alpha_of(s, U) == O.alpha(cfg, U)[0]
    s.close()


@pytest.mark.parametrize("gamma", [1.4, 1.01, 1.001, 1.0001, 1.00001, 1 + 1e-8])
@pytest.mark.parametrize("n", SHAPES)
def test_gamma_near_one_fp32_bulk(W, n, gamma):
    rng = np.random.default_rng(len(n))
    cfg = O.Cfg(dim=len(n), n=n, gamma=gamma)
    h, cfl = 1.0 / max(n), 1e-9
    s = solver(W, n, gamma, precision=W.FP32_BULK, cfl=cfl)
    for _ in range(24):
        U = state(rng, n, gamma)
        want = O.alpha(cfg, U)[0]
        assert abs(alpha_of(s, U) - want) <= 2.0 ** -18 * want
    if gamma < 1.001:  # (the jumps of E, ~1 / (gamma - 1), to the eighth power leave the FP32 range of the weights)
        return s.close()
    t, Ud = [], [torch.from_numpy(U).cuda() for _ in range(2)]
    for k in range(2):  # and of the state a step leaves, through the second step's dt
        s.set_time(0.0)
        s.run(Ud[k], 1e30, max_steps=k + 1, graph_steps=k + 1)
        t.append(s.time()[0])
    want = O.alpha(cfg, Ud[0].cpu().numpy())[0]
    assert abs(cfl * h / (t[1] - t[0]) - want) <= 2.0 ** -18 * want
    s.close()


@pytest.mark.parametrize("mode", [O.ALPHA_GLOBAL_NORM, O.ALPHA_PER_DIR])
@pytest.mark.parametrize("gamma", [1.4, 1.00001, 1 + 1e-8])
@pytest.mark.parametrize("n", SHAPES)
def test_alpha_of_the_state_a_step_leaves(W, n, gamma, mode):
    """weno_run takes the second step's dt from the first step's last stage.  (dt 1e-9 of a cell's crossing: the state
    keeps its competing cells.)"""
    rng = np.random.default_rng(7 + len(n))
    cfg = O.Cfg(dim=len(n), n=n, gamma=gamma)
    h, cfl = 1.0 / max(n), 1e-9
    for _ in range(6):
        U = torch.from_numpy(state(rng, n, gamma)).cuda()
        s, V = solver(W, n, gamma, cfl=cfl, alpha_mode=mode), U.clone()
        s.set_time(0.0)
        s.run(V, 1e30, max_steps=1, graph_steps=1)
        t1 = s.time()[0]
        assert t1 == cfl * h / O.alpha(cfg, U.cpu().numpy())[0]
        s.set_time(0.0)
        s.run(U, 1e30, max_steps=2, graph_steps=2)
        assert s.time()[0] == t1 + cfl * h / O.alpha(cfg, V.cpu().numpy())[0]
        s.close()


@pytest.mark.parametrize("rho,speed", [(1e10, 1e-20), (1e6, 1e-19), (1.0, 1e-15), (1e-14, 1e-13), (1e-20, 1.0), (1e20, 1e12)])
@pytest.mark.parametrize("n", SHAPES)
def test_speeds_far_from_one(W, n, rho, speed):
    rng = np.random.default_rng(3 + len(n))
    cfg = O.Cfg(dim=len(n), n=n)
    s = solver(W, n, 1.4)
    for _ in range(12):
        U = state(rng, n, 1.4, rho, speed)
        assert alpha_of(s, U) == O.alpha(cfg, U)[0]
    s.close()
