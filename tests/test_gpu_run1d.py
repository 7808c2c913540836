"""Small 1D FP64 Euler grids, whose steps run inside one cluster kernel (k_run1d): against the oracle at the sizes where
the split over 8 CTAs of at most 256 cells can go wrong (CTAs without cells, halos that reach past a neighbour, full
CTAs, the first size of the per-stage kernels), for every boundary rule and both alpha modes, and several launches
against one.  Tolerance: 1e-12 per step of the field's scale, the parity bound of one FP64 step."""
import numpy as np
import pytest

import oracle as O
from paper_2405_12301_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

BCS = [((O.PERIODIC, O.PERIODIC),), ((O.TRANSMISSIVE, O.REFLECTIVE),), ((O.REFLECTIVE, O.TRANSMISSIVE),),
       ((O.INFLOW, O.TRANSMISSIVE),), ((O.REFLECTIVE, O.INFLOW),)]


@pytest.fixture(scope="module")
def W():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2405_12301_gb300 import build, weno
    build.build()
    weno.lib()
    return weno


@pytest.mark.parametrize("mode", [O.ALPHA_GLOBAL_NORM, O.ALPHA_PER_DIR])
@pytest.mark.parametrize("bc", BCS)
@pytest.mark.parametrize("n", [3, 7, 8, 9, 17, 100, 255, 256, 257, 1024, 2047, 2048, 2049])
def test_steps_match_oracle(W, n, bc, mode):
    st = [[[1.1, 0.3, 2.6, 0.0, 0.0], [0.9, -0.2, 2.2, 0.0, 0.0]]] + [[[0.0] * 5] * 2] * 2
    bc3 = bc + ((O.PERIODIC, O.PERIODIC),) * 2
    cfg = O.Cfg(dim=1, n=(n,), bc=bc3, alpha_mode=mode, bc_state=[[s[:3] + [0.0, 0.0] for s in d] for d in st])
    U0 = I.random_state(1, (n,), seed=n, jumps=n > 16)
    steps = 5
    U, t = U0, 0.0
    for _ in range(steps):
        dt = O.cfl_dt(cfg, U, 0.4)
        U = O.ssprk3_step(cfg, U, dt)
        t += dt
    outs = []
    for graph_steps in (5, 2, 0):
        s = W.Solver(1, (n,), (0.0,), (1.0,), bc=bc3, cfl=0.4, alpha_mode=mode, bc_state=cfg.bc_state)
        Ud = torch.from_numpy(np.ascontiguousarray(U0)).cuda()
        s.set_time(0.0)
        assert s.run(Ud, 1e9, max_steps=steps, graph_steps=graph_steps) == steps
        tg, taken = s.time()
        assert taken == steps and abs(tg - t) <= 1e-12 * t
        outs.append(Ud.cpu().numpy())
        s.close()
    for f in range(3):
        assert np.abs(outs[0][f] - U[f]).max() <= steps * 1e-12 * max(np.abs(U[f]).max(), 1e-3)
    assert np.array_equal(outs[0], outs[1]) and np.array_equal(outs[0], outs[2])


def test_run_lands_on_t_end_and_stops(W):
    s = W.Solver(1, (64,), (0.0,), (2.0,), cfl=0.5)
    U = torch.from_numpy(I.density_wave(1, (64,))).cuda()
    s.set_time(0.0)
    steps = s.run(U, 0.1, graph_steps=16)
    assert s.time() == (0.1, steps) and steps > 1
    before = U.clone()
    assert s.run(U, 0.1, max_steps=3, graph_steps=4) == 0
    assert torch.equal(U, before)
