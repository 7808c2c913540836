"""Grids at the edges of what the FP64 kernels cut into tiles: fewer cells than a tile, tiles of one row, a last tile
of a few cells, rows and columns far longer than a tile, and sizes whose fitted extents differ.  L(U) and one step
against the FP64 oracle, with the tolerances (and their derivation) of the parity tests of the Euler equations and of
the scalar laws."""
import numpy as np
import pytest

import oracle as O
import test_gpu_parity as E
import test_gpu_scalar as S
from paper_2405_12301_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
P, T, R = O.PERIODIC, O.TRANSMISSIVE, O.REFLECTIVE
BC = ((T, R), (P, P), (R, T))
W = E.W


@pytest.mark.parametrize("model", ["euler", "burgers"])
@pytest.mark.parametrize("n", [(3, 3), (4, 70), (9, 17), (16, 16), (17, 33), (100, 5), (257, 31), (512, 300), (3, 3, 3),
                               (8, 9, 70), (70, 4, 5), (33, 17, 11), (97, 6, 22), (128, 5, 3)])
def test_rhs_and_step(W, n, model):
    dim = len(n)
    if model == "euler":
        cfg = O.Cfg(dim=dim, n=n, bc=BC[:dim])
        U = I.random_state(dim, n, seed=40 + sum(n), jumps=True)
        s = E.solver(W, cfg)
        Rref, aref = O.residual(cfg, U)
        tol = E.fp64_rhs_tol(cfg, U, Rref, aref[0])
    else:
        cfg = O.Cfg(dim=dim, n=n, bc=BC[:dim], model=O.BURGERS)
        U = S.scalar_state(dim, n, seed=40 + sum(n))
        s = S.solver(W, cfg)
        Rref, aref = O.residual(cfg, U)
        tol = S.rhs_tol(cfg, U, Rref, aref[0])
    Ud, Rd = E.dev(U), torch.empty(U.shape, dtype=torch.float64, device="cuda")
    s.rhs(Ud, Rd)
    err = np.abs(E.host(Rd) - Rref)
    assert (err <= tol).all(), float((err / tol).max())
    dt = O.cfl_dt(cfg, U, 0.5)
    s.set_time(0.0)
    s.step(Ud)
    assert E.rel_field_err(E.host(Ud), O.ssprk3_step(cfg, U, dt)) <= 1e-12
    s.close()
