"""FP32 steps in the small tile (16x8, while all of a grid's tiles run at once) and in the large one, on ragged grids
on both sides of the rule: against the oracle's step from the same state within the FP32 step bound."""
import numpy as np
import pytest

import hydro_problems as hp
import oracle
from paper_1306_6883_gb300 import hydro as H
from paper_1306_6883_gb300.solver import Solver, params_for

pytestmark = pytest.mark.gpu
NG = 4


# on 152 SMs: 1, 4, 18, 128 and 456 tiles of 16x8 (the most), then 475 (32x16 tiles)
@pytest.mark.parametrize("nx,ny", [(1, 1), (17, 9), (47, 41), (128, 128), (300, 190), (300, 193)])
@pytest.mark.parametrize("kw", [{}, {"riemann_solver": 1}, {"reconstruction": 1}, {"riemann_solver": 1, "reconstruction": 1}])
def test_tile_shapes_step_like_the_oracle(nx, ny, kw):
    pr = hp.quad(nx, ny, seed=nx)
    xmin, xmax, ymin, ymax = pr.domain
    po = oracle.params(nx, ny, bc=pr.bc, gamma=pr.gamma, cfl=pr.cfl, xmin=xmin, xmax=xmax, ymin=ymin, ymax=ymax, **kw)
    for fused in (True, False):
        s = Solver(params_for(pr, H.HYDRO_FP32, **kw), pr.U)
        s.advance(3)  # consecutive steps, each launched ahead of the end of the one before
        s.fill_ghost()
        U = s.state_numpy().astype(np.float64)
        dt = s.cfl_dt()
        if fused:
            t0 = s.time()[0]
            s.step_fused()
            dt = s.time()[0] - t0
        else:
            s.step(dt)
        H.hydro_sync_status(s.ctx)
        got = s.interior().astype(np.float64)
        s.close()
        oracle.fill_ghost(po, U)
        c = np.sqrt(1.4 * 0.4 * np.abs(U[3] / U[0])).max()  # momenta are measured against rho c too
        oracle.step(po, U, dt)
        ref = U[:, NG:-NG, NG:-NG]
        scale = np.abs(ref).reshape(4, -1).max(axis=1)
        scale[1:3] = np.maximum(scale[1:3], scale[0] * c)
        assert np.all(np.abs(got - ref).reshape(4, -1).max(axis=1) <= 2e-5 * scale), (fused, nx, ny)
