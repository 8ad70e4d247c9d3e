"""FP64 steps with either tile shape (16x8 where its tiles find an SM each, else 16x16) on ragged grids: bit for
bit the oracle's, through the driver loop's fused and unfused calls."""
import numpy as np
import pytest

import hydro_problems as hp
import oracle
from paper_1306_6883_gb300 import hydro as H
from paper_1306_6883_gb300.solver import Solver, params_for

pytestmark = pytest.mark.gpu


# on 152 SMs: 16x8 for the first two (few tiles; one round of 16x8 tiles against one of 16x16), 16x16 for the
# others (two rounds of 16x8 tiles against one; many rounds)
@pytest.mark.parametrize("nx,ny", [(17, 9), (127, 121), (150, 131), (403, 217)])
@pytest.mark.parametrize("riemann,recon", [("two-shock", "plm"), ("hllc", "ppm")])
def test_tile_shapes_step_like_the_oracle(nx, ny, riemann, recon):
    pr = hp.quad(nx, ny, seed=nx)
    po = oracle.params(nx, ny, bc=pr.bc, gamma=pr.gamma, cfl=pr.cfl, riemann_solver=int(riemann == "hllc"),
                       reconstruction=int(recon == "ppm"))
    U = np.array(pr.U)
    oracle.advance(po, U, nsteps=3)
    for fused in (True, False):
        s = Solver(params_for(pr, riemann_solver=riemann, reconstruction=recon), pr.U)
        if fused:
            s.advance(3)
        else:
            for _ in range(3):
                s.fill_ghost()
                s.step(s.cfl_dt())
        H.hydro_sync_status(s.ctx)
        got = s.interior()
        s.close()
        assert np.array_equal(got, U[:, 4:-4, 4:-4]), (fused, np.abs(got - U[:, 4:-4, 4:-4]).max())
