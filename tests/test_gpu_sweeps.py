"""FP32 sweeps of the dimensionally split step (sweep_march.cuh): one step in either order against the oracle's from the
same state within the FP32 step bound, and the oracle's count of solves, on grids with every remainder of the pieces
(chunks of 56 cells, pairs of rows, segments) and with an odd number of ghost cells (unaligned pairs)."""
import numpy as np
import pytest

import hydro_problems as hp
import oracle
from paper_1306_6883_gb300 import hydro as H
from paper_1306_6883_gb300.solver import Solver, params_for

pytestmark = pytest.mark.gpu


def _problem(name, nx, ny, ng):
    rng = np.random.default_rng(nx + 7 * ny)
    shape = (ny, nx)
    bc = {"periodic": ("periodic",) * 4, "outflow": ("outflow",) * 4,
          "walls": ("reflect", "outflow", "hydrostatic", "reflect")}[name]
    U = hp._pack(1.0 + 0.5 * rng.random(shape), rng.uniform(-0.5, 0.5, shape), rng.uniform(-0.5, 0.5, shape),
                 1.0 + rng.random(shape), 1.4, ng)
    return hp.Problem(name, nx, ny, U, bc, ng=ng, grav=-1.0 if name == "walls" else 0.0)


@pytest.mark.parametrize("nx,ny,ng", [(1, 1, 4), (5, 4, 4), (55, 7, 4), (57, 64, 4), (112, 33, 5), (201, 131, 4),
                                      (1030, 41, 4), (6, 900, 5), (700, 500, 4)])
@pytest.mark.parametrize("name", ["periodic", "outflow", "walls"])
@pytest.mark.parametrize("kw", [{}, {"riemann_solver": 1}, {"reconstruction": 1}, {"riemann_solver": 1, "reconstruction": 1},
                                {"limiter": 1, "use_flattening": 0, "cvisc": 0.0}])
def test_a_split_step_is_the_oracles(nx, ny, ng, name, kw):
    if name != "outflow" and min(nx, ny) < ng:
        pytest.skip("periodic and reflecting sides need as many cells as ghost cells")
    pr = _problem(name, nx, ny, ng)
    po = oracle.params(nx, ny, ng=ng, bc=pr.bc, gamma=pr.gamma, cfl=pr.cfl, grav=pr.grav, **kw)
    for fused in (True, False):
        s = Solver(params_for(pr, H.HYDRO_FP32, split=1, **kw), pr.U)
        for first in (0, 1):
            s.fill_ghost()
            U = s.state_numpy().astype(np.float64)
            t0, solves0, dt = s.time()[0], s.status()[1][0], s.cfl_dt()
            if fused:
                s.step_fused()
                dt = s.time()[0] - t0
            else:
                s.step(dt)
            got = s.interior().astype(np.float64)
            assert s.status()[1][0] - solves0 == (nx + 1) * ny + nx * (ny + 1)
            oracle.fill_ghost(po, U)
            c = np.sqrt(1.4 * 0.4 * np.abs(U[3] / U[0])).max()  # momenta are measured against rho c too
            oracle.step_split(po, U, dt, first)
            ref = U[:, ng:-ng, ng:-ng]
            scale = np.abs(ref).reshape(4, -1).max(axis=1)
            scale[1:3] = np.maximum(scale[1:3], scale[0] * c)
            err = np.abs(got - ref).reshape(4, -1).max(axis=1)
            assert np.all(err <= 2e-5 * scale), (fused, first, err / scale)
        s.close()
