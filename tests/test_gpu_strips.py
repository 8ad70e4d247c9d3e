"""FP32 steps in marching strips (ctu_march.cuh), on grids whose strips and segments have every kind of remainder:
against the oracle's step from the same state within the FP32 step bound, and cut differently (the bands of a host
step against the whole step) bit for bit."""
import numpy as np
import pytest

import hydro_problems as hp
import oracle

pytestmark = pytest.mark.gpu
NG = 4


def _problem(name, nx, ny):
    if name == "walls":  # reflecting x walls, a hydrostatic and a reflecting y wall, gravity
        pr = hp.bubble(nx, ny)
        return hp.Problem("walls", nx, ny, pr.U, ("reflect", "reflect", "hydrostatic", "reflect"), domain=pr.domain,
                          grav=pr.grav)
    return {"kh": lambda: hp.kh(nx, ny, seed=1), "quad": lambda: hp.quad(nx, ny, seed=2)}[name]()


# on 152 SMs the first three run in strips (ragged last strips and segments), the second and fourth with some of the
# options or sides, the others in tiles: too few rows to a segment, or too few tiles
SIZES = [(1030, 700), (317, 951), (100, 5000), (130, 2000), (700, 1100), (120, 130), (1500, 40), (1, 700)]


@pytest.mark.parametrize("nx,ny", SIZES)
@pytest.mark.parametrize("name", ["kh", "quad", "walls"])
@pytest.mark.parametrize("kw", [{}, {"riemann_solver": 1}, {"reconstruction": 1}, {"riemann_solver": 1, "reconstruction": 1},
                                {"limiter": 1, "use_flattening": 0, "cvisc": 0.0}])
def test_a_step_is_the_oracles(nx, ny, name, kw):
    from paper_1306_6883_gb300 import hydro as H
    from paper_1306_6883_gb300.solver import Solver, params_for
    if (name == "kh" and min(nx, ny) < NG) or (name == "walls" and min(nx, ny) < NG):
        pytest.skip("periodic and reflecting sides need four cells")
    pr = _problem(name, nx, ny)
    xmin, xmax, ymin, ymax = pr.domain
    po = oracle.params(nx, ny, bc=pr.bc, gamma=pr.gamma, cfl=pr.cfl, xmin=xmin, xmax=xmax, ymin=ymin, ymax=ymax,
                       grav=pr.grav, **kw)
    for fused in (True, False):
        s = Solver(params_for(pr, H.HYDRO_FP32, **kw), pr.U)
        s.fill_ghost()
        U = s.state_numpy().astype(np.float64)
        dt = s.cfl_dt()
        if fused:
            s.step_fused()
            dt = s.time()[0]
        else:
            s.step(dt)
        H.hydro_sync_status(s.ctx)
        got = s.interior().astype(np.float64)
        s.close()
        oracle.fill_ghost(po, U)
        c = np.sqrt(1.4 * 0.4 * np.abs(U[3] / U[0])).max()  # a sound speed: momenta are measured against rho c too
        oracle.step(po, U, dt)
        ref = U[:, NG:-NG, NG:-NG]
        scale = np.abs(ref).reshape(4, -1).max(axis=1)
        scale[1:3] = np.maximum(scale[1:3], scale[0] * c)
        assert np.all(np.abs(got - ref).reshape(4, -1).max(axis=1) <= 2e-5 * scale), (fused, nx, ny)


@pytest.mark.parametrize("nx,ny", [(1030, 700), (130, 2000), (1500, 1100)])
def test_strips_cut_into_bands_give_the_same_state(nx, ny):
    import torch
    from paper_1306_6883_gb300 import hydro as H
    from paper_1306_6883_gb300.solver import Solver, params_for
    pr = hp.kh(nx, ny, seed=4)
    a, b = (Solver(params_for(pr, H.HYDRO_FP32), pr.U) for _ in range(2))
    host = [torch.from_numpy(np.ascontiguousarray(pr.U)).float().pin_memory() for _ in range(2)]
    for k in range(3):
        a.step_host(host[k % 2], host[(k + 1) % 2], chained=True)
        b.step_fused()
    assert a.time() == b.time()
    np.testing.assert_array_equal(a.interior(), b.interior())
    a.close()
    b.close()


@pytest.mark.parametrize("nx,ny", [(1030, 700), (2100, 1800)])  # in tiles, in strips (sixteen waves of tiles)
@pytest.mark.parametrize("gate", [None, (0.0, 0.0), (40.0, 1e9)])  # default, every face past it, none
def test_learned_strips_hand_their_strong_faces_to_tiles(gate, nx, ny):
    # an untrained network: its proposals change where the iterations start, not what they converge to
    import torch
    from paper_1306_6883_gb300 import hydro as H
    from paper_1306_6883_gb300.solver import Model, Solver, params_for
    pr = hp.quad(nx, ny, seed=7)
    po = oracle.params(pr.nx, pr.ny, bc=pr.bc)
    m = Model(seed=3)
    if gate:
        m.set_gate(*gate)
    host = [torch.from_numpy(np.ascontiguousarray(pr.U)).float().pin_memory() for _ in range(2)]
    solvers = [Solver(params_for(pr, H.HYDRO_FP32, use_learned_guess=1), pr.U) for _ in range(3)]
    for s in solvers:
        H.hydro_set_riemann_model(s.ctx, m.m)
    U = solvers[0].state_numpy().astype(np.float64)
    solvers[0].step_fused()
    solvers[1].step_host(host[0], host[1])  # bands
    dt = solvers[0].time()[0]
    solvers[2].fill_ghost()
    solvers[2].step(dt)
    oracle.fill_ghost(po, U)
    oracle.step(po, U, dt)
    ref = U[:, NG:-NG, NG:-NG]
    scale = np.abs(ref).reshape(4, -1).max(axis=1)[:, None, None]
    got = [s.interior() for s in solvers]
    for s, g in zip(solvers, got):
        st, stats = s.status()
        assert st == 0 and stats[2] == 0
        assert np.all(np.abs(g - ref) <= 2e-5 * scale)
    np.testing.assert_array_equal(got[0], got[1])
    # the work area is left ready for the next step
    for _ in range(3):
        solvers[0].step_fused()
    assert solvers[0].status()[0] == 0 and solvers[0].time()[1] == 4
    for s in solvers:
        s.close()
    m.close()
