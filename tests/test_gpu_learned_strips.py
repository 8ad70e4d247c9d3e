"""Learned steps in strips (ctu_march.cuh, learned_tiles_kernel): which cells are stepped from the network's proposals
is a matter of the faces their update reads, not of how the grid is cut into strips, and the time step and the counters
are those of the cells as they are in the end."""
import numpy as np
import pytest

import hydro_problems as hp

pytestmark = pytest.mark.gpu
NG = 4
# Untrained weights: the start then shows in the last bits of every face past the gate.  None: the default gate.
GATES = [None, (0.1, 0.1)]


@pytest.fixture(scope="module")
def torch():
    t = pytest.importorskip("torch")
    if not t.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1306_6883_gb300 import build
    build.build()
    t.cuda.set_device(0)
    return t


def _noisy_blast(nx, ny):
    pr = hp.kh(nx, ny, seed=11)
    rng = np.random.default_rng(5)
    x = (np.arange(nx) + 0.5) / nx
    y = (np.arange(ny) + 0.5) / ny
    r2 = (x[None, :] - 0.4) ** 2 + (y[:, None] - 0.55) ** 2
    U = pr.U
    inner = U[:, NG:-NG, NG:-NG]
    inner[:] *= 1.0 + 0.02 * rng.random((ny, nx))
    inner[3] *= np.where(r2 < 0.05 ** 2, 30.0, 1.0)
    return pr


def _evolved(torch, nx, ny):
    from paper_1306_6883_gb300 import hydro as H
    from paper_1306_6883_gb300.solver import Solver, params_for
    pr = _noisy_blast(nx, ny)
    s = Solver(params_for(pr, H.HYDRO_FP32), pr.U)
    s.advance(60)
    assert s.status()[0] == 0
    U = s.state_numpy()
    s.close()
    return pr, U


@pytest.mark.parametrize("gate", GATES + [False])  # False: no network
@pytest.mark.parametrize("nx,ny", [(2100, 1800), (3001, 1500)])  # strips: sixteen waves of tiles and more
def test_bands_and_whole_steps_agree_in_evolved_flow(torch, gate, nx, ny):
    from paper_1306_6883_gb300 import hydro as H
    from paper_1306_6883_gb300.solver import Model, Solver, params_for
    pr, U = _evolved(torch, nx, ny)
    m = Model(seed=3)
    if gate:
        m.set_gate(*gate)
    learned = gate is not False
    a, b, c = (Solver(params_for(pr, H.HYDRO_FP32, use_learned_guess=int(learned)), U) for _ in range(3))
    if learned:
        for s in (a, b, c):
            H.hydro_set_riemann_model(s.ctx, m.m)
    ha, hb = ([torch.from_numpy(np.ascontiguousarray(U)).pin_memory() for _ in range(2)] for _ in range(2))
    t = 0.0
    for k in range(4):
        dt = c.cfl_dt()
        a.step_host(ha[k % 2], ha[(k + 1) % 2], chained=True)
        b.step_host(hb[k % 2], hb[(k + 1) % 2])
        c.step_fused()
        t += dt  # each time step is the CFL condition of the state it starts from
        assert a.time()[0] == b.time()[0] == c.time()[0] == t
        got = [s.interior() for s in (a, b, c)]
        np.testing.assert_array_equal(got[0], got[2])
        np.testing.assert_array_equal(got[1], got[2])
    for s in (a, b, c):
        st, stats = s.status()
        assert st == 0 and stats[2] == 0
        s.close()
    m.close()


# (0, 0): every face is past the gate, and the strips leave all that one iteration does not solve
@pytest.mark.parametrize("gate", GATES + [(0.0, 0.0)])
@pytest.mark.parametrize("fused", [True, False])
def test_no_cell_keeps_what_a_strip_left_unsolved(torch, gate, fused):
    from paper_1306_6883_gb300 import hydro as H
    from paper_1306_6883_gb300.solver import Model, Solver, params_for
    pr, U = _evolved(torch, 2100, 1800)
    m = Model(seed=3)
    if gate:
        m.set_gate(*gate)
    a, b = (Solver(params_for(pr, H.HYDRO_FP32, use_learned_guess=k), U) for k in (1, 0))
    H.hydro_set_riemann_model(a.ctx, m.m)
    for _ in range(2):
        b.set_state(a.state_numpy())
        dt = a.cfl_dt()
        for s in (a, b):
            s.fill_ghost()
            s.step_fused() if fused else s.step(dt)
        got, ref = a.interior(), b.interior()
        scale = np.abs(ref).reshape(4, -1).max(axis=1)[:, None, None]
        assert np.all(np.abs(got - ref) <= 4e-5 * scale)  # twice the FP32 step bound against the oracle
        st, stats = a.status()
        assert st == 0 and stats[2] == 0
    assert a.time() == b.time() or not fused
    a.close()
    b.close()
    m.close()


def test_a_cell_stepped_by_both_launches_counts_once(torch):
    # the blast lists half a percent of the tiles; a tile solves a tenth more faces per cell than a strip
    from paper_1306_6883_gb300 import hydro as H
    from paper_1306_6883_gb300.solver import Model, Solver, params_for
    pr, U = _evolved(torch, 2100, 1800)
    m = Model(seed=3)
    counts = []
    for learned, gate, maxiter in ((0, None, 16), (1, (40.0, 1e9), 16), (1, (0.35, 1.0), 16), (1, (0.35, 1.0), 300)):
        s = Solver(params_for(pr, H.HYDRO_FP32, use_learned_guess=learned, riemann_maxiter=maxiter), U)
        if learned:
            m.set_gate(*gate)
            H.hydro_set_riemann_model(s.ctx, m.m)
        s.step_fused()
        counts.append(s.status()[1])
        s.close()
    assert counts[0] == counts[1]  # nothing listed
    assert counts[2] == counts[3]  # two ways of summing a warp's iterations, by how many there can be
    assert counts[0][0] < counts[2][0] < 1.001 * counts[0][0]
    m.close()
