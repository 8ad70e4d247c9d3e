"""Steps by the kernel that a grid reaches, asked from the library: TMA and plain tile loads give the same bits, and
strips take the same steps as the oracle and as the bands of a host step, on sizes far from the rule's line."""
import numpy as np
import pytest

import hydro_problems as hp
import oracle

pytestmark = pytest.mark.gpu
NG = 4


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1306_6883_gb300 import build
    build.build()
    torch.cuda.set_device(0)


# 32x16 tiles with interior ones (loaded by TMA when ng = 4, cell by cell when ng = 6), ragged on both sides
@pytest.mark.parametrize("nx,ny", [(420, 380), (333, 333)])
@pytest.mark.parametrize("kw", [{}, {"riemann_solver": 1}, {"reconstruction": 1}])
def test_tma_and_plain_tile_loads_give_the_same_bits(nx, ny, kw):
    from paper_1306_6883_gb300 import hydro as H
    from paper_1306_6883_gb300.solver import Solver, params_for
    pr = hp.kh(nx, ny, seed=3)
    inner = pr.U[:, NG:-NG, NG:-NG]
    for fused in (True, False):
        outs = []
        for ng in (4, 6):
            p = params_for(pr, H.HYDRO_FP32, **kw)
            p.ng = ng
            U = np.zeros((4, ny + 2 * ng, nx + 2 * ng))
            U[:, ng:-ng, ng:-ng] = inner
            s = Solver(p, U)
            assert H.hydro_step_cut(s.ctx) == ("tiles", 32, 16)
            assert H.hydro_tma_enabled(s.ctx) == (ng == 4)
            if fused:
                s.advance(5)
            else:
                for _ in range(5):
                    s.fill_ghost()
                    s.step(s.cfl_dt())
            assert s.status()[0] == 0
            outs.append(s.state_numpy()[:, ng:-ng, ng:-ng])
            s.close()
        np.testing.assert_array_equal(outs[0], outs[1])


# ragged strips and segments: one, few and many strips, segments of 16 to 64 rows
@pytest.mark.parametrize("nx,ny", [(1030, 1400), (100, 9000), (2050, 900)])
@pytest.mark.parametrize("kw", [{}, {"riemann_solver": 1}, {"reconstruction": 1}, {"riemann_solver": 1, "reconstruction": 1}])
def test_strips_step_like_the_oracle_and_like_their_bands(nx, ny, kw):
    import torch
    from paper_1306_6883_gb300 import hydro as H
    from paper_1306_6883_gb300.solver import Solver, params_for
    pr = hp.kh(nx, ny, seed=4)
    a, b = (Solver(params_for(pr, H.HYDRO_FP32, **kw), pr.U) for _ in range(2))
    assert H.hydro_step_cut(a.ctx)[0] == "strips"
    host = [torch.from_numpy(np.ascontiguousarray(pr.U)).float().pin_memory() for _ in range(2)]
    for k in range(3):
        a.step_host(host[k % 2], host[(k + 1) % 2], chained=True)
        b.step_fused()
        assert a.time() == b.time()
        np.testing.assert_array_equal(a.interior(), b.interior())
    b.fill_ghost()
    U = b.state_numpy().astype(np.float64)
    dt = b.cfl_dt()
    b.step(dt)
    got = b.interior()
    assert b.status()[0] == 0
    po = oracle.params(nx, ny, bc=pr.bc, gamma=pr.gamma, cfl=pr.cfl, **kw)
    oracle.fill_ghost(po, U)
    oracle.step(po, U, dt)
    ref = U[:, NG:-NG, NG:-NG]
    c = np.sqrt(1.4 * 0.4 * np.abs(ref[3] / ref[0])).max()
    scale = np.abs(ref).reshape(4, -1).max(axis=1)
    scale[1:3] = np.maximum(scale[1:3], scale[0] * c)  # momenta are measured against rho c too
    assert np.all(np.abs(got - ref).reshape(4, -1).max(axis=1) <= 2e-5 * scale)
    a.close()
    b.close()


@pytest.mark.parametrize("precision,nx,ny,cut", [(0, 64, 64, (16, 8)), (0, 1024, 1024, (16, 16)), (1, 64, 64, (16, 8)),
                                                 (1, 384, 384, (32, 16))])
def test_small_grids_run_in_small_tiles(precision, nx, ny, cut):
    from paper_1306_6883_gb300 import hydro as H
    from paper_1306_6883_gb300.solver import Solver, params_for
    pr = hp.kh(nx, ny)
    s = Solver(params_for(pr, precision), pr.U)
    assert H.hydro_step_cut(s.ctx) == ("tiles",) + cut
    s.close()
    t = Solver(params_for(pr, precision, split=1), pr.U)
    with pytest.raises(H.HydroError):
        H.hydro_step_cut(t.ctx)
    t.close()
    assert H.load().hydro_step_cut(None, None, None, None) == H.HYDRO_EINVAL
