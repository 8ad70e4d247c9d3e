"""Several solvers at once, each on a stream of its own: every one gets the state it gets alone, and they share the
SMs rather than take turns."""
import time

import numpy as np
import pytest

import hydro_problems as hp

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    t = pytest.importorskip("torch")
    if not t.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1306_6883_gb300 import build
    build.build()
    t.cuda.set_device(0)
    return t


def _solvers(torch, n, precision, nx, ny, **kw):
    from paper_1306_6883_gb300.solver import Solver, params_for
    out = []
    for k in range(n):
        pr = hp.kh(nx, ny, seed=k)
        out.append(Solver(params_for(pr, precision, **kw), pr.U, stream=torch.cuda.Stream()))
    return out


# one to three blocks per SM, tiles of both precisions and sizes, strips, sweeps
@pytest.mark.parametrize("precision,nx,ny,kw", [(0, 128, 128, {}), (0, 64, 40, {"split": 1}), (1, 64, 64, {}),
                                                (1, 256, 256, {}), (1, 384, 384, {}), (1, 1030, 700, {}),
                                                (1, 200, 200, {"split": 1})])
def test_interleaved_solvers_match_their_runs_alone(torch, precision, nx, ny, kw):
    together, alone = _solvers(torch, 3, precision, nx, ny, **kw), _solvers(torch, 3, precision, nx, ny, **kw)
    for _ in range(6):
        for s in together:
            s.advance(2)
    for a, b in zip(together, alone):
        for _ in range(6):
            b.advance(2)
        assert a.time() == b.time()
        np.testing.assert_array_equal(a.interior(), b.interior())
        a.close()
        b.close()


def test_small_solvers_on_their_own_streams_share_the_sms(torch):
    # KH 256^2 has fewer tiles than a GB300 has SMs, and an SM holds three: four solvers cost 1.5 times one (held
    # to one tile per SM, 2.4 times)
    def per_step(n, rounds=50):
        ss = _solvers(torch, n, 1, 256, 256)
        best = 1e9
        for _ in range(8):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            for _ in range(rounds):
                for s in ss:
                    s.advance(4)
            torch.cuda.synchronize()
            best = min(best, time.perf_counter() - t0)
        for s in ss:
            s.close()
        return best

    assert per_step(4) < 2.0 * per_step(1)
