"""Ensembles in every shape the autotuner may choose (ids 0 to 3 tiles, 4 to 7 strips), each set for all members: the
members have every kind of remainder and differ in their sides, and evolve as the same problems alone."""
import numpy as np
import pytest

import hydro_problems as hp
from paper_1306_6883_gb300 import hydro as H

pytestmark = pytest.mark.gpu
NG = 4
TILES = [(32, 16), (16, 16), (32, 8), (32, 16), (88, 16), (120, 16), (56, 16), (88, 32)]


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1306_6883_gb300 import build
    build.build()
    torch.cuda.set_device(0)


def _members():
    return [hp.quad(300, 97, seed=1), hp.kh(177, 48, seed=2), hp.bubble(96, 200), hp.quad(1, 1, seed=3),
            hp.quad(89, 33, seed=4), hp.rt(64, 130), hp.quad(121, 65, seed=5), hp.kh(56, 16, seed=6)]


def _ensemble(precision=1, **kw):
    from paper_1306_6883_gb300.solver import Ensemble, params_for
    return Ensemble([params_for(p, precision, **kw) for p in _members()], [p.U for p in _members()])


@pytest.fixture(scope="module")
def alone():
    from paper_1306_6883_gb300.solver import Solver, params_for
    out = []
    for pr in _members():
        s = Solver(params_for(pr, H.HYDRO_FP32), pr.U)
        s.advance(5)
        out.append((s.interior(), s.time()[0]))
        s.close()
    return out


@pytest.mark.parametrize("shape", range(8))
def test_members_evolve_as_alone_in_every_shape(shape, alone):
    e = _ensemble()
    e.run(1)  # steps before the change, through a graph that it drops
    e.set_shape(shape)
    assert all(c["tile"] == TILES[shape] for c in e.classes())
    e.run(2)
    e.run(2, use_graph=False)
    assert e.status()[0] == 0
    for i, (ref, t_ref) in enumerate(alone):
        got = e.state_numpy(i)[:, NG:-NG, NG:-NG]
        scale = np.abs(ref).max(axis=(1, 2), keepdims=True)
        scale[1:3] = np.maximum(scale[1:3], scale[0])  # momenta that vanish: against rho times a unit sound speed
        # FP32 rounding: the kernels may fuse different multiply-adds
        assert np.all(np.abs(got - ref) <= 2.0 ** -24 * 256 * scale), (i, np.abs(got - ref).max())
        assert e.time(i)[0] == pytest.approx(t_ref, rel=2.0 ** -24 * 16) and e.time(i)[1] == 5
    e.close()


def test_a_shape_that_the_members_do_not_have_is_refused():
    for kw, n in (({}, 8), ({"use_learned_guess": 1}, 4), ({"precision": 0}, 1)):
        e = _ensemble(**kw)
        for bad in (-1, n, 8, 100):
            with pytest.raises(H.HydroError) as err:
                e.set_shape(bad)
            assert err.value.status == H.HYDRO_EINVAL
        e.set_shape(n - 1)
        e.close()
    assert H.load().hydro_batch_set_shape(None, 0) == H.HYDRO_EINVAL
