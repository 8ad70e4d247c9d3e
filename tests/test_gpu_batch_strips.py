"""Ensembles in strips (batch_march_kernel): every shape the autotuner may choose, on members whose strips and segments
have every kind of remainder and that differ in their sides, against the same problems stepped alone."""
import numpy as np
import pytest

import hydro_problems as hp
from paper_1306_6883_gb300 import hydro as H
from paper_1306_6883_gb300.solver import Ensemble, Solver, params_for

pytestmark = pytest.mark.gpu
NG = 4


def _members():
    return [hp.quad(300, 97, seed=1), hp.kh(177, 48, seed=2), hp.bubble(96, 200), hp.quad(1, 1, seed=3),
            hp.quad(89, 33, seed=4), hp.rt(64, 130), hp.quad(300, 97, seed=5), hp.kh(900, 700, seed=6)]


def test_a_tuned_ensemble_of_mixed_sizes_evolves_as_its_members_alone():
    probs = _members()
    seen = set()
    for n in (2, 5, 8):  # the tuner's choice depends on what runs together
        e = Ensemble([params_for(p, H.HYDRO_FP32) for p in probs[:n]], [p.U for p in probs[:n]])
        seen |= set(e.autotune(reps=2))
        e.run(3)
        e.run(2, use_graph=False)
        assert e.status()[0] == 0
        for i, pr in enumerate(probs[:n]):
            s = Solver(params_for(pr, H.HYDRO_FP32), pr.U)
            s.advance(5)
            ref = s.interior()
            t_ref = s.time()[0]
            s.close()
            got = e.state_numpy(i)[:, NG:-NG, NG:-NG]
            scale = np.abs(ref).max(axis=(1, 2), keepdims=True)
            scale[1:3] = np.maximum(scale[1:3], scale[0])  # momenta that vanish: against rho times a unit sound speed
            # FP32 rounding: the kernels may fuse different multiply-adds
            assert np.all(np.abs(got - ref) <= 2.0 ** -24 * 256 * scale), (n, i, np.abs(got - ref).max())
            assert e.time(i)[0] == pytest.approx(t_ref, rel=2.0 ** -24 * 16) and e.time(i)[1] == 5
        e.close()
    assert seen and all(0 <= k < 8 for k in seen)
