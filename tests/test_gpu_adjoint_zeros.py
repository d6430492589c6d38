"""The FP64 HH gradient where factors of its entries vanish -- a drive of zero, gates of zero, V on a reversal potential or
on a removable singularity of the rates -- against the oracle's, to 1e-12 of the largest entry."""
import numpy as np
import pytest

import oracle
from paper_1103_4887_gb300 import pimc, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("drive", [True, False])
@pytest.mark.parametrize("gates", [True, False])
def test_vanishing_factors(drive, gates):
    prob = synth.hh_problem(600, data_seed=3, free="all")
    if not drive:
        prob.I = np.zeros(prob.M)
    X = synth.random_path_near(prob, prob.X_true, np.array([1.0, 0.05, 0.05, 0.05]), 4)
    X[0, ::5], X[0, 3::5], X[0, 4::11] = -40.0, -55.0, prob.p_init[5]
    if not gates:
        X[1:, ::7] = 0.0
    g = pimc.Sampler.from_problem(prob)
    o = oracle.Chain(prob.model, prob.M, prob.dt, prob.Rm, prob.Rf)
    o.set_data(prob.y, prob.I)
    o.set_params(prob.p_init, prob.lo, prob.hi, prob.free)
    for h in (g, o):
        h.set_path(X)
    for a, b in zip(g.grad(), o.grad()):
        assert np.all(np.abs(a - b) <= 1e-12 * np.abs(b).max())
