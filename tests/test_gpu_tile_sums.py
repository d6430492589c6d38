"""The resident form's CTA sum of a parameter move's terms in tiles of up to 224 sites, with terms of one sign and like
size (as a far proposal of a parameter that acts alike on every site gives): the sums are exact, so every decision is that
of the general form and of a whole chain in one CTA.  The paths lie on the model's own trajectory and do not move (site
steps of zero); R_f is set so that a parameter move of one step changes the action by `term` a site."""
import numpy as np
import pytest

from paper_1103_4887_gb300 import pimc, synth

pytestmark = pytest.mark.gpu


def _problem(kind, M):
    if kind == "hh":  # E_L
        prob = synth.hh_problem(M, data_seed=2, free=("EL",), substeps=2)
        prob.p_init = prob.p_true.copy()
        prob.sig_p = np.where(prob.free, 2.0, 0.0)
        s = pimc.Sampler.from_problem(prob)
        path, l = s.forecast(M, prob.I, 1, 0, 1)[0], 5
    else:             # the origin is a fixed point of the undriven linear model
        prob = synth.lingauss_problem(M)
        prob.I, prob.sig_p, prob.scheme = np.zeros(M), np.ones(1), int(kind == "trapezoid")
        path, l = np.zeros((2, M + 1)), 0
    prob.Rf = np.eye(prob.D)[0]
    prob.sig_x = np.zeros(prob.D)
    s = pimc.Sampler.from_problem(prob)
    s.set_path(path)
    return prob, path, s.param_delta(l, prob.p_init[l] + prob.sig_p[l]) / M


@pytest.mark.parametrize("term", [200.0, 450.0, 0.3, 1.2e-5])
@pytest.mark.parametrize("M,grid", [(447, 2), (431, 2), (257, 2), (32768, 0)])
@pytest.mark.parametrize("kind", ["rk4", "trapezoid", "hh"])
def test_terms_of_one_sign(kind, M, grid, term):
    prob, path, one = _problem(kind, M)
    prob.Rf = prob.Rf * (term / one)
    got = []
    for form in ("auto", "general", "batch"):
        s = pimc.Sampler.from_problem(prob, precision=pimc.FP32_MIXED)
        s.set_path(path)
        s.set_param_trace(300)
        run = s
        if form == "batch":
            run = pimc.Batch([s])
            run.set_tuning(256, 1, 1)
        else:
            s.set_grid(grid)
            s.set_sweep_form(form)
            assert s.sweep_form() == ("resident" if form == "auto" else "general") and s.launch_info()[0] > 1
        run.sweep(300, 5)
        got.append((s.param_trace(), *s.state(), *s.accept_stats()))
        if form == "batch":
            run.close()
    for other in got[1:]:
        for x, y in zip(got[0], other):
            assert np.array_equal(x, y)
