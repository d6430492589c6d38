"""Parameter moves whose sums leave the counted words' range (2^15 a CTA, infinities) and ordinary ones: the resident
and the general form's counted exchange decide them as the exact Fix3 sum of a whole chain in one CTA does (a batched
launch of one whole chain, which uses no counted words), bit for bit."""
import numpy as np
import pytest

from paper_1103_4887_gb300 import pimc, synth

pytestmark = pytest.mark.gpu


def _sampler(prob, precision, form):
    s = pimc.Sampler.from_problem(prob, precision=precision)
    s.set_sweep_form(form)
    s.set_schedule(n_init=0, n_skip=3)
    s.set_param_trace(64)
    return s


@pytest.mark.parametrize("precision", [pimc.FP32_MIXED, pimc.FP64])
@pytest.mark.parametrize("scale", [1.0, 1e3, 1e6, 1e12, 1e36])
@pytest.mark.parametrize("M", [1000, 449])
def test_sums_out_of_range(precision, scale, M):
    prob = synth.hh_problem(M, data_seed=4, free="all")
    prob.Rf = prob.Rf * scale
    prob.sig_p = prob.sig_p * 5.0
    ref = _sampler(prob, precision, "general")
    b = pimc.Batch([ref])
    b.set_tuning(256, 1, 1)
    b.sweep(9, 17)
    b.sweep(8, 17)
    Xr, pr = ref.state()
    mr, vr, Jr = ref.moments()
    for form in ("auto", "general"):
        s = _sampler(prob, precision, form)
        assert s.launch_info()[0] > 1
        s.sweep(9, 17)
        s.sweep(8, 17)
        X, p = s.state()
        assert np.array_equal(X, Xr) and np.array_equal(p, pr)
        assert np.array_equal(s.param_trace(), ref.param_trace())
        m, v, J = s.moments()
        assert J == Jr and np.array_equal(m, mr, equal_nan=True) and np.array_equal(v, vr, equal_nan=True)
        for x, y in zip(s.residual_moments(), ref.residual_moments()):
            assert np.array_equal(np.asarray(x), np.asarray(y), equal_nan=True)
        assert all(np.array_equal(x, y) for x, y in zip(s.accept_stats(), ref.accept_stats()))
    b.close()


@pytest.mark.parametrize("scheme", [0, 1])
@pytest.mark.parametrize("M,grid", [(12, 6), (15, 8), (255, 2), (447, 2), (300, 3)])
def test_tile_edges(M, grid, scheme):
    """Tiles of one site, of two, of the resident form's largest size and ragged last ones: boundary sites by packets
    (resident), by flags (general) and in one CTA, over burn-in with adaptation and annealing, then recording, in three
    launches."""
    prob = synth.hh_problem(M, data_seed=8, free="all")
    prob.scheme = scheme
    got = []
    for form in ("auto", "general", "batch"):
        s = pimc.Sampler.from_problem(prob, precision=pimc.FP32_MIXED)
        if form != "batch":
            s.set_grid(grid)
            s.set_sweep_form(form)
            assert s.sweep_form() == ("resident" if form == "auto" else "general") and s.launch_info()[0] > 1
        s.set_schedule(n_init=7, n_skip=3, beta0=0.3, n_cool=5, f_acc=0.4, alpha=0.3)
        s.set_param_trace(40)
        run = s
        if form == "batch":
            run = pimc.Batch([s])
            run.set_tuning(256, 1, 1)
        for n in (5, 1, 17):
            run.sweep(n, 23)
        got.append((*s.state(), *s.moments(), *s.residual_moments(), s.param_trace(), *s.steps(), *s.accept_stats(),
                    np.array(s.sweep_counter())))
        if form == "batch":
            run.close()
    for other in got[1:]:
        for x, y in zip(got[0], other):
            assert np.array_equal(np.asarray(x), np.asarray(y), equal_nan=True)
