"""Moments and residual moments on both sides of the size from which they are formed on the device, and where the staging
buffer's length cuts them, against sums formed here from the states of every recorded sweep."""
import numpy as np
import pytest

from paper_1103_4887_gb300 import pimc, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [pimc.FP32_MIXED, pimc.FP64])
@pytest.mark.parametrize("M", [1, 10922, 10923, 16382, 16383])  # 3 M and 2 (M + 1) + 1 around 32768 quantities
def test_read_moments(M, precision):
    prob = synth.lingauss_problem(M)
    s = pimc.Sampler.from_problem(prob, precision=precision)
    s.set_schedule(n_init=0, n_skip=1)
    y = prob.y.astype(np.float32).astype(np.float64) if precision == pimc.FP32_MIXED else prob.y
    x, r, J = [], [], 5
    for _ in range(J):
        s.sweep(1, 11)
        X, p = s.state()
        x.append(np.concatenate([X.ravel(), p]))
        r.append((X[0] - y)[1:])

    def moments(v, shift):  # in the kernels' order of additions
        s1 = s2 = np.zeros_like(v[0])
        for a in v:
            s1, s2 = s1 + (a - shift), s2 + (a - shift) ** 2
        return shift + s1 / J, (s2 - s1 * s1 / J) / (J - 1), s2
    mean, var, n = s.moments()
    m, v, s2 = moments(x, x[0])
    assert n == J and np.array_equal(mean, m)
    # a fused multiply-add of the device saves one rounding a record: J 2^-53 of the sum, and of the difference
    assert np.all(np.abs(var - v) <= 2 * J * 2.0 ** -53 * s2 / (J - 1))
    mean, var, n = s.residual_moments()
    m, v, s2 = moments(r, 0.0)
    assert n == J and mean.size == 3 * M and np.array_equal(mean[2 * M:], m)
    assert np.all(np.abs(var[2 * M:] - v) <= 2 * J * 2.0 ** -53 * s2 / (J - 1))
    assert np.all(np.isfinite(mean)) and np.all(np.isfinite(var))
