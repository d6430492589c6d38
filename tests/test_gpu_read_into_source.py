"""The state read into the page-locked memory whose data is still waiting on the handle's stream to be uploaded: the upload
takes the data, the read comes after it.  (FP64: every bit of the data shows in the residuals.)"""
import numpy as np
import pytest

from paper_1103_4887_gb300 import pimc, synth

pytestmark = pytest.mark.gpu


def test_state_into_the_uploaded_arrays():
    import torch

    M = 20000
    prob, new = synth.hh_problem(M, data_seed=1, substeps=2), synth.hh_problem(M, data_seed=2, substeps=2)
    got = []
    for shared in (False, True):
        s = pimc.Sampler.from_problem(prob)
        s.set_schedule(n_init=0, n_skip=65)
        arena = torch.zeros((4 if shared else 2) * (M + 1), dtype=torch.float64).pin_memory()
        a = arena.numpy()
        a[:M + 1], a[M + 1:2 * M + 1] = new.y, new.I
        s.sweep(60, 3, sync=False)  # the stream is busy while the uploads wait
        s.load_data(arena.data_ptr(), arena.data_ptr() + 8 * (M + 1))
        X = a if shared else np.zeros(4 * (M + 1))
        s._ck(s._L.pimc_get_state(s._h, X.ctypes.data, None))
        s.sweep(6, 4)  # the record of sweep 65 holds x - y of the new data
        got.append((X.copy(), *s.state(), *s.residual_moments()))
    for x, y in zip(*got):
        assert np.array_equal(x, y, equal_nan=True)
