"""Device memory of handles: the first-stage buffer of the FP64 moves (40 bytes a site) is held only where they read it."""
import numpy as np
import pytest

from paper_1103_4887_gb300 import pimc, synth

pytestmark = pytest.mark.gpu

M = 1 << 20


def _free():
    import torch

    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def _used(make):
    before = _free()
    s = make()
    used = before - _free()
    s.close()
    return used


def test_first_stage_buffer():
    p = synth.hh_problem(M, data_seed=1, substeps=1)

    def handle(precision, scheme=0):
        s = pimc.Sampler(p.model, M, p.dt, p.Rm, p.Rf, precision)
        s.set_scheme(scheme)
        s.set_data(p.y, p.I)
        return s

    handle(pimc.FP64).close()  # what the context and the library take once
    buffer = 40 * (M + 1)
    fp64 = _used(lambda: handle(pimc.FP64))
    assert _used(lambda: handle(pimc.FP32_MIXED)) <= fp64 - 0.9 * buffer
    assert _used(lambda: handle(pimc.FP64, 1)) <= fp64 - 0.9 * buffer
    # a handle that changes: the buffer comes and goes, and the chain is the same
    s, t = handle(pimc.FP32_MIXED), handle(pimc.FP64)
    s.set_precision(pimc.FP64)
    for h in (s, t):
        h.set_data(p.y, p.I)
        h.set_params(p.p_init, p.lo, p.hi, p.free)
        h.set_steps(p.sig_x, p.sig_p)
        h.sweep(2, 9)
    assert all(np.array_equal(a, b) for a, b in zip(s.state(), t.state()))
    before = _free()
    s.set_precision(pimc.FP32_MIXED)
    assert _free() - before >= 0.9 * buffer
    s.sweep(1, 9)
    assert np.all(np.isfinite(s.state()[0]))
