"""Batches of fewer chains than the device holds CTAs, without tuning: long chains are cut into tiles, one a CTA, and every
chain stays bit for bit what it is whole in one CTA."""
import numpy as np
import pytest

from paper_1103_4887_gb300 import pimc, synth

pytestmark = pytest.mark.gpu

MAKE = {"hh": lambda M, k: synth.hh_problem(M, data_seed=k, free="all" if k % 2 else ("gNa", "gK", "gL"), substeps=2),
        "paper": lambda M, k: synth.paper_problem(M, data_seed=k, substeps=2),
        "lingauss": lambda M, k: synth.lingauss_problem(M, data_seed=k)}


def _chains(kind, prec, Ms):
    out = []
    for k, M in enumerate(Ms):
        s = pimc.Sampler.from_problem(MAKE[kind](M, k), precision=prec)
        s.set_chain(k)
        s.set_schedule(n_init=4, n_skip=3, beta0=0.5, n_cool=3, f_acc=0.4, alpha=0.3)
        out.append(s)
    return out


@pytest.mark.parametrize("prec", [pimc.FP32_MIXED, pimc.FP64])
@pytest.mark.parametrize("kind", list(MAKE))
@pytest.mark.parametrize("Ms,split", [([3100, 700, 5, 2048, 1023, 4501], True), ([34000, 1, 3000], True),
                                      ([900, 30, 1022], False)])
def test_few_chains(kind, prec, Ms, split):
    if kind == "paper":
        Ms = [min(M, 6000) for M in Ms]
    whole, cut = _chains(kind, prec, Ms), _chains(kind, prec, Ms)
    b1, b2 = pimc.Batch(whole), pimc.Batch(cut)
    b1.set_tuning(256, 1, 1)
    assert b1.info()[2] == 0 and (b2.info()[2] > 0) == split and (b2.info()[0] > len(Ms)) == split
    for n in (8, 6):
        b1.sweep(n, 19)
        b2.sweep(n, 19)
    b1.sync(), b2.sync()
    for s1, s2 in zip(whole, cut):
        for x, y in zip((*s1.state(), *s1.moments(), *s1.residual_moments(), *s1.accept_stats(), *s1.steps()),
                        (*s2.state(), *s2.moments(), *s2.residual_moments(), *s2.accept_stats(), *s2.steps())):
            assert np.array_equal(np.asarray(x), np.asarray(y), equal_nan=True)
    b1.close(), b2.close()
