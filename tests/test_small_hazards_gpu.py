"""Couplings so weak that neighbouring decay values of the candidate search differ by less than their
rounding, on lists longer than the shared head: the switch against the oracle."""
import numpy as np
import pytest

import oracle as O
import paper_1503_03295_gb300 as sco

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D", [1e-4, 1e-9, 1e-11, 1e-12, 1e-13, 1e-15, 1e-17, 1e-300])
@pytest.mark.parametrize("Lx,Ly", [(120, 90), (3, 3000)])
def test_weak_couplings(Lx, Ly, D):
    o = O.Chain(O.make_params(Lx, Ly, T=0.7, D=D, J=0.3, seed=4))
    o.sweep(1)
    for prec in (sco.FP64, sco.FP32_GUARDED):
        p = sco.make_params(Lx, Ly, T=0.7, D=D, J=0.3, seed=4, precision=prec)
        g = sco.Lattice(p)
        g.sweep(1)
        assert np.array_equal(g.graph()[1], o.graph()[1])
        assert np.array_equal(g.spins(), o.spins())
        with sco.Batch([p, sco.make_params(16, T=0.5, precision=prec)]) as b:
            b.run(1)
            assert np.array_equal(b.spins(0), o.spins())
