"""Sweeps at low temperatures: the first decisions take the sites there too (they are counted when they
are left to FP64, in the FP32-guarded form, or to double-double), with the oracle's results."""
import numpy as np
import pytest

import oracle as O
import paper_1503_03295_gb300 as sco

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Lx,Ly,T,J,D", [(40, 33, 0.02, 0.0, 1.0), (64, 20, 0.005, 0.0, 1.0), (33, 30, 0.002, 0.0, 1.0)])
def test_errors_that_add_up_beside_wide_margins(Lx, Ly, T, J, D):
    _compare(Lx, Ly, T, J, D)


@pytest.mark.parametrize("Lx,Ly,T,J,D", [
    (40, 33, 0.0015, 1.0, 0.1), (40, 33, 0.0015, -1.0, 0.01),  # beta J = 667
    (31, 30, 1e-4, 1.0, 0.0), (31, 30, 2e-5, -1.0, 1e-3),      # 1e4, 5e4
])
def test_strong_exchange(Lx, Ly, T, J, D):
    _compare(Lx, Ly, T, J, D)


@pytest.mark.parametrize("Lx,Ly,T,J,D", [(20, 17, 4e-4, 0.0, 1.0), (20, 17, 2e-5, 0.0, 1.0), (17, 12, 2e-5, 1.0, 0.1)])
def test_strong_pairs(Lx, Ly, T, J, D):
    # beta (Vmax - V) up to 2e5: the FP64 form (the FP32-guarded one leaves these sites to FP64)
    _compare(Lx, Ly, T, J, D, guarded=False)


def _compare(Lx, Ly, T, J, D, guarded=True):
    n = 3
    o = O.Chain(O.make_params(Lx, Ly, T=T, J=J, D=D, seed=11))
    o.sweep(n)
    for prec in (sco.FP64, sco.FP32_GUARDED):
        p = sco.make_params(Lx, Ly, T=T, J=J, D=D, seed=11, precision=prec)
        g = sco.Lattice(p)
        g.sweep(n)
        assert np.array_equal(g.accepts(), o.accepts()), prec
        assert np.array_equal(g.spins(), o.spins()), prec
        ob = g.observables()
        if not guarded and prec == sco.FP32_GUARDED:
            continue
        assert ob["guard_hits_fp32"] + ob["guard_hits_fp64"] < g.N * n // 5, ob
        with sco.Batch([p, sco.make_params(16, T=0.5, precision=prec)]) as b:
            b.run(n)
            assert np.array_equal(b.spins(0), o.spins()), prec
