"""The sweeps of both precisions against the oracle where their dispatch changes: lanes per site by
class size, the trailing colours left to one block, one block for a small lattice, pairs and exchange
factors outside the range of the first decision (settled in FP64 / double-double)."""
import numpy as np
import pytest

import oracle as O
import paper_1503_03295_gb300 as sco

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Lx,Ly,T,J,D,n", [
    (1000, 700, 0.8, 0.0, 1.0, 1),    # largest classes above half the grid: 2 lanes per site
    (257, 131, 0.6, 0.0, 1.0, 2),     # a few thousand sites: 8, then 32 lanes per site
    (24, 24, 2e-4, 0.0, 1.0, 2),      # beta (Vmax - V) up to 2e4: beyond the float-float range
    (24, 24, 2e-3, 0.0, 1.0, 2),      # up to 2000: exponents in the thousands, rows of hundreds
    (40, 33, 0.05, 1.0, 0.1, 3),      # exchange factors e^(+-80)
    (40, 33, 0.0015, 1.0, 0.1, 2),    # beta J = 667: exchange factor out of range
    (31, 17, 0.4, -0.5, 1.0, 3),      # antiferromagnetic exchange
    (16, 16, 3.0, 0.0, 1e-9, 2),      # pair constants near 1e-9
    (1, 37, 0.3, 0.0, 1.0, 3),        # a chain (Lx = 1)
    (45, 45, 0.5, 1.0, 0.1, 3), (46, 45, 0.5, 1.0, 0.1, 3),  # one block of the sweep, and more
])
def test_sweep_matches_oracle(Lx, Ly, T, J, D, n):
    o = O.Chain(O.make_params(Lx, Ly, T=T, J=J, D=D, seed=11))
    o.sweep(n)
    for prec in (sco.FP64, sco.FP32_GUARDED):
        p = sco.make_params(Lx, Ly, T=T, J=J, D=D, seed=11, precision=prec)
        g = sco.Lattice(p)
        g.sweep(n)
        assert np.array_equal(g.accepts(), o.accepts()), prec
        assert np.array_equal(g.spins(), o.spins()), prec
        with sco.Batch([p, sco.make_params(16, T=0.5, precision=prec)]) as b:
            b.run(n)
            assert np.array_equal(b.spins(0), o.spins()), prec
