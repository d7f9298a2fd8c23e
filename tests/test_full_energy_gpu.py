"""The full energy by transforms against the oracle's direct sum: sides that are powers of two, one
off them, either side the longer, the smallest lattices, the largest side, and one that takes the
direct sum.  Tolerance: 1e-12 of max(|E|, N), the summation-order bound
of the other energies (the transforms' rounding, 2^-52 log2(points) per term of mean size 1/N, stays
below 1e-14 N)."""
import numpy as np
import pytest

import oracle as O
import paper_1503_03295_gb300 as sco

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Lx,Ly,J,D", [
    (32, 32, 0.0, 1.0), (31, 33, 1.0, 0.1), (33, 32, 0.0, 1.0), (65, 100, -0.5, 1.0),
    (1024, 1, 0.0, 1.0), (1, 1024, 0.0, 1.0), (1024, 17, 1.0, 0.1), (128, 129, 0.0, 3.0),
    (1, 1, 0.0, 1.0), (2, 1, 1.0, 1.0), (16, 16, 1.0, 0.1),
    (1025, 3, 0.0, 1.0),  # direct sum
])
def test_full_energy_matches_oracle(Lx, Ly, J, D):
    g = sco.Lattice(sco.make_params(Lx, Ly, T=0.6, J=J, D=D, seed=4))
    o = O.Chain(O.make_params(Lx, Ly, T=0.6, J=J, D=D, seed=4))
    for _ in range(2):  # the workspace is made, then reused
        a, b = g.observables(full=True)["e_full"], o.observables(full=True)["e_full"]
        assert abs(a - b) <= 1e-12 * max(abs(b), float(Lx * Ly))
    # ferromagnetic and antiparallel columns: large coherent sums
    s = np.zeros((3, Ly, Lx))
    s[0] = 1.0
    s[0, :, 1::2] = -1.0
    g.set_spins(s.ravel())
    o.set_spins(s.ravel())
    a, b = g.observables(full=True)["e_full"], o.observables(full=True)["e_full"]
    assert abs(a - b) <= 1e-12 * max(abs(b), float(Lx * Ly))
