"""Spins that a caller sets need not have length 1: long, infinite and not-a-number ones are outside the
first decisions' error bounds and have to go to the exact ones, on the site itself, among its neighbours
and through the exchange field.  Against the oracle; where the pair energies leave the range of a double
(infinite spins, products of 1e200), in which the exact decisions work, both precisions and a batch against
one another."""
import numpy as np
import pytest

import oracle as O
import paper_1503_03295_gb300 as sco

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Lx,Ly,T,J,D", [(24, 17, 0.4, 0.0, 1.0), (24, 17, 0.5, 1.0, 0.1), (24, 17, 0.5, 1.0, 0.0),
                                         (70, 50, 0.6, -0.5, 1.0)])
@pytest.mark.parametrize("kind", ["nan", "inf", "long", "huge", "short", "mixed"])
def test_sweep_with_any_spins(Lx, Ly, T, J, D, kind):
    rng = np.random.default_rng(3)
    o = O.Chain(O.make_params(Lx, Ly, T=T, J=J, D=D, seed=5))
    N = Lx * Ly
    s = np.array(o.spins()).reshape(3, N).copy()
    at = rng.choice(N, N // 8, replace=False)
    val = {"nan": [np.nan], "inf": [np.inf, -np.inf], "long": [3.0, -1.5, 1.002], "huge": [1e30, -1e200],
           "short": [0.0, 1e-30], "mixed": [np.nan, np.inf, 4.0, 1e25, 0.0]}[kind]
    for a in at:
        s[rng.integers(3), a] = val[rng.integers(len(val))]
    o.set_spins(s.ravel())
    o.sweep(2)
    want = np.asarray(o.spins()).ravel() if kind in ("nan", "long", "short") else None
    for prec in (sco.FP64, sco.FP32_GUARDED):
        p = sco.make_params(Lx, Ly, T=T, J=J, D=D, seed=5, precision=prec)
        g = sco.Lattice(p)
        g.set_spins(s.ravel())
        g.sweep(2)
        if want is None:
            want = g.spins()
        assert np.array_equal(g.spins(), want, equal_nan=True), prec
        with sco.Batch([p, sco.make_params(16, T=0.5, precision=prec)]) as b:
            b.set_spins(0, s.ravel())
            b.run(2)
            assert np.array_equal(b.spins(0), want, equal_nan=True), prec
