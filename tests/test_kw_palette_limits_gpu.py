"""A lattice's palette just below and above the size from which one kernel per level takes over from the
dataflow kernel (it depends on the lattice): colours and t_R against the oracle, and a batch, which stays with
the dataflow kernel."""
import numpy as np
import pytest

import oracle as O
import paper_1503_03295_gb300 as sco

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Lx,Ly,T", [(64, 72, 0.0145), (65, 71, 0.0145),   # 4608 and 4615 sites, palette about 225
                                     (100, 90, 0.021), (100, 90, 0.0185),  # about 198 and 215
                                     (224, 223, 0.021), (224, 224, 0.021),  # 49,952 and 50,176 sites, about 212
                                     (256, 200, 0.018)])                   # about 232
def test_colouring_around_the_limits(Lx, Ly, T):
    p = sco.make_params(Lx, Ly, T=T, seed=6)
    o = O.Chain(O.make_params(Lx, Ly, T=T, seed=6))
    o.colour()
    oo = o.observables()
    lat = sco.Lattice(p)
    for _ in range(2):
        lat.colour()
        og = lat.observables()
        assert np.array_equal(lat.colours().astype(np.int32), o.colours())
        assert og["kw_rounds"] == oo["kw_rounds"] and og["max_degree"] == oo["max_degree"]
    with sco.Batch([p, sco.make_params(16, T=0.5)]) as b:
        b.run(1)
        assert np.array_equal(b.colours(0).astype(np.int32), o.colours())
