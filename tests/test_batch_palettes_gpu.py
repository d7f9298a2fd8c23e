"""A batch whose palette capacity has grown past what the bucketed colouring kernel takes (2048) and
whose palettes are small again: the kernel of one level per launch must leave a colouring alone that
the dataflow kernel has made."""
import numpy as np
import pytest

import paper_1503_03295_gb300 as sco

pytestmark = pytest.mark.gpu


def test_small_palettes_after_a_palette_above_2048():
    # 2116 sites at T = 1e-6 D: nearly every pair survives; then T = 0.5 D, palette below 64
    ps = [sco.make_params(46, T=1e-6, seed=1), sco.make_params(40, T=0.7, seed=2)]
    lats = [sco.Lattice(p) for p in ps]
    with sco.Batch(ps) as b:
        b.run(1)
        lats[0].sweep(1)
        lats[1].sweep(1)
        assert b.sizes(0)[3] > 2048
        for r, lat in enumerate(lats):
            assert np.array_equal(b.colours(r), lat.colours()), r
        b.set_temperature(0, 0.5)
        lats[0].set_temperature(0.5)
        b.run(2)
        for r, lat in enumerate(lats):
            lat.sweep(2)
            assert b.sizes(r)[3] < 64
            assert np.array_equal(b.colours(r), lat.colours()), r
            assert b.observables(r)["kw_rounds"] == lat.observables()["kw_rounds"], r
            assert np.array_equal(b.spins(r), lat.spins()), r
