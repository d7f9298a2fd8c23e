"""The switch at temperatures where beta (Vmax - V) leaves the exponential's range: the survival test
needs no double-double there, and the graph is the oracle's."""
import numpy as np
import pytest

import oracle as O
import paper_1503_03295_gb300 as sco

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T", [1e-3, 4e-4, 1e-4, 1e-5, 1e-6])
def test_strong_pairs(T):
    o = O.Chain(O.make_params(20, 17, T=T, seed=11))
    o.switch()
    ro, co = o.graph()
    for prec in (sco.FP64, sco.FP32_GUARDED):
        p = sco.make_params(20, 17, T=T, seed=11, precision=prec)
        g = sco.Lattice(p)
        g.switch()
        rg, cg = g.graph()
        assert np.array_equal(rg.astype(np.int64), ro) and np.array_equal(cg, co)
        assert g.observables()["guard_hits_fp64"] <= 5
        with sco.Batch([p, sco.make_params(16, T=0.5, precision=prec)]) as b:
            b.run(1)
            assert np.array_equal(b.graph(0)[1], co)


@pytest.mark.parametrize("Lx,Ly,T", [(1, 1, 0.5), (6, 6, 1e-6), (33, 1, 1e-9), (8, 8, 1e-9), (13, 5, 1e-9), (70, 60, 0.05),
                                     (46, 45, 1e-6)])
def test_rows_of_any_length_come_sorted(Lx, Ly, T):
    # rows around 32 and 64 entries, and of 2000; twice, as the copy's workspace is kept
    lat = sco.Lattice(sco.make_params(Lx, Ly, T=T, J=1.0, seed=2))
    o = O.Chain(O.make_params(Lx, Ly, T=T, J=1.0, seed=2))
    lat.switch()
    o.switch()
    ro, co = o.graph()
    for _ in range(2):
        rg, cg = lat.graph()
        assert np.array_equal(rg.astype(np.int64), ro) and np.array_equal(cg, co)


@pytest.mark.parametrize("Lx,Ly", [(183, 180), (181, 180)])  # 32,940 and 32,580 sites: both row orders
def test_rows_of_palettes_above_255(Lx, Ly):
    p = sco.make_params(Lx, Ly, T=0.0105, seed=3)
    o = O.Chain(O.make_params(Lx, Ly, T=0.0105, seed=3))
    o.colour()
    ro, co = o.graph()
    lat = sco.Lattice(p)
    lat.colour()
    assert lat.sizes()[3] > 255
    with sco.Batch([p, sco.make_params(16, T=0.5)]) as b:
        b.run(1)
        for rg, cg, c in (*[(*lat.graph(), lat.colours())], *[(*b.graph(0), b.colours(0))]):
            assert np.array_equal(rg.astype(np.int64), ro) and np.array_equal(cg, co)
            assert np.array_equal(c.astype(np.int32), o.colours())
