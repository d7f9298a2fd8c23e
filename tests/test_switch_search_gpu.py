"""The switch's guided candidate search against the oracle where its ranges change: lists shorter
than the shared head, just past it and far beyond it, decay values that underflow, and long thin
lattices; both precisions, and the batched switch on the same lattices."""
import numpy as np
import pytest

import oracle as O
import paper_1503_03295_gb300 as sco

pytestmark = pytest.mark.gpu

CASES = [
    (2, 1, 0.3),       # one displacement
    (31, 32, 0.5),     # 1921 displacements: all of them in the shared head
    (32, 33, 0.5),     # 2047
    (33, 32, 0.5),     # 2047 + 1 row's worth
    (200, 150, 0.6),   # far guide in use
    (3, 4000, 0.4), (4000, 3, 0.4),
    (90, 80, 0.05),    # total hazard 361: targets down to e^-361
    (60, 50, 0.012),   # beyond e^-690: the decay bits underflow, the logarithm decides
    (150, 150, 40.0),  # a handful of candidates per site, mostly far
]


@pytest.mark.parametrize("Lx,Ly,T", CASES)
def test_graph_matches_oracle(Lx, Ly, T):
    o = O.Chain(O.make_params(Lx, Ly, T=T, seed=5))
    o.switch()
    ro, co = o.graph()
    for prec in (sco.FP64, sco.FP32_GUARDED):
        p = sco.make_params(Lx, Ly, T=T, seed=5, precision=prec)
        g = sco.Lattice(p)
        g.switch()
        rg, cg = g.graph()
        assert np.array_equal(rg.astype(np.int64), ro) and np.array_equal(cg, co), prec
        if Lx * Ly <= 30000 and T > 0.02:
            with sco.Batch([p, sco.make_params(16, T=0.5, precision=prec)]) as b:
                b.run(1)
                rb, cb = b.graph(0)
                assert np.array_equal(rb.astype(np.int64), ro) and np.array_equal(cb, co), prec
