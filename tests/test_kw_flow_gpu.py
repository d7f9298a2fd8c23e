"""The dataflow colouring kernel where its shape changes, against the oracle (colours, t_R): one
block and many, short last groups, palettes of 1 and above its limit (which take the other
kernels), lattices too large for the blocks' shared memory; the static entry point on rows that
may not be read by whole sectors; a batch that mixes palettes."""
import numpy as np
import pytest

import oracle as O
import paper_1503_03295_gb300 as sco

pytestmark = pytest.mark.gpu


def _compare(g, o):
    g.colour()
    o.colour()
    assert np.array_equal(g.colours().astype(np.int32), o.colours())
    og, oo = g.observables(), o.observables()
    assert og["kw_rounds"] == oo["kw_rounds"] and og["max_degree"] == oo["max_degree"]


@pytest.mark.parametrize("Lx,Ly,T,J", [
    (1, 1, 0.5, 0.0), (2, 1, 0.5, 0.0), (5, 3, 0.4, 1.0),
    (45, 46, 1e12, 0.0),     # no pairs: palette 1, 2070 vertices, 12 levels
    (64, 32, 0.5, 0.0),      # 2048 vertices: one block of 1024 right-half ones
    (64, 33, 0.5, 0.0),      # just above
    (32, 32, 0.85, 1.0), (33, 32, 0.85, 1.0),  # palettes up to 24: one block of 512, several of 256
    (301, 299, 0.6, 0.0), (700, 301, 0.9, 1.0),
    (1024, 700, 0.3, 0.0),   # larger blocks, mean degree 30: lists read in parts
    (40, 40, 0.1, 0.0), (301, 200, 0.1, 0.0),  # palettes of 65 to 255: colours above 31 looked up again
    # near parts of the rows: none (one column), of a few levels, of every level
    (1, 700, 0.2, 0.0), (7, 900, 0.4, 0.0), (900, 2, 0.3, 0.0),
    (40, 40, 0.006, 0.0), (200, 150, 0.011, 0.0),  # palettes above 255: the other kernels
])
def test_colouring_matches_oracle(Lx, Ly, T, J):
    D = 1.0 if J == 0.0 else 0.1
    _compare(sco.Lattice(sco.make_params(Lx, Ly, T=T, J=J, D=D, seed=3)),
             O.Chain(O.make_params(Lx, Ly, T=T, J=J, D=D, seed=3)))


def test_lattice_beyond_the_blocks_shared_memory():
    _compare(sco.Lattice(sco.make_params(3500, T=6.0, seed=1)), O.Chain(O.make_params(3500, T=6.0, seed=1)))


@pytest.mark.parametrize("offset", [0, 1, 8])
def test_static_rows_at_any_alignment(offset):
    import torch

    lat = sco.Lattice(sco.make_params(150, 90, T=0.5, seed=2))
    lat.colour()
    rp, col = lat.graph()
    # the rows start `offset` entries into a buffer that ends with the last entry
    buf = torch.zeros(col.size + offset, dtype=torch.int32, device="cuda")
    buf[offset:] = torch.from_numpy(col.view(np.int32).copy()).cuda()
    d_rp = torch.from_numpy(rp.view(np.int32).copy()).cuda()
    out = torch.full((lat.N,), -1, dtype=torch.int32, device="cuda")
    sco.kw_colour_static(d_rp.data_ptr(), buf.data_ptr() + 4 * offset, lat.N, out.data_ptr(),
                         stream=torch.cuda.current_stream().cuda_stream)
    assert np.array_equal(out.cpu().numpy().view(np.uint32), lat.colours())


@pytest.mark.parametrize("cold", [0.5, 0.1, 0.006])  # one replica's palette above 64, above 255
def test_batch_matches_single_lattices(cold):
    ps = [sco.make_params(36, T=cold, seed=1), sco.make_params(3, 2, T=0.5, seed=2),
          sco.make_params(90, 70, T=0.7, seed=3), sco.make_params(64, T=1e12, seed=4)]
    with sco.Batch(ps) as b:
        b.run(2)
        for r, p in enumerate(ps):
            lat = sco.Lattice(p)
            lat.sweep(2)
            assert np.array_equal(b.colours(r), lat.colours()), r
            assert b.observables(r)["kw_rounds"] == lat.observables()["kw_rounds"], r
            assert np.array_equal(b.spins(r), lat.spins()), r
