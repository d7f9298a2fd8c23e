"""Bounded waits that run out (limit 0) on the paths that test_wait_limit_gpu.py does not take: the
status is SCO_ETIMEOUT, later calls are refused, and a step whose colouring gave up changes no spin."""
import numpy as np
import pytest

import oracle as O
import paper_1503_03295_gb300 as sco

pytestmark = pytest.mark.gpu


def _status(call):
    try:
        call()
    except sco.ScoError as e:
        return e.status
    return sco.SCO_OK


def _refuses(obj, run):
    assert _status(obj.sync) == sco.SCO_ETIMEOUT
    assert _status(run) == sco.SCO_ETIMEOUT
    obj.close()
    # the device still works
    g, o = sco.Lattice(sco.make_params(32, T=0.5, seed=2)), O.Chain(O.make_params(32, T=0.5, seed=2))
    g.sweep(2)
    o.sweep(2)
    assert np.array_equal(g.spins(), o.spins())
    g.close()


def _spins_after(get, n):
    import torch

    s = torch.empty(3 * n, dtype=torch.float64, device="cuda")
    assert _status(lambda: get(s.data_ptr())) == sco.SCO_ETIMEOUT  # copied, then refused
    return s.cpu().numpy()


@pytest.mark.parametrize("use_graph", [0, 1])
@pytest.mark.parametrize("precision", [sco.FP64, sco.FP32_GUARDED])
def test_first_step_of_a_batch_whose_colouring_gives_up(precision, use_graph):
    # no class has ever been built: the sweep must not walk what the arrays hold
    ps = [sco.make_params(L, T=0.3, seed=L, precision=precision) for L in (64, 128, 96)]
    b = sco.Batch(ps)
    b.set_tuning(steps_per_graph=2, sweep_blocks_per_sm=2, kw_blocks_per_sm=2, use_graph=use_graph)
    first = [b.spins(r) for r in range(len(ps))]
    b.set_wait_limit(0)
    assert _status(lambda: b.run(2)) == sco.SCO_ETIMEOUT
    for r, s in enumerate(first):
        got = _spins_after(lambda p: b.get_spins_device(r, p), b.N[r])
        assert np.array_equal(got, s.ravel()), r
    _refuses(b, lambda: b.run(1))


def test_first_step_of_a_lattice_whose_colouring_gives_up():
    lat = sco.Lattice(sco.make_params(256, T=0.3, seed=1))
    first = lat.spins()
    lat.set_wait_limit(0)
    _status(lambda: lat.sweep(1))
    assert _status(lat.sync) == sco.SCO_ETIMEOUT
    assert np.array_equal(_spins_after(lat.get_spins_device, lat.N), first.ravel())
    _refuses(lat, lambda: lat.sweep(1))


@pytest.mark.parametrize("precision", [sco.FP64, sco.FP32_GUARDED])
def test_sweep_barrier_of_a_lattice_runs_out(precision):
    # coloured with the normal limit: only the barriers between the classes are left to wait
    lat = sco.Lattice(sco.make_params(256, T=0.4, seed=1, n_sw=4, precision=precision))
    lat.sweep(1)
    lat.sync()
    lat.set_wait_limit(0)
    _status(lambda: lat.sweep(1))
    _refuses(lat, lambda: lat.sweep(1))


@pytest.mark.parametrize("use_graph", [0, 1])
def test_sweep_barrier_of_a_batch_runs_out(use_graph):
    b = sco.Batch([sco.make_params(L, T=0.4, seed=L, n_sw=4) for L in (128, 200)])
    b.set_tuning(steps_per_graph=1, sweep_blocks_per_sm=1, kw_blocks_per_sm=1, use_graph=use_graph)
    b.run(1)
    b.set_wait_limit(0)
    assert _status(lambda: b.run(1)) == sco.SCO_ETIMEOUT
    _refuses(b, lambda: b.run(1))


@pytest.mark.parametrize("Lx,Ly,T", [(60, 50, 0.006),   # palette above 255: one kernel per level
                                     (3500, 3500, 6.0)])  # beyond the dataflow kernel: bucketed grid barriers
def test_colouring_by_the_other_kernels_runs_out(Lx, Ly, T):
    lat = sco.Lattice(sco.make_params(Lx, Ly, T=T, seed=1))
    lat.switch()
    lat.set_wait_limit(0)
    assert _status(lambda: lat.colour()) == sco.SCO_ETIMEOUT
    _refuses(lat, lambda: lat.sweep(1))


@pytest.mark.parametrize("kw_schedule", [0, 1])
def test_batch_colouring_by_the_other_kernels_runs_out(kw_schedule):
    # palettes above 255: buckets in one kernel (0), one kernel per level (1)
    ps = [sco.make_params(60, 50, T=0.006, seed=1), sco.make_params(64, T=0.5, seed=2)]
    b = sco.Batch(ps)
    b.set_tuning(steps_per_graph=1, sweep_blocks_per_sm=1, kw_blocks_per_sm=2, kw_schedule=kw_schedule)
    b.run(1)
    s = [b.spins(r) for r in range(2)]
    b.set_wait_limit(0)
    assert _status(lambda: b.run(1)) == sco.SCO_ETIMEOUT
    for r in range(2):
        assert np.array_equal(_spins_after(lambda p: b.get_spins_device(r, p), b.N[r]), s[r]), r
    _refuses(b, lambda: b.run(1))
