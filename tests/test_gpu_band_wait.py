"""Bounded waits of the band-resident kernels: a band that sends nothing makes
its neighbours' waits run out, the launch ends normally and the host sees the
error; nothing of it stays behind for the next launch."""
import ctypes
import time

import numpy as np
import pytest

import oracle
import paper_1209_0296_gb300 as lt
from paper_1209_0296_gb300._lib import check

pytestmark = pytest.mark.gpu
ETIMEOUT = -4
POLLS = 1 << 18   # about a tenth of a second


@pytest.fixture
def hook():
    lib = lt.load()
    yield lib.lattice_test_band_wait
    lib.lattice_test_band_wait(0, 0)


def _pair(L, model=lt.ISING, J=1.0, h=0.0, par=2.3, two_S=1, seed=5, **kw):
    init = lt.INIT_EQUILIBRIUM if model == lt.NE else lt.INIT_RANDOM
    a = (2, L, two_S, model, J, h, par)
    return lt.Lattice(*a, seed=seed, init=init, **kw), oracle.Lattice(*a, seed=seed, init=init)


def _times_out(g):
    with pytest.raises(lt.LatticeError) as e:
        g.synchronize()
    assert e.value.code == ETIMEOUT


def _silence(hook, g, band, n=12):
    """Run g in a batch of its own, `band` of it silent."""
    b = lt.Batch()
    hook(POLLS, band)
    b.add(g, n)
    b.run()
    _times_out(g)
    hook(0, 0)
    b.close()


# every form: one chunk a thread, a byte a site with several, bits, North-East in one chunk a thread and on bits
@pytest.mark.parametrize("kw", [dict(L=256), dict(L=1602, h=0.3), dict(L=1632), dict(L=300, model=lt.NE, J=0.0, par=0.3),
                                dict(L=1632, model=lt.NE, J=0.0, par=0.3)])
@pytest.mark.parametrize("band", [1, 4])
def test_a_silent_band_ends_the_launch(hook, kw, band):
    g, o = _pair(**kw)
    spins, flags, _ = g.get_state()
    _silence(hook, g, band)
    g.set_state(spins, flags, 0)         # whole again
    g.set_kernel(lt.KERNEL_WIDE)
    g.sweep(12)
    o.sweep(12)
    assert np.array_equal(g.get_spins(), o.spins)
    g.close()


def test_a_batch_waits_as_long_after_a_time_out(hook):
    b = lt.Batch()
    took = []
    for rep in range(2):
        (g, _), (f, o) = _pair(512, seed=rep), _pair(300, seed=10 + rep)
        hook(POLLS, 1)                   # a band of the larger lattice
        b.add(g, 8)
        b.add(f, 8)
        t0 = time.perf_counter()
        b.run()
        try:
            b.synchronize()
        except lt.LatticeError as e:
            assert e.code == ETIMEOUT
        took.append(time.perf_counter() - t0)
        _times_out(g)
        o.sweep(8)
        assert np.array_equal(f.get_spins(), o.spins)   # the other lattice is not touched
        g.close()
        f.close()
    # the first run's give-up mark does not cut the second run's waits short (they would end after 1024 polls)
    assert took[1] > 0.25 * took[0], took
    b.close()


def _codes(*calls):
    out = []
    for f in calls:
        try:
            f()
            out.append(0)
        except lt.LatticeError as e:
            out.append(e.code)
    return out


# after a time-out every call that reads, advances or refers to the state says so, set_state ends it
def test_every_call_on_a_lattice_that_timed_out(hook):
    L = 512
    g, o = _pair(L, lt.NE, 0.0, 0.0, 0.3)
    spins, flags, _ = g.get_state()
    g.set_kernel(lt.KERNEL_WIDE)
    g.set_reference()
    _silence(hook, g, 2, 8)
    b = lt.Batch()
    n = ctypes.c_int64()
    calls = [lambda: g.sweep(1), lambda: g.sweep(8), lambda: g.series(0, 8), g.observables, g.set_reference,
             lambda: g.autocorrelation(0, 8), g.get_spins, lambda: g.set_spins(spins), g.get_state, g.device_spins,
             lambda: check(lt.load().lattice_get_state(g.handle, None, None, ctypes.byref(n)), "get_state"),
             g.synchronize, lambda: b.add(g, 4)]
    assert _codes(*calls) == [ETIMEOUT] * len(calls)
    g.set_state(spins, flags, 0)
    b.add(g, 6)
    b.run()
    b.synchronize()
    o.sweep(6)
    assert np.array_equal(g.get_spins(), o.spins)
    b.close()
    g.close()


def test_a_batch_reports_a_time_out_once(hook):
    b = lt.Batch()
    (g, _), (f, o) = _pair(512), _pair(300, seed=8)
    b.add(g, 8)
    b.add(f, 8)
    hook(POLLS, 1)
    b.run()
    assert _codes(b.synchronize, b.synchronize) == [ETIMEOUT, 0]
    hook(0, 0)
    b.add(f, 4)
    b.run()                              # the healthy lattice goes on
    b.synchronize()
    o.sweep(12)
    assert np.array_equal(f.get_spins(), o.spins)
    b.close()


def test_a_run_with_a_lattice_that_timed_out_meanwhile(hook):
    b = lt.Batch()
    (g, _), (f, o) = _pair(512), _pair(300, seed=8)
    b.add(g, 8)                          # added while it was whole
    b.add(f, 8)
    _silence(hook, g, 3)
    assert _codes(b.run) == [ETIMEOUT]
    assert f.sweeps() == 0 and np.array_equal(f.get_spins(), o.spins)   # nothing was queued
    b.close()


def test_a_server_request_that_timed_out_ends_alone(hook):
    hook(POLLS, 1)                       # a band of the larger lattice, in the first round that has both
    s = lt.Server(max_slots=8, chunk_sweeps=32)
    ids = [s.submit(2, L, 1, lt.ISING, 1.0, 0.0, 2.3, seed=L, sweeps=1280, keep_spins=True) for L in (600, 200)]
    s.drain(60.0)
    spins = np.empty(200 * 200, dtype=np.int8)
    assert s.poll(ids[0])["status"] == ETIMEOUT
    assert s.poll(ids[1], spins)["status"] == 0
    s.close()
    o = oracle.Lattice(2, 200, 1, lt.ISING, 1.0, 0.0, 2.3, seed=200, init=lt.INIT_RANDOM)
    o.sweep(1280)
    assert np.array_equal(spins, o.spins)
