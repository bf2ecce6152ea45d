"""Bounded waits of the band-resident kernels: a band that sends nothing makes
its neighbours' waits run out, the launch ends normally and the host sees the
error; nothing of it stays behind for the next launch."""
import time

import numpy as np
import pytest

import oracle
import paper_1209_0296_gb300 as lt

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


# every form: one chunk a thread, int8 in several, bits, North-East on bits, Potts planes, bit-packed
@pytest.mark.parametrize("kw", [dict(L=256), dict(L=1632, h=0.3), dict(L=1632), dict(L=1632, model=lt.NE, J=0.0, par=0.3),
                                dict(L=1632, model=lt.POTTS, two_S=2, par=0.995), dict(L=1664, layout=lt.BITPACKED)])
@pytest.mark.parametrize("band", [1, 4])
def test_a_silent_band_ends_the_launch(hook, kw, band):
    g, o = _pair(**kw)
    g.set_kernel(lt.KERNEL_AUTO if kw.get("layout") or kw.get("two_S") else lt.KERNEL_WIDE)
    spins, flags, _ = g.get_state()
    hook(POLLS, band)
    g.sweep(6)
    _times_out(g)
    hook(0, 0)
    g.set_state(spins, flags, 0)         # whole again
    g.sweep(6)
    o.sweep(6)
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
