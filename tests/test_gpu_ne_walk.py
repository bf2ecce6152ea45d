"""The c-mode North-East kernels (draws queued per warp, "unflipped" carried
from sweep to sweep) against the CPU oracle, bit for bit: both directions of
the certain move (c below, at and above 1/2), chunk and group remainders,
the counter's carry over other kernels and over a restored state."""
import numpy as np
import pytest

import oracle
import paper_1209_0296_gb300 as lt

pytestmark = pytest.mark.gpu


def _make(L, c, seed):
    a = (2, L, 1, lt.NE, 0.0, 0.0, c)
    init = lt.INIT_EQUILIBRIUM
    return lt.Lattice(*a, seed=seed, init=init), oracle.Lattice(*a, seed=seed, init=init)


def _check(g, o, first, ser_o, n):
    spins, flags, _ = g.get_state()
    assert np.array_equal(spins, o.spins)
    assert np.array_equal(flags, o.flags)
    ser = g.series(first, n)
    for k in ("bond", "mag", "up", "unflipped"):
        assert np.array_equal(ser[k], ser_o[k]), k


@pytest.mark.parametrize("L,c", [(2, 0.3), (4, 0.7), (6, 0.5), (30, 0.05), (34, 0.95), (62, 0.6), (64, 0.5),
                                 (96, 0.9), (126, 0.999), (160, 0.3), (254, 0.45), (288, 0.8), (1056, 0.6)])
def test_c_on_both_sides_of_one_half(L, c):
    g, o = _make(L, c, 70 + L)
    n = 12 if L < 500 else 3
    g.set_kernel(lt.KERNEL_WIDE)
    g.set_reference()
    o.set_reference()
    ser_o = o.sweep(n)
    g.sweep(n)
    _check(g, o, 0, ser_o, n)
    assert np.array_equal(g.autocorrelation(0, n, m=0.0)[0], ser_o["overlap"])
    g.close()


def test_unflipped_carries_over_kernels_and_restored_states():
    g, o = _make(64, 0.35, 5)
    for kernel, n in [(lt.KERNEL_WIDE, 3), (lt.KERNEL_GENERIC, 2), (lt.KERNEL_WIDE, 4), (lt.KERNEL_TILED, 1),
                      (lt.KERNEL_WIDE, 2), (lt.KERNEL_RESIDENT, 2), (lt.KERNEL_WIDE, 200)]:
        g.set_kernel(kernel)
        first = g.sweeps()
        ser_o = o.sweep(n)
        g.sweep(n)
        _check(g, o, first, ser_o, n)
    spins, flags, done = g.get_state()
    h, _ = _make(64, 0.35, 5)
    h.set_kernel(lt.KERNEL_WIDE)
    h.set_state(spins, flags, done)     # the series restarts here
    ser_o = o.sweep(5)
    h.sweep(5)
    _check(h, o, done, ser_o, 5)
    g.close()
    h.close()


def test_batched_above_one_half():
    b = lt.Batch()
    pairs = [_make(L, c, 300 + L) for L, c in [(132, 0.7), (160, 0.55), (610, 0.9), (704, 0.2), (130, 0.5)]]
    for g, _ in pairs:
        b.add(g, 9)
    b.run()
    b.synchronize()
    for g, o in pairs:
        _check(g, o, 0, o.sweep(9), 9)
        g.close()
    b.close()
