"""Batched lattices on the band-resident kernel: uneven sizes and models share
one launch, each with its own number of sweeps, and end bit for bit where
the CPU oracle ends; more lattices than SMs run in several launches."""
import numpy as np
import pytest

import oracle
import paper_1209_0296_gb300 as lt

pytestmark = pytest.mark.gpu


def _make(L, ne, par, seed, h=0.0):
    a = (2, L, 1, lt.NE, 0.0, 0.0, par) if ne else (2, L, 1, lt.ISING, 1.0, h, par)
    init = lt.INIT_EQUILIBRIUM if ne else lt.INIT_RANDOM
    return lt.Lattice(*a, seed=seed, init=init), oracle.Lattice(*a, seed=seed, init=init)


def _check(g, o, n, ne, reference=False):
    first = g.sweeps() - n
    ser_o = o.sweep(n)
    ser = g.series(first, n)
    spins, flags, _ = g.get_state()
    assert np.array_equal(spins, o.spins)
    for k in ("bond", "mag", "up") + (("unflipped",) if ne else ()):
        assert np.array_equal(ser[k], ser_o[k]), k
    if ne:
        assert np.array_equal(flags, o.flags)
    if reference:
        assert np.array_equal(g.autocorrelation(first, n, m=0.0)[0], ser_o["overlap"])


def test_uneven_lattices_share_a_launch():
    spec = [(610, False, 2.2, 0.0, 9), (132, True, 0.3, 0.0, 31), (448, False, 2.5, 0.2, 12), (700, True, 0.7, 0.0, 6),
            (250, False, 1.9, 0.0, 31), (160, True, 0.1, 0.0, 4), (1090, False, 2.269185, 0.0, 5),
            (130, False, 3.0, -0.4, 64)]
    pairs = [_make(L, ne, par, 40 + L, h) for L, ne, par, h, _ in spec]
    for i, (g, o) in enumerate(pairs):
        if i % 3 == 0:
            g.set_reference()
            o.set_reference()
    b = lt.Batch()
    for rep in range(2):                 # the second run starts at odd sweep counts, with used packets
        ns = [n + rep for *_, n in spec]
        for (g, _), n in zip(pairs, ns):
            b.add(g, n)
        b.run()
        b.synchronize()
        for i, ((g, o), n) in enumerate(zip(pairs, ns)):
            _check(g, o, n, spec[i][1], reference=i % 3 == 0)
    g, o = pairs[0]
    g.sweep(7)                           # alone, after the batch
    _check(g, o, 7, False, reference=True)
    b.close()


def test_more_lattices_than_sms():
    pairs = [_make(130 + 2 * (i % 9), i % 4 == 1, 0.25 if i % 4 == 1 else 2.3, 900 + i) for i in range(170)]
    b = lt.Batch()
    for g, _ in pairs:
        b.add(g, 40)
    b.run()
    b.synchronize()
    for i in range(0, 170, 13):
        _check(*pairs[i], 40, i % 4 == 1)
    b.close()
