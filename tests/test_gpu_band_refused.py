"""Bands refused (no memory for the packets, fewer usable SMs than the device
reports): the launches do the sweeps, whoever asked for them, and the results
and counts are those of the CPU oracle."""
import numpy as np
import pytest

import oracle
import paper_1209_0296_gb300 as lt

pytestmark = pytest.mark.gpu


@pytest.fixture
def lib():
    l = lt.load()
    yield l
    l.lattice_test_band_refuse(0)
    l.lattice_test_fail_alloc(0)


def _make(L, seed, ne=False):
    a = (2, L, 1, lt.NE, 0.0, 0.0, 0.3) if ne else (2, L, 1, lt.ISING, 1.0, 0.0, 2.3)
    init = lt.INIT_EQUILIBRIUM if ne else lt.INIT_RANDOM
    return lt.Lattice(*a, seed=seed, init=init), oracle.Lattice(*a, seed=seed, init=init)


def _check(g, o, ser_o, first, n):
    assert g.sweeps() == first + n
    assert np.array_equal(g.get_spins(), o.spins)
    ser = g.series(first, n)
    for k in ("bond", "mag", "up"):
        assert np.array_equal(ser[k], ser_o[k]), k


# the tuning call: no memory at its first band launch; that launch, its second and a later one refused
# (sizes no other test tunes, so that each call times its candidates)
@pytest.mark.parametrize("L,how,at", [(214, "memory", 1), (218, "launch", 1), (222, "launch", 2), (226, "launch", 3),
                                      (352, "memory", 1), (416, "launch", 2), (672, "launch", 3)])
def test_tuning_call(lib, L, how, at):
    g, o = _make(L, L)
    (lib.lattice_test_fail_alloc if how == "memory" else lib.lattice_test_band_refuse)(at)
    before = lib.lattice_test_band_launches()
    g.sweep(60)
    assert lib.lattice_test_band_refuse(0) == 0
    _check(g, o, o.sweep(60), 0, 60)
    g.sweep(9)
    _check(g, o, o.sweep(9), 60, 9)
    if L % 32:                                            # (else the tuner may have found another kernel)
        assert lib.lattice_test_band_launches() > before  # bands again
    g.close()


# 170 lattices go in two band launches or more: none, the second or a later one is refused
@pytest.mark.parametrize("at", [1, 2])
def test_batch(lib, at):
    pairs = [_make(130 + 2 * (i % 9), 700 + i, i % 4 == 1) for i in range(170)]
    b = lt.Batch()
    for rep in range(2):                 # the second run follows on what both forms left
        lib.lattice_test_band_refuse(at if rep == 0 else 0)
        before = lib.lattice_test_band_launches()
        for i, (g, _) in enumerate(pairs):
            b.add(g, 20 + i % 3)
        b.run()
        b.synchronize()
        assert (lib.lattice_test_band_launches() - before) == (at - 1) or rep == 1
        for i in range(0, 170, 11):
            g, o = pairs[i]
            n = 20 + i % 3
            _check(g, o, o.sweep(n), rep * n, n)
    b.close()


def test_batch_without_memory_for_the_packets(lib):
    b = lt.Batch()
    pairs = [_make(L, L) for L in (300, 512, 610)]
    for g, _ in pairs:
        g.sweep(1)
        b.add(g, 12)
    lib.lattice_test_fail_alloc(2)       # the band descriptors, then the packets
    b.run()
    lib.lattice_test_fail_alloc(0)
    for g, o in pairs:
        o.sweep(1)
        _check(g, o, o.sweep(12), 1, 12)
    b.close()
