"""The band-resident forms with several chunks of a byte a site per thread
(general tables: a field, J < 0, bonds in a field, field signs), with and
without a reference, alone and in a batch, against the CPU oracle; and a
batch cut into several launches.  Each test sees that bands were launched."""
import numpy as np
import pytest

import oracle
import paper_1209_0296_gb300 as lt

pytestmark = pytest.mark.gpu


@pytest.fixture
def bands():
    """bands(): band launches since the last call of it."""
    last = [lt.load().lattice_test_band_launches()]

    def since():
        now = lt.load().lattice_test_band_launches()
        n, last[0] = now - last[0], now
        return n

    return since


def _pair(L, J, h, T, seed, kind, reference):
    g = lt.Lattice(2, L, 1, lt.ISING, J, h, T, seed=seed, init=lt.INIT_RANDOM)
    o = oracle.Lattice(2, L, 1, lt.ISING, J, h, T, seed=seed, init=lt.INIT_RANDOM)
    g.set_kernel(lt.KERNEL_WIDE)
    rng = np.random.default_rng(seed)
    sign = lambda n: np.where(rng.random(n) < 0.5, -1, 1).astype(np.int8)
    b = sign(2 * L * L) if kind in ("bonds", "both") else None
    f = sign(L * L) if kind in ("fields", "both") else None
    for x in (g, o):
        if b is not None:
            x.set_couplings(b)
        if f is not None:
            x.set_fields(f)
        if reference:
            x.set_reference()
    return g, o


def _check(g, o, n, kind, reference):
    first = g.sweeps() - n
    ser_o = o.sweep(n)
    ser = g.series(first, n)
    for k in ("bond", "mag", "up"):
        assert np.array_equal(ser[k], ser_o[k]), k
    if reference:
        assert np.array_equal(g.autocorrelation(first, n, m=0.0)[0], ser_o["overlap"])
    if kind in ("fields", "both"):
        assert np.array_equal(g.field_series(first, n), ser_o["field"])
    assert np.array_equal(g.get_spins(), o.spins)


# rows ending inside a chunk (1602: one chunk and a bit a thread, 2606: nearly three) and whole chunks (2048)
@pytest.mark.parametrize("L,J,h,kind,ref,calls", [
    (1602, 1.0, 0.3, None, True, [8, 9]), (1602, -0.7, 0.0, None, False, [9]), (2606, 1.0, -0.2, None, False, [8]),
    (2048, 1.0, 0.3, None, True, [5, 6]), (2048, -0.7, 0.0, None, False, [5]), (2048, 1.0, 0.4, "bonds", True, [5, 6]),
    (1664, 1.0, 0.6, "fields", True, [12, 13]), (2048, 1.0, 0.6, "both", False, [5, 6]),
    (2048, 1.0, 0.0, "fields", True, [5])])
def test_general_tables(bands, L, J, h, kind, ref, calls):
    g, o = _pair(L, J, h, 1.9, L, kind, ref)
    for n in calls:
        g.sweep(n)
        _check(g, o, n, kind, ref)
        assert bands() == 1
    g.close()


def test_general_tables_in_a_batch(bands):
    pairs = [_pair(L, J, h, 2.1, L, None, ref) for L, J, h, ref in
             ((1602, 1.0, 0.3, True), (1632, -0.7, 0.0, False), (704, 1.0, 0.2, True), (610, 1.0, 0.0, True))]
    b = lt.Batch()
    for rep in range(2):
        for i, (g, _) in enumerate(pairs):
            b.add(g, 9 + i)
        b.run()
        b.synchronize()
        assert bands() >= 1
        for i, (g, o) in enumerate(pairs):
            _check(g, o, 9 + i, None, i != 1)
    b.close()


# long runs are cut into launches of a quarter second; a lattice of few sweeps has none in some of them
def test_a_batch_in_several_launches(bands):
    spec = [(130, 900000, 2.3), (132, 4, 2.0), (200, 7, 2.5)]
    make = lambda i: lt.Lattice(2, spec[i][0], 1, lt.ISING, 1.0, 0.0, spec[i][2], seed=60 + i, init=lt.INIT_RANDOM)
    a, c = [make(i) for i in range(3)], [make(i) for i in range(3)]
    b = lt.Batch()
    for g, (_, n, _) in zip(a, spec):
        b.add(g, n)
    b.run()
    b.synchronize()
    assert bands() >= 5
    for g, f, (_, n, _) in zip(a, c, spec):
        f.set_kernel(lt.KERNEL_WIDE)
        f.sweep(n)
        k = min(n, 50)
        sg, sf = g.series(n - k, k), f.series(n - k, k)
        assert all(np.array_equal(sg[x], sf[x]) for x in ("bond", "mag", "up"))
        assert np.array_equal(g.get_spins(), f.get_spins())
    b.close()
