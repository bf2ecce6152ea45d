"""The band-resident kernel (many sweeps per launch, rows of a lattice split
over the SMs) against the CPU oracle, bit for bit: two bands to one per SM,
bands of two rows, rows of any byte alignment, partial chunks and groups,
odd and even sweep counts mixed with single sweeps (other kernels), every
table kind, disorder, a reference state."""
import numpy as np
import pytest

import oracle
import paper_1209_0296_gb300 as lt

pytestmark = pytest.mark.gpu


def _run(args, seed, init, calls, reference=False, bonds=None, fields=None):
    g = lt.Lattice(*args, seed=seed, init=init)
    o = oracle.Lattice(*args, seed=seed, init=init)
    g.set_kernel(lt.KERNEL_WIDE)
    if bonds is not None:
        g.set_couplings(bonds)
        o.set_couplings(bonds)
    if fields is not None:
        g.set_fields(fields)
        o.set_fields(fields)
    if reference:
        g.set_reference()
        o.set_reference()
    done = 0
    for n in calls:
        ser_o = o.sweep(n)
        g.sweep(n)
        ser = g.series(done, n)
        for k in ("bond", "mag", "up") + (("unflipped",) if args[3] == lt.NE else ()):
            assert np.array_equal(ser[k], ser_o[k]), (k, n)
        if reference:
            assert np.array_equal(g.autocorrelation(done, n, m=0.0)[0], ser_o["overlap"])
        if fields is not None:
            assert np.array_equal(g.field_series(done, n), ser_o["field"])
        spins, flags, _ = g.get_state()
        assert np.array_equal(spins, o.spins), n
        if args[3] == lt.NE:
            assert np.array_equal(flags, o.flags), n
        done += n
    g.close()


CALLS = [5, 1, 4, 7]


@pytest.mark.parametrize("L", [4, 6, 34, 62, 64, 100, 130, 250, 304, 306, 610])
@pytest.mark.parametrize("J,h", [(1.0, 0.0), (1.0, 0.3), (-0.7, 0.0), (0.0, 0.0)])
def test_ising(L, J, h):
    _run((2, L, 1, lt.ISING, J, h, 2.3), 17 + L, lt.INIT_RANDOM, CALLS, reference=L in (6, 64, 250))


@pytest.mark.parametrize("L,c", [(4, 0.4), (6, 0.3), (34, 0.7), (62, 0.1), (64, 0.5), (130, 0.3), (304, 0.05),
                                 (306, 0.9), (510, 0.35)])
def test_north_east(L, c):
    _run((2, L, 1, lt.NE, 0.0, 0.0, c), 5 + L, lt.INIT_EQUILIBRIUM, CALLS, reference=L in (6, 64, 306))


@pytest.mark.parametrize("model", [lt.ISING, lt.NE])
@pytest.mark.parametrize("L", [1000, 2050])
def test_large(L, model):
    a = (0.0, 0.0, 0.25) if model == lt.NE else (1.0, 0.0, 2.269185)
    _run((2, L, 1, model) + a, 3, lt.INIT_EQUILIBRIUM if model == lt.NE else lt.INIT_RANDOM, [4])


@pytest.mark.parametrize("L", [32, 96, 320])
@pytest.mark.parametrize("kind", ["bonds", "bonds_h", "fields", "both"])
def test_disorder(L, kind):
    rng = np.random.default_rng(L)
    sign = lambda n: np.where(rng.random(n) < 0.5, -1, 1).astype(np.int8)
    bonds = sign(2 * L * L) if kind != "fields" else None
    fields = sign(L * L) if kind in ("fields", "both") else None
    h = 0.0 if kind == "bonds" else 0.6
    _run((2, L, 1, lt.ISING, 1.0, h, 1.7), 9, lt.INIT_RANDOM, CALLS, reference=L == 96, bonds=bonds, fields=fields)


@pytest.mark.parametrize("L", [64, 128, 320, 704, 2112])
def test_bit_packed(L):
    a = (2, L, 1, lt.ISING, 1.0, 0.0, 2.269185)
    g = lt.Lattice(*a, seed=L, init=lt.INIT_RANDOM, layout=lt.BITPACKED)
    o = oracle.Lattice(*a, seed=L, init=lt.INIT_RANDOM)
    if L in (128, 704):
        g.set_reference()
        o.set_reference()
    done = 0
    for n in ([17, 1, 16, 5] if L < 1000 else [5]):
        ser_o = o.sweep(n)
        g.sweep(n)
        ser = g.series(done, n)
        for k in ("bond", "mag", "up"):
            assert np.array_equal(ser[k], ser_o[k]), (k, n)
        if L in (128, 704):
            assert np.array_equal(g.autocorrelation(done, n, m=0.0)[0], ser_o["overlap"])
        assert np.array_equal(g.get_spins(), o.spins), n
        done += n
    g.close()


# bands of more than one 16-site chunk a thread hold one bit a site: rows that
# end inside a word, both directions of the certain move, references, bonds
@pytest.mark.parametrize("L,ne,par,ref", [(1630, False, 2.3, True), (1602, False, 2.0, False), (1664, False, 2.5, False),
                                          (1630, True, 0.3, True), (1602, True, 0.8, False), (1664, True, 0.1, True),
                                          (1700, True, 0.5, False)])
def test_bits_on_chip(L, ne, par, ref):
    a = (2, L, 1, lt.NE, 0.0, 0.0, par) if ne else (2, L, 1, lt.ISING, 1.0, 0.0, par)
    _run(a, 3 + L, lt.INIT_EQUILIBRIUM if ne else lt.INIT_RANDOM, [3, 1, 4], reference=ref)


def test_bits_on_chip_with_bonds():
    rng = np.random.default_rng(8)
    L = 1632
    bonds = np.where(rng.random(2 * L * L) < 0.5, -1, 1).astype(np.int8)
    _run((2, L, 1, lt.ISING, 1.0, 0.0, 1.2), 4, lt.INIT_RANDOM, [5, 6], reference=True, bonds=bonds)


@pytest.mark.parametrize("L,c", [(64, 0.3), (320, 0.7), (1728, 0.15)])
def test_bit_packed_north_east(L, c):
    a = (2, L, 1, lt.NE, 0.0, 0.0, c)
    g = lt.Lattice(*a, seed=L, init=lt.INIT_EQUILIBRIUM, layout=lt.BITPACKED)
    o = oracle.Lattice(*a, seed=L, init=lt.INIT_EQUILIBRIUM)
    done = 0
    for n in ([17, 1, 18] if L < 1000 else [3, 2, 4]):
        ser_o = o.sweep(n)
        g.sweep(n)
        ser = g.series(done, n)
        for k in ("bond", "mag", "up", "unflipped"):
            assert np.array_equal(ser[k], ser_o[k]), (k, n)
        spins, flags, _ = g.get_state()
        assert np.array_equal(spins, o.spins) and np.array_equal(flags, o.flags)
        done += n
    g.close()


# words of 32 sites, partial last words, two-row bands, dE = 0 and infinite-T moves, references
@pytest.mark.parametrize("L,J,T", [(4, 1.0, 0.9), (6, 1.0, 1.5), (62, 1.0, 0.995), (64, 0.0, 1.0), (66, 1.0, 0.3),
                                   (130, 0.7, 0.7), (306, 1.0, 0.995), (610, 1.0, 2.0), (896, 0.0, 1.0), (1632, 1.0, 0.995)])
def test_potts3(L, J, T):
    a = (2, L, 2, lt.POTTS, J, 0.0, T)
    g = lt.Lattice(*a, seed=L, init=lt.INIT_RANDOM)
    o = oracle.Lattice(*a, seed=L, init=lt.INIT_RANDOM)
    ref = L in (62, 306, 896)
    if ref:
        g.set_reference()
        o.set_reference()
    done = 0
    for n in ([17, 1, 16, 5] if L < 1000 else [4, 3]):
        ser_o = o.sweep(n)
        g.sweep(n)
        ser = g.series(done, n)
        for k in ("bond", "mag", "up"):
            assert np.array_equal(ser[k], ser_o[k]), (k, n)
        if ref:
            assert np.array_equal(g.autocorrelation(done, n, m=0.0)[0], ser_o["overlap"])
        assert np.array_equal(g.get_spins(), o.spins), n
        done += n
    g.close()


# one lattice through kinds with packets of different sizes: bits, then fields (int8; h = 0, so that they are not
# felt), bonds (bits), uniform again; in bands and, one sweep, in launches
def test_kinds_of_one_lattice():
    rng = np.random.default_rng(1)
    L, n = 1632, 4
    a = (2, L, 1, lt.ISING, 1.0, 0.0, 1.6)
    g = lt.Lattice(*a, seed=2, init=lt.INIT_RANDOM)
    o = oracle.Lattice(*a, seed=2, init=lt.INIT_RANDOM)
    g.set_kernel(lt.KERNEL_WIDE)
    sign = lambda m: np.where(rng.random(m) < 0.5, -1, 1).astype(np.int8)
    for step in ("uniform", "fields", "bonds", "none"):
        fields = sign(L * L) if step == "fields" else None
        bonds = sign(2 * L * L) if step == "bonds" else None
        for x in (g, o):
            x.set_fields(fields)
            x.set_couplings(bonds)
        for m in (n, 1):
            g.sweep(m)
            o.sweep(m)
            assert np.array_equal(g.get_spins(), o.spins), (step, m)
    g.close()


# bands of more than 1024 words: North-East with twice the threads, rows ending inside a word
def test_north_east_more_threads():
    _run((2, 3202, 1, lt.NE, 0.0, 0.0, 0.3), 6, lt.INIT_EQUILIBRIUM, [5, 6], reference=True)


# the one-CTA kernel for L = 32 and 64: runs of one, two and many sweeps, every table kind, references
@pytest.mark.parametrize("L", [32, 64])
@pytest.mark.parametrize("model,J,h,par", [(lt.ISING, 1.0, 0.0, 2.3), (lt.ISING, 1.0, 0.3, 2.0), (lt.ISING, -0.7, 0.0, 1.5),
                                           (lt.NE, 0.0, 0.0, 0.3), (lt.NE, 0.0, 0.0, 0.7)])
@pytest.mark.parametrize("ref", [False, True])
def test_resident_words(L, model, J, h, par, ref):
    a = (2, L, 1, model, J, h, par)
    init = lt.INIT_EQUILIBRIUM if model == lt.NE else lt.INIT_RANDOM
    g = lt.Lattice(*a, seed=L, init=init)
    o = oracle.Lattice(*a, seed=L, init=init)
    g.set_kernel(lt.KERNEL_RESIDENT)
    if ref:
        g.set_reference()
        o.set_reference()
    done = 0
    for n in (1, 2, 3, 40):
        ser_o = o.sweep(n)
        g.sweep(n)
        ser = g.series(done, n)
        for k in ("bond", "mag", "up") + (("unflipped",) if model == lt.NE else ()):
            assert np.array_equal(ser[k], ser_o[k]), (k, n)
        if ref:
            assert np.array_equal(g.autocorrelation(done, n, m=0.0)[0], ser_o["overlap"])
        spins, flags, _ = g.get_state()
        assert np.array_equal(spins, o.spins), n
        if model == lt.NE:
            assert np.array_equal(flags, o.flags), n
        done += n
    g.close()
