"""The two-launch sweeps (a graph size keeps the bands away) against the CPU
oracle, bit for bit: one chunk a thread and row walks, bands of threads that
begin inside a warp, rows of any byte alignment, every table kind, references,
graph replays and direct launches; and the batch's step loop over the same."""
import numpy as np
import pytest

import oracle
import paper_1209_0296_gb300 as lt

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def no_bands():
    before = lt.load().lattice_test_band_launches()
    yield
    assert lt.load().lattice_test_band_launches() == before   # these tests are for the other kernels


def _pair(args, seed, init, kind=None, reference=False, layout=lt.INT8, graph=4):
    g = lt.Lattice(*args, seed=seed, init=init, layout=layout)
    o = oracle.Lattice(*args, seed=seed, init=init)
    L = args[1]
    for x, s in ((g, np.random.default_rng(seed)), (o, np.random.default_rng(seed))):
        sign = lambda n: np.where(s.random(n) < 0.5, -1, 1).astype(np.int8)
        if kind in ("bonds", "both"):
            x.set_couplings(sign(2 * L * L))
        if kind in ("fields", "both"):
            x.set_fields(sign(L * L))
        if reference:
            x.set_reference()
    g.set_kernel(lt.KERNEL_AUTO if layout == lt.BITPACKED else lt.KERNEL_WIDE, 0, 0, graph)
    return g, o


def _check(g, o, ser_o, n, kind=None, reference=False):
    first, ne = g.sweeps() - n, g.model == lt.NE
    ser = g.series(first, n)
    for k in ("bond", "mag", "up") + (("unflipped",) if ne else ()):
        assert np.array_equal(ser[k], ser_o[k]), (k, n)
    if reference:
        assert np.array_equal(g.autocorrelation(first, n, m=0.0)[0], ser_o["overlap"])
    if kind in ("fields", "both"):
        assert np.array_equal(g.field_series(first, n), ser_o["field"])
    spins, flags, _ = g.get_state()
    assert np.array_equal(spins, o.spins)
    if ne:
        assert np.array_equal(flags, o.flags)


def _run(args, seed, init, calls, **kw):
    g, o = _pair(args, seed, init, **kw)
    kw.pop("layout", None)
    kw.pop("graph", None)
    for n in calls:
        g.sweep(n)
        _check(g, o, o.sweep(n), n, **kw)
    g.close()


# one chunk a thread (to two waves of threads), then row walks of two rows or three, then of ten and more (16-bit
# acceptance for symmetric tables)
@pytest.mark.parametrize("L", [34, 62, 64, 250, 256, 1000, 1024, 2050, 2300, 2400])
@pytest.mark.parametrize("J,h", [(1.0, 0.0), (1.0, 0.3), (-0.7, 0.0)])
def test_ising(L, J, h):
    _run((2, L, 1, lt.ISING, J, h, 2.3), 11 + L, lt.INIT_RANDOM, [1, 6, 3] if L < 1000 else [2], reference=L in (62, 256, 2300, 2400))


@pytest.mark.parametrize("L", [4998, 5024])
@pytest.mark.parametrize("h,ref", [(0.0, False), (0.0, True), (0.2, False)])
def test_ising_long_walks(L, h, ref):
    _run((2, L, 1, lt.ISING, 1.0, h, 2.269185), 4, lt.INIT_RANDOM, [2], reference=ref)


@pytest.mark.parametrize("L", [32, 96, 2400, 5024])
@pytest.mark.parametrize("kind,h", [("bonds", 0.0), ("bonds", 0.4), ("fields", 0.6), ("fields", 0.0), ("both", 0.5)])
def test_disorder(L, kind, h):
    if L > 3000 and (kind, h) in (("fields", 0.0), ("both", 0.5)):
        pytest.skip("the same kernel as fields")
    _run((2, L, 1, lt.ISING, 1.0, h, 1.7), 3, lt.INIT_RANDOM, [1, 5] if L < 100 else [2], kind=kind, reference=L in (96, 2400))


# c on both sides of 1/2 and at it, where no move needs a draw; walks of two or three rows, and of row pairs
@pytest.mark.parametrize("L", [6, 62, 64, 250, 256, 1000, 1024, 2734, 2752])
@pytest.mark.parametrize("c", [0.2, 0.5, 0.8])
def test_north_east(L, c):
    _run((2, L, 1, lt.NE, 0.0, 0.0, c), 2 + L, lt.INIT_EQUILIBRIUM, [1, 6, 3] if L < 1000 else [2],
         reference=L in (62, 256, 2734, 2752))


@pytest.mark.parametrize("L,c", [(4736, 0.3), (4740, 0.3), (4740, 0.7)])
def test_north_east_row_pairs(L, c):
    _run((2, L, 1, lt.NE, 0.0, 0.0, c), 8, lt.INIT_EQUILIBRIUM, [2], reference=L == 4740)


# bit-packed: a word or two a thread (table look-ups), more (two draws a compare)
@pytest.mark.parametrize("L,h,ref", [(64, 0.0, False), (320, 0.0, True), (2112, 0.0, False), (2112, 0.2, True),
                                     (3776, 0.0, True), (3776, 0.0, False)])
def test_bit_packed(L, h, ref):
    _run((2, L, 1, lt.ISING, 1.0, h, 2.269185), 21, lt.INIT_RANDOM, [1, 6] if L < 1000 else [2], reference=ref,
         layout=lt.BITPACKED)


# the batch's step loop: its North-East and Ising items, aligned rows and others
def test_step_loop():
    spec = [((2, L, 1, lt.NE, 0.0, 0.0, c), c > 0.4) for L, c in
            ((132, 0.7), (160, 0.55), (610, 0.9), (704, 0.2), (130, 0.5), (1056, 0.3), (160, 0.3))]
    spec += [((2, L, 1, lt.ISING, J, h, 2.2), L > 400) for L, J, h in
             ((130, 1.0, 0.0), (160, 1.0, 0.2), (610, -0.7, 0.0), (704, 1.0, 0.0))]
    spec += [((2, 256, 1, lt.NE, 1.0, 0.2, 2.0), False)]
    pairs = [_pair(a, 50 + i, lt.INIT_EQUILIBRIUM if a[3] == lt.NE and a[4] == 0.0 else lt.INIT_RANDOM, reference=r)
             for i, (a, r) in enumerate(spec)]
    b = lt.Batch()
    for rep in range(2):
        for i, (g, _) in enumerate(pairs):
            b.add(g, 7 + i % 3)
        b.run()
        b.synchronize()
        for i, ((g, o), (_, r)) in enumerate(zip(pairs, spec)):
            _check(g, o, o.sweep(7 + i % 3), 7 + i % 3, reference=r)
    b.close()
