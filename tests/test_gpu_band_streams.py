"""Band-resident launches on several streams: none waits for what another
stream waits for, small lattices that meet overlap their launches, large ones
take turns; results are those of the CPU oracle whichever way they ran."""
import numpy as np
import pytest

import oracle
import paper_1209_0296_gb300 as lt

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _make(L, stream, seed):
    a = (2, L, 1, lt.ISING, 1.0, 0.0, 2.3)
    return (lt.Lattice(*a, seed=seed, init=lt.INIT_RANDOM, stream=stream),
            oracle.Lattice(*a, seed=seed, init=lt.INIT_RANDOM))


def _check(g, o, n):
    first = g.sweeps() - n
    ser_o = o.sweep(n)
    assert np.array_equal(g.get_spins(), o.spins)
    assert np.array_equal(g.series(first, n)["mag"], ser_o["mag"])


@pytest.mark.parametrize("L", [512, 1632])
def test_a_busy_stream_holds_no_other_back(L):
    s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
    (g, o), (f, q) = _make(L, s1, 1), _make(L, s2, 2)
    for x, y in ((g, o), (f, q)):        # every kernel loaded, no launch in flight
        for n in (1, 2, 8):
            x.sweep(n)
            _check(x, y, n)
    end = torch.cuda.Event()
    with torch.cuda.stream(s1):
        torch.cuda._sleep(1_000_000_000)   # half a second on s1, as work of the caller's own
    g.sweep(8)
    end.record(s1)
    f.sweep(8)
    f.synchronize()
    assert not end.query()               # s2's lattice is done while s1 still waits
    _check(f, q, 8)
    _check(g, o, 8)
    g.close()
    f.close()


def test_large_lattices_take_turns():
    pairs = [_make(1632, torch.cuda.Stream(), 5 + i) for i in range(3)]
    for g, o in pairs:
        g.set_kernel(lt.KERNEL_WIDE)     # (no tuning calls)
        g.sweep(8)
        _check(g, o, 8)
    torch.cuda.synchronize()
    before = lt.load().lattice_test_band_launches()
    for g, _ in pairs:
        g.sweep(60)
    assert lt.load().lattice_test_band_launches() - before == 3
    for g, o in pairs:
        _check(g, o, 60)
        g.close()


def test_small_lattices_that_meet_go_back_to_launches():
    pairs = [_make(256, torch.cuda.Stream(), 9 + i) for i in range(4)]
    for g, o in pairs:
        g.sweep(70)
        _check(g, o, 70)
    count = lt.load().lattice_test_band_launches
    before = count()
    for rep in range(10):
        for g, _ in pairs:
            g.sweep(100)
        torch.cuda.synchronize()
    assert count() - before < 10         # 40 calls
    for g, o in pairs:
        o.sweep(900)
        _check(g, o, 100)
    before = count()                     # alone again: bands after a while
    for _ in range(40):
        pairs[0][0].sweep(4)
        pairs[0][0].synchronize()
    assert count() - before >= 5
    o = pairs[0][1]
    o.sweep(156)
    _check(pairs[0][0], o, 4)
    for g, _ in pairs:
        g.close()


def test_batches_on_two_streams():
    bs = [lt.Batch(stream=torch.cuda.Stream()) for _ in range(2)]
    sets = [[_make(L, torch.cuda.Stream(), 30 + L + i) for L in (300, 512, 700)] for i in range(2)]
    for rep in range(3):
        for b, pairs in zip(bs, sets):
            for g, _ in pairs:
                b.add(g, 20)
            b.run()
        for b in bs:
            b.synchronize()
    for pairs in sets:
        for g, o in pairs:
            o.sweep(40)
            _check(g, o, 20)
    for b in bs:
        b.close()


# threads with a lattice and a stream each: whoever meets whom, the sweeps are the same
def test_threads():
    import threading

    sizes = [300, 512, 1000, 1632, 1632, 300]
    make = lambda i, s: lt.Lattice(2, sizes[i], 1, lt.ISING, 1.0, 0.0, 2.2, seed=80 + i, init=lt.INIT_RANDOM, stream=s)
    lats = [make(i, torch.cuda.Stream()) for i in range(len(sizes))]
    for g in lats:
        g.set_kernel(lt.KERNEL_WIDE)
    failed = []

    def work(g):
        try:
            for k in range(60):
                g.sweep(5 + k % 7)
                if k % 5 == 0:
                    g.synchronize()
            g.synchronize()
        except Exception as e:
            failed.append(e)

    threads = [threading.Thread(target=work, args=(g,)) for g in lats]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed
    n = sum(5 + k % 7 for k in range(60))
    for i, g in enumerate(lats):
        f = make(i, None)
        f.set_kernel(lt.KERNEL_WIDE, 0, 0, 8)    # launches
        f.sweep(n)
        assert np.array_equal(f.get_spins(), g.get_spins())
        assert np.array_equal(f.series(0, n)["bond"], g.series(0, n)["bond"])
        f.close()
        g.close()
