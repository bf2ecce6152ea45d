"""Sweeps beside and under a caller's stream capture: what the library
allocates on the way does not break a capture on another stream, and a
lattice whose captured sweeps are replayed goes on from the device's count."""
import os
import subprocess
import sys

import numpy as np
import pytest

import oracle
import paper_1209_0296_gb300 as lt

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# a process of its own: the first band launch, event and read-back of a process allocate
BESIDE = """
import sys; sys.path.insert(0, %r)
import numpy as np, torch
import oracle, paper_1209_0296_gb300 as lt
s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
a = (2, 512, 1, lt.ISING, 1.0, 0.0, 2.3)
g = lt.Lattice(*a, seed=3, init=lt.INIT_RANDOM, stream=s2)
o = oracle.Lattice(*a, seed=3, init=lt.INIT_RANDOM)
x = torch.zeros(16, device="cuda")
torch.cuda.synchronize()
graph = torch.cuda.CUDAGraph()
with torch.cuda.graph(graph, stream=s1):      # global capture mode
    x += 1
    g.sweep(6)                                # on another stream: bands
    x += 1
graph.replay()
torch.cuda.synchronize()
assert x.sum().item() == 32.0
o.sweep(6)
assert np.array_equal(g.get_spins(), o.spins)
assert lt.load().lattice_test_band_launches() == 1
print("fine")
"""


def test_beside_a_capture():
    r = subprocess.run([sys.executable, "-c", BESIDE % ROOT], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip().endswith("fine"), r.stderr[-2000:]


# host count 2, device count 2 per replay: direct, band and resident sweeps follow the device's
@pytest.mark.parametrize("L,ne,then", [(512, False, [1, 20, 2]), (300, False, [20, 1]), (64, False, [1, 3, 40]),
                                       (512, True, [1, 20]), (64, True, [2, 30])])
def test_after_replays_of_a_captured_sweep(L, ne, then):
    s = torch.cuda.Stream()
    a = (2, L, 1, lt.NE, 0.0, 0.0, 0.3) if ne else (2, L, 1, lt.ISING, 1.0, 0.0, 2.3)
    init = lt.INIT_EQUILIBRIUM if ne else lt.INIT_RANDOM
    g = lt.Lattice(*a, seed=4, init=init, stream=s)
    o = oracle.Lattice(*a, seed=4, init=init)
    g.sweep(2)                                # kernels loaded
    g.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s):
        g.sweep(2)
    with torch.cuda.stream(s):
        for _ in range(3):
            graph.replay()
    o.sweep(2 + 6)
    for n in then:
        g.sweep(n)
        o.sweep(n)
        spins, flags, _ = g.get_state()
        assert np.array_equal(spins, o.spins), n
        if ne:
            assert np.array_equal(flags, o.flags), n
    g.close()


def test_a_batch_after_replays_of_a_captured_sweep():
    s = torch.cuda.Stream()
    a = (2, 300, 1, lt.ISING, 1.0, 0.0, 2.3)
    g = lt.Lattice(*a, seed=4, init=lt.INIT_RANDOM, stream=s)
    o = oracle.Lattice(*a, seed=4, init=lt.INIT_RANDOM)
    g.sweep(2)
    g.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s):
        g.sweep(2)
    with torch.cuda.stream(s):
        for _ in range(3):
            graph.replay()
    b = lt.Batch(stream=s)
    b.add(g, 12)
    b.run()
    b.synchronize()
    o.sweep(2 + 6 + 12)
    assert np.array_equal(g.get_spins(), o.spins)
    b.close()
    g.close()
