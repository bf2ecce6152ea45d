"""Sweeps beside a caller's stream capture: what the library
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
