"""The sweeps this library is used for, as timed cases.

A case is one program's inner loop: lattices that live on the GPU are
advanced by some sweeps and the per-sweep counters (energy and magnetisation
sums) are read back, through the Python binding of the C ABI.  Every output
is a whole number (spins, exact counters), the same on every correct build.
"""
import math

import numpy as np
import torch

import paper_1209_0296_gb300 as lt

TC = 2.0 / math.log(1.0 + math.sqrt(2.0))   # 2D Ising critical temperature


def _case(name, kind, **kw):
    c = {"kind": kind, "dims": 2, "L": 64, "two_S": 1, "J": 1.0, "h": 0.0, "T": 2.269185, "bits": False,
         "cold": False, "reference": False, "sweeps": 1, "read": True}
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the paper's smallest lattice advanced one sweep per call, as a
        # program that looks at every configuration does: launches only
        _case("ising2d_L64_single", "ising", L=64, sweeps=1, read=False),
        # the same lattice, cold start, a whole run of 1000 recorded sweeps
        _case("ising2d_L64_run", "ising", L=64, cold=True, sweeps=1000),
        # the headline lattice: L = 4096 near T_c, int8 spins
        _case("ising2d_L4096", "ising", L=4096, sweeps=100),
        # the same in the one-bit layout
        _case("ising2d_L4096_bits", "ising", L=4096, bits=True, T=2.0, sweeps=100),
        # a size that is no multiple of 32, in a field
        _case("ising2d_L1000_field", "ising", L=1000, h=0.15, sweeps=200),
        # 3D spin-1 lattice of the temperature scan
        _case("ising3d_spin1_L256", "ising", dims=3, L=256, two_S=2, T=2.933333333, sweeps=20),
        # the North-East model at equilibrium, the largest lattice
        _case("ne_L8192", "ne", J=0.0, L=8192, T=0.3, sweeps=20),
        # the North-East autocorrelation Phi(t) at an odd size and low density
        _case("ne_L1022_phi", "ne", J=0.0, L=1022, T=0.1, reference=True, sweeps=200),
        # the paper's own North-East algorithm: random sites in 32 x 32 sub-lattices
        _case("ne_random_site_L2048", "rsite", J=0.0, L=2048, T=0.42, tile=32, lam=16, sweeps=10),
        # a served mix: uneven Ising and North-East lattices advanced together
        _case("batch_served_mix", "batch", lattices=16, Lmin=132, Lmax=2048, mix=99, sweeps=64),
        # 3-state Potts model at its critical temperature
        _case("potts_q3_L2048", "potts", L=2048, two_S=2, T=1.0 / math.log(1.0 + math.sqrt(3.0)), sweeps=40),
        # +-J spin glass: Eq. 1 with a random sign per bond
        _case("spin_glass_L2048", "glass", L=2048, T=1.0, sweeps=40),
    ]


def _even(rng, lo, hi, step=2):
    """Log-uniform multiple of `step` in [lo, hi]."""
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return min(hi, max(lo, int(round(v / step)) * step))


def draw(rng):
    kind = rng.choice(["ising", "ising", "ising", "bits", "spin3d", "ne", "ne", "rsite", "batch", "potts", "glass",
                       "fields"])
    work = math.exp(rng.uniform(math.log(2e6), math.log(4e8)))   # site updates of the pass
    c = None
    if kind == "ising":
        L = _even(rng, 32, 6000, rng.choice([2, 32]))
        c = _case(None, "ising", L=L, T=rng.uniform(1.5, 3.5), h=rng.choice([0.0, 0.0, rng.uniform(-0.5, 0.5)]),
                  J=rng.choice([1.0, 1.0, -1.0]), reference=rng.random() < 0.2)
    elif kind == "bits":
        c = _case(None, "ising", L=_even(rng, 64, 8192, 64), bits=True, T=rng.uniform(1.5, 3.5))
    elif kind == "spin3d":
        c = _case(None, "ising", dims=3, L=_even(rng, 16, 256, rng.choice([2, 16])), two_S=rng.choice([1, 2, 2, 3]),
                  T=rng.uniform(2.0, 4.5))
        work /= 4
    elif kind == "ne":
        c = _case(None, "ne", J=0.0, L=_even(rng, 64, 8192, rng.choice([2, 32])), T=rng.uniform(0.05, 0.6),
                  reference=rng.random() < 0.3)
    elif kind == "rsite":
        c = _case(None, "rsite", J=0.0, L=_even(rng, 256, 4096, 128), T=rng.uniform(0.1, 0.45),
                  tile=rng.choice([16, 32, 64]), lam=rng.choice([8, 16, 32]))
        work /= 8
    elif kind == "batch":
        c = _case(None, "batch", lattices=rng.randrange(4, 24), Lmin=132, Lmax=_even(rng, 512, 2048),
                  mix=rng.randrange(1, 1 << 20))
        return dict(c, sweeps=rng.randrange(8, 65))
    elif kind == "potts":
        c = _case(None, "potts", L=_even(rng, 64, 3000, rng.choice([2, 16, 16])), two_S=rng.choice([1, 2, 2, 3, 4]),
                  T=rng.uniform(0.7, 1.4))
        work /= 4
    else:
        c = _case(None, kind, L=_even(rng, 64, 3000, 32), T=rng.uniform(0.8, 2.5),
                  h=rng.uniform(0.2, 1.2) if kind == "fields" else 0.0)
        work /= 2
    sites = c["L"] ** c["dims"]
    return dict(c, sweeps=max(1, min(400, int(work / sites))))


def _mix(case):
    """(model, L, T or c) of a batch case: 70% Ising, 30% North-East, L log-uniform and even."""
    r = np.random.default_rng(case["mix"])
    out = []
    for _ in range(case["lattices"]):
        ne = r.random() < 0.3
        L = int(round(math.exp(r.uniform(math.log(case["Lmin"]), math.log(case["Lmax"]))) / 2)) * 2
        out.append((lt.NE if ne else lt.ISING, L, r.uniform(0.05, 0.3) if ne else r.uniform(1.5, 3.5)))
    return out


class _DeviceSpins:
    """Lets torch see lattice_device_spins' buffer; torch keeps this object,
    and with it the lattice that owns the memory, as long as the tensor."""

    def __init__(self, lat, ptr, nbytes):
        self.owner = lat
        self.__cuda_array_interface__ = {"shape": (nbytes,), "typestr": "|i1", "data": (ptr, False), "version": 3}


class _State:
    def __init__(self, case):
        self.case = case
        self.lats = []
        self.batch = None
        self.views = {}

    def spins(self, lat):
        """The lattice's current spins on the device (two buffers take turns)."""
        ptr, nbytes = lat.device_spins()
        if ptr not in self.views:
            self.views[ptr] = torch.as_tensor(_DeviceSpins(lat, ptr, nbytes), device="cuda")
        return self.views[ptr]


def prepare(case, seed):
    s = _State(case)
    rng = np.random.default_rng(seed)
    key = int(rng.integers(1 << 62))
    kind = case["kind"]
    if kind == "batch":
        for i, (model, L, T) in enumerate(_mix(case)):
            ne = model == lt.NE
            s.lats.append(lt.Lattice(2, L, 1, model, 0.0 if ne else 1.0, 0.0, T, seed=key + i,
                                     init=lt.INIT_EQUILIBRIUM if ne else lt.INIT_RANDOM))
        s.batch = lt.Batch()
        return s
    model = {"ne": lt.NE, "rsite": lt.NE, "potts": lt.POTTS}.get(kind, lt.ISING)
    init = lt.INIT_EQUILIBRIUM if model == lt.NE else lt.INIT_COLD if case["cold"] else lt.INIT_RANDOM
    lat = lt.Lattice(case["dims"], case["L"], case["two_S"], model, case["J"], case["h"], case["T"], seed=key,
                     init=init, layout=lt.BITPACKED if case["bits"] else lt.INT8)
    n = lat.N
    if kind == "glass":
        lat.set_couplings((2 * rng.integers(0, 2, case["dims"] * n, dtype=np.int8) - 1).astype(np.int8))
    if kind == "fields":
        lat.set_fields((2 * rng.integers(0, 2, n, dtype=np.int8) - 1).astype(np.int8))
    if kind == "rsite":
        lat.set_dynamics(lt.DYNAMICS_RANDOM_SITE, case["tile"], case["lam"])
    if case["reference"]:
        lat.set_reference()
    s.lats.append(lat)
    return s


def run(state):
    case = state.case
    n = case["sweeps"]
    if state.batch is not None:
        for lat in state.lats:
            state.batch.add(lat, n)
        state.batch.run()
    else:
        state.lats[0].sweep(n)
    out = {"spins": [state.spins(lat) for lat in state.lats]}
    if case["read"]:
        firsts = [lat.sweeps() - n for lat in state.lats]
        series = [lat.series(f, n) for lat, f in zip(state.lats, firsts)]
        out["series"] = {k: np.concatenate([s[k] for s in series]) for k in series[0]}
        if case["reference"]:
            out["overlap"] = state.lats[0].autocorrelation(firsts[0], n)[0]
        if case["kind"] == "fields":
            out["field"] = state.lats[0].field_series(firsts[0], n)
    return out


def work(case):
    """Bytes: the spins (and persistence flags, disorder signs, reference)
    read once and the new ones and the counters written once.  Operations,
    as integer operations: a Philox4x32-10 call is 18 wide products and 19
    logic operations for 4 sites of spin 1/2 or 2 sites otherwise; a site
    adds its neighbours, compares and updates itself; a North-East site
    draws only where the move is free and not certain."""
    n = case["sweeps"]

    def one(kind, L, dims, two_S, T):
        sites = L ** dims
        per = 2.0 * sites * (0.125 if case["bits"] else 1.0)
        if kind in ("ne", "rsite"):
            per += 0.5 * sites
        per += sites * (case["reference"] + (kind in ("glass", "fields")))
        draws = 37.0 / (4.0 if two_S == 1 else 2.0)
        if kind == "ne":
            draws *= T * T
        if kind == "rsite":
            draws = 37.0 / 2.0
        return per + 32.0 * n, n * sites * (draws + 2.0 * dims + 2.0)

    if case["kind"] == "batch":
        parts = [one("ne" if m == lt.NE else "ising", L, 2, 1, T) for m, L, T in _mix(case)]
    else:
        parts = [one(case["kind"], case["L"], case["dims"], case["two_S"], case["T"])]
    return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}


def exact(case, seed):
    """No output is a rounded number: spins and counters are whole."""
    return None
