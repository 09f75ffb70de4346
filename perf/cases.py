"""The work that programs have this library do, as timed cases.

A case is a dict of plain values.  Four kinds:

  ising    an L x L lattice (swgpu.Lattice), plain at temperature T or PCC:
           one pass runs `sweeps` sweeps on the resident lattice, then reads
           the per-sweep observables and the final spins back
  potts    the same for swgpu.PottsLattice (dim, q; pcc ignores T)
  batch    `jobs` replicas submitted to a swgpu.Server together and waited for
  static   one sweep on caller-owned torch tensors (sw_sweep_static)

Every output is a whole number (spins, labels, per-sweep integer sums), so two
implementations agree bit for bit or not at all.
"""
import ctypes
import math

import numpy as np
import torch

from paper_0808_2109_gb300 import swgpu
from paper_0808_2109_gb300.workloads import T_CRITICAL_ROUNDED as TC

# Critical temperatures of the Potts cases: exact in 2D (1 / ln(1 + sqrt(q))),
# the estimates that the Potts benchmark uses in 3D.
POTTS_TC = {(2, q): 1.0 / math.log(1.0 + math.sqrt(q)) for q in (2, 3, 4)}
POTTS_TC.update({(3, 2): 2.2557, (3, 3): 1.8164})

# Integer operations of a Philox4x32-10 block: ten rounds of two 32 x 32 -> 64
# products (a low and a high half each), four xors and two key additions.
PHILOX_OPS = 100

# Sweeps from the hot start before anything is measured.
EQUILIBRATION = 30


def listed():
    return [
        # A measurement loop on a small lattice: one sweep a call, its
        # observables read every time (the smallest call there is).
        {"name": "ising_L64_step", "kind": "ising", "L": 64, "T": TC, "sweeps": 1},
        # The small configured run: 1000 sweeps of a one-tile lattice.
        {"name": "ising_L64_run", "kind": "ising", "L": 64, "T": TC, "sweeps": 1000},
        # A side that no tile divides, with open boundaries, cluster sizes and
        # the topological rule: every option of a finite-size study at once.
        {"name": "ising_L1001_options", "kind": "ising", "L": 1001, "T": TC, "sweeps": 100,
         "open": True, "csize": True, "wind": True},
        # The temperature regimes of the configured L=4096 runs: a giant
        # cluster below T_c, many small ones above.
        {"name": "ising_L4096_cold", "kind": "ising", "L": 4096, "T": 2.0, "sweeps": 100},
        {"name": "ising_L4096_hot", "kind": "ising", "L": 4096, "T": 3.0, "sweeps": 100},
        # The benchmark lattice: 268M sites at T_c, 50 sweeps.
        {"name": "ising_L16384_critical", "kind": "ising", "L": 16384, "T": TC, "sweeps": 50},
        # The configured PCC lattice, a stretch of its chain.
        {"name": "pcc_L2048", "kind": "ising", "L": 2048, "sweeps": 200, "pcc": True},
        # The configured replica mix (L from 64 to 1024 on a temperature
        # ladder) through the batch server.
        {"name": "batch_mix", "kind": "batch", "jobs": 512, "Lmin": 64, "Lmax": 1024, "sweeps": 100},
        # Potts, 2D and 3D, at the benchmark's sizes.
        {"name": "potts2d_L8192_q3", "kind": "potts", "dim": 2, "L": 8192, "q": 3, "T": POTTS_TC[2, 3],
         "sweeps": 20},
        {"name": "potts3d_L512_q2", "kind": "potts", "dim": 3, "L": 512, "q": 2, "T": POTTS_TC[3, 2],
         "sweeps": 10},
        # A small 3D percolation chain (PCC with the topological rule) on a
        # side that 4 does not divide.
        {"name": "potts3d_L50_pcc", "kind": "potts", "dim": 3, "L": 50, "q": 2, "T": 1.0, "sweeps": 50,
         "pcc": True, "wind": True},
        # A sweep inside somebody else's program: device tensors in and out,
        # no allocation.
        {"name": "static_L300", "kind": "static", "L": 300, "T": TC},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _flags(rng):
    return {k: True for k in ("open", "csize", "wind") if rng.random() < 0.3}


def draw(rng):
    kind = rng.choice(["ising", "ising", "ising", "pcc", "potts2", "potts3", "batch", "static"])
    if kind == "static":
        return {"kind": "static", "L": _log_int(rng, 2, 1024), "T": rng.uniform(1.8, 3.2)}
    if kind == "batch":
        # at most the listed mix's site updates: 64 x 512^2 x 100 sites
        lmax = _log_int(rng, 64, 512)
        return {"kind": "batch", "jobs": _log_int(rng, 4, 64), "Lmin": 32, "Lmax": lmax,
                "sweeps": _log_int(rng, 10, 100)}
    if kind in ("potts2", "potts3"):
        dim = 2 if kind == "potts2" else 3
        L = _log_int(rng, 16, 8192) if dim == 2 else _log_int(rng, 8, 400)
        q = rng.choice([2, 3, 4]) if dim == 2 else rng.choice([2, 3])
        sweeps = max(1, min(100, _log_int(rng, 1, 100), int(6e8 / L ** dim)))
        c = {"kind": "potts", "dim": dim, "L": L, "q": q, "sweeps": sweeps,
             "T": POTTS_TC[dim, q] * rng.uniform(0.9, 1.3)}
        c.update(_flags(rng))
        if rng.random() < 0.2:
            c["pcc"] = True
        return c
    L = _log_int(rng, 16, 8192)
    c = {"kind": "ising", "L": L, "sweeps": max(1, min(1000, _log_int(rng, 1, 1000), int(2e9 / (L * L))))}
    if kind == "pcc":
        c["pcc"] = True
        c["sweeps"] = min(c["sweeps"], 200)
    else:
        c["T"] = rng.uniform(1.8, 3.2)
    if rng.random() < 0.4:
        c.update(_flags(rng))
    return c


# --------------------------------------------------------------- what a user holds

def _host_bytes(n):
    """Pinned host memory that the spins are read back into."""
    return torch.empty(n, dtype=torch.uint8, pin_memory=True).numpy()


def _options(case):
    return {k: bool(case.get(k)) for k in ("open", "csize", "wind")}


def _mix(case, seed):
    """Replica specs: every side of the ladder is a power of two in the
    configured mix (weights .4 .25 .2 .1 .05), any side otherwise; temperatures
    on a 32-point ladder around T_c."""
    rng = np.random.default_rng(20260)
    n, lo, hi = case["jobs"], case["Lmin"], case["Lmax"]
    if (lo, hi) == (64, 1024):
        sides = rng.choice([64, 128, 256, 512, 1024], size=n, p=[0.4, 0.25, 0.2, 0.1, 0.05])
    else:
        sides = np.rint(np.exp(rng.uniform(math.log(lo), math.log(hi), size=n)))
    return [{"L": int(sides[r]), "T": 2.0 + 0.6 * (r % 32) / 31.0, "seed": 1000 * seed + r,
             "sweeps": case["sweeps"]} for r in range(n)]


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        # a server that has served one batch before, as a long-lived one has
        srv, specs = swgpu.Server(), _mix(case, seed)
        _serve(srv, [dict(sp, sweeps=1) for sp in specs])
        return {"case": case, "srv": srv, "specs": specs}
    if kind == "static":
        L = case["L"]
        g = torch.Generator(device="cuda").manual_seed(seed)
        state = {"case": case, "seed": seed, "thr": swgpu.sw_threshold(1.0, case["T"]),
                 "spins": torch.randint(0, 2, (L * L,), dtype=torch.uint8, device="cuda", generator=g),
                 "out": torch.empty(L * L, dtype=torch.uint8, device="cuda"),
                 "labels": torch.empty(L * L, dtype=torch.int32, device="cuda"),
                 "obs": torch.empty(swgpu.OBS_DTYPE.itemsize // 8, dtype=torch.int64, device="cuda")}
        for k in range(EQUILIBRATION):   # in place
            _static_sweep(state, state["spins"], k)
        return state
    if kind == "potts":
        lat = swgpu.PottsLattice(case["dim"], case["L"], case["q"], T=case["T"], seed=seed,
                                 pcc=bool(case.get("pcc")), **_options(case))
        n = case["L"] ** case["dim"]
    else:
        # the largest lattices run at the tile height that the autotuner finds
        th = swgpu.sw_autotune(case["L"], case["T"]) if case["L"] > 8192 and "T" in case else 0
        lat = swgpu.Lattice(case["L"], T=case.get("T"), seed=seed, pcc=bool(case.get("pcc")), tile_h=th,
                            **_options(case))
        n = case["L"] ** 2
    # past the hot start: measurements are taken on an equilibrated lattice
    lat.sweep(EQUILIBRATION)
    lat.observables()
    return {"case": case, "lat": lat, "spins": _host_bytes(n)}


# ------------------------------------------------------------------------ one pass

def _ints(obs):
    """Observables records as rows of 64-bit words."""
    return obs.view("<i8").reshape(-1, swgpu.OBS_DTYPE.itemsize // 8)


def _static_sweep(state, out, k):
    swgpu.sw_sweep_static(state["spins"].data_ptr(), out.data_ptr(), state["labels"].data_ptr(),
                          state["obs"].data_ptr(), state["case"]["L"], state["thr"], state["seed"], k,
                          torch.cuda.current_stream())


def _serve(srv, specs):
    ids = srv.submit(specs)
    srv.wait_all()
    return [srv.poll(i)[1]["obs"] for i in ids]


def run(state):
    case = state["case"]
    if case["kind"] == "batch":
        return {"obs": _ints(np.concatenate(_serve(state["srv"], state["specs"])))}
    if case["kind"] == "static":
        # the chain's next sweep, on the same input spins every time
        _static_sweep(state, state["out"], EQUILIBRATION)
        return {"spins": state["out"], "labels": state["labels"], "obs": state["obs"]}
    lat, spins = state["lat"], state["spins"]
    lat.sweep(case["sweeps"])
    obs = lat.observables(case["sweeps"])
    swgpu._check(swgpu.lib().sw_get_spins(lat.h, ctypes.c_void_p(spins.ctypes.data)), "sw_get_spins")
    return {"obs": _ints(obs), "spins": spins}


def _sweep_work(sites, dim, potts):
    """Philox blocks of one sweep: a word per link (dim links a site, four
    words a block); the cluster's new state costs a word a site at most (one
    bit a site on the Ising path), drawn per cluster root: counted for an
    eighth of the sites."""
    return sites * (dim / 4.0 + (1.0 / 32.0 if potts else 1.0 / 1024.0))


def work(case):
    """Bytes: the spins read and written once, the last sweep's labels and
    bonds and the observables written once.  Operations: the Philox draws of
    every sweep.  (The state between sweeps, a bit or a byte a site, fits on
    the chip for most lattices and is not counted.)"""
    if case["kind"] == "batch":
        sides = [sp["L"] for sp in _mix(case, 0)]
        sites, n, dim, potts = sum(L * L for L in sides), case["sweeps"], 2, False
        obs = len(sides) * n * swgpu.OBS_DTYPE.itemsize
    else:
        dim, potts = case.get("dim", 2), case["kind"] == "potts"
        sites, n = case["L"] ** dim, case.get("sweeps", 1)
        obs = n * swgpu.OBS_DTYPE.itemsize
    return {"bytes": sites * (1 + 1 + 4 + 1) + obs, "flops": PHILOX_OPS * n * _sweep_work(sites, dim, potts)}


def exact(case, seed):
    """No output is a rounded number: spins, labels and sums are whole numbers
    and have to be equal."""
    return None
