"""What the performance of this library is measured on.

Each case is work that a user has the library do, through its public entry
points: the five workloads of the benchmark table (one small instance, a large
Gaussian batch, a multispin-coded chimera batch, uneven sizes in one shared
launch, served requests), large instances in the default layout and on
thread-block clusters, diluted and 4D lattices, a step from host buffers to
host observables, simulated annealing, and site percolation.

A simulation pass runs the chains on by a few sweeps and reads the state the
user works with (spins and energies, on the device).  No 64-bit reference is
given: the outputs are states of Monte Carlo chains.  One rounding that falls
on the other side of an acceptance test changes all that follows, so a chain in
64 bits is another chain; spins, counts and sizes are whole numbers that have
to be equal, and the energies belong to exactly these spins.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1501_05630_gb300 import icmpt
from paper_1501_05630_gb300 import inputs as I
from paper_1501_05630_gb300.serve import Request, Server

LATTICE = {"2d": I.SQUARE2D, "3d": I.CUBIC3D, "chimera": I.CHIMERA, "4d": I.HYPERCUBIC4D}
DEGREE = {"2d": 4, "3d": 6, "chimera": 6, "4d": 8}
T_MAX = {"2d": 1.5, "3d": 2.0, "chimera": 3.0, "4d": 3.0}
T_ICM = {"2d": 1.0, "3d": 1.0, "chimera": 1.5, "4d": 1.5}
T_MIN = 0.2
# threads per instance of the shared group kernel, by 3D size
TEAM = {4: 32, 6: 64, 8: 128, 10: 224, 12: 448}
MIXED_COUNTS = {4: 4096, 6: 2048, 8: 1024, 10: 512, 12: 256}
ANNEAL_STEPS = 16
# the served mix: lattice, size, disorder kind
MENU = (("2d", 16, "pmj"), ("2d", 32, "pmj"), ("2d", 64, "pmj"), ("3d", 6, "gauss"), ("3d", 8, "gauss"),
        ("3d", 12, "gauss"), ("chimera", 8, "pmj"), ("chimera", 12, "pmj"))


def listed():
    return [
        # one instance of the smallest workload, a few sweeps at a time: the latency of one step
        dict(name="one_2d_pmj_L8", kind="chain", lattice="2d", L=8, disorder="pmj", n_inst=1, n_T=16, sweeps=64,
             K=0, threads=0, dilution=0.0),
        # the 3D Gaussian workload: 1000 instances in one launch
        dict(name="batch_3d_gauss_L8", kind="chain", lattice="3d", L=8, disorder="gauss", n_inst=1000, n_T=24,
             sweeps=32, K=0, threads=0, dilution=0.0),
        # the chimera workload: 10^4 +-J instances, 30 temperatures (60 replicas: a partly used second word)
        dict(name="batch_chimera_pmj_C8", kind="chain", lattice="chimera", L=8, disorder="pmj", n_inst=10000, n_T=30,
             sweeps=16, K=0, threads=0, dilution=0.0),
        # the mixed-size workload: 3D L = 4..12 in one persistent launch
        dict(name="mixed_3d_gauss", kind="mixed", sizes="4,6,8,10,12", share=1.0, n_T=24, sweeps=16),
        # the largest 2D size served, on thread-block clusters
        dict(name="cluster_2d_pmj_L128", kind="chain", lattice="2d", L=128, disorder="pmj", n_inst=20, n_T=32,
             sweeps=16, K=8, threads=1024, dilution=0.0),
        # the largest 3D size served, on thread-block clusters
        dict(name="cluster_3d_gauss_L16", kind="chain", lattice="3d", L=16, disorder="gauss", n_inst=20, n_T=32,
             sweeps=32, K=8, threads=256, dilution=0.0),
        # a size above one CTA's shared memory in the layout a new batch gets
        dict(name="default_2d_pmj_L64", kind="chain", lattice="2d", L=64, disorder="pmj", n_inst=40, n_T=24,
             sweeps=16, K=0, threads=0, dilution=0.0),
        # diluted 4D lattices (absent bonds: per-instance neighbour tables)
        dict(name="diluted_4d_pmj_L6", kind="chain", lattice="4d", L=6, disorder="pmj", n_inst=200, n_T=16, sweeps=16,
             K=0, threads=0, dilution=0.3),
        # new disorder from pinned host buffers, a measured run, observables back on the host
        dict(name="host_3d_gauss_L8", kind="host", lattice="3d", L=8, disorder="gauss", n_inst=1000, n_T=24,
             sweeps=16),
        # simulated annealing with cluster moves: two replicas per instance, one temperature at a time
        dict(name="anneal_3d_gauss_L6", kind="anneal", lattice="3d", L=6, disorder="gauss", n_inst=512, sweeps=32),
        # site percolation near the chimera threshold
        dict(name="percolation_chimera_C32", kind="percolation", lattice="chimera", L=32, p=0.387, n_masks=20000),
        # requests of mixed kinds and sizes, each run to the thermalization test
        dict(name="serve_mixed", kind="serve", requests=48, n_T=16, max_sweeps=512),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["one", "batch", "batch", "chimera", "mixed", "cluster2d", "cluster3d", "default", "diluted", "host",
                       "anneal", "percolation", "serve"])
    if kind == "one":
        return dict(kind="chain", lattice="2d", L=2 * rng.randint(2, 8), disorder="pmj", n_inst=rng.randint(1, 4),
                    n_T=rng.randint(8, 32), sweeps=rng.randint(16, 128), K=0, threads=0, dilution=0.0)
    if kind == "batch":
        lat = rng.choice(["3d", "2d"])
        L = rng.choice([4, 6, 8, 10]) if lat == "3d" else rng.choice([8, 12, 16, 24])
        N = L ** 3 if lat == "3d" else L * L
        return dict(kind="chain", lattice=lat, L=L, disorder=rng.choice(["gauss", "gauss", "pmj"]),
                    n_inst=_log_int(rng, 50, 512000 // N), n_T=rng.randint(16, 32), sweeps=rng.randint(8, 32),
                    K=0, threads=0, dilution=0.0)
    if kind == "chimera":
        M = rng.randint(3, 10)
        return dict(kind="chain", lattice="chimera", L=M, disorder="pmj", n_inst=_log_int(rng, 100, 2000000 // (8 * M * M)),
                    n_T=rng.randint(16, 32), sweeps=rng.randint(8, 16), K=0, threads=0, dilution=0.0)
    if kind == "mixed":
        sizes = sorted(rng.sample([4, 6, 8, 10, 12], rng.randint(2, 4)))
        return dict(kind="mixed", sizes=",".join(map(str, sizes)), share=round(rng.uniform(0.1, 0.6), 3),
                    n_T=rng.randint(16, 24), sweeps=rng.randint(8, 16))
    if kind == "cluster2d":
        return dict(kind="chain", lattice="2d", L=rng.choice([64, 96, 128]), disorder=rng.choice(["pmj", "pmj", "gauss"]),
                    n_inst=rng.randint(1, 36), n_T=rng.randint(16, 32), sweeps=rng.randint(8, 16),
                    K=8, threads=rng.choice([768, 1024]), dilution=0.0)
    if kind == "cluster3d":
        return dict(kind="chain", lattice="3d", L=16, disorder=rng.choice(["gauss", "gauss", "pmj"]),
                    n_inst=rng.randint(1, 36), n_T=rng.randint(16, 32), sweeps=rng.randint(8, 32),
                    K=rng.choice([4, 8]), threads=rng.choice([256, 512]), dilution=0.0)
    if kind == "default":
        lat, L = rng.choice([("2d", 48), ("2d", 64), ("2d", 80), ("3d", 12), ("3d", 14), ("chimera", 20)])
        return dict(kind="chain", lattice=lat, L=L, disorder=rng.choice(["pmj", "gauss"]), n_inst=rng.randint(1, 80),
                    n_T=rng.randint(16, 32), sweeps=rng.randint(8, 16), K=0, threads=0, dilution=0.0)
    if kind == "diluted":
        lat, L = rng.choice([("4d", 4), ("4d", 6), ("3d", 6), ("3d", 8), ("2d", 16), ("chimera", 7)])
        return dict(kind="chain", lattice=lat, L=L, disorder=rng.choice(["pmj", "gauss"]), n_inst=rng.randint(20, 300),
                    n_T=rng.randint(8, 24), sweeps=rng.randint(8, 32), K=0, threads=0,
                    dilution=round(rng.uniform(0.05, 0.5), 3))
    if kind == "host":
        L = rng.choice([4, 6, 8])
        return dict(kind="host", lattice="3d", L=L, disorder=rng.choice(["gauss", "pmj"]),
                    n_inst=_log_int(rng, 50, 512000 // L ** 3), n_T=rng.randint(16, 24), sweeps=rng.randint(8, 32))
    if kind == "anneal":
        lat, L = rng.choice([("3d", 6), ("3d", 8), ("chimera", 6), ("2d", 16)])
        return dict(kind="anneal", lattice=lat, L=L, disorder=rng.choice(["gauss", "gauss", "pmj"]),
                    n_inst=_log_int(rng, 50, 1000), sweeps=rng.randint(8, 32))
    if kind == "percolation":
        lat, L = rng.choice([("chimera", 8), ("chimera", 16), ("chimera", 48), ("2d", 64), ("2d", 128), ("3d", 12), ("3d", 20)])
        N = 8 * L * L if lat == "chimera" else L ** int(lat[0])
        return dict(kind="percolation", lattice=lat, L=L, p=round(rng.uniform(0.25, 0.65), 4),
                    n_masks=_log_int(rng, 200, 40000000 // N))
    return dict(kind="serve", requests=rng.randint(8, 48), n_T=rng.choice([16, 24]), max_sweeps=rng.choice([256, 512]))


# ------------------------------------------------------------------ inputs

def _gen(seed, salt):
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) * 1000003 + salt) & 0x7FFFFFFFFFFFFFFF)
    return g


def _couplings(g, n, nb, disorder, dilution=0.0):
    if disorder == "gauss":
        J = torch.randn(n, nb, generator=g, device="cuda", dtype=torch.float32)
        J = torch.where(J == 0, torch.full_like(J, 0.5), J)      # an exact 0 would be an absent bond
    else:
        J = torch.randint(0, 2, (n, nb), generator=g, device="cuda", dtype=torch.int8) * 2 - 1
    if dilution:
        J = J * (torch.rand(n, nb, generator=g, device="cuda") >= dilution).to(J.dtype)
    return J.contiguous()


def _spins(g, n, R, N):
    return (torch.randint(0, 2, (n, R, N), generator=g, device="cuda", dtype=torch.int8) * 2 - 1).contiguous()


def _batch(ctx, g, seed, lattice, L, disorder, n, n_T, dilution=0.0, first_id=0, J=None, s=None):
    lat = LATTICE[lattice]
    N, nb = icmpt.lattice_size(lat, L)
    if J is None:
        J = _couplings(g, n, nb, disorder, dilution)
        s = _spins(g, n, 2 * n_T, N)
    T = I.ladder(T_MIN, T_MAX[lattice], n_T)
    return icmpt.Batch(ctx, lat, L, I.GAUSS if disorder == "gauss" else I.PM_J, J, T, T_ICM[lattice],
                       0x1501056300000000 + int(seed), spins=s, instance_ids=np.arange(first_id, first_id + n))


def _buffers(b):
    return dict(spins=torch.empty(b.n_inst, b.R, b.N, dtype=torch.int8, device="cuda"),
                energies=torch.empty(b.n_inst, b.R, dtype=torch.float64, device="cuda"))


def prepare(case, seed):
    kind = case["kind"]
    if kind == "serve":
        return _prepare_serve(case, seed)
    ctx = icmpt.Context(0, stream=torch.cuda.current_stream())
    g = _gen(seed, 17)
    if kind == "chain":
        b = _batch(ctx, g, seed, case["lattice"], case["L"], case["disorder"], case["n_inst"], case["n_T"],
                   case["dilution"])
        if case["K"]:
            b.set_cluster(case["K"], case["threads"])
        return dict(kind=kind, ctx=ctx, batch=b, sweeps=case["sweeps"], out=_buffers(b))
    if kind == "mixed":
        batches, first = [], 0
        sizes = [int(x) for x in case["sizes"].split(",")]
        for L in sizes:
            n = max(1, int(MIXED_COUNTS[L] * case["share"]))
            batches.append(_batch(ctx, g, seed, "3d", L, "gauss", n, case["n_T"], first_id=first))
            first += n
        grp = icmpt.Group(ctx, batches, case["sweeps"], shared=True, team_threads=[TEAM[L] for L in sizes])
        return dict(kind=kind, ctx=ctx, batches=batches, group=grp, out=[_buffers(b) for b in batches])
    if kind in ("host", "anneal"):
        lat = LATTICE[case["lattice"]]
        N, nb = icmpt.lattice_size(lat, case["L"])
        n, n_T = case["n_inst"], case.get("n_T", 1)
        J = _couplings(g, n, nb, case["disorder"])
        s = _spins(g, n, 2 * n_T, N)
        if kind == "host":
            b = _batch(ctx, g, seed, case["lattice"], case["L"], case["disorder"], n, n_T, J=J, s=s)
            return dict(kind=kind, ctx=ctx, batch=b, sweeps=case["sweeps"], J=J.cpu().pin_memory(),
                        s=s.cpu().pin_memory())
        ts = 3.0 * (0.05 / 3.0) ** (np.arange(ANNEAL_STEPS) / (ANNEAL_STEPS - 1))
        b = icmpt.Batch(ctx, lat, case["L"], I.GAUSS if case["disorder"] == "gauss" else I.PM_J, J, ts[:1], 1e300,
                        0x1501056300000000 + int(seed), spins=s)
        b.set_schedule(swap_every=0, t_meas=1 << 62)
        return dict(kind=kind, ctx=ctx, batch=b, sweeps=case["sweeps"], J=J, s=s, ts=ts, out=_buffers(b))
    if kind == "percolation":
        return dict(kind=kind, ctx=ctx, lattice=LATTICE[case["lattice"]], L=case["L"], p=case["p"],
                    n=case["n_masks"], seed=0x1501056300000000 + int(seed))
    raise ValueError(kind)


def _prepare_serve(case, seed):
    rng = np.random.default_rng(int(seed))
    reqs = []
    for i in range(case["requests"]):
        name, L, disorder = MENU[i % len(MENU)]
        lat = LATTICE[name]
        N, nb = icmpt.lattice_size(lat, L)
        gauss = disorder == "gauss"
        J = rng.standard_normal(nb).astype(np.float32) if gauss else (1 - 2 * rng.integers(0, 2, nb)).astype(np.int8)
        s = (1 - 2 * rng.integers(0, 2, (2 * case["n_T"], N))).astype(np.int8)
        reqs.append(Request(lat, L, I.GAUSS if gauss else I.PM_J, I.ladder(T_MIN, T_MAX[name], case["n_T"]), T_ICM[name],
                            0x1501056300000000 + int(seed), i, J, s))
    return dict(kind="serve", server=Server(0, slots_per_class=16, quantum=64, max_sweeps=case["max_sweeps"]),
                requests=reqs)


# ------------------------------------------------------------------ one pass

def run(state):
    kind = state["kind"]
    if kind == "chain":
        b, out = state["batch"], state["out"]
        b.run(state["sweeps"])
        b.read_spins(out["spins"])
        b.read_energies(out["energies"])
        return out
    if kind == "mixed":
        state["group"].run(1)
        for b, out in zip(state["batches"], state["out"]):
            b.read_spins(out["spins"])
            b.read_energies(out["energies"])
        return state["out"]
    if kind == "host":
        b = state["batch"]
        b.load(state["J"], state["s"])
        b.run(state["sweeps"])
        o = b.read_observables(hist=False)
        return dict(accE=o.accE, acc_n=o.acc_n, acc_q2=o.acc_q2, acc_pmin=o.acc_pmin, acc_d=o.acc_d, n_meas=o.n_meas)
    if kind == "anneal":
        b, out = state["batch"], state["out"]
        b.load(state["J"], state["s"])
        for T in state["ts"]:
            b.set_temperatures([T], 1e300)
            b.run(state["sweeps"])
        b.read_spins(out["spins"])
        b.read_energies(out["energies"])
        return out
    if kind == "percolation":
        return icmpt.largest_clusters_random(state["ctx"], state["lattice"], state["L"], state["p"], state["seed"],
                                             state["n"])
    srv = state["server"]
    tickets = [srv.submit(r) for r in state["requests"]]
    srv.run_until_idle()
    res = [srv.poll(t) for t in tickets]
    return dict(sweeps=np.array([r.sweeps for r in res], dtype=np.int64),
                thermalized=np.array([r.status == "thermalized" for r in res], dtype=np.int64),
                acc_d=np.array([r.acc_d for r in res], dtype=np.int64),
                n_meas=np.array([r.n_meas for r in res], dtype=np.int64),
                e=np.array([r.e for r in res]), q_l=np.array([r.q_l for r in res]), accE=np.array([r.accE for r in res]))


# ------------------------------------------------------------------ the work of one pass

def _sites(lattice, L):
    N, nb = (L * L, 2 * L * L) if lattice == "2d" else (L ** 3, 3 * L ** 3) if lattice == "3d" else \
        (L ** 4, 4 * L ** 4) if lattice == "4d" else (8 * L * L, 16 * L * L + 8 * L * (L - 1))
    return N, nb


def _chain_work(lattice, L, disorder, n, R, sweeps):
    """Spin updates x the method's operations per update (a Philox4x32-10 draw
    24.5, field and acceptance 12.5, for Gaussian couplings z + 1 more); the
    packed spins read and written, the couplings read, the results written."""
    N, nb = _sites(lattice, L)
    ops = 37.0 + (DEGREE[lattice] + 1 if disorder == "gauss" else 0)
    words = 4 * ((R + 31) // 32)
    return (n * (2 * N * words + nb * (4 if disorder == "gauss" else 1) + R * N + 8 * R), float(n) * N * R * sweeps * ops)


def work(case):
    kind = case["kind"]
    if kind == "chain":
        by, fl = _chain_work(case["lattice"], case["L"], case["disorder"], case["n_inst"], 2 * case["n_T"], case["sweeps"])
    elif kind == "mixed":
        by = fl = 0.0
        for L in (int(x) for x in case["sizes"].split(",")):
            b, f = _chain_work("3d", L, "gauss", max(1, int(MIXED_COUNTS[L] * case["share"])), 2 * case["n_T"], case["sweeps"])
            by, fl = by + b, fl + f
    elif kind == "host":
        by, fl = _chain_work(case["lattice"], case["L"], case["disorder"], case["n_inst"], 2 * case["n_T"], case["sweeps"])
    elif kind == "anneal":
        by, fl = _chain_work(case["lattice"], case["L"], case["disorder"], case["n_inst"], 2, case["sweeps"] * ANNEAL_STEPS)
    elif kind == "percolation":
        # per site one Philox draw (98 operations), one union per bond and one root lookup, at least
        N, nb = _sites(case["lattice"], case["L"])
        by, fl = 4.0 * case["n_masks"], float(case["n_masks"]) * (N * 99 + nb)
    else:
        by = fl = 0.0
        for i in range(case["requests"]):
            lat, L, disorder = MENU[i % len(MENU)]
            b, f = _chain_work(lat, L, disorder, 1, 2 * case["n_T"], case["max_sweeps"])
            by, fl = by + b, fl + f
    return {"bytes": float(by), "flops": float(fl)}


def exact(case, seed):
    """None: see the module's docstring (chain states; the others are whole numbers)."""
    return None
