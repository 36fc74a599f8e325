"""The global-resident layout (instances too large for one CTA's shared memory):
every case checks that the batch is in it, by a CTA's shared memory that could not
hold one word per site.  +-J: equal to the oracle, bit for bit.  Gaussian: the
same chain as a wide CTA with its instance in shared memory, bit for bit (the
same sums in the same order); for instances that fit nowhere else, energies and
cluster moves against the spins to 1e-5 sum|J|, as in the other layouts."""
import json
import os
import subprocess
import sys

import numpy as np
import pytest

from oracle import oracle as O
from paper_1501_05630_gb300 import inputs as I
from test_gpu_parity import TRACE_KEYS, _check_icm_only_step, _e64, _setup, icm  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


def _batch(icmpt, ctx, kind, L, dis, n_inst, T, T_icm, seed, dilution, threads):
    g, J, s0, ids = _setup(kind, L, dis, n_inst, T, seed)
    if dilution:
        J = I.dilute(J, dilution, seed, ids)
    b = icmpt.Batch(ctx, kind, L, dis, J, T, T_icm, seed, spins=s0)
    if threads:
        b.set_threads(threads)
    return b, g, J, s0


def _global_resident(b):
    return b.info()["threads"] > 128 and b.info()["smem_bytes"] < 4 * b.N


@pytest.mark.parametrize("kind,L,nT,T_hi,T_icm,dilution,threads", [
    (O.CUBIC3D, 22, 16, 2.0, 1.0, 0.0, None),
    (O.CUBIC3D, 22, 17, 2.0, 1.0, 0.25, 512),         # two spin words, absent bonds
    (O.CHIMERA, 32, 30, 3.0, 1.5, 0.0, None),         # per-site degrees, padded neighbour lists
    (O.CHIMERA, 36, 9, 3.0, 1.5, 0.2, 352),
    (O.HYPERCUBIC4D, 10, 8, 3.0, 1.5, 0.0, None),
    (O.HYPERCUBIC4D, 10, 5, 3.0, 1.5, 0.3, 512),
    (O.SQUARE2D, 128, 8, 1.5, 1.0, 0.1, None),        # absent bonds: word per site
    (O.SQUARE2D, 130, 8, 1.5, 1.0, 0.0, None),        # no row form above L = 128
    (O.SQUARE2D, 128, 8, 1.5, 1.0, 0.0, 256),         # row form
])
def test_pmj_equals_oracle(icm, kind, L, nT, T_hi, T_icm, dilution, threads):
    icmpt, ctx = icm
    T = I.ladder(0.2, T_hi, nT)
    seed = 0x1700 + L
    b, g, J, s0 = _batch(icmpt, ctx, kind, L, I.PM_J, 2, T, T_icm, seed, dilution, threads)
    assert _global_resident(b)
    b.set_schedule(trace=1, t_meas=2)
    refs = [O.Instance(g, J[a].astype(np.float64), T, s0[a], pm=True, T_icm=T_icm, seed=seed, inst=a, t_meas=2)
            for a in range(2)]
    for _ in range(3):
        b.run(2)
        trs = [r.run(2, trace=True) for r in refs]
        spins, E, tr, cm = b.read_spins(), b.read_energies(), b.read_trace(), b.read_cluster_masks()
        for a, r in enumerate(refs):
            assert np.array_equal(spins[a], r.s) and np.array_equal(E[a], r.E)
            assert np.array_equal(cm[a], trs[a]["cmask"])
            for key in TRACE_KEYS + ("swap_acc",):
                assert np.array_equal(tr[key][a], trs[a][key]), key
    o = b.read_observables()
    for a, r in enumerate(refs):
        for f in ("accE", "acc_n", "acc_q2", "acc_pmin", "acc_d", "hist"):
            assert np.array_equal(getattr(o, f)[a], getattr(r, f)), f
    b.close()


@pytest.mark.parametrize("kind,L,dilution", [(O.CUBIC3D, 12, 0.0), (O.CUBIC3D, 12, 0.3), (O.CHIMERA, 15, 0.0),
                                             (O.HYPERCUBIC4D, 6, 0.0), (O.HYPERCUBIC4D, 6, 0.2), (O.SQUARE2D, 50, 0.0),
                                             (O.SQUARE2D, 50, 0.1)])
def test_gauss_equals_the_shared_memory_layout(icm, kind, L, dilution):
    """Three instances an SM do not fit in shared memory at 256 threads, a few
    instances do: the same first instances, the same chains."""
    icmpt, ctx = icm
    import torch
    T = I.ladder(0.2, 2.0, 24)
    few, many = 6, 3 * torch.cuda.get_device_properties(0).multi_processor_count
    out = []
    for n in (many, few):
        b, g, J, s0 = _batch(icmpt, ctx, kind, L, I.GAUSS, n, T, 1.0, 0x1710, dilution, 256)
        assert _global_resident(b) == (n == many)
        b.set_schedule(trace=1, t_meas=3)
        b.run(9)
        o, tr = b.read_observables(), b.read_trace()
        out.append([x[:few] for x in (b.read_spins(), b.read_energies(), o.accE, o.acc_n, o.acc_d, o.hist,
                                      *(tr[k] for k in TRACE_KEYS))])
        b.close()
    for x, y in zip(*out):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("kind,L,nT,T_hi,dilution", [
    (O.HYPERCUBIC4D, 8, 24, 3.0, 0.0),                # four sites a thread: growth in registers
    (O.HYPERCUBIC4D, 8, 24, 3.0, 0.3),
    (O.CUBIC3D, 18, 8, 2.0, 0.0),                     # six sites a thread
    (O.SQUARE2D, 80, 32, 1.5, 0.0),                   # row form
    (O.SQUARE2D, 128, 6, 1.5, 0.1),
])
def test_gauss_conservation_and_consistency(icm, kind, L, nT, T_hi, dilution):
    icmpt, ctx = icm
    T = I.ladder(0.2, T_hi, nT)
    b, g, J, s0 = _batch(icmpt, ctx, kind, L, I.GAUSS, 3, T, 1.0, 0x1720 + L, dilution, None)
    assert _global_resident(b)
    b.set_schedule(trace=1)
    scale = np.abs(J).astype(np.float64).sum(1)
    moves = 0
    for _ in range(2):
        b.run(5)
        tr = b.read_trace()
        k = tr["n_pre"] >= 0
        assert np.all(np.abs(tr["esum_after"] - tr["esum_before"])[k] <= 1e-5 * np.repeat(scale[:, None], nT, 1)[k])
        spins, E = b.read_spins(), b.read_energies()
        assert np.all(np.abs(E - _e64(J, spins, g)) <= 1e-5 * scale[:, None])
        moves += _check_icm_only_step(b, g, J, T, 1.0)
    assert moves > 0
    b.close()


def test_checked_build_finds_no_out_of_range_index():
    here = os.path.dirname(os.path.abspath(__file__))
    r = subprocess.run([sys.executable, os.path.join(here, "checked_wide_run.py")], capture_output=True, text=True,
                       timeout=900)
    assert r.returncode == 0, r.stdout + r.stderr
    out = json.loads(r.stdout.strip().splitlines()[-1])
    assert out == {"rc": 0, "check": [0, 0, 0, 0], "mismatch": [], "elsewhere": []}
