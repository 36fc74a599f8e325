"""2 x 2 growth blocks on thread-block clusters (2D, four sites a thread, word per
site: lattices with absent bonds)."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1501_05630_gb300 import inputs as I
from test_gpu_parity import _setup, icm  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


def test_diluted_block_growth_sees_the_reversed_spins(icm):
    """2D L=128 with 1% of the bonds absent on 8 x 512: a thread grows sites that
    other threads reversed in step 2a.  Two CTAs share some SMs.  The same chain
    as without blocks (8 x 1024), the same twice, and the oracle's."""
    icmpt, ctx = icm
    T = I.ladder(0.2, 1.5, 32)
    g, J, s0, ids = _setup(O.SQUARE2D, 128, I.PM_J, 20, T, 0x1603)
    J = I.dilute(J, 0.01, 0x1603, ids)
    runs = []
    for threads in (1024, 512, 512):
        b = icmpt.Batch(ctx, O.SQUARE2D, 128, I.PM_J, J, T, 1.0, 0x1603, spins=s0)
        b.set_cluster(8, threads)
        b.run(8)
        runs.append((b.read_spins(), b.read_energies()))
        b.close()
    for s, e in runs[1:]:
        assert np.array_equal(s, runs[0][0]) and np.array_equal(e, runs[0][1])
    r = O.Instance(g, J[0].astype(np.float64), T, s0[0], pm=True, T_icm=1.0, seed=0x1603, inst=0)
    r.run(8)
    assert np.array_equal(runs[0][0][0], r.s) and np.array_equal(runs[0][1][0], r.E)


def test_block_order_only_where_it_is_read(icm):
    """The blocks' order takes two bytes per own site of a CTA's shared memory, on
    the word-per-site scans alone: absent bonds bring it, the row form and
    union-find do without."""
    icmpt, ctx = icm
    T = I.ladder(0.2, 1.5, 32)
    g, J, s0, ids = _setup(O.SQUARE2D, 128, I.PM_J, 1, T, 0x1605)
    b = icmpt.Batch(ctx, O.SQUARE2D, 128, I.PM_J, J, T, 1.0, 0x1605, spins=s0)
    smem = {}
    for name, couplings in (("rows", J), ("scans", I.dilute(J, 0.05, 0x1605, ids))):
        b.load(couplings=couplings)
        for threads in (512, 544):                # 544: not four sites a thread, no blocks
            b.set_cluster(8, threads)
            smem[name, threads] = b.info()["smem_bytes"]
    part = 64 * 4                                  # one more warp's partial energies
    assert smem["rows", 544] - smem["rows", 512] == part
    assert smem["scans", 544] - smem["scans", 512] == part - 2 * (g.N // 8)
    b.close()
