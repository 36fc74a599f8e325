"""Changes of a clustered batch's shape: whatever a call answers, the chain that
follows is the oracle's, bit for bit (+-J, no tolerance)."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1501_05630_gb300 import inputs as I
from test_gpu_parity import _setup, icm  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


def _equals_oracle(b, g, J, s0, T, seed, sweeps):
    spins, E = b.read_spins(), b.read_energies()
    for a in range(b.n_inst):
        r = O.Instance(g, J[a].astype(np.float64), T, s0[a], pm=True, T_icm=1.0, seed=seed, inst=a)
        r.run(sweeps)
        assert np.array_equal(spins[a], r.s), a
        assert np.array_equal(E[a], r.E), a


def test_refused_shape_keeps_the_batch(icm):
    """2D L=128 with 64 replicas on K = 8; K = 2 needs 243,728 bytes of shared
    memory a CTA and is refused: the batch runs on with K = 8, then with K = 4."""
    icmpt, ctx = icm
    T = I.ladder(0.2, 1.5, 32)
    g, J, s0, _ = _setup(O.SQUARE2D, 128, I.PM_J, 1, T, 0x1601)
    b = icmpt.Batch(ctx, O.SQUARE2D, 128, I.PM_J, J, T, 1.0, 0x1601, spins=s0)
    for K, threads in ((8, 512), (4, 512)):
        b.set_cluster(K, threads)
        b.run(1)
        before = b.info()
        for bad in ((2, 512), (2, 1024), (16, 256), (4, 48)):
            with pytest.raises(icmpt.IcmError):
                b.set_cluster(*bad)
        assert b.cluster() == K
        after = b.info()
        assert [after[k] for k in ("threads", "grid", "smem_bytes")] == [before[k] for k in ("threads", "grid", "smem_bytes")]
        b.run(1)
    _equals_oracle(b, g, J, s0, T, 0x1601, 4)
    b.close()


@pytest.mark.parametrize("kind,L,first,second,dilution", [
    (O.CUBIC3D, 8, (4, 64), (8, 32), 0.0),
    (O.SQUARE2D, 32, (4, 64), (2, 128), 0.2),         # 2 x 2 growth blocks in both
], ids=["3d", "2d_blocks"])
def test_change_beyond_the_budget_keeps_the_batch(icm, kind, L, first, second, dilution):
    """Another K whose tables exceed the context's memory budget: refused, or done
    with the memory that is there; either way the chain goes on."""
    icmpt, _ = icm
    T = I.ladder(0.3, 2.0, 8)
    g, J, s0, ids = _setup(kind, L, I.PM_J, 2, T, 0x1602)
    if dilution:
        J = I.dilute(J, dilution, 0x1602, ids)
    budget = 0
    for _ in range(2):                                # without a budget, then with what that took
        ctx = icmpt.Context(0, hbm_budget=budget)
        b = icmpt.Batch(ctx, kind, L, I.PM_J, J, T, 1.0, 0x1602, spins=s0)
        b.set_cluster(*first)
        if not budget:
            budget = ctx.memory()[0]
        else:
            b.run(3)
            try:
                b.set_cluster(*second)
                assert b.cluster() == second[0]
            except icmpt.IcmError:
                assert b.cluster() == first[0] and b.info()["threads"] == first[1]
            b.run(3)
            _equals_oracle(b, g, J, s0, T, 0x1602, 6)
        b.close()
        ctx.close()


@pytest.mark.parametrize("kind,L,shapes,dilution", [
    (O.CUBIC3D, 8, ((8, 32), (4, 64), (2, 128)), 0.0),
    (O.SQUARE2D, 32, ((8, 32), (4, 64), (2, 128)), 0.2),       # 2 x 2 growth blocks in all
    (O.SQUARE2D, 32, ((2, 128), (8, 32), (4, 64)), 0.0),       # row form
], ids=["3d", "2d_blocks", "2d_rows"])
def test_captured_group_keeps_its_tables(icm, kind, L, shapes, dilution):
    """A group captured on one cluster shape runs on unchanged while the batch takes
    other shapes, by request and by the tuner; without a group the shapes share
    their memory."""
    icmpt, ctx = icm
    T = I.ladder(0.3, 2.0, 8)
    g, J, s0, ids = _setup(kind, L, I.PM_J, 2, T, 0x1604)
    if dilution:
        J = I.dilute(J, dilution, 0x1604, ids)
    b = icmpt.Batch(ctx, kind, L, I.PM_J, J, T, 1.0, 0x1604, spins=s0)
    b.set_cluster(*shapes[0])
    grp = icmpt.Group(ctx, [b], sweeps_per_launch=2)
    for shape in shapes[1:]:
        grp.run(1)
        b.set_cluster(*shape)
        grp.run(1)
        b.run(1)
    b.autotune(1)
    grp.run(1)
    _equals_oracle(b, g, J, s0, T, 0x1604, 12)
    grp.close()
    held = 0
    for i in range(6):
        b.set_cluster(*shapes[i % 3])
        b.run(1)
        if i == 2:
            held = ctx.memory()[0]
    assert ctx.memory()[0] == held
    _equals_oracle(b, g, J, s0, T, 0x1604, 18)
    b.close()
