"""Packing, unpacking and initial energies at their edges: host, device and
odd-address device arrays give the same bytes; the initial energies of +-J
equal the integers of the spins, those of Gaussian couplings the fp32 sums in
their documented order, bit for bit (no tolerance)."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1501_05630_gb300 import inputs as I
from test_gpu_parity import _setup, icm  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu

SHAPES = [(O.SQUARE2D, 2, 1, 3), (O.SQUARE2D, 6, 17, 2), (O.CUBIC3D, 4, 24, 2), (O.CHIMERA, 1, 5, 2), (O.CHIMERA, 3, 32, 2),
          (O.HYPERCUBIC4D, 4, 9, 1), (O.SQUARE2D, 40, 3, 1)]


@pytest.mark.parametrize("kind,L,nT,n_inst", SHAPES)
def test_device_and_odd_addresses(icm, kind, L, nT, n_inst):
    import torch
    icmpt, ctx = icm
    T = I.ladder(0.3, 2.0, nT)
    g, J, s0, _ = _setup(kind, L, I.PM_J, n_inst, T, 0x51)
    b = icmpt.Batch(ctx, kind, L, I.PM_J, J, T, 1.0, 0x51, spins=s0)
    assert np.array_equal(b.read_spins(), s0)
    dJ = torch.from_numpy(J).cuda()
    for off in (0, 1, 2):
        raw = torch.zeros(s0.size + 4, dtype=torch.int8, device="cuda")
        raw[off:off + s0.size] = torch.from_numpy(-s0.reshape(-1)).cuda()
        view = raw[off:off + s0.size].view(s0.shape)
        b.load(dJ, view)
        assert np.array_equal(b.read_spins(), -s0)
        out = torch.full((s0.size + 4,), 7, dtype=torch.int8, device="cuda")
        b.read_spins(out[off:off + s0.size].view(s0.shape))
        got = out.cpu().numpy()
        assert np.array_equal(got[off:off + s0.size], -s0.reshape(-1))
        assert (got[:off] == 7).all() and (got[off + s0.size:] == 7).all()
    e = torch.empty(b.n_inst, b.R, dtype=torch.float64, device="cuda")
    b.read_energies(e)
    want = -np.einsum("ib,irb->ir", J.astype(np.int64), s0[:, :, g.bi].astype(np.int64) * s0[:, :, g.bj])
    assert np.array_equal(e.cpu().numpy(), want) and np.array_equal(b.read_energies(), want)


@pytest.mark.parametrize("kind,L,nT,n_inst", [(O.SQUARE2D, 4, 1, 2), (O.CUBIC3D, 6, 9, 2), (O.CHIMERA, 3, 17, 1),
                                              (O.HYPERCUBIC4D, 4, 32, 1)])
def test_gauss_initial_energies_keep_their_order(icm, kind, L, nT, n_inst):
    icmpt, ctx = icm
    T = I.ladder(0.3, 2.0, nT)
    g, J, s0, _ = _setup(kind, L, I.GAUSS, n_inst, T, 0x52)
    b = icmpt.Batch(ctx, kind, L, I.GAUSS, J, T, 1.0, 0x52, spins=s0)
    inc = [[] for _ in range(g.N)]                     # incident bonds in bond order
    for e in range(g.Nb):
        inc[g.bi[e]].append(e)
        inc[g.bj[e]].append(e)
    color = np.asarray(g.color)
    ones = np.flatnonzero(color == 1)                  # colour-1 sites, ascending
    got = b.read_energies()
    for a in range(n_inst):
        acc = np.zeros((128, 2 * nT), dtype=np.float32)
        for i, site in enumerate(ones):
            for e in inc[site]:
                x = s0[a, :, g.bi[e]].astype(np.float32) * s0[a, :, g.bj[e]]
                acc[i % 128] = acc[i % 128] - np.float32(J[a, e]) * x
        n = 64
        while n:
            acc[:n] = acc[:n] + acc[n:2 * n]
            n //= 2
        assert np.array_equal(got[a], acc[0].astype(np.float64))
