"""Gaussian batches with one temperature run in a kernel of their own; the shared
group kernel runs the same instances in the general passes at the same width:
equal spins and energies, bit for bit (the same sums in the same order)."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1501_05630_gb300 import inputs as I
from test_gpu_parity import _setup, icm  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,L,width", [(O.SQUARE2D, 4, 32), (O.SQUARE2D, 16, 128), (O.CUBIC3D, 6, 128), (O.CUBIC3D, 8, 64),
                                          (O.CHIMERA, 5, 128), (O.HYPERCUBIC4D, 4, 128)])
@pytest.mark.parametrize("T,T_icm", [(0.4, 1e300), (2.5, 0.0)])
def test_pair_kernel_equals_general_passes(icm, kind, L, width, T, T_icm):
    icmpt, ctx = icm
    g, J, s0, _ = _setup(kind, L, I.GAUSS, 9, np.array([T]), 0x61 + L)
    out = []
    for shared in (False, True):
        b = icmpt.Batch(ctx, kind, L, I.GAUSS, J, [T], T_icm, 0x61, spins=s0)
        if shared:
            grp = icmpt.Group(ctx, [b], 12, shared=True, team_threads=[width])
            grp.run(2)
        else:
            b.set_threads(width)
            b.run(24)
        o = b.read_observables()
        out.append((b.read_spins(), b.read_energies(), o.accE, o.acc_n, o.acc_d, o.hist))
        if shared:
            grp.close()
        b.close()
    for a, c in zip(*out):
        assert np.array_equal(a, c)
