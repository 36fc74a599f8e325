"""Edges of the bit-sliced +-J sweep and of the PT pass's move masks, bit for
bit against the oracle: replica counts that end inside a group of 8, a pass of
16 or a word of 32; site degrees of both parities (chimera C_1: 4, C_2: 5 and
6); warp groups that share out the replica groups; overlap masks of one word,
of an odd and of an even number of words.  Tolerance: none, every value is a
whole number."""
import pytest

from oracle import oracle as O
from test_gpu_parity import _compare_sweeps, icm  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,L,nT,n_inst,threads", [
    (O.SQUARE2D, 4, 1, 2, None),        # two replicas: one group of 8, no swaps
    (O.SQUARE2D, 4, 3, 2, None),        # R = 6
    (O.SQUARE2D, 8, 5, 2, 32),          # R = 10: the second group partly used
    (O.SQUARE2D, 8, 9, 1, 128),         # R = 18: four warp groups share three groups of 8
    (O.SQUARE2D, 8, 17, 2, 64),         # R = 34: a share crosses the word boundary
    (O.SQUARE2D, 6, 31, 1, 96),         # R = 62: three warp groups share eight groups of 8
    (O.CHIMERA, 1, 7, 3, None),         # degree 4 in a graph of degree 6
    (O.CHIMERA, 2, 12, 2, None),        # degrees 5 and 6
    (O.CUBIC3D, 6, 32, 2, 32),          # seven mask words, every swap position used
    (O.HYPERCUBIC4D, 2, 11, 2, None),   # degree 8 with doubled bonds
])
def test_sweep_edges(icm, kind, L, nT, n_inst, threads):
    _compare_sweeps(icm, kind, L, nT, 0.2, 2.0, 1.2, n_inst, 24, 0xE0 + L + nT, threads=threads)


@pytest.mark.parametrize("L,nT,n_inst,threads", [
    (2, 4, 2, None), (10, 20, 2, None), (14, 7, 1, 64), (16, 32, 1, None), (18, 6, 2, None), (30, 17, 1, 128),
    (32, 5, 1, None), (34, 6, 1, None), (50, 18, 1, 256), (64, 4, 1, None), (68, 3, 1, None), (70, 3, 1, None),
    (100, 2, 1, None),
])
def test_row_shapes(icm, L, nT, n_inst, threads):
    """Every row shape of the 2D cluster moves (70: none, word per site), more and
    fewer pairs than the team's warps take at once, shared-memory and wide CTAs."""
    _compare_sweeps(icm, O.SQUARE2D, L, nT, 0.2, 1.5, 1.2, n_inst, 8, 0xF0 + L, threads=threads)
