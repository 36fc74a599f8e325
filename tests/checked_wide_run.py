"""Run by tests/test_gpu_wide_layout.py in a child process (it is not a test
module): the checked build of the library on instances that only the
global-resident layout holds, +-J against the oracle, then the check words as
JSON (see checked_run.py)."""
import ctypes
import json
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import numpy as np  # noqa: E402

from oracle import oracle as O  # noqa: E402
from paper_1501_05630_gb300 import build, icmpt, inputs as I  # noqa: E402

lib = icmpt.load_library(build.build(checked=True))
lib.icm_debug_check.argtypes = [ctypes.c_void_p, ctypes.c_int]
lib.icm_debug_check.restype = ctypes.c_int
ctx = icmpt.Context(0)

CASES = [  # lattice, L, disorder, n_T, dilution
    (O.CUBIC3D, 22, I.PM_J, 16, 0.0),
    (O.CHIMERA, 32, I.PM_J, 30, 0.2),
    (O.SQUARE2D, 128, I.PM_J, 8, 0.0),
    (O.SQUARE2D, 130, I.PM_J, 8, 0.0),
    (O.HYPERCUBIC4D, 8, I.GAUSS, 24, 0.0),
    (O.SQUARE2D, 80, I.GAUSS, 32, 0.1),
]
mismatch, elsewhere = [], []
for ci, (lat, L, dis, nT, dil) in enumerate(CASES):
    g = O.Geometry(lat, L)
    T = I.ladder(0.2, 2.0, nT)
    J = I.couplings(g.Nb, dis, 70 + ci, range(2))
    if dil:
        J = I.dilute(J, dil, 70 + ci, range(2))
    s0 = I.initial_spins(g.N, 2 * nT, 70 + ci, range(2))
    b = icmpt.Batch(ctx, lat, L, dis, J, T, 1.0, 70 + ci, spins=s0)
    if b.info()["smem_bytes"] >= 4 * b.N:
        elsewhere.append(ci)
    b.set_schedule(trace=1)
    b.run(6)
    if dis == I.PM_J:
        spins, E = b.read_spins(), b.read_energies()
        for a in range(2):
            r = O.Instance(g, J[a].astype(np.float64), T, s0[a], pm=True, T_icm=1.0, seed=70 + ci, inst=a)
            r.run(6)
            if not (np.array_equal(spins[a], r.s) and np.array_equal(E[a], r.E)):
                mismatch.append([ci, a])
    b.close()
ctx.sync()
word = (ctypes.c_uint * 4)()
rc = lib.icm_debug_check(word, 1)
print(json.dumps({"rc": rc, "check": list(word), "mismatch": mismatch, "elsewhere": elsewhere}))
