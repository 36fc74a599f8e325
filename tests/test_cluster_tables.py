"""Host tables of the thread-block-cluster layout (cluster_tables), on the CPU:
a small program linked against the library checks, for every lattice kind and
K, that each neighbour entry names the neighbour's site (own or halo), that
each halo entry is filled by exactly one copy of its owner, and that every
index stays in its table."""
import os
import subprocess

import pytest

from paper_1501_05630_gb300 import build as B

SRC = r"""
#include "icm_internal.h"
#include <cstdio>
#include <cstdlib>
int main(int argc, char **argv)
{
    const int kind = atoi(argv[1]), L = atoi(argv[2]), K = atoi(argv[3]);
    icm::HostTables h;
    if (!icm::host_tables(kind, L, h)) return 2;
    const int N = h.N, Z = h.Z, half = N / 2, hs = half / K, nls = 2 * hs;
    icm::ClusterTables t;
    icm::cluster_tables(h.nbr.data(), N, Z, K, t);
    auto pos = [&](int r, int li) { const int c = li >= hs; return c * half + r * hs + (li - c * hs); };
    long copies = 0, entries = 0;
    for (int r = 0; r < K; ++r)
        for (int li = 0; li < nls; ++li) {
            for (int d = 0; d < Z; ++d) {
                const int q = t.nb[((size_t)r * nls + li) * Z + d], want = h.nbr[(size_t)pos(r, li) * Z + d];
                if (q >= nls + t.nh) return 3;
                if ((q < nls ? pos(r, q) : (int)t.hpos[(size_t)r * t.nh + q - nls]) != want) return 4;
                if (q >= nls) {
                    const unsigned o = t.hown[(size_t)r * t.nh + q - nls];
                    if ((int)(o >> 16) >= K || (int)(o & 0xffff) >= nls || pos(o >> 16, o & 0xffff) != want) return 5;
                }
            }
            int x = t.xoff[(size_t)r * nls + li];
            if (x == 0xffff) continue;
            for (;;) {
                if (x >= t.nx) return 6;
                const unsigned v = t.xl[(size_t)r * t.nx + x++];
                const int c = (v >> 16) & 0xff, e = v & 0xffff;
                if (c >= K || c == r || e >= t.nh || t.hpos[(size_t)c * t.nh + e] != pos(r, li)) return 7;
                ++copies;
                if (v >> 31) break;
            }
        }
    for (size_t i = 0; i < t.hpos.size(); ++i) entries += t.hpos[i] != 0xffff;
    return copies == entries ? 0 : 8;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    B.build()
    d = tmp_path_factory.mktemp("cluster_tables")
    (d / "t.cpp").write_text(SRC)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", B.CSRC, "-I", os.path.join(B.ROOT, "include"),
                    "-I", os.path.join(cuda, "include"), str(d / "t.cpp"), B.LIB, "-Wl,-rpath," + B.BUILD,
                    "-o", str(d / "t")], check=True)
    return str(d / "t")


@pytest.mark.parametrize("kind,L,K", [(0, 16, 4), (0, 32, 8), (0, 128, 8), (0, 128, 2), (1, 8, 2), (1, 8, 8), (1, 16, 4),
                                      (1, 16, 8), (2, 4, 2), (2, 16, 8), (3, 4, 2), (3, 8, 8)])
def test_tables(program, kind, L, K):
    assert subprocess.run([program, str(kind), str(L), str(K)]).returncode == 0
