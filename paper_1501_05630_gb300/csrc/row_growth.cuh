// row_growth.cuh -- cluster moves of one ICM pair on 2D lattices with the sites
// along the bits of a word (steps 2a and 2b: count, reversal decision, seed,
// connected component).  Included into an anonymous namespace of each
// translation unit, after icm_device.cuh.
//
// The word-per-site form grows all pairs at once, but only one or two bonds per
// scan, and a 2D cluster is 130-300 bonds deep (L = 64, 128).  Here a pair's
// q = -1 sites are rows of bits held in the registers of one warp (or of 2 or
// 8 lanes for small L): a step along a row is a shift of whole words, a step
// between rows of a lane is an AND-OR of registers, and between lanes a
// shuffle.  No shared memory and no barrier is
// touched until the component is complete.  Measured against the word-per-site
// scans: see cluster_moves (pt_icm.cu) and cl_cluster_moves (cluster_icm.cu).
//
// Shapes (KParams::row_kind; L even):
//   kRows8    L <= 8    four rows to a word, a word to a lane, 2 lanes a pair
//   kRows16   L <= 16   two rows to a word, a word to a lane, 8 lanes a pair
//   kRows32   L <= 32   a row to a word, a word to a lane, a warp a pair
//   kRows64   L <= 64   two words to a row, two rows to a lane, a warp a pair
//   kRows128  L <= 128  four words to a row, four rows to a lane (L % 4 == 0)
// Word j of a pair's rows (row_words of them, lane-major) and bit i hold the
// site of row_site(kind, j, i).
#pragma once

template <int KIND>
struct RowShape {
    static constexpr int FB = KIND == kRows8 ? 8 : KIND == kRows16 ? 16 : 32;   // bits of a row in a word
    static constexpr int U = KIND == kRows8 ? 2 : KIND == kRows16 ? 8 : 32;     // lanes of a pair
    static constexpr int W = KIND == kRows128 ? 4 : KIND == kRows64 ? 2 : 1;    // words of a row
    static constexpr int RPL = W;                                               // rows (or packed words) of a lane
    static constexpr int NW = W * RPL;                                          // words of a lane
};

// (x, y) of bit i of word j; outside the lattice when x or y >= L.
__device__ __forceinline__ void row_site(int kind, int j, int i, int &x, int &y)
{
    const int fb = kind == kRows8 ? 3 : kind == kRows16 ? 4 : 5;
    const int wl = kind == kRows128 ? 2 : kind == kRows64 ? 1 : 0;
    y = ((j >> wl) << (5 - fb)) + (i >> fb);
    x = ((j & ((1 << wl) - 1)) << 5) + (i & ((1 << fb) - 1));
}

// Component of the seeds c in the domain m, one packed word per lane.  Lanes of
// a pair are consecutive; ul is the lane in the pair, nl the pair's lanes in use.
template <int KIND>
__device__ __forceinline__ int grow_packed(uint32_t m, uint32_t &c, int L, int lane, int ul, int nl)
{
    constexpr int FB = RowShape<KIND>::FB, U = RowShape<KIND>::U, RPW = 32 / FB;
    constexpr uint32_t lo = FB == 8 ? 0x01010101u : FB == 16 ? 0x00010001u : 1u;   // bit 0 of every row
    const int base = lane & ~(U - 1);
    const int prv = base + (ul == 0 ? nl - 1 : (ul - 1) & (U - 1)), nxt = base + (ul >= nl - 1 ? 0 : ul + 1);
    // row index, in its word, of the last row of this lane and of the lane before
    const int f = ul == nl - 1 ? (L - 1) % RPW : RPW - 1, fp = ul == 0 ? (L - 1) % RPW : RPW - 1;
    int rounds = 0;
    uint32_t old;
    do {
        old = c;
        const uint32_t up = __shfl_sync(kFull, c, nxt), dn = __shfl_sync(kFull, c, prv);
        uint32_t v;
        if constexpr (FB == 32) v = up | dn;
        else v = (c >> FB) | (up << (FB * f)) | (c << FB) | (dn >> (FB * fp));
        c |= m & v;
        const uint32_t h = ((c << 1) & ~lo) | ((c >> 1) & ~(lo << (FB - 1))) | ((c >> (L - 1)) & lo) |
                           ((c & lo) << (L - 1));
        c |= m & h;
        if constexpr (FB == 32) {          // the rest of the run to the right, one more to the left
            c |= m & ~(m + c);
            c |= m & (c >> 1);
        }
        ++rounds;
    } while (__any_sync(kFull, c != old));
    return rounds;
}

// As above with rows of W words, RPL rows per lane (lane l holds rows RPL l ..):
// down through the lane's rows, each filling its runs to higher x, and up
// again, each with two bonds to lower x.  A warp has a pair and few warps share
// an SM sub-partition: bound by the ALU instructions of a pass, so the test for
// completion and the rows' periodic seam come once in three passes.  Passes and
// word operations per row on 128 x 128 sites at 0.57: this form 25 x 32, one
// bond either way in both directions 25 x 40, runs and two bonds in both 17 x
// 64.
template <int KIND>
__device__ __forceinline__ int grow_rows(const uint32_t (&m)[RowShape<KIND>::NW], uint32_t (&c)[RowShape<KIND>::NW],
                                         int L, int lane, int nl)
{
    constexpr int W = RowShape<KIND>::W, RPL = RowShape<KIND>::RPL;
    const int prv = lane == 0 ? nl - 1 : lane - 1, nxt = lane >= nl - 1 ? 0 : lane + 1;
    const int bl = (L - 1) & 31;
    const bool last3 = W == 4 && ((L - 1) >> 5) == 3;      // a row's last word: 3 or 2 (W = 4), 1 (W = 2)
    auto row_end = [&](const uint32_t *w) { return W == 2 ? w[1] : last3 ? w[W - 1] : w[W - 2]; };
    // across the seam of the periodic row, both ways
    auto seam = [&](int r) {
        uint32_t *cr = c + r * W;
        const uint32_t *mr = m + r * W;
        const uint32_t wrap = (cr[0] & 1u) << bl;
        cr[0] |= mr[0] & ((row_end(cr) >> bl) & 1u);
        if constexpr (W == 2) cr[1] |= mr[1] & wrap;
        else {
            cr[W - 1] |= mr[W - 1] & (last3 ? wrap : 0u);
            cr[W - 2] |= mr[W - 2] & (last3 ? 0u : wrap);
        }
    };
    // to higher x: m + c carries from every member through the ones of the domain
    // to the end of its run
    auto run = [&](int r) {
        uint32_t *cr = c + r * W;
        const uint32_t *mr = m + r * W;
        uint32_t t[W];
        if constexpr (W == 2) {
            asm("add.cc.u32 %0, %2, %4;\n\taddc.u32 %1, %3, %5;"
                : "=&r"(t[0]), "=r"(t[1]) : "r"(mr[0]), "r"(mr[1]), "r"(cr[0]), "r"(cr[1]));
        } else {
            asm("add.cc.u32 %0, %4, %8;\n\taddc.cc.u32 %1, %5, %9;\n\taddc.cc.u32 %2, %6, %10;\n\taddc.u32 %3, %7, %11;"
                : "=&r"(t[0]), "=&r"(t[1]), "=&r"(t[W - 2]), "=r"(t[W - 1])
                : "r"(mr[0]), "r"(mr[1]), "r"(mr[W - 2]), "r"(mr[W - 1]), "r"(cr[0]), "r"(cr[1]), "r"(cr[W - 2]),
                  "r"(cr[W - 1]));
        }
#pragma unroll
        for (int j = 0; j < W; ++j) cr[j] |= mr[j] & ~t[j];
    };
    // to lower x: two bonds
    auto back = [&](int r) {
        uint32_t *cr = c + r * W;
        const uint32_t *mr = m + r * W;
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            uint32_t t[W];
#pragma unroll
            for (int j = 0; j < W; ++j) t[j] = __funnelshift_r(cr[j], j + 1 < W ? cr[j + 1] : 0u, 1);
#pragma unroll
            for (int j = 0; j < W; ++j) cr[j] |= mr[j] & t[j];
        }
    };
    int rounds = 0;
    for (;;) {
#pragma unroll 1
        for (int it = 0; it < 3; ++it) {
            uint32_t n[W];
#pragma unroll
            for (int j = 0; j < W; ++j) n[j] = __shfl_sync(kFull, c[(RPL - 1) * W + j], prv);
#pragma unroll
            for (int r = 0; r < RPL; ++r) {
#pragma unroll
                for (int j = 0; j < W; ++j) c[r * W + j] |= m[r * W + j] & (r ? c[(r - 1) * W + j] : n[j]);
                run(r);
            }
#pragma unroll
            for (int j = 0; j < W; ++j) n[j] = __shfl_sync(kFull, c[j], nxt);
#pragma unroll
            for (int r = RPL - 1; r >= 0; --r) {
#pragma unroll
                for (int j = 0; j < W; ++j) c[r * W + j] |= m[r * W + j] & (r < RPL - 1 ? c[(r + 1) * W + j] : n[j]);
                back(r);
            }
        }
        rounds += 3;
#pragma unroll
        for (int r = 0; r < RPL; ++r) seam(r);
        // complete when no site of the domain outside has a neighbour inside
        uint32_t open = 0u;
        uint32_t up[W], dn[W];
#pragma unroll
        for (int j = 0; j < W; ++j) {
            dn[j] = __shfl_sync(kFull, c[(RPL - 1) * W + j], prv);
            up[j] = __shfl_sync(kFull, c[j], nxt);
        }
#pragma unroll
        for (int r = 0; r < RPL; ++r) {
            const uint32_t *cr = c + r * W;
            const uint32_t first = (row_end(cr) >> bl) & 1u, wrap = (cr[0] & 1u) << bl;
#pragma unroll
            for (int j = 0; j < W; ++j) {
                uint32_t v = (r ? c[(r - 1) * W + j] : dn[j]) | (r < RPL - 1 ? c[(r + 1) * W + j] : up[j]);
                v |= (cr[j] << 1) | (j ? cr[j - 1] >> 31 : first);
                v |= __funnelshift_r(cr[j], j + 1 < W ? cr[j + 1] : 0u, 1);
                if (W == 2 ? j == 1 : j == (last3 ? W - 1 : W - 2)) v |= wrap;
                open |= v & m[r * W + j] & ~cr[j];
            }
        }
        if (!__any_sync(kFull, open)) return rounds;
    }
}

struct RowMove {
    int n_pre, seed, rounds;      // q = -1 sites before step 2a; seed site, -1: none; growth rounds
    int size;                     // this lane's share of the cluster's sites
    bool flipped;
};

// Steps 2a and 2b of the pair whose q = -1 bits are the words at row (this
// lane's, before step 2a; `mine`: the lane has words): they become its cluster
// (0 when it has none).  Every lane of the warp calls; lanes without a pair
// pass have = false.  Not inlined: the rows take half of the 64 registers of
// the wide kernels, and next to the caller's values they were spilled inside
// the growth loop (2D L=128 on 8 x 512: 47 of 105 us per sweep).
template <int KIND>
__device__ __noinline__ RowMove rows_move(uint32_t *row, bool have, bool mine, uint32_t draw, bool enable_2a, int L)
{
    using S = RowShape<KIND>;
    const int lane = threadIdx.x & 31;
    uint32_t w[S::NW];
#pragma unroll
    for (int k = 0; k < S::NW; ++k) w[k] = mine ? row[k] : 0u;
    constexpr int U = S::U, W = S::W, NW = S::NW, FB = S::FB;
    const int ul = lane & (U - 1), half = L * L / 2;
    const int nl = S::W > 1 ? L / S::RPL : (L + 32 / FB - 1) / (32 / FB);
    // colour-0 bits of word k of this lane
    auto col0 = [&](int k) -> uint32_t {
        if constexpr (FB == 8) return 0xAA55AA55u;
        else if constexpr (FB == 16) return 0xAAAA5555u;
        else return ((W == 1 ? ul : k / W) & 1) ? 0xAAAAAAAAu : 0x55555555u;
    };
    int n = 0, n0 = 0;
#pragma unroll
    for (int k = 0; k < NW; ++k) {
        n += __popc(w[k]);
        n0 += __popc(w[k] & col0(k));
    }
#pragma unroll
    for (int o = U / 2; o >= 1; o >>= 1) {
        n += __shfl_xor_sync(kFull, n, o);
        n0 += __shfl_xor_sync(kFull, n0, o);
    }
    RowMove mv;
    mv.n_pre = n;
    mv.flipped = have && enable_2a && 2 * n > 2 * half;
    if (mv.flipped) {
        n = 2 * half - n;
        n0 = half - n0;
#pragma unroll
        for (int k = 0; k < NW; ++k) {
            uint32_t valid;
            if constexpr (W > 1) {
                const int left = ul < nl ? L - 32 * (k % W) : 0;
                valid = left >= 32 ? kFull : left > 0 ? (1u << left) - 1u : 0u;
            } else {
                const uint32_t row = L == FB ? kFull >> (32 - FB) : (1u << L) - 1u;
                valid = 0u;
#pragma unroll
                for (int f = 0; f < 32 / FB; ++f)
                    if (ul * (32 / FB) + f < L) valid |= row << (FB * f);
            }
            w[k] = ~w[k] & valid;
        }
    }
    // the seed: the rank-th site in (colour, site) order
    uint32_t rank = __umulhi(draw, (uint32_t)n);
    const bool second = rank >= (uint32_t)n0;
    if (second) rank -= (uint32_t)n0;
    int cnt = 0;
#pragma unroll
    for (int k = 0; k < NW; ++k) cnt += __popc(w[k] & (second ? ~col0(k) : col0(k)));
    int incl = cnt;
#pragma unroll
    for (int o = 1; o < U; o <<= 1) {
        const int v = __shfl_up_sync(kFull, incl, o);
        if (ul >= o) incl += v;
    }
    rank -= (uint32_t)(incl - cnt);        // wraps far above cnt in the lanes past the seed
    uint32_t c[NW];
    int seed = -1;
    {
        uint32_t sel = 0u, rr = 0u;
        int at = -1;
#pragma unroll
        for (int k = 0; k < NW; ++k) {
            const uint32_t v = w[k] & (second ? ~col0(k) : col0(k));
            const uint32_t pc = (uint32_t)__popc(v);
            if (at < 0 && n > 0 && rank < pc) {
                at = k;
                sel = v;
                rr = rank;
            }
            if (at < 0) rank -= pc;
        }
        if (incl <= 0 || cnt == 0) at = -1;
        const int bit = at >= 0 ? nth_set_bit(sel, rr) : 0;
#pragma unroll
        for (int k = 0; k < NW; ++k) c[k] = k == at ? 1u << bit : 0u;
        if (at >= 0) {
            int x, y;
            row_site(KIND, ul * NW + at, bit, x, y);
            seed = y * L + x;
        }
    }
#pragma unroll
    for (int o = U / 2; o >= 1; o >>= 1) seed = max(seed, __shfl_xor_sync(kFull, seed, o));
    mv.seed = seed;
    if constexpr (W == 1) mv.rounds = grow_packed<KIND>(w[0], c[0], L, lane, ul, nl);
    else mv.rounds = grow_rows<KIND>(w, c, L, lane, nl);
    mv.size = 0;
#pragma unroll
    for (int k = 0; k < NW; ++k) {
        if (mine) row[k] = c[k];
        mv.size += __popc(c[k]);
    }
    return mv;
}
