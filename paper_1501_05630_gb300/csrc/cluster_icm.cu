// cluster_icm.cu -- the simulation step of pt_icm.cu for one instance spread
// over a thread-block cluster of K CTAs (K SMs), for instances whose single
// CTA would be slow (2D L=128, 3D L=16 and larger).
//
// CTA r of the cluster owns the positions [c half + r hs, c half + (r+1) hs)
// of each colour c and keeps their spin words, couplings, cluster words and
// neighbour table in its own shared memory, with copies (the halo) of the
// spin and cluster words of every site in another CTA that borders one of
// its own.  The neighbour table holds the shared-memory offset of the
// neighbour's cluster word, own or halo, in 16 bits, so every neighbour access
// is a plain shared-memory load; reading the owner's word through the cluster
// window (ld.shared::cluster) cost two to nine times the latency and most of
// the growth's time.  What changes a word keeps its copies up to date:
//  * the sweep and the growth store a changed border word into the halos that
//    hold it (st.shared::cluster; one writer per word, nobody waits for it);
//  * step 2a, the cluster flip and the PT permutation are the same function of
//    a site's words everywhere, so every CTA applies them to its halo itself.
// Phases are separated by cluster barriers (barrier.cluster arrive.release /
// wait.acquire):
//  * sweep: colour 0, barrier, colour 1; each CTA stores its energy sums into
//    every CTA, barrier, every CTA adds the K shares in rank order (the same E
//    in all);
//  * ICM: overlap counts stored into every CTA, barrier, every CTA finds the
//    seed's owner from the K counts (position order = (colour, rank, local)),
//    the owner plants it; growth in rounds of a few in-place scans without
//    barriers, each round ending with a barrier after which every CTA reads
//    the round stamp that growing warps stored into all CTAs; flip, copy-a
//    energies exchanged as above;
//  * PT: every CTA holds the same energies and draws the same numbers, so
//    all make the same decisions and permute their own and halo words;
//  * observables: counts stored into rank 0, the barrier that ends the step,
//    rank 0 accumulates.
// Every buffer another CTA writes is written only after a barrier that
// both have passed since its last read.  Random keys are those of the
// single-CTA kernels, so the chain is the same, bit for bit for +-J.
#include "icm_internal.h"
#include "icm_device.cuh"

#include <algorithm>
#include <type_traits>

// The file is compiled three times so that the kernels build in parallel:
// ICM_PART 0 = layout and dispatch (the default), 1 = kernels for +-J couplings,
// 2 = Gaussian (cluster_pmj.cu and cluster_gauss.cu define the macro and include
// this file).
#ifndef ICM_PART
#define ICM_PART 0
#endif

namespace icm {
cudaError_t launch_cluster_pmj(const KParams &P, const ClusterLayout &L, int threads, int n_clusters, uint32_t n_sweeps,
                               cudaStream_t st);
cudaError_t launch_cluster_gauss(const KParams &P, const ClusterLayout &L, int threads, int n_clusters,
                                 uint32_t n_sweeps, cudaStream_t st);
cudaError_t cluster_occupancy_pmj(int Z, bool dil, bool lean, int K, int threads, int smem, int *clusters);
cudaError_t cluster_occupancy_gauss(int Z, bool dil, bool lean, int K, int threads, int smem, int *clusters);
int debug_check_cluster_pmj(unsigned int *out, int reset);
int debug_check_cluster_gauss(unsigned int *out, int reset);
}  // namespace icm

#if ICM_PART != 0
namespace icm {
namespace {

#include "row_growth.cuh"

__device__ __forceinline__ uint32_t cl_rank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

__device__ __forceinline__ uint32_t cl_id()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%clusterid.x;" : "=r"(r));
    return r;
}

__device__ __forceinline__ uint32_t cl_count()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%nclusterid.x;" : "=r"(r));
    return r;
}

// Every thread of every CTA of the cluster; orders shared-memory accesses
// across the cluster (release before, acquire after).
__device__ __forceinline__ void cl_sync()
{
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Cluster-window address of the shared-memory byte `local` (a shared-window
// address of this CTA) in CTA `rank`.
__device__ __forceinline__ uint32_t cl_map(uint32_t local, uint32_t rank)
{
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(local), "r"(rank));
    return r;
}

// (trace only: everything else is stored into the CTA that reads it)
__device__ __forceinline__ uint32_t cl_ld(uint32_t addr)
{
    uint32_t v;
    asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
    return v;
}


// A word of this CTA's shared memory by its shared-window address.
__device__ __forceinline__ uint32_t sh_ld(uint32_t addr)
{
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
    return v;
}

__device__ __forceinline__ void cl_st(uint32_t addr, uint32_t v)
{
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}

// Relaxed cluster-scope accesses of the union-find labels, which other
// threads of the cluster change while they are read.
__device__ __forceinline__ uint32_t cl_ld_rlx(uint32_t addr)
{
    uint32_t v;
    asm volatile("ld.relaxed.cluster.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
    return v;
}

__device__ __forceinline__ uint32_t cl_cas(uint32_t addr, uint32_t cmp, uint32_t v)
{
    uint32_t old;
    asm volatile("atom.relaxed.cluster.shared::cluster.cas.b32 %0, [%1], %2, %3;"
                 : "=r"(old) : "r"(addr), "r"(cmp), "r"(v) : "memory");
    return old;
}

// This CTA's view: pointers into its shared memory and cluster addresses.
struct CS {
    uint32_t *s, *C;
    uint16_t *nb, *xoff;
    uint32_t *xl, *hlab;
    float *Jd;
    uint8_t *Jb, *zdeg;
    void *E, *Epart, *Esw, *Epair, *esum;   // Esw [K][R], Epair [K][32]: every CTA's share
    uint32_t *thr;
    float *b2l;
    uint32_t *mask, *lab, *sadr, *sroot;
    uint32_t *rowm, *rowc, *rowi;
    uint16_t *gord;
    int *cntloc, *cntobs, *flags, *seed, *csz, *cnt_n, *cnt_d;   // cntloc [K][2][32], cntobs [2][K][2][32]
    uint32_t *flipw;
    uint32_t *swap_x;
    uint64_t *swap_mask;
    double *accE;
    long long *acc64, *nmeas;
    unsigned long long *icmst;
    uint32_t base;        // shared-window address of this CTA's dynamic shared memory
    uint32_t win;         // where this CTA's shared window starts (its rank << 24)
    uint32_t dCs;         // a cluster word's address minus this: the site's spin word 0
    uint32_t rank, K;
    int hs, nls, ns;      // ns: own and halo sites, the stride of the two spin words
};

__device__ __forceinline__ CS make_cs(unsigned char *smem, const ClusterLayout &L)
{
    CS S;
    S.s = (uint32_t *)(smem + L.s);
    S.C = (uint32_t *)(smem + L.C);
    S.nb = (uint16_t *)(smem + L.nb);
    S.xoff = (uint16_t *)(smem + L.xoff);
    S.xl = (uint32_t *)(smem + L.xl);
    S.hlab = (uint32_t *)(smem + L.hlab);
    S.Jd = (float *)(smem + L.coup);
    S.Jb = (uint8_t *)(smem + L.coup);
    S.zdeg = (uint8_t *)(smem + L.zdeg);
    S.E = smem + L.E;
    S.Epart = smem + L.Epart;
    S.Esw = smem + L.Esw;
    S.Epair = smem + L.Epair;
    S.esum = smem + L.esum;
    S.thr = (uint32_t *)(smem + L.rtab);
    S.b2l = (float *)(smem + L.rtab);
    S.mask = (uint32_t *)(smem + L.mask);
    S.lab = (uint32_t *)(smem + L.lab);
    S.rowm = (uint32_t *)(smem + L.rowm);
    S.rowc = (uint32_t *)(smem + L.rowc);
    S.rowi = (uint32_t *)(smem + L.rowi);
    S.sadr = (uint32_t *)(smem + L.sadr);
    S.sroot = (uint32_t *)(smem + L.sroot);
    S.gord = L.gord >= 0 ? (uint16_t *)(smem + L.gord) : nullptr;
    S.cntloc = (int *)(smem + L.cntloc);
    S.cntobs = (int *)(smem + L.cntobs);
    S.flags = (int *)(smem + L.flags);
    S.seed = (int *)(smem + L.seed);
    S.csz = (int *)(smem + L.csz);
    S.cnt_n = (int *)(smem + L.cnt_n);
    S.cnt_d = (int *)(smem + L.cnt_d);
    S.flipw = (uint32_t *)(smem + L.flipw);
    S.swap_x = (uint32_t *)(smem + L.swap_x);
    S.swap_mask = (uint64_t *)(smem + L.swap_mask);
    S.accE = (double *)(smem + L.accE);
    S.acc64 = (long long *)(smem + L.acc64);
    S.nmeas = (long long *)(smem + L.nmeas);
    S.icmst = (unsigned long long *)(smem + L.icmst);
    S.base = (uint32_t)__cvta_generic_to_shared(smem);
    S.win = S.base & 0xFF000000u;
    S.dCs = (uint32_t)(L.C - L.s);
    S.rank = cl_rank();
    S.K = (uint32_t)L.K;
    S.hs = L.hs;
    S.nls = L.nls;
    S.ns = L.ns;
    return S;
}

// The neighbour row of own site li: the offsets of the neighbours' cluster
// words in the CTA's shared window, two to a 32-bit word.
template <int Z>
__device__ __forceinline__ void nb_row(const uint16_t *nb, int li, uint32_t (&e)[Z / 2])
{
    const uint16_t *row = nb + li * Z;
    if constexpr (Z == 4) {
        const uint2 v = *reinterpret_cast<const uint2 *>(row);
        e[0] = v.x;
        e[1] = v.y;
    } else if constexpr (Z == 8) {
        const uint4 v = *reinterpret_cast<const uint4 *>(row);
        e[0] = v.x;
        e[1] = v.y;
        e[2] = v.z;
        e[3] = v.w;
    } else {
#pragma unroll
        for (int i = 0; i < Z / 2; ++i) e[i] = reinterpret_cast<const uint32_t *>(row)[i];
    }
}
// The shared-window address of entry d.  In a cluster the window of CTA r starts
// at r << 24 (win, S.win): the 16-bit offset alone would name another CTA's
// window, which ld.shared must not touch.
__device__ __forceinline__ uint32_t nb_addr(uint32_t pair, int d, uint32_t win)
{
    return __byte_perm(pair, win, (d & 1) ? 0x7632 : 0x7610);
}

// Spin word `off` bytes from the cluster word of each neighbour of li.
template <int Z>
__device__ __forceinline__ void nb_words(const CS &S, int li, uint32_t off, uint32_t (&w)[Z])
{
    uint32_t e[Z / 2];
    nb_row<Z>(S.nb, li, e);
#pragma unroll
    for (int d = 0; d < Z; ++d) w[d] = sh_ld(nb_addr(e[d >> 1], d, S.win) + off);
}

// Apply f to the addresses of the copies of own site li's cluster word in the
// halos of other CTAs (none for an inner site).  The last one has bit 0 set.
template <typename F>
__device__ __forceinline__ void for_copies(const CS &S, int li, F f)
{
    uint32_t i = S.xoff[li];
    if (i == 0xffffu) return;
    uint32_t a;
    do {
        a = S.xl[i++];
        f(a & ~1u);
    } while (!(a & 1u));
}

// Store v at word `i` of row `rank` of the [K][n] array at byte offset `off`
// of every CTA's shared memory.
template <typename ET>
__device__ __forceinline__ void cl_share(const CS &S, int off, int n, int i, ET v)
{
    uint32_t w;
    if constexpr (std::is_same<ET, float>::value) w = __float_as_uint(v);
    else w = (uint32_t)v;
    const uint32_t a = S.base + off + 4u * (uint32_t)((int)S.rank * n + i);
    for (uint32_t r = 0; r < S.K; ++r) cl_st(cl_map(a, r), w);
}

// Sum of entry i over the K rows, in rank order (the same result in every CTA).
template <typename ET>
__device__ __forceinline__ ET row_sum(const CS &S, const void *rows, int n, int i)
{
    ET v = ET(0);
    for (uint32_t r = 0; r < S.K; ++r) v += ((const ET *)rows)[(int)r * n + i];
    return v;
}

// Global position of local site li of CTA `rank`.
__device__ __forceinline__ int pos_of(const KParams &P, const CS &S, int li)
{
    const int c = li >= S.hs;
    return c * P.half + (int)S.rank * S.hs + (li - c * S.hs);
}

// ---------------------------------------------------------------------------
// Step 1, Gaussian couplings: one 16-bit pass of colour COLOR over word g
// (see gauss_pass in pt_icm.cu).
template <int Z, bool DIL>
__device__ __forceinline__ void cl_gauss_pass(const KParams &P, const CS &S, uint32_t t, uint32_t inst, int g,
                                              int COLOR, int H, bool tie)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nth = blockDim.x;
    const int rbase = 32 * g + 16 * H;
    const int sh0 = 16 * H;
    const int npairs8 = (P.R - rbase + 7) >> 3;
    const uint32_t goff = (uint32_t)(g * S.ns * 4) - S.dCs;    // cluster word -> spin word g
    uint32_t *sg = S.s + g * S.ns;
    float acc[16];
#pragma unroll
    for (int b = 0; b < 16; ++b) acc[b] = 0.f;
    for (int j = threadIdx.x; j < S.hs; j += nth) {
        const int li = COLOR * S.hs + j;
        const uint32_t sw0 = sg[li];
        const uint32_t sw = sw0 >> sh0;
        const uint32_t site = __ldg(P.pos2site + pos_of(P, S, li));
        uint32_t nw[Z];
        nb_words<Z>(S, li, goff, nw);
        uint32_t flip = 0;
        float J[Z];
        float Jsum = 0.f;
#pragma unroll
        for (int d = 0; d < Z; ++d) {
            nw[d] >>= sh0;
            J[d] = S.Jd[li * Z + d];
            Jsum += J[d];
        }
        const float *b2l = S.b2l + (rbase >> 1);
#pragma unroll
        for (int qq = 0; qq < 2; ++qq) {
            if (qq < npairs8) {
                uint32_t x[4], y[4];
                philox10x2(site, t, (uint32_t)(rbase >> 2) + 2 * qq, inst, P.key, x, y);
                const float4 bl4 = *reinterpret_cast<const float4 *>(b2l + 4 * qq);   // four temperatures
                const float bl[4] = {bl4.x, bl4.y, bl4.z, bl4.w};
                uint32_t f8 = 0u;
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int b = 8 * qq + i;
                    float h = Jsum;
#pragma unroll
                    for (int d = 0; d < Z; ++d)
                        if ((nw[d] >> b) & 1u) h = fmaf(J[d], -2.f, h);
                    const float sh = neg_if(h, sw & (1u << b));
                    const uint32_t xr = i < 4 ? x[i] : y[i - 4];
                    const uint32_t thr = __float2uint_rz(ex2_approx(fmaf(bl[i >> 1], sh, 32.f)));
                    bool a;
                    if constexpr (DIL)   // diluted instance: Delta E = 0 accepted with probability 1/2
                        a = (sh < 0.f) || (sh == 0.f ? (!tie || xr < 0x80000000u) : (xr < thr));
                    else
                        a = (sh <= 0.f) || (xr < thr);
                    acc[b] -= sh;
                    if (a) {
                        f8 |= 1u << i;
                        acc[b] += 2.f * sh;
                    }
                }
                flip |= f8 << (8 * qq);
            }
        }
        const uint32_t w = sw0 ^ (flip << sh0);
        sg[li] = w;
        for_copies(S, li, [&](uint32_t a) { cl_st(a + goff, w); });
    }
    if (COLOR == 1) {
        const float v = transpose_reduce16(acc, lane);
        const int r = rbase + (lane >> 1);
        if (!(lane & 1) && r < P.R) ((float *)S.Epart)[warp * P.R + r] = v;
    }
}

// Step 1, +-J couplings: the replica groups [q0, q1) of word g of colour COLOR
// (see pmj_pass in pt_icm.cu).  When warp groups share out the replicas
// (`shared`), the flips go into the word by atomic XOR and the caller stores
// the copies.
template <int Z, bool DIL>
__device__ __forceinline__ void cl_pmj_pass(const KParams &P, const CS &S, uint32_t t, uint32_t inst, int g, int COLOR,
                                            int q0, int q1, int j0, int jstride, bool shared, bool tie)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t goff = (uint32_t)(g * S.ns * 4) - S.dCs;
    uint32_t *sg = S.s + g * S.ns;
    const int left = P.R - 32 * g;
    const uint32_t live = left >= 32 ? kFull : (1u << left) - 1u;
    const int end = 8 * q1 < left ? 8 * q1 : min(32, (left + 15) & ~15);
    const uint32_t mine = (kFull >> (32 - end)) & (kFull << (8 * q0));
    uint32_t pl[kPlanes];
#pragma unroll
    for (int i = 0; i < kPlanes; ++i) pl[i] = 0u;
    for (int j = j0; j < S.hs; j += jstride) {
        const int li = COLOR * S.hs + j;
        const uint32_t sw = sg[li];
        const uint32_t site = __ldg(P.pos2site + pos_of(P, S, li));
        const uint32_t jb = S.Jb[li];
        uint32_t u[Z], c[4];
        nb_words<Z>(S, li, goff, u);
#pragma unroll
        for (int d = 0; d < Z; ++d) u[d] ^= sw ^ (0u - ((jb >> d) & 1u));
        csa_count<Z>(u, c[0], c[1], c[2], c[3]);
        const int z = (!DIL && Z != 6) ? Z : (!DIL && P.const_z) ? P.const_z : (int)S.zdeg[li];   // bonds present
        const uint32_t flip = pmj_flips<Z, DIL>(c, z, tie, live, S.thr + 16 * g * kThrRow, site, t, 8u * (uint32_t)g,
                                                inst, P.key, q0, q1) & mine;
        if (shared) {
            atomicXor(sg + li, flip);
        } else {
            sg[li] = sw ^ flip;
            for_copies(S, li, [&](uint32_t a) { cl_st(a + goff, sw ^ flip); });
        }
        if (COLOR == 1) pmj_count(pl, c, z, flip, mine & live);
    }
    if (COLOR == 1) {
        const int v = warp_vcount(pl, P.cnt_planes, lane);
        if (lane < left) ((int *)S.Epart)[warp * P.R + 32 * g + lane] = v;
    }
}

// Step 1 for all replicas; this CTA's share of the energies goes into every
// CTA's row.  The barrier that ends the phase is the caller's.
template <bool GAUSS, int Z, bool DIL>
__device__ __forceinline__ void cl_metropolis(const KParams &P, const ClusterLayout &L, const CS &S, uint32_t t,
                                              uint32_t inst, bool tie)
{
    using ET = typename std::conditional<GAUSS, float, int>::type;
    const int nth = blockDim.x, nwarps = nth >> 5, tid = threadIdx.x;
    if constexpr (GAUSS) {
        const int npass = (P.R + 15) >> 4;
        for (int it = 0; it < 2 * npass; ++it) {
            const int color = it >= npass;
            const int pass = it - color * npass;
            cl_gauss_pass<Z, DIL>(P, S, t, inst, pass >> 1, color, pass & 1, tie);
            if (pass == npass - 1) {
                if (color == 0) cl_sync();            // colour 1 reads the copies of colour 0
                else __syncthreads();
            }
        }
    } else {
        const int n8 = (P.R + 7) >> 3;                // groups of 8 replicas
        const int conc = min(nth / S.hs, n8);         // hs is a multiple of 32
        const bool split = conc >= 2;
        const int group = split ? tid / S.hs : 0;
        const int per = split ? (n8 + conc - 1) / conc : n8;
        const int lo = group * per, hi = min(lo + per, n8);
        const int j0 = tid - (split ? group * S.hs : 0), jstride = split ? S.hs : nth;
        if (split)
            for (int i = tid; i < nwarps * P.R; i += nth) ((int *)S.Epart)[i] = 0;   // before the barrier below
        for (int color = 0; color < 2; ++color) {
            for (int g = lo >> 2; lo < hi && 4 * g < hi; ++g)
                cl_pmj_pass<Z, DIL>(P, S, t, inst, g, color, max(lo - 4 * g, 0), min(hi - 4 * g, 4), j0, jstride, split,
                                    tie);
            if (split) {                              // the words are complete: store the copies
                __syncthreads();
                for (int i = tid; i < P.G * S.hs; i += nth) {
                    const int g = i >= S.hs, li = color * S.hs + i - g * S.hs;
                    const uint32_t w = S.s[g * S.ns + li], goff = (uint32_t)(g * S.ns * 4) - S.dCs;
                    for_copies(S, li, [&](uint32_t a) { cl_st(a + goff, w); });
                }
            }
            if (color == 0) cl_sync();
            else __syncthreads();
        }
    }
    for (int r = tid; r < P.R; r += nth) {
        ET e = ET(0);
        for (int w = 0; w < nwarps; ++w) e += ((const ET *)S.Epart)[w * P.R + r];
        cl_share<ET>(S, L.Esw, P.R, r, e);
    }
}

// ---------------------------------------------------------------------------
// Union-find over the cluster's shared memory.  A label word holds the
// cluster-window address of its parent's label word; a root holds its own
// address.  Roots are linked by a fixed random priority of their addresses
// (a bijective hash): a root is hooked, by compare-and-swap on the root, only
// under a root of higher priority, so priorities increase strictly along
// every path (no cycle forms, a walk ends within N steps) and the trees stay
// shallow, where linking by address would chain the sites of a row.  Words
// of this CTA are reached through its own shared window, which is faster
// than the cluster window.  In the phase where only this CTA's threads touch
// its words (LOCAL) the accesses are plain; otherwise they are relaxed at
// cluster scope, so that compare-and-swaps from every CTA are atomic with
// one another.
struct Uf {
    uint32_t lab;     // cluster-window address of this CTA's first label word
    uint32_t loc;     // its shared-window address
    uint32_t span;    // bytes of this CTA's label words in use
    int limit;        // N + 1
};

__device__ __forceinline__ uint32_t uf_prio(uint32_t x)
{
    x *= 0x9E3779B1u;
    x ^= x >> 15;
    x *= 0x85EBCA77u;
    return x ^ (x >> 13);
}

template <bool LOCAL>
__device__ __forceinline__ uint32_t uf_ld(const Uf &U, uint32_t a)
{
    const uint32_t o = a - U.lab;
    uint32_t v;
    if (LOCAL) v = sh_ld(U.loc + o);
    else if (o < U.span)
        asm volatile("ld.relaxed.cluster.shared::cta.u32 %0, [%1];" : "=r"(v) : "r"(U.loc + o) : "memory");
    else v = cl_ld_rlx(a);
    return v;
}

template <bool LOCAL>
__device__ __forceinline__ uint32_t uf_cas(const Uf &U, uint32_t a, uint32_t cmp, uint32_t v)
{
    const uint32_t o = a - U.lab;
    uint32_t old;
    if (LOCAL)
        asm volatile("atom.shared.cas.b32 %0, [%1], %2, %3;" : "=r"(old) : "r"(U.loc + o), "r"(cmp), "r"(v) : "memory");
    else if (o < U.span)
        asm volatile("atom.relaxed.cluster.shared::cta.cas.b32 %0, [%1], %2, %3;"
                     : "=r"(old) : "r"(U.loc + o), "r"(cmp), "r"(v) : "memory");
    else old = cl_cas(a, cmp, v);
    return old;
}

// The root of x (after the unions: nothing changes the labels any more).
__device__ __forceinline__ uint32_t uf_root(const Uf &U, uint32_t x)
{
    for (int i = 0; i < U.limit; ++i) {
        const uint32_t p = uf_ld<false>(U, x);
        if (p == x) return x;
        x = p;
    }
    (void)ICM_IDX(U.limit, U.limit, 23);
    return x;
}

// Union over the bonds of this CTA's colour-1 sites whose two ends have
// q = -1 in a group pair, each bond once: those inside this CTA (REMOTE
// false) or those to other CTAs (REMOTE true).  The lanes of a warp run in
// lockstep: each iteration, every lane with a union in hand reads the
// parents of both ends and climbs one level, or, at two distinct roots,
// hooks the lower-priority root under the other (a failed swap goes on from
// the root's new parent); a lane without one first takes its next bond.
// Every iteration ends in a warp vote, so the lanes' loads issue together
// (lanes that ran their own loops fell apart and waited for their loads one
// by one).  `it` is bounded (never reached: each union ends within N climbs
// and N failed swaps).
template <int Z, bool REMOTE>
__device__ __forceinline__ void uf_unions(const Uf &U, const CS &S, uint32_t gm0, uint32_t gm1, int n0,
                                          uint32_t qstride)
{
    const int nls = S.nls, ns = S.ns, hs = S.hs, nth = blockDim.x;
    const uint32_t cw0 = (uint32_t)__cvta_generic_to_shared(S.C) - S.win;
    int j = (int)threadIdx.x - nth, li = 0, d = Z;
    uint32_t x0 = 0u, x1 = 0u, y0 = 0u, y1 = 0u, ea = 0u, eb = 0u, a = 0u, b = 0u;
    bool more = true, busy = false;
    // iterations a lane can need: its bonds x pairs x (N climbs + N failed swaps + 1)
    const long long cap = (long long)(hs / nth + 1) * Z * 32 * (2ll * U.limit + 1);
    for (long long it = 0;; ++it) {
        if (!busy && more) {
            while (!(y0 | y1)) {                     // the next bond with a pair to link
                if (d == Z) {
                    j += nth;
                    if (j >= hs) {
                        more = false;
                        break;
                    }
                    li = hs + j;
                    const uint32_t w0 = S.s[li];
                    x0 = (w0 ^ (w0 >> 1)) & gm0;
                    x1 = 0u;
                    if (gm1) {
                        const uint32_t w1 = S.s[ns + li];
                        x1 = (w1 ^ (w1 >> 1)) & gm1;
                    }
                    d = (x0 | x1) ? 0 : Z;
                    ea = U.lab + 4u * (uint32_t)li;
                    continue;
                }
                const int q = (int)((S.nb[li * Z + d] - cw0) >> 2);   // own site or halo entry
                ++d;
                if ((q >= nls) != REMOTE) continue;
                if (x0) {
                    const uint32_t v = S.s[q];
                    y0 = x0 & (v ^ (v >> 1));
                }
                if (x1) {
                    const uint32_t v = S.s[ns + q];
                    y1 = x1 & (v ^ (v >> 1));
                }
                eb = REMOTE ? S.hlab[q - nls] : U.lab + 4u * (uint32_t)q;
            }
            if (y0 | y1) {
                uint32_t q;
                if (y0) {
                    q = (uint32_t)__popc(gm0 & ((y0 & (0u - y0)) - 1u));
                    y0 &= y0 - 1u;
                } else {
                    q = (uint32_t)(n0 + __popc(gm1 & ((y1 & (0u - y1)) - 1u)));
                    y1 &= y1 - 1u;
                }
                a = ea + q * qstride;
                b = eb + q * qstride;
                busy = true;
            }
        }
        if (!__any_sync(kFull, busy)) break;
        if (it >= cap) {
            (void)ICM_IDX(U.limit, U.limit, 23);
            break;
        }
        if (busy) {
            const uint32_t pa = uf_ld<!REMOTE>(U, a), pb = uf_ld<!REMOTE>(U, b);
            if (pa != a || pb != b) {
                a = pa;
                b = pb;
            } else if (a == b) {
                busy = false;
            } else {
                if (uf_prio(a) < uf_prio(b)) {
                    const uint32_t x = a;
                    a = b;
                    b = x;
                }
                const uint32_t old = uf_cas<!REMOTE>(U, b, b, a);   // hook the lower-priority root under the other
                if (old == b) busy = false;
                else b = old;
            }
        }
    }
}

// The own sites in the seed's component of each group pair: their cluster
// bits are set.  Lockstep as above: each iteration a lane climbs one level
// from its site's label toward the root.
__device__ __forceinline__ void uf_mark(const Uf &U, const CS &S, uint32_t gm0, uint32_t gm1, int n0)
{
    const int nls = S.nls, nth = blockDim.x;
    int li = (int)threadIdx.x - nth, q = 0;
    uint32_t x0 = 0u, x1 = 0u, bit = 0u, c = 0u, c0 = 0u, c1 = 0u;
    bool word1 = false, more = true, busy = false;
    const long long cap = (long long)(nls / nth + 1) * 32 * (U.limit + 1);   // sites x pairs x (N climbs + 1)
    for (long long it = 0;; ++it) {
        if (!busy && more) {
            while (!(x0 | x1)) {
                if (li >= 0 && (c0 | c1)) {          // the last site's bits are complete
                    S.C[li] |= c0 | (c1 << 1);
                    c0 = c1 = 0u;
                }
                li += nth;
                if (li >= nls) {
                    more = false;
                    break;
                }
                const uint32_t w0 = S.s[li];
                x0 = (w0 ^ (w0 >> 1)) & gm0;
                if (gm1) {
                    const uint32_t w1 = S.s[S.ns + li];
                    x1 = (w1 ^ (w1 >> 1)) & gm1;
                }
            }
            if (x0 | x1) {
                word1 = !x0;
                uint32_t &x = word1 ? x1 : x0;
                bit = x & (0u - x);
                x &= x - 1u;
                q = word1 ? n0 + __popc(gm1 & (bit - 1u)) : __popc(gm0 & (bit - 1u));
                c = U.lab + 4u * (uint32_t)(q * nls + li);
                busy = true;
            }
        }
        if (!__any_sync(kFull, busy)) break;
        if (it >= cap) {
            (void)ICM_IDX(U.limit, U.limit, 23);
            break;
        }
        if (busy) {
            const uint32_t p = uf_ld<false>(U, c);
            if (p != c) {
                c = p;
            } else {
                if (c == S.sroot[q]) (word1 ? c1 : c0) |= bit;
                busy = false;
            }
        }
    }
    if (li < nls && (c0 | c1)) S.C[li] |= c0 | (c1 << 1);
}

// Step 2b(c) by union-find: the seed's component of q = -1 sites of every
// moving pair, set in the cluster words of the own sites (the seed's
// bit is already set).  Pairs go in groups of L.ufg (act0 / act1: pair j of
// word w at bit 2j of act_w).  Per group: labels reset (every site its own
// root); union over the bonds inside this CTA, where every walk stays in this
// CTA; cluster barrier; union over the bonds to other CTAs; cluster barrier;
// every own site compares its root with the seed's.  The components are those
// of the propagation in the other branch, so the cluster words are the same,
// bit for bit.
template <int Z>
__device__ __forceinline__ void cl_grow_uf(const KParams &P, const ClusterLayout &L, const CS &S, uint32_t act0,
                                           uint32_t act1)
{
    const int tid = threadIdx.x, nth = blockDim.x;
    const int nls = S.nls, g = L.ufg;
    Uf U;
    U.lab = cl_map(S.base + L.lab, S.rank);
    U.loc = S.base + (uint32_t)L.lab;
    U.limit = P.N + 1;
    const uint32_t qstride = 4u * (uint32_t)nls;            // label arrays of consecutive group pairs
    uint32_t rest0 = act0, rest1 = act1;
    int groups = 0;
    while (rest0 | rest1) {
        uint32_t gm0 = 0u, gm1 = 0u;                 // the next (up to) g pairs, in pair order
        for (int q = 0; q < g && (rest0 | rest1); ++q) {
            if (rest0) {
                gm0 |= rest0 & (0u - rest0);
                rest0 &= rest0 - 1u;
            } else {
                gm1 |= rest1 & (0u - rest1);
                rest1 &= rest1 - 1u;
            }
        }
        const int n0 = __popc(gm0), ng = n0 + __popc(gm1);
        U.span = (uint32_t)ng * qstride;
        ++groups;
        for (int i = tid; i < ng * nls; i += nth) S.lab[i] = U.lab + 4u * (uint32_t)i;
        __syncthreads();
        uf_unions<Z, false>(U, S, gm0, gm1, n0, qstride);
        cl_sync();                                   // every CTA's own unions are done
        uf_unions<Z, true>(U, S, gm0, gm1, n0, qstride);
        cl_sync();
        if (tid < ng) {                              // the root of the tid-th group pair's seed
            uint32_t m0 = gm0, m1 = gm1;
            for (int q = 0; q < tid; ++q) {
                if (m0) m0 &= m0 - 1u;
                else m1 &= m1 - 1u;
            }
            const int k = m0 ? (__ffs(m0) - 1) >> 1 : 16 + ((__ffs(m1) - 1) >> 1);
            S.sroot[tid] = uf_root(U, S.sadr[k] + (uint32_t)L.lab + (uint32_t)tid * qstride);
        }
        __syncthreads();
        uf_mark(U, S, gm0, gm1, n0);
        if (rest0 | rest1) cl_sync();                // walks through these labels end before the reset
    }
    __syncthreads();
    for (int li = tid; li < nls; li += nth) {        // the marked words into the halos
        const uint32_t c = S.C[li];
        if (c) for_copies(S, li, [&](uint32_t a) { cl_st(a, c); });
    }
    cl_sync();
    if (S.rank == 0 && tid == 0) {
        S.icmst[0] += (unsigned)(__popc(act0) + __popc(act1));
        S.icmst[1] += 4u * (unsigned)groups;         // passes over the own sites
    }
}

// Steps 2a and 2b in the row form (row_growth.cuh): every CTA stores its rows of
// a pair into the CTA that takes the pair (k mod K), whose warp counts,
// reverses, seeds and grows it on its own and stores the cluster's rows back
// into the CTAs that hold them or their halo copies.  Two cluster barriers,
// where the scans took one each round of six.  2D L=128 x 20 on 8 x 1024, 16
// sweeps: 4.72 to 1.82 ms; on 8 x 512 189 to 90 us per sweep.
template <int KIND>
__device__ __forceinline__ void cl_rows_pairs(const KParams &P, const ClusterLayout &L, const CS &S, int slot, bool trace)
{
    using Sh = RowShape<KIND>;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    const int ul = lane & (Sh::U - 1), per = 32 / Sh::U, K = (int)S.K, pairs = (P.n_icm + K - 1) / K;
    const int stride = L.rw + 2 * L.rh;
    for (int s0 = warp * per; s0 < pairs; s0 += nwarps * per) {
        const int s = s0 + lane / Sh::U, k = s * K + (int)S.rank;
        const bool have = s < pairs && k < P.n_icm;
        const bool mine = have && ul * Sh::NW < L.rs;
        uint32_t *row = S.rowm + s * L.rs + ul * Sh::NW;
        const RowMove mv = rows_move<KIND>(row, have, mine, have ? (uint32_t)S.seed[k] : 0u, P.enable_2a != 0, P.L);
        if (mine)
#pragma unroll 1
            for (int i = 0; i < Sh::NW; ++i) {
                const int j = ul * Sh::NW + i, r = j / L.rw, jl = j - r * L.rw;   // CTA of the row, word in its rows
                const uint32_t at = S.base + (uint32_t)L.rowc + 4u * (uint32_t)(k * stride), w = row[i];
                cl_st(cl_map(at + 4u * (uint32_t)jl, (uint32_t)r), w);
                if (jl < L.rh)                     // the first rows follow the CTA before
                    cl_st(cl_map(at + 4u * (uint32_t)(L.rw + L.rh + jl), (uint32_t)((r + K - 1) & (K - 1))), w);
                if (jl >= L.rw - L.rh)             // the last ones precede the CTA after
                    cl_st(cl_map(at + 4u * (uint32_t)(L.rw + jl - (L.rw - L.rh)), (uint32_t)((r + 1) & (K - 1))), w);
            }
        int size = mv.size;
        if (trace)
            for (int o = Sh::U / 2; o >= 1; o >>= 1) size += __shfl_xor_sync(kFull, size, o);
        if (have && ul == 0) {
            const uint32_t info = (uint32_t)(mv.seed >= 0) | ((uint32_t)mv.flipped << 1) | ((uint32_t)mv.rounds << 2);
            for (int r = 0; r < K; ++r) cl_st(cl_map(S.base + (uint32_t)L.rowi + 4u * (uint32_t)k, (uint32_t)r), info);
            if (trace) {
                const size_t o = (size_t)slot * P.nT + k;
                P.tr_n_pre[o] = mv.n_pre;
                P.tr_flip2a[o] = mv.flipped ? 1 : 0;
                P.tr_seed[o] = mv.seed;
                P.tr_csize[o] = size;
            }
        }
    }
}

template <bool GAUSS>
__device__ __forceinline__ void cl_row_moves(const KParams &P, const ClusterLayout &L, const CS &S, int slot, bool trace,
                                             uint32_t &act0, uint32_t &act1)
{
    using ET = typename std::conditional<GAUSS, float, int>::type;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    const int tid = threadIdx.x, nth = blockDim.x;
    const int Lx = P.L, nicm = P.n_icm, kind = P.row_kind, K = (int)S.K, rank = (int)S.rank;
    const int ns = S.ns, hs = S.hs, rows = Lx / K, y0 = rank * rows;
    const bool two = P.G > 1;
    const ET *E = (const ET *)S.E;
    ET *esum = (ET *)S.esum;
    const int kp = pair_of_bit(lane);
    // local index of lane's site of the pair's word j of this CTA's rows, or -1
    auto own_of = [&](int j) {
        int x, y;
        row_site(kind, rank * L.rw + j, lane, x, y);
        return x < Lx ? ((x + y) & 1) * hs + (((y - y0) * Lx + x) >> 1) : -1;
    };
    for (int j = warp; j < L.rw; j += nwarps) {
        const int li = own_of(j);
        const uint32_t x = li >= 0 ? overlap_word(S.s[li], two ? S.s[ns + li] : 0u) : 0u;
        const uint32_t col = warp_transpose32(x, lane);
        if (kp < nicm) {
            const int s = kp / K;
            cl_st(cl_map(S.base + (uint32_t)L.rowm + 4u * (uint32_t)(s * L.rs + rank * L.rw + j), (uint32_t)(kp - s * K)), col);
        }
    }
    for (int k = tid; k < nicm; k += nth) {
        esum[k] = E[2 * k] + E[2 * k + 1];
        if (trace && rank == 0)
            P.tr_eb[(size_t)slot * P.nT + k] = P.tr_ea[(size_t)slot * P.nT + k] = (float)(E[2 * k] + E[2 * k + 1]);
    }
    cl_sync();
    switch (kind) {
    case kRows16: cl_rows_pairs<kRows16>(P, L, S, slot, trace); break;
    case kRows32: cl_rows_pairs<kRows32>(P, L, S, slot, trace); break;
    case kRows64: cl_rows_pairs<kRows64>(P, L, S, slot, trace); break;
    default: cl_rows_pairs<kRows128>(P, L, S, slot, trace); break;
    }
    cl_sync();
    const uint32_t info = lane < nicm ? S.rowi[lane] : 0u;
    const uint32_t act = __ballot_sync(kFull, info & 1u), fl = __ballot_sync(kFull, info & 2u);
    const uint32_t rounds = __reduce_max_sync(kFull, info >> 2);
    if (tid < nicm) S.seed[tid] = (int)(info & 1u);
    act0 = spread16(act & 0xFFFFu);
    act1 = spread16(act >> 16);
    const uint32_t f0 = spread16(fl & 0xFFFFu) << 1, f1 = spread16(fl >> 16) << 1;
    if (rank == 0 && tid == 0) {
        S.icmst[0] += (unsigned)(__popc(act0) + __popc(act1));
        S.icmst[1] += rounds;
    }
    // flip the own sites, then the two halo rows (entries by colour, row, x)
    const int stride = L.rw + 2 * L.rh;
    const int ya = (y0 + Lx - 1) % Lx, yb = (y0 + rows) % Lx;
    for (int j = warp; j < stride; j += nwarps) {
        const uint32_t c = warp_transpose32(kp < nicm ? S.rowc[kp * stride + j] : 0u, lane);
        int li;
        if (j < L.rw) {
            li = own_of(j);
        } else {
            // the row before in the last row of its words, the row after in the first of its own
            const bool after = j >= L.rw + L.rh;
            const int jh = j - L.rw - (after ? L.rh : 0);
            int x, y;
            row_site(kind, jh, lane, x, y);
            const int want = !after && kind == kRows16 ? 1 : 0;
            y = y == want && x < Lx ? (after ? yb : ya) : -1;
            const bool upper = after ? yb > ya : ya > yb;      // the larger of the two rows
            li = y < 0 ? -1 : S.nls + ((x + y) & 1) * Lx + (upper ? Lx / 2 : 0) + (x >> 1);
        }
        if (li < 0) continue;
        const uint32_t e0 = c & 0x55555555u, e1 = (c >> 1) & 0x55555555u;
        S.s[li] ^= f0 ^ (e0 | (e0 << 1));
        if (two) S.s[ns + li] ^= f1 ^ (e1 | (e1 << 1));
        if (trace && P.tr_cmask && li < S.nls) {
            uint32_t *cm = P.tr_cmask + ((size_t)slot * P.N + pos_of(P, S, li)) * 2;
            cm[0] = e0;
            cm[1] = e1;
        }
    }
    __syncthreads();
}

// Steps 2a and 2b word by word (see site_moves in pt_icm.cu), or by union-find.
template <bool GAUSS, int Z>
__device__ __forceinline__ void cl_site_moves(const KParams &P, const ClusterLayout &L, const CS &S, uint32_t t, int slot,
                                              bool trace, uint32_t &act0, uint32_t &act1)
{
    using ET = typename std::conditional<GAUSS, float, int>::type;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    const int tid = threadIdx.x, nth = blockDim.x;
    const int N = P.N, nicm = P.n_icm, G = P.G, nls = S.nls, ns = S.ns, hs = S.hs, NWl = L.NWl;
    const ET *E = (const ET *)S.E;
    ET *esum = (ET *)S.esum;

    // (a) overlap masks of the own sites and their counts per colour block
    // (cnt_n: colour 0, cnt_d: colour 1); clear the cluster words
    const int kp = pair_of_bit(lane);
    int cnt[2] = {0, 0};
    for (int m = warp; m < NWl; m += nwarps) {
        const int li = 32 * m + lane;
        const uint32_t col = warp_transpose32(overlap_word(S.s[li], G > 1 ? S.s[ns + li] : 0u), lane);
        cnt[32 * m >= hs] += __popc(col);
        if (kp < nicm) S.mask[kp * NWl + m] = col;
    }
    if (kp < nicm) {
        if (cnt[0]) atomicAdd(&S.cnt_n[kp], cnt[0]);
        if (cnt[1]) atomicAdd(&S.cnt_d[kp], cnt[1]);
    }
    for (int i = tid; i < ns; i += nth) S.C[i] = 0u;
    if (tid < 2) S.flipw[tid] = 0u;
    if (tid < 32) S.csz[tid] = 0;
    __syncthreads();
    for (int i = tid; i < 2 * nicm; i += nth) {
        const int c = i >= nicm, k = i - c * nicm;
        int *v = (c ? S.cnt_d : S.cnt_n) + k;
        cl_share<int>(S, L.cntloc, 64, 32 * c + k, *v);
        *v = 0;                                       // as the observables expect it
    }
    cl_sync();

    // (b) per pair, in every CTA alike: n, step 2a, the seed's owner by rank;
    // the owner plants the seed
    for (int k = tid; k < nicm; k += nth) {
        int n = row_sum<int>(S, S.cntloc, 64, k) + row_sum<int>(S, S.cntloc, 64, 32 + k);
        const int n_pre = n;
        const bool flipped = P.enable_2a && 2 * n > N;
        if (flipped) {
            n = N - n;
            atomicOr(&S.flipw[(2 * k + 1) >> 5], 1u << ((2 * k + 1) & 31));
        }
        bool moves = false;
        if (n > 0) {
            uint32_t rank = (uint32_t)(((uint64_t)(uint32_t)S.seed[k] * (uint32_t)n) >> 32);
            const uint32_t inv = flipped ? kFull : 0u;
            for (int cr = 0; cr < 2 * (int)S.K; ++cr) {
                const int c = cr >= (int)S.K, r = cr - c * (int)S.K;
                int cn = S.cntloc[64 * r + 32 * c + k];
                if (flipped) cn = hs - cn;
                if (rank < (uint32_t)cn) {
                    moves = true;
                    if (r == (int)S.rank) {           // this CTA owns the seed: find the local site
                        for (int m = c * (hs / 32); m < (c + 1) * (hs / 32); ++m) {
                            const uint32_t w = S.mask[k * NWl + m] ^ inv;
                            const uint32_t pc = (uint32_t)__popc(w);
                            if (rank < pc) {
                                const int li = 32 * m + nth_set_bit(w, rank);
                                const uint32_t bit = 1u << (2 * (k & 15) + (k >> 4));
                                atomicOr(S.C + ICM_IDX(li, nls, 21), bit);
                                if (L.ufg) {           // the seed's site address, for the union-find roots
                                    const uint32_t sa = cl_map(S.base, S.rank) + 4u * (uint32_t)li;
                                    for (uint32_t r2 = 0; r2 < S.K; ++r2) cl_st(cl_map(S.base + L.sadr + 4 * k, r2), sa);
                                }
                                if (trace) P.tr_seed[(size_t)slot * P.nT + k] = (int)__ldg(P.pos2site + pos_of(P, S, li));
                                break;
                            }
                            rank -= pc;
                        }
                    }
                    break;
                }
                rank -= (uint32_t)cn;
            }
        }
        S.seed[k] = moves;
        esum[k] = E[2 * k] + E[2 * k + 1];
        if (trace && S.rank == 0) {
            const size_t o = (size_t)slot * P.nT + k;
            P.tr_n_pre[o] = n_pre;
            P.tr_flip2a[o] = flipped ? 1 : 0;
            if (!moves) P.tr_seed[o] = -1;
            P.tr_csize[o] = 0;
            P.tr_eb[o] = (float)(E[2 * k] + E[2 * k + 1]);
            P.tr_ea[o] = (float)(E[2 * k] + E[2 * k + 1]);
        }
    }
    // The growth below stores the seeds' copies first and runs at least two
    // rounds, so that they are seen before the rounds can end; the union-find
    // needs every CTA's seed addresses.
    if (L.ufg) cl_sync();
    else __syncthreads();

    // (c) step 2a on the own and halo sites, then the clusters of all pairs at once
    act0 = act1 = 0u;
    for (int k = 0; k < nicm; ++k)
        if (S.seed[k]) {
            if (k < 16) act0 |= 1u << (2 * k);
            else act1 |= 1u << (2 * (k - 16));
        }
    const uint32_t f0 = S.flipw[0], f1 = S.flipw[1];
    if (f0 | f1)
        for (int li = tid; li < ns; li += nth) {
            S.s[li] ^= f0;
            if (G > 1) S.s[ns + li] ^= f1;
        }
    __syncthreads();                                 // below a thread reads sites that others reversed
    if (!(act0 | act1)) return;                      // the same decision in every CTA
    // One cluster word per site holds every pair: bit 2j = pair j, bit 2j + 1
    // = pair 16 + j, so that the domain word is q of the first spin word | q
    // of the second << 1 and a neighbour is one load.
    // Growth in cluster rounds of kScansPerRound in-place scans of the own
    // sites, reading the halo words as they are; a border site that grew is
    // stored into its copies.  A warp that grew a site writes the round's
    // stamp into the stamp word of every CTA of the cluster; after the
    // round's barrier each CTA reads its own word, so all CTAs decide alike.
    // The growth ends after a round, the second at the earliest, in which
    // nothing grew: every read of that round saw the state that the previous
    // barrier published, and no site could grow from it, so it is the fixed
    // point, each seed's component of q = -1.  Stamps are (t << 16) + round +
    // 1 (at most N < 2^16 rounds), so words need no reset; a stale equal value
    // could only add one empty round.
    constexpr int kScansPerRound = 6;
    const uint32_t actc = act0 | (act1 << 1);
    // with at most four own sites per thread, each thread keeps their
    // neighbour addresses, domain and cluster words in registers across the
    // scans.  On 2D lattices with four sites per thread the host gives each
    // thread a 2 x 2 block of sites, taken around the block (S.gord): a scan
    // then carries the growth across the block and into the next lane's block
    // (a model of the in-place scans on this workload's domains: 118 scans per
    // sweep instead of 155).  With more, the domain words take the place of
    // the overlap masks, which are dead once the seeds are planted.
    const bool in_regs = nls <= 4 * nth;
    uint32_t *dom = S.lab;
    uint32_t dm[4], cw[4], own2[2], e[4][Z / 2];
    if (!L.ufg && in_regs) {
        own2[0] = own2[1] = 0u;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            dm[j] = cw[j] = 0u;
#pragma unroll
            for (int i = 0; i < Z / 2; ++i) e[j][i] = 0u;
            if (tid + j * nth < nls) {
                const int li = S.gord ? (int)S.gord[4 * tid + j] : tid + j * nth;
                own2[j >> 1] |= (uint32_t)li << (16 * (j & 1));
                dm[j] = overlap_word(S.s[li], G > 1 ? S.s[ns + li] : 0u) & actc;
                cw[j] = S.C[li];
                nb_row<Z>(S.nb, li, e[j]);
                if (cw[j]) for_copies(S, li, [&](uint32_t a) { cl_st(a, cw[j]); });
            }
        }
    } else if (!L.ufg) {
        for (int li = tid; li < nls; li += nth) {
            dom[li] = overlap_word(S.s[li], G > 1 ? S.s[ns + li] : 0u) & actc;
            const uint32_t c = S.C[li];
            if (c) for_copies(S, li, [&](uint32_t a) { cl_st(a, c); });
        }
    }
    if (L.ufg) cl_grow_uf<Z>(P, L, S, act0, act1);
    else for (int round = 0;; ++round) {
        int grew = 0;
        for (int scan = 0; scan < kScansPerRound; ++scan) {
            if (in_regs) {
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    if (dm[j] == cw[j]) continue;    // nothing left to absorb
                    uint32_t nb = 0u;
#pragma unroll
                    for (int d = 0; d < Z; ++d) nb |= sh_ld(nb_addr(e[j][d >> 1], d, S.win));
                    const uint32_t n = cw[j] | (dm[j] & nb);
                    if (n != cw[j]) {
                        const int li = (int)((own2[j >> 1] >> (16 * (j & 1))) & 0xffffu);
                        S.C[li] = n;
                        cw[j] = n;
                        grew = 1;
                        for_copies(S, li, [&](uint32_t a) { cl_st(a, n); });
                    }
                }
            } else {
                for (int li = tid; li < nls; li += nth) {
                    const uint32_t d0 = dom[li], c = S.C[li];
                    if (d0 == c) continue;
                    uint32_t w[Z], nb = 0u;
                    nb_words<Z>(S, li, 0u, w);
#pragma unroll
                    for (int d = 0; d < Z; ++d) nb |= w[d];
                    const uint32_t n = c | (d0 & nb);
                    if (n != c) {
                        S.C[li] = n;
                        grew = 1;
                        for_copies(S, li, [&](uint32_t a) { cl_st(a, n); });
                    }
                }
            }
        }
        const uint32_t stamp = (t << 16) + (uint32_t)round + 1u;
        if (__any_sync(kFull, grew) && lane == 0)
            for (uint32_t r = 0; r < S.K; ++r) cl_st(cl_map(S.base + L.flags + 4 * (round & 1), r), stamp);
        cl_sync();
        if (round > 0 && (uint32_t)S.flags[round & 1] != stamp) {
            if (S.rank == 0 && tid == 0) {
                S.icmst[0] += (unsigned)(__popc(act0) + __popc(act1));
                S.icmst[1] += (unsigned)(round + 1) * kScansPerRound;   // scans of the own sites
            }
            break;
        }
    }

    // (d) flip the own and halo sites; copy-a energies of the moved pairs
    for (int li = tid; li < ns; li += nth) {
        const uint32_t cw = S.C[li];
        const uint32_t c0 = cw & 0x55555555u, c1 = (cw >> 1) & 0x55555555u;
        if (c0) S.s[li] ^= c0 | (c0 << 1);
        if (c1) S.s[ns + li] ^= c1 | (c1 << 1);
        if (trace && li < nls) {
            for (int w = 0; w < 2; ++w)
                for (uint32_t b = w ? c1 : c0; b; b &= b - 1u) atomicAdd(&S.csz[16 * w + ((__ffs(b) - 1) >> 1)], 1);
            if (P.tr_cmask) {
                uint32_t *cm = P.tr_cmask + ((size_t)slot * N + pos_of(P, S, li)) * 2;
                cm[0] = c0;
                cm[1] = c1;
            }
        }
    }
    __syncthreads();
}

// Steps 2a and 2b (see cluster_moves in pt_icm.cu).  S.seed holds the seed
// draws on entry.
template <bool GAUSS, int Z, bool DIL>
__device__ void cl_cluster_moves(const KParams &P, const ClusterLayout &L, const CS &S, uint32_t t, int slot,
                                 bool trace)
{
    using ET = typename std::conditional<GAUSS, float, int>::type;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    const int tid = threadIdx.x, nth = blockDim.x;
    const int nicm = P.n_icm, G = P.G, ns = S.ns, hs = S.hs;
    const int kp = pair_of_bit(lane);
    ET *E = (ET *)S.E;
    const ET *esum = (const ET *)S.esum;
    uint32_t act0 = 0u, act1 = 0u;
    bool by_rows = false;
    if constexpr (Z == 4 && !DIL) by_rows = L.rw > 0;
    if (by_rows) {
        if constexpr (Z == 4 && !DIL) cl_row_moves<GAUSS>(P, L, S, slot, trace, act0, act1);
    } else {
        cl_site_moves<GAUSS, Z>(P, L, S, t, slot, trace, act0, act1);
    }
    if (!(act0 | act1)) return;                      // the same decision in every CTA
    // copy-a energies of the moved pairs (cb = 0); a traced sweep then also
    // recomputes the copy-b energies (cb = 1) and records E_a + E_b of the two
    // recomputed energies, so that the trace tests the conservation of E_a + E_b
    ET *part = (ET *)S.Epart;
    for (int cb = 0; cb < (trace ? 2 : 1); ++cb) {
        if (cb) cl_sync();                           // every CTA has read the copy-a shares
        if constexpr (GAUSS) {
            for (int g = 0; g < G; ++g) {
                const uint32_t act = g ? act1 : act0;
                if (!act) continue;
                const uint32_t goff = (uint32_t)(g * ns * 4) - S.dCs;   // cluster word -> spin word g
                const uint32_t *sg = S.s + g * ns;
                float acc[16];
#pragma unroll
                for (int j = 0; j < 16; ++j) acc[j] = 0.f;
                for (int j = tid; j < hs; j += nth) {
                    const int li = hs + j;           // colour-1 sites: every bond once
                    const uint32_t sw = sg[li] >> cb;
                    uint32_t nw[Z];
                    nb_words<Z>(S, li, goff, nw);
                    float J[Z];
                    float Jsum = 0.f;
#pragma unroll
                    for (int d = 0; d < Z; ++d) {
                        nw[d] >>= cb;
                        J[d] = S.Jd[li * Z + d];
                        Jsum += J[d];
                    }
#pragma unroll
                    for (int jj = 0; jj < 16; ++jj) {
                        if (!((act >> (2 * jj)) & 1u)) continue;
                        const int b = 2 * jj;
                        float h = Jsum;
#pragma unroll
                        for (int d = 0; d < Z; ++d)
                            if ((nw[d] >> b) & 1u) h = fmaf(J[d], -2.f, h);
                        acc[jj] += ((sw >> b) & 1u) ? h : -h;
                    }
                }
                const float v = transpose_reduce16(acc, lane);
                if (!(lane & 1)) part[warp * 32 + 16 * g + (lane >> 1)] = v;
            }
        } else {
            uint32_t pl[kPlanes];
#pragma unroll
            for (int i = 0; i < kPlanes; ++i) pl[i] = 0u;
            const uint32_t o1 = (uint32_t)(ns * 4);
            for (int j = tid; j < hs; j += nth) {
                const int li = hs + j;               // colour-1 sites: every bond once
                const uint32_t y = copy_word(S.s[li], G > 1 ? S.s[ns + li] : 0u, cb);
                const uint32_t jb = S.Jb[li];
                uint32_t r[Z / 2], u[Z], c0, c1, c2, c3;
                nb_row<Z>(S.nb, li, r);
#pragma unroll
                for (int d = 0; d < Z; ++d) {
                    const uint32_t a = nb_addr(r[d >> 1], d, S.win) - S.dCs;
                    u[d] = y ^ copy_word(sh_ld(a), G > 1 ? sh_ld(a + o1) : 0u, cb) ^ (0u - ((jb >> d) & 1u));
                }
                csa_count<Z>(u, c0, c1, c2, c3);
                vadd4(pl, c0, c1, c2, c3);
            }
            part[warp * 32 + kp] = warp_vcount(pl, P.cnt_planes, lane);
        }
        __syncthreads();
        for (int k = tid; k < nicm; k += nth) {
            ET es = ET(0);
            if (S.seed[k])
                for (int w = 0; w < nwarps; ++w) es += part[w * 32 + k];
            cl_share<ET>(S, L.Epair, 32, k, es);
        }
        cl_sync();
        for (int k = tid; k < nicm; k += nth) {
            if (!S.seed[k]) continue;
            ET es = row_sum<ET>(S, S.Epair, 32, k);
            if constexpr (!GAUSS) es = 2 * es - (P.diluted ? P.nb_inst[slot] : P.Nb);   // E = 2 U - N_b (bonds present)
            if (cb == 0) {
                E[2 * k] = es;
                E[2 * k + 1] = esum[k] - es;
            }
            if (trace && S.rank == 0) {
                const size_t o = (size_t)slot * P.nT + k;
                if (cb == 0) {
                    if (by_rows) continue;           // counted by the pair's warp
                    int cs = 0;
                    for (uint32_t r = 0; r < S.K; ++r) cs += (int)cl_ld(cl_map(S.base + L.csz + 4 * k, r));
                    P.tr_csize[o] = cs;
                } else {
                    P.tr_ea[o] = (float)(E[2 * k] + es);
                }
            }
        }
        __syncthreads();
    }
}

// Step 3 (see pt_pass in pt_icm.cu): the same energies and draws in every
// CTA give the same decisions; each CTA permutes its own and halo words.
template <bool GAUSS>
__device__ void cl_pt_pass(const KParams &P, const CS &S, int slot, bool trace)
{
    using ET = typename std::conditional<GAUSS, float, int>::type;
    const int np = P.nT - 1, ns = S.ns;
    // every CTA decides alike (the same energies and draws); rank 0 traces
    if (threadIdx.x < 32)
        pt_warp<GAUSS, ET>((ET *)S.E, P.R, np, S.swap_x, P.dbeta_l2e, S.swap_mask,
                           trace && S.rank == 0 ? P.tr_swap + (size_t)slot * 2 * np : nullptr);
    __syncthreads();
    SwapMasks m;
    if (swap_masks(S.swap_mask, m)) {
        const bool two = P.G > 1;
        for (int li = threadIdx.x; li < ns; li += blockDim.x) {
            const uint64_t x = (uint64_t)S.s[li] | (two ? (uint64_t)S.s[ns + li] << 32 : 0ull);
            const uint64_t y = swap_apply(m, x);
            S.s[li] = (uint32_t)y;
            if (two) S.s[ns + li] = (uint32_t)(y >> 32);
        }
    }
    __syncthreads();
}

// Observables (see measure in pt_icm.cu): this CTA's counts, stored into rank
// 0's rows.  The barrier before rank 0 adds them is the one that ends the step.
template <int Z>
__device__ __forceinline__ void cl_count(const KParams &P, const ClusterLayout &L, const CS &S, int parity)
{
    const int lane = threadIdx.x & 31, nth = blockDim.x;
    const int nT = P.nT, nls = S.nls, ns = S.ns, hs = S.hs;
    const bool two = P.G > 1;
    const uint32_t o1 = (uint32_t)(ns * 4);
    uint32_t pn[kPlanes], pd[kPlanes];
#pragma unroll
    for (int i = 0; i < kPlanes; ++i) pn[i] = pd[i] = 0u;
    for (int li = threadIdx.x; li < nls; li += nth) {
        const uint32_t x = overlap_word(S.s[li], two ? S.s[ns + li] : 0u);
        vadd(pn, x);
        if (li < hs) continue;
        uint32_t r[Z / 2], y[Z], c0, c1, c2, c3;   // a padding entry points at the site itself: y = 0
        nb_row<Z>(S.nb, li, r);
#pragma unroll
        for (int d = 0; d < Z; ++d) {
            const uint32_t a = nb_addr(r[d >> 1], d, S.win) - S.dCs;
            y[d] = x ^ overlap_word(sh_ld(a), two ? sh_ld(a + o1) : 0u);
        }
        csa_count<Z>(y, c0, c1, c2, c3);
        vadd4(pd, c0, c1, c2, c3);
    }
    const int k = pair_of_bit(lane);
    const int n = warp_vcount(pn, P.cnt_planes, lane), d = warp_vcount(pd, P.cnt_planes, lane);
    if (k < nT) {
        atomicAdd(S.cnt_n + k, n);
        atomicAdd(S.cnt_d + k, d);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < 2 * nT; i += nth) {
        const int c = i >= nT, kk = i - c * nT;
        int *v = (c ? S.cnt_d : S.cnt_n) + kk;
        cl_st(cl_map(S.base + L.cntobs + 4u * (uint32_t)((parity * (int)S.K + (int)S.rank) * 64 + 32 * c + kk), 0u),
              (uint32_t)*v);
        *v = 0;
    }
}

// rank 0, after the barrier; the rows alternate between steps, since the next
// step may count without another barrier
template <bool GAUSS>
__device__ __forceinline__ void cl_accumulate(const KParams &P, const CS &S, int slot, int parity)
{
    using ET = typename std::conditional<GAUSS, float, int>::type;
    const int N = P.N, nT = P.nT;
    const int *rows = S.cntobs + parity * (int)S.K * 64;
    for (int k = threadIdx.x; k < nT; k += blockDim.x) {
        const long long n = row_sum<int>(S, rows, 64, k), d = row_sum<int>(S, rows, 64, 32 + k);
        const ET *E = (const ET *)S.E;
        S.accE[k] += (double)E[2 * k] + (double)E[2 * k + 1];
        S.acc64[0 * nT + k] += n;
        S.acc64[1 * nT + k] += (N - 2 * n) * (N - 2 * n);
        S.acc64[2 * nT + k] += n < N - n ? n : N - n;
        S.acc64[3 * nT + k] += d;
        atomicAdd(&P.hist[((size_t)slot * nT + k) * (N + 1) + ICM_IDX(n, N + 1, 22)], 1ull);
    }
    if (threadIdx.x == 0) S.nmeas[0] += 1;
}

// ---------------------------------------------------------------------------
// MAXT: the widest CTA of the variant, which sets its registers a thread: 64
// (1024) or 128 (512).  At 64 the kernel spills; at 128 fewer CTAs share an SM.
// 3D Gaussian L=16 on 8 x 256, us per sweep: 20 instances 52.8 (64 registers) and
// 42.9 (128), one 43.1 and 34.4, but 72 instances, more than the clusters
// resident at 128 registers, 87.6 and 92.3.  So the host takes 128 where every
// instance is resident with them (ClusterLayout::lean).
template <bool GAUSS, int Z, bool DIL, int MAXT>
__global__ void __launch_bounds__(MAXT, 1) cluster_kernel(const KParams P, const ClusterLayout L, uint32_t n_sweeps)
{
    using ET = typename std::conditional<GAUSS, float, int>::type;
    extern __shared__ __align__(16) unsigned char smem[];
    const CS S = make_cs(smem, L);
    const int tid = threadIdx.x, nth = blockDim.x;
    const int N = P.N, R = P.R, nT = P.nT, G = P.G, nls = S.nls, ns = S.ns;

    if (tid < 2) S.flags[tid] = 0;   // growth round stamps (the same in every CTA at all times)
    if (tid < 32) {
        S.cnt_n[tid] = 0;
        S.cnt_d[tid] = 0;
    }
    // neighbour table: the offset of each neighbour's cluster word in the shared
    // window, own or halo, by the batch's lattice; an instance's absent bonds (diluted
    // batches) point at the site itself
    const uint32_t cadr = S.base + (uint32_t)L.C;
    const uint16_t *tab = P.cl_nb + (size_t)S.rank * nls * Z;
    auto neighbour_table = [&](const uint16_t *nbr, const uint8_t *zdeg) {
        for (int i = tid; i < nls * Z; i += nth) {
            const int li = i / Z, d = i - li * Z;
            int q = ICM_IDX(tab[i], ns, 20);
            if constexpr (DIL) {
                const int p = pos_of(P, S, li);
                if (nbr[p * Z + d] == p) q = li;
            }
            S.nb[i] = (uint16_t)(cadr - S.win + 4u * (uint32_t)q);
        }
        if (!GAUSS && (DIL || !P.const_z))
            for (int li = tid; li < nls; li += nth) S.zdeg[li] = zdeg[pos_of(P, S, li)];
    };
    if constexpr (!DIL) neighbour_table(P.nbr, P.zdeg);
    for (int li = tid; li < nls; li += nth) S.xoff[li] = P.cl_xoff[S.rank * nls + li];
    for (int i = tid; i < L.nx; i += nth) {          // copies: (CTA, halo entry, last) -> cluster-window address
        const uint32_t v = P.cl_xl[S.rank * L.nx + i];
        S.xl[i] = cl_map(cadr + 4u * ((uint32_t)nls + (v & 0xffffu)), (v >> 16) & 0xffu) | (v >> 31);
    }
    if (L.ufg)
        for (int i = tid; i < L.nh; i += nth) {      // halo entry -> the owner's first label word
            const uint32_t v = P.cl_hown[S.rank * L.nh + i];
            S.hlab[i] = cl_map(S.base + L.lab + 4u * (v & 0xffffu), v >> 16);
        }
    const uint16_t *hpos = P.cl_hpos + S.rank * L.nh;
    if (L.gord >= 0)
        for (int i = tid; i < nls; i += nth) S.gord[i] = P.cl_order[i];
    if constexpr (GAUSS) {
        for (int k = tid; k < 16 * G; k += nth) S.b2l[k] = k < nT ? P.b2l[2 * k] : 0.f;
    } else {
        load_thr_rows<Z>(S.thr, P.thr_metro, R, G, tid, nth);
    }

    for (int slot = (int)cl_id(); slot < P.n_inst; slot += (int)cl_count()) {
        if (P.active && !P.active[slot]) continue;   // the same for every CTA of the cluster
        for (int i = tid; i < G * ns; i += nth) {
            const int g = i >= ns, li = i - g * ns;
            const int p = li < nls ? pos_of(P, S, li) : (int)hpos[li - nls];
            if (p != 0xffff) S.s[i] = P.spins[((size_t)slot * G + g) * N + p];   // fewer entries than nh: unused
        }
        if constexpr (GAUSS) {
            for (int i = tid; i < nls * Z; i += nth)
                S.Jd[i] = P.Jd[((size_t)slot * N + pos_of(P, S, i / Z)) * Z + i % Z];
            for (int r = tid; r < R; r += nth) ((float *)S.E)[r] = P.Ef[(size_t)slot * R + r];
        } else {
            for (int li = tid; li < nls; li += nth) S.Jb[li] = P.Jb[(size_t)slot * N + pos_of(P, S, li)];
            for (int r = tid; r < R; r += nth) ((int *)S.E)[r] = P.Ei[(size_t)slot * R + r];
        }
        if (S.rank == 0) {
            for (int k = tid; k < nT; k += nth) {
                S.accE[k] = P.accE[(size_t)slot * nT + k];
                for (int a = 0; a < 4; ++a) S.acc64[a * nT + k] = P.acc64[((size_t)a * P.n_inst + slot) * nT + k];
            }
            if (tid == 0) {
                S.nmeas[0] = P.n_meas[slot];
                S.icmst[0] = S.icmst[1] = 0ull;
            }
        }
        // a diluted instance: its own neighbour table (absent bonds point at the
        // site itself) and degrees, and zero-energy proposals accepted with
        // probability 1/2
        bool tie = false;
        if constexpr (DIL) {
            neighbour_table(P.nbr_inst + (size_t)slot * N * Z, P.zdeg_inst + (size_t)slot * N);
            tie = P.nb_inst[slot] < P.Nb;
        }
        const uint32_t inst = P.inst_id[slot];
        const long long t_meas = P.t_meas_inst ? P.t_meas_inst[slot] : P.t_meas;
        uint32_t t = P.tsweep[slot];
        cl_sync();

        for (uint32_t step = 0; step < n_sweeps; ++step, ++t) {
            const bool trace = P.trace && step + 1 == n_sweeps;
            if (trace && S.rank == 0) {
                for (int k = tid; k < nT; k += nth) {
                    const size_t o = (size_t)slot * nT + k;
                    P.tr_n_pre[o] = -1;
                    P.tr_flip2a[o] = 0;
                    P.tr_seed[o] = -1;
                    P.tr_csize[o] = 0;
                    P.tr_eb[o] = 0.f;
                    P.tr_ea[o] = 0.f;
                }
                for (int i = tid; i < 2 * (nT - 1); i += nth) P.tr_swap[(size_t)slot * 2 * (nT - 1) + i] = 0;
            }
            if (trace && P.tr_cmask)                 // every CTA clears its own positions
                for (int li = tid; li < nls; li += nth) {
                    uint32_t *cm = P.tr_cmask + ((size_t)slot * N + pos_of(P, S, li)) * 2;
                    cm[0] = 0u;
                    cm[1] = 0u;
                }
            const bool icm = P.icm_every > 0 && t % (uint32_t)P.icm_every == 0 && P.n_icm > 0;
            const bool pt = P.swap_every > 0 && t % (uint32_t)P.swap_every == 0 && nT > 1;
            const bool meas = (long long)t >= t_meas;
            if (P.enable_metropolis) cl_metropolis<GAUSS, Z, DIL>(P, L, S, t, inst, tie);
            {   // the draws of steps 2b and 3, by the threads that share no energy
                const int nicm = icm ? P.n_icm : 0, np = nT - 1, n = nicm + (pt ? 2 * np : 0);
                const int at = ((R + 31) & ~31) < nth ? (R + 31) & ~31 : 0;
                for (int i = tid < at ? tid + nth - at : tid - at; i < n; i += nth) {
                    if (i < nicm) {
                        uint32_t x[4];
                        philox10k((uint32_t)i, t, 0u, (1u << 24) | inst, P.key, x);
                        S.seed[i] = (int)x[0];
                    } else {
                        pt_draw<GAUSS>(i - nicm, np, t, inst, P.key, S.swap_x, P.thr_swap, P.swap_off, P.swap_len,
                                       P.dbeta_l2e);
                    }
                }
            }
            if (P.enable_metropolis) {
                cl_sync();
                for (int r = tid; r < R; r += nth) {
                    ET e = row_sum<ET>(S, S.Esw, R, r);
                    if constexpr (!GAUSS) e = 2 * e - (DIL ? P.nb_inst[slot] : P.Nb);   // E = 2 U - (bonds present)
                    ((ET *)S.E)[r] = e;
                }
            }
            __syncthreads();
            if (icm) cl_cluster_moves<GAUSS, Z, DIL>(P, L, S, t, slot, trace);
            if (pt) cl_pt_pass<GAUSS>(P, S, slot, trace);
            if (meas) cl_count<Z>(P, L, S, (int)(step & 1u));
            cl_sync();               // ends the step: no CTA reads this step's words any more
            if (meas && S.rank == 0) cl_accumulate<GAUSS>(P, S, slot, (int)(step & 1u));
        }
        __syncthreads();

        for (int i = tid; i < G * nls; i += nth) {
            const int g = i >= nls, li = i - g * nls;
            P.spins[((size_t)slot * G + g) * N + pos_of(P, S, li)] = S.s[g * ns + li];
        }
        if (S.rank == 0) {
            for (int r = tid; r < R; r += nth) {
                if constexpr (GAUSS) P.Ef[(size_t)slot * R + r] = ((float *)S.E)[r];
                else P.Ei[(size_t)slot * R + r] = ((int *)S.E)[r];
            }
            for (int k = tid; k < nT; k += nth) {
                P.accE[(size_t)slot * nT + k] = S.accE[k];
                for (int a = 0; a < 4; ++a) P.acc64[((size_t)a * P.n_inst + slot) * nT + k] = S.acc64[a * nT + k];
            }
            if (tid == 0) {
                P.n_meas[slot] = S.nmeas[0];
                P.tsweep[slot] = t;
                if (P.icm_stats) {
                    P.icm_stats[2 * (size_t)slot] += S.icmst[0];
                    P.icm_stats[2 * (size_t)slot + 1] += S.icmst[1];
                }
            }
        }
        cl_sync();
    }
}

template <bool GAUSS, int Z, bool DIL, int MAXT>
cudaError_t launch_cluster_t(const KParams &P, const ClusterLayout &L, int threads, int n_clusters, uint32_t n_sweeps,
                             cudaStream_t st)
{
    auto kern = cluster_kernel<GAUSS, Z, DIL, MAXT>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, L.total);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(n_clusters * L.K), 1, 1);
    cfg.blockDim = dim3((unsigned)threads, 1, 1);
    cfg.dynamicSmemBytes = (size_t)L.total;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)L.K;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, P, L, n_sweeps);
}

template <bool GAUSS, int Z, bool DIL, int MAXT>
cudaError_t cluster_occupancy_t(int K, int threads, int smem, int *clusters)
{
    auto kern = cluster_kernel<GAUSS, Z, DIL, MAXT>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)K, 1, 1);
    cfg.blockDim = dim3((unsigned)threads, 1, 1);
    cfg.dynamicSmemBytes = (size_t)smem;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)K;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaOccupancyMaxActiveClusters(clusters, kern, &cfg);
}


constexpr bool kPartGauss = ICM_PART == 2;

template <int Z, bool DIL>
cudaError_t launch_part_zd(const KParams &P, const ClusterLayout &L, int threads, int n_clusters, uint32_t n_sweeps,
                           cudaStream_t st)
{
    return L.lean ? launch_cluster_t<kPartGauss, Z, DIL, kLeanThreads>(P, L, threads, n_clusters, n_sweeps, st)
                  : launch_cluster_t<kPartGauss, Z, DIL, kMaxThreadsWide>(P, L, threads, n_clusters, n_sweeps, st);
}

template <int Z>
cudaError_t launch_part_z(const KParams &P, const ClusterLayout &L, int threads, int n_clusters, uint32_t n_sweeps,
                          cudaStream_t st)
{
    return P.diluted ? launch_part_zd<Z, true>(P, L, threads, n_clusters, n_sweeps, st)
                     : launch_part_zd<Z, false>(P, L, threads, n_clusters, n_sweeps, st);
}

cudaError_t launch_part(const KParams &P, const ClusterLayout &L, int threads, int n_clusters, uint32_t n_sweeps,
                        cudaStream_t st)
{
    switch (P.Z) {
    case 4: return launch_part_z<4>(P, L, threads, n_clusters, n_sweeps, st);
    case 6: return launch_part_z<6>(P, L, threads, n_clusters, n_sweeps, st);
    case 8: return launch_part_z<8>(P, L, threads, n_clusters, n_sweeps, st);
    default: return cudaErrorInvalidValue;
    }
}

template <int Z>
cudaError_t occupancy_part_z(bool dil, bool lean, int K, int threads, int smem, int *clusters)
{
    if (lean)
        return dil ? cluster_occupancy_t<kPartGauss, Z, true, kLeanThreads>(K, threads, smem, clusters)
                   : cluster_occupancy_t<kPartGauss, Z, false, kLeanThreads>(K, threads, smem, clusters);
    return dil ? cluster_occupancy_t<kPartGauss, Z, true, kMaxThreadsWide>(K, threads, smem, clusters)
               : cluster_occupancy_t<kPartGauss, Z, false, kMaxThreadsWide>(K, threads, smem, clusters);
}

cudaError_t occupancy_part(int Z, bool dil, bool lean, int K, int threads, int smem, int *clusters)
{
    switch (Z) {
    case 4: return occupancy_part_z<4>(dil, lean, K, threads, smem, clusters);
    case 6: return occupancy_part_z<6>(dil, lean, K, threads, smem, clusters);
    case 8: return occupancy_part_z<8>(dil, lean, K, threads, smem, clusters);
    default: return cudaErrorInvalidValue;
    }
}

int check_part(unsigned int *out, int reset)
{
#ifdef ICM_CHECKED
    if (cudaMemcpyFromSymbol(out, g_icm_check, sizeof(unsigned int) * 4) != cudaSuccess) return -4;
    if (reset) {
        unsigned int z[4] = {};
        if (cudaMemcpyToSymbol(g_icm_check, z, sizeof(z)) != cudaSuccess) return -4;
    }
    return 0;
#else
    (void)out;
    (void)reset;
    return -7;
#endif
}

}  // namespace

#if ICM_PART == 1
#define ICM_CL_NAME(f) f##_pmj
#else
#define ICM_CL_NAME(f) f##_gauss
#endif
cudaError_t ICM_CL_NAME(launch_cluster)(const KParams &P, const ClusterLayout &L, int threads, int n_clusters,
                                        uint32_t n_sweeps, cudaStream_t st)
{
    return launch_part(P, L, threads, n_clusters, n_sweeps, st);
}
cudaError_t ICM_CL_NAME(cluster_occupancy)(int Z, bool dil, bool lean, int K, int threads, int smem, int *clusters)
{
    return occupancy_part(Z, dil, lean, K, threads, smem, clusters);
}
int ICM_CL_NAME(debug_check_cluster)(unsigned int *out, int reset) { return check_part(out, reset); }

}  // namespace icm

#else  // ICM_PART == 0

namespace icm {
namespace {
int align_up16(int v) { return (v + 15) / 16 * 16; }
}  // namespace

ClusterLayout cluster_layout(int N, int Z, int R, int G, int nT, int K, int nwarps, bool gauss, int ufg,
                             bool order, int nh, int nx, int row_kind, int Lx)
{
    ClusterLayout L{};
    L.K = K;
    L.ufg = ufg;
    L.hs = (N / 2) / K;
    L.nls = 2 * L.hs;
    L.NWl = L.nls / 32;
    L.nh = nh;
    L.nx = nx;
    L.ns = L.nls + nh;
    int o = 0;
    auto take = [&](int bytes) {
        o = align_up16(o);
        const int at = o;
        o += bytes;
        return at;
    };
    const int nls = L.nls, ns = L.ns;
    if (row_kind) {
        L.rs = row_words_of(row_kind, Lx);
        L.rw = L.rs / K;
        L.rh = L.rs / Lx > 1 ? L.rs / Lx : 1;       // words of a row (or the word that holds it)
    }
    // in the row form the pairs' clusters take the place of the cluster words and
    // the pairs' rows that of the masks
    const int c_bytes = std::max(ns * 4, row_kind ? nT * (L.rw + 2 * L.rh) * 4 : 0);
    const int m_bytes = std::max((ufg > 1 ? ufg : 1) * nls * 4, row_kind ? (nT + K - 1) / K * L.rs * 4 : 0);
    L.C = take(c_bytes);           // first: its addresses fit the 16 bits of the neighbour table
    L.rowc = L.C;
    L.s = take(G * ns * 4);
    L.nb = take(nls * Z * 2);
    L.xoff = take(nls * 2);
    L.xl = take(nx * 4);
    L.hlab = ufg ? take(nh * 4) : 0;
    L.coup = take(gauss ? nls * Z * 4 : nls);
    L.zdeg = take(nls);
    L.E = take(R * 4);
    L.Epart = take(nwarps * (R > 32 ? R : 32) * 4);
    L.Esw = take(K * R * 4);
    L.Epair = take(K * 32 * 4);
    L.rtab = take(gauss ? G * 32 * 4 : G * 16 * 8 * 4);
    // the overlap masks are dead once the seeds are planted: the domain words
    // or the union-find labels take their place (one pair's labels are as
    // large as the masks)
    L.lab = take(m_bytes);
    L.mask = L.rowm = L.lab;
    L.rowi = take(32 * 4);
    L.sadr = take(32 * 4);
    L.sroot = take(kMaxUfGroup * 4);
    L.gord = order ? take(nls * 2) : -1;
    L.cntloc = take(K * 64 * 4);
    L.cntobs = take(2 * K * 64 * 4);
    L.flags = take(2 * 4);
    L.seed = take(32 * 4);
    L.esum = take(32 * 4);
    L.flipw = take(2 * 4);
    L.csz = take(32 * 4);
    L.swap_x = take(2 * 32 * 4);
    L.swap_mask = take(6 * 8);
    L.cnt_n = take(32 * 4);
    L.cnt_d = take(32 * 4);
    L.accE = take(nT * 8);
    L.acc64 = take(4 * nT * 8);
    L.nmeas = take(8);
    L.icmst = take(16);
    L.total = align_up16(o);
    return L;
}

cudaError_t launch_cluster(const KParams &P, const ClusterLayout &L, bool gauss, int threads, int n_clusters,
                           uint32_t n_sweeps, cudaStream_t st)
{
    if (threads > (L.lean ? kLeanThreads : kMaxThreadsWide) || L.K < 1 || L.hs % 32) return cudaErrorInvalidValue;
    if (P.diluted && (!P.nbr_inst || !P.zdeg_inst || !P.nb_inst)) return cudaErrorInvalidValue;
    return gauss ? launch_cluster_gauss(P, L, threads, n_clusters, n_sweeps, st)
                 : launch_cluster_pmj(P, L, threads, n_clusters, n_sweeps, st);
}

cudaError_t cluster_occupancy(bool gauss, int Z, bool dil, bool lean, int K, int threads, int smem, int *clusters)
{
    return gauss ? cluster_occupancy_gauss(Z, dil, lean, K, threads, smem, clusters)
                 : cluster_occupancy_pmj(Z, dil, lean, K, threads, smem, clusters);
}

}  // namespace icm

#ifdef ICM_CHECKED
// Checked builds: the check words of the thread-block-cluster kernels (guarded
// neighbour positions, seed sites and histogram bins; site codes 20-23), read
// like icm_debug_check reads those of the fused kernels.
extern "C" int icm_debug_check_cluster(unsigned int *out, int reset)
{
    unsigned int a[4], b[4];
    int rc = icm::debug_check_cluster_pmj(a, reset);
    if (!rc) rc = icm::debug_check_cluster_gauss(b, reset);
    if (rc) return rc;
    out[0] = a[0] + b[0];
    for (int i = 1; i < 4; ++i) out[i] = a[0] ? a[i] : b[i];
    return 0;
}
#endif

#endif  // ICM_PART
