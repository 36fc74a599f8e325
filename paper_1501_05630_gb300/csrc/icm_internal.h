// Internal declarations shared by the host half (icm_api.cpp) and the device
// half (pt_icm.cu) of the library.  Not part of the public ABI.
#pragma once
#include <cstdint>
#include <vector>
#include <cuda_runtime.h>

namespace icm {

constexpr int kMaxZ = 8;          // largest degree of the supported graphs (4D hypercubic)
constexpr int kMaxR = 64;         // replicas per instance (2 N_T, N_T <= 32)
constexpr int kMaxThreads = 128;  // threads per CTA of the fused kernel, kLayoutShared
constexpr int kMaxThreadsWide = 1024;  // threads per CTA of the fused kernel, kLayoutWide and kLayoutBig
// One-CTA layouts: the instance in shared memory with CTAs up to kMaxThreads;
// in global memory with wider CTAs; in shared memory with wider CTAs.
constexpr int kLayoutShared = 0, kLayoutWide = 1, kLayoutBig = 2;
constexpr int kPlanes = 8;        // bit-planes of the vertical counters (counts < 256 per thread)

// Entries per replica of the +-J Metropolis threshold table, indexed by
// m = s_i h_i = 0..Z (m = 0: the probability-1/2 entry of diluted instances).
#ifdef __CUDACC__
__host__ __device__
#endif
constexpr int thr_stride(int Z) { return Z > 7 ? 16 : 8; }

// Words from one pair's overlap mask to the next: odd, so that the threads of
// the seed search (one per pair) read different banks.
#ifdef __CUDACC__
__host__ __device__
#endif
constexpr int mask_stride(int NW) { return NW | 1; }

// Row forms of the cluster moves on undiluted 2D lattices (row_growth.cuh), by
// the lattice's size; 0: the word-per-site form (other lattices, absent bonds,
// L above 128 or not divisible into lanes of four rows).
constexpr int kRows8 = 1, kRows16 = 2, kRows32 = 3, kRows64 = 4, kRows128 = 5;
inline int row_kind_of(bool square2d, int L)
{
    if (!square2d) return 0;
    return L <= 8 ? kRows8 : L <= 16 ? kRows16 : L <= 32 ? kRows32 : L <= 64 ? kRows64
                                                        : L <= 128 && L % 4 == 0 ? kRows128 : 0;
}
// the row form on K CTAs, each with L / K whole rows in whole words
inline int cluster_row_kind(int kind, int L, int K)
{
    const int per = kind == kRows8 ? 4 : kind == kRows16 ? 2 : 1;   // rows of a word
    return kind && L % K == 0 && (L / K) % per == 0 ? kind : 0;
}
// words of one pair's rows
inline int row_words_of(int kind, int L)
{
    return kind == kRows8 ? (L + 3) / 4 : kind == kRows16 ? L / 2 : kind == kRows32 ? L : kind == kRows64 ? 2 * L : 4 * L;
}

// Bit-planes for the counts of a thread that takes `sites` sites, `half_sites`
// of them of colour 1 with Z bonds each (at most kPlanes: the launch-shape
// checks bound both counts by 255).
inline int count_planes(int sites, int half_sites, int Z)
{
    const int most = half_sites * Z > sites ? half_sites * Z : sites;
    int n = 1;
    while (n < kPlanes && (most >> n)) ++n;
    return n;
}

// Byte offsets into the fused kernel's dynamic shared memory.  In the
// global-resident ("wide") layout the spins, couplings, neighbour table,
// overlap masks and cluster words stay in global memory (size 0 here).
struct SmemLayout {
    int spins;      // uint32 [G][N]
    int nbr;        // uint16 [N][Z]   neighbour positions, padding = self
    int zdeg;       // uint8  [N]      degree (+-J only)
    int coup;       // float [N][Z] (Gaussian) or uint8 [N] bit d = (J < 0) (+-J)
    int E;          // float or int32 [R]
    int Epart;      // float or int32 [nwarps][max(R, 32)]
    int rtab;       // uint32 [16 G][8] threshold rows (+-J) or float [16 G] -2 beta log2(e) (Gaussian)
    int icm_mask;   // uint32 [n_icm][mask_stride(NW)] overlap masks per ICM pair
    int icm_C;      // uint32 [N]        cluster bits of every pair (bit 2k: pair k, bit 2k + 1: pair 16 + k)
    int swap_x;     // uint32 [2][32]
    int swap_mask;  // uint64 [3][2]   PT moves as bit masks (pt_warp), per copy
    int swap_tab;   // [3][32]         per neighbouring pair k: dbeta log2(e) (float), +-J table offset and length
    int flipw;      // uint32 [2]      step-2a reversal masks of the two words
    int icm_seed;   // int32 [32]      seed position per ICM pair (-1: none)
    int icm_esum;   // float or int32 [32]  E_a + E_b of each ICM pair before the move
    int cnt_n;      // int32 [32]
    int cnt_d;      // int32 [32]
    int accE;       // double [nT]
    int acc64;      // int64 [4][nT]  n, q2, pmin, d
    int nmeas;      // int64 [1]
    int icmst;      // uint64 [2]      this instance's cluster moves (pairs with n > 0) and growth scans
    int total;
};

// Everything the fused kernel reads or writes.  Device pointers.
struct KParams {
    int N, Nb, nT, R, G, Z, n_inst, n_icm, half, NW;
    int const_z;                  // degree when uniform (lattices), 0 = per-site table
    int wide;                     // kLayoutShared, kLayoutWide or kLayoutBig
    int diluted;                  // 1: some instance has absent bonds (J = 0): per-instance tables below
    int scratch_words;            // wide layout: uint32 words of scratch per CTA (cluster words, masks)
    uint32_t *scratch;            // wide layout: [grid][scratch_words]
    int row_kind, row_words;      // row form of the cluster moves and words per pair (row_kind 0: none)
    int L;                        // lattice size
    int cnt_planes;               // bit-planes that hold a thread's counts of sites and bonds
    // geometry, shared by all instances of the batch
    const uint16_t *nbr;          // [N][Z]
    const uint8_t *zdeg;          // [N]
    const uint16_t *pos2site;     // [N]
    // per instance, used when `diluted`: neighbour positions with absent bonds
    // replaced by the site itself, degree = bonds present, bonds present
    const uint16_t *nbr_inst;     // [n_inst][N][Z]
    const uint8_t *zdeg_inst;     // [n_inst][N]
    const int32_t *nb_inst;       // [n_inst]
    // per instance
    const float *Jd;              // [n_inst][N][Z]  (Gaussian)
    const uint8_t *Jb;            // [n_inst][N]     (+-J)
    uint32_t *spins;              // [n_inst][G][N]
    float *Ef;                    // [n_inst][R]     (Gaussian)
    int32_t *Ei;                  // [n_inst][R]     (+-J)
    uint32_t *tsweep;             // [n_inst]
    const uint32_t *inst_id;      // [n_inst]
    // temperature tables
    const uint32_t *thr_metro;    // [R][thr_stride(Z)]
    const float *b2l;             // [R]
    const double *beta;           // [nT]
    const float *dbeta_l2e;       // [nT-1] (beta_k - beta_{k+1}) log2(e)
    const uint32_t *thr_swap;     // concatenated per pair k
    const int32_t *swap_off;      // [nT-1]
    const int32_t *swap_len;      // [nT-1]
    // schedule
    int icm_every, swap_every, enable_2a, enable_metropolis, trace;
    long long t_meas;
    const long long *t_meas_inst;  // [n_inst] per-instance measurement start, or null (t_meas for all)
    const uint8_t *active;         // [n_inst] 0 = free slot (skipped), or null (all active)
    uint32_t seed_lo, seed_hi;
    // Philox4x32-10 key schedule of the seed: key[2i] = seed_lo + i 0x9E3779B9,
    // key[2i+1] = seed_hi + i 0xBB67AE85 (mod 2^32), the round keys i = 0..9;
    // read from the kernel parameters, so no round recomputes them
    uint32_t key[20];
    // observables
    double *accE;                 // [n_inst][nT]
    long long *acc64;             // [4][n_inst][nT]: n, (N-2n)^2, min(n,N-n), d
    unsigned long long *hist;     // [n_inst][nT][N+1]
    long long *n_meas;            // [n_inst]
    // ICM counters, accumulated over launches (cleared with the observables):
    // [n_inst][2] = pairs moved (n > 0 after step 2a), growth scans (passes over the sites)
    unsigned long long *icm_stats;
    // trace of the last sweep
    int32_t *tr_n_pre, *tr_flip2a, *tr_seed, *tr_csize;  // [n_inst][nT]
    float *tr_eb, *tr_ea;                                // [n_inst][nT]
    uint8_t *tr_swap;                                    // [n_inst][2][nT-1]
    uint32_t *tr_cmask;   // [n_inst][N][2] cluster words of the traced sweep, by position (NULL = off)
    // thread-block-cluster layout of 2D lattices: the own site that thread t
    // of a CTA grows as its j-th, at [4 t + j] (2 x 2 blocks of sites), or null
    const uint16_t *cl_order;     // [nls]
    // thread-block-cluster layout: ClusterTables of the lattice and K
    const uint16_t *cl_nb, *cl_hpos, *cl_xoff;
    const uint32_t *cl_xl, *cl_hown;
    SmemLayout sm;
};

// The shared group kernel (pt_icm.cu): one persistent CTA of kTeamThreads
// threads per SM runs tiles of instances of several batches (sizes) of one
// disorder kind and degree; a tile of batch c is `count` instances side by
// side, one team of team_threads[c] threads each (a divisor of
// kTeamThreads), each team with its own shared memory (KParams::sm of its
// batch, laid out for the team's width) and its own barrier.
constexpr int kTeamThreads = 896;   // 7 x 128: the threads of seven fused-kernel CTAs
constexpr int kTeamClasses = 8;     // batches per shared group
struct TeamItem {
    int cls, slot0, count;
};
struct TeamParams {
    KParams cls[kTeamClasses];
    int team_threads[kTeamClasses];
    const TeamItem *items;         // [n_items], in the order the CTAs take them
    int n_items;
    int *counters;                 // [2]: next item, CTAs done; zero between launches
    uint32_t key[20];              // Philox round keys of the common seed
};

// Host-built position tables of one lattice (see host_tables in icm_api.cpp).
struct HostTables {
    int N = 0, Nb = 0, Z = 0;
    std::vector<uint16_t> nbr;        // [N][Z]
    std::vector<uint16_t> pos2site;   // [N]
    std::vector<int32_t> edge_bond;   // [N][Z]
};
bool host_tables(int lattice, int L, HostTables &t);

SmemLayout smem_layout(int N, int Z, int R, int G, int nT, int n_icm, int nwarps, bool gauss, bool wide);

// Thread-block-cluster layout (cluster_icm.cu): one instance per cluster of
// K CTAs.  CTA r owns the positions [c half + r hs, c half + (r+1) hs) of
// each colour c (hs = half / K), stored as local index li = c hs + i; the
// local indices nls .. ns-1 are its halo, copies of the sites of other CTAs
// that border its own (cluster_tables).  The spin and cluster words have
// stride 4 bytes per local site, so the address of a neighbour's cluster word
// also locates its spin words.  Byte offsets into each CTA's dynamic shared
// memory:
struct ClusterLayout {
    int lean;              // 1: the variant with 128 registers a thread (CTAs up to kLeanThreads)
    int K, hs, nls, NWl;   // CTAs, own sites per colour, own sites (2 hs), mask words (nls / 32)
    int nh, nx, ns;        // halo entries, copies of own sites in other halos, nls + nh
    int C;          // uint32 [ns]       cluster word: bit 2j = pair j, bit 2j + 1 = pair 16 + j
    int s;          // uint32 [G][ns]    spin words
    int nb;         // uint16 [nls][Z]   offset of the neighbour's cluster word C in the shared window
    int xoff;       // uint16 [nls]      first entry of the site's copies in xl, 0xffff = none
    int xl;         // uint32 [nx]       cluster-window address of a copy's cluster word, bit 0 = the site's last
    int hlab;       // uint32 [nh]       cluster-window address of the halo site's first label word (union-find)
    int coup;       // float [nls][Z] (Gaussian) or uint8 [nls] sign bits (+-J)
    int zdeg;       // uint8 [nls]
    int E;          // float or int32 [R]       energies (the same in every CTA)
    int Epart;      // float or int32 [nwarps][max(R, 32)]
    int Esw;        // float or int32 [K][R]    every CTA's share of the sweep energies (written remotely)
    int Epair;      // float or int32 [K][32]   every CTA's share of the copy-a energies (written remotely)
    int rtab;       // thresholds (+-J) or -2 beta log2(e) (Gaussian), as in SmemLayout
    int mask;       // uint32 [32][NWl]         overlap masks of the ICM pairs (in the lab region)
    int lab;        // uint32 [max(ufg, 1)][nls] union-find parents: the cluster-window address of the
                    //                          parent's label word (a root holds its own address);
                    //                          growth by scans: the domain words
    // row form (undiluted 2D lattices whose CTAs hold whole row words): words of
    // this CTA's rows of a pair, the two halo rows' words, row words of a pair's
    // slot (0: word-per-site form)
    int rw, rh, rs;
    int rowm;       // uint32 [pairs of this CTA][rs]   whole pairs, every CTA's rows (written remotely, lab region)
    int rowc;       // uint32 [nT][rw + 2 rh]           clusters: own rows, the row before, the row after (written
                    //                                  remotely, C region)
    int rowi;       // uint32 [32]              per pair: moves | flipped << 1 | rounds << 2 (written remotely)
    int ufg;        // pairs per union-find group; 0 = growth by in-place scans (no labels)
    int sadr;       // uint32 [32]              cluster-window address of each pair's seed site (written remotely)
    int sroot;      // uint32 [8]               root of each group pair's seed
    int gord;       // uint16 [nls]             KParams::cl_order in shared memory, or -1 (site tid + j nth)
    int cntloc;     // int32 [K][2][32]         every CTA's q = -1 sites per colour block and pair (written remotely)
    int cntobs;     // int32 [2][K][2][32]      every CTA's observable counts, by step parity (written remotely, rank 0)
    int flags;      // uint32 [2]               growth-round stamps, by round parity (written remotely)
    int seed;       // int32 [32]               seed draws, then 1 = the pair moves
    int esum;       // float or int32 [32]
    int flipw;      // uint32 [2]
    int csz;        // int32 [32]               this CTA's cluster sites per pair (read remotely)
    int swap_x, swap_mask;                      // as in SmemLayout
    int cnt_n, cnt_d;   // int32 [32]           this CTA's counts
    int accE, acc64, nmeas;                     // observables (rank 0)
    int icmst;      // uint64 [2]               cluster moves and growth scans of this instance (rank 0)
    int total;
};
constexpr int kLeanThreads = 512;
// ufg: pairs per union-find group (1..kMaxUfGroup), or 0 for growth by scans.
constexpr int kMaxUfGroup = 8;
ClusterLayout cluster_layout(int N, int Z, int R, int G, int nT, int K, int nwarps, bool gauss, int ufg,
                             bool order, int nh, int nx, int row_kind, int L);
// Host-built tables of the layout for one lattice and K, every CTA's in turn:
// the neighbours' local indices, the positions of its halo entries (0xffff =
// unused), the first copy of each own site, the copies ((last << 31) | CTA
// << 16 | halo entry) and the halo entries' owners (CTA << 16 | local index).
struct ClusterTables {
    int nh = 0, nx = 0;
    std::vector<uint16_t> nb, hpos, xoff;   // [K][nls][Z], [K][nh], [K][nls]
    std::vector<uint32_t> xl, hown;         // [K][nx], [K][nh]
};
void cluster_tables(const uint16_t *nbr, int N, int Z, int K, ClusterTables &t);
cudaError_t launch_cluster(const KParams &P, const ClusterLayout &CL, bool gauss, int threads, int n_clusters,
                           uint32_t n_sweeps, cudaStream_t st);
cudaError_t cluster_occupancy(bool gauss, int Z, bool dil, bool lean, int K, int threads, int smem, int *clusters);
int fused_threads(int N);
int fused_threads_wide(int N);
// uint32 words of per-CTA scratch of the wide layout (the cluster words and the
// overlap-mask rows), rounded to 16 bytes.
int wide_scratch_words(int N);

// Host-callable launchers (pt_icm.cu).  Return a cudaError_t.
cudaError_t fused_occupancy(bool gauss, int Z, int layout, int threads, int smem, int *ctas_per_sm);
cudaError_t launch_fused(const KParams &P, bool gauss, int threads, int grid, uint32_t n_sweeps,
                         cudaStream_t st);
// Spins int8 [n_inst][R][N] by site <-> packed words [n_inst][G][N] by position
// (cells: chimera).  Unpacking writes 4 bytes at a time: dst is 4-byte aligned.
cudaError_t launch_pack_spins(const int8_t *src, uint32_t *dst, const uint16_t *pos2site, int n_inst,
                              int R, int G, int N, bool cells, cudaStream_t st);
cudaError_t launch_unpack_spins(const uint32_t *src, int8_t *dst, const uint16_t *pos2site, int n_inst,
                                int R, int G, int N, bool cells, cudaStream_t st);
cudaError_t launch_expand_couplings(const void *bond_J, bool gauss, const int32_t *edge_bond, int n_inst,
                                    int N, int Z, int Nb, float *Jd, uint8_t *Jb, cudaStream_t st);
// Per-instance tables of a diluted batch from the bond couplings: neighbour
// positions (absent bond -> the site itself), degree and bonds present, and
// the number of invalid couplings (not finite; +-J outside -1, 0, +1) per
// instance in bad.  nb_inst and bad must be zero on entry (the kernel adds).
cudaError_t launch_expand_dilution(const void *bond_J, bool gauss, const int32_t *edge_bond, const uint16_t *nbr,
                                   int n_inst, int N, int Z, int Nb, uint16_t *nbr_inst, uint8_t *zdeg_inst,
                                   int32_t *nb_inst, int32_t *bad, cudaStream_t st);
cudaError_t launch_init_energies(const KParams &P, bool gauss, cudaStream_t st);
// The shared group kernel: grid persistent CTAs of kTeamThreads threads with
// `smem` bytes of dynamic shared memory each.
cudaError_t launch_team(const TeamParams &TP, bool gauss, int Z, int grid, int smem, uint32_t n_sweeps,
                        cudaStream_t st);
cudaError_t team_occupancy(bool gauss, int Z, int smem, int *ctas_per_sm);
cudaError_t launch_energies_to_double(const KParams &P, bool gauss, double *out, cudaStream_t st);

}  // namespace icm
