// Internal definitions of the sm_103a NSGA-III selection library.
//
// Data layout in HBM, per population ("problem"):
//   * up to five objectives the points are ranked by a two-level tree of
//     bounding boxes: leaves of 32 points in the order of a grid's Morton cells
//     (k_order.cu), nodes of 32 leaves (k_fronts.cu). There is no dominance
//     matrix;
//   * with more objectives, and for TensorHypE's sample counts and the
//     caller-order matrix, they are put in lexicographic order of their objective
//     vectors (stable LSD radix sort).  In that order p < q implies that q cannot
//     dominate p, so the dominance matrix is strictly upper triangular;
//   * that triangle is stored as 4 KB tiles of 32 rows x 1024 columns
//     (32 rows x 32 uint32 words).  Row block rb = rows [32 rb, 32 rb + 32),
//     column block cb = columns [1024 cb, 1024 cb + 1024); tile (rb, cb)
//     exists for cb >= rb / 32.  Tiles of a row block are contiguous; inside
//     a tile, word w of row r (columns 32 w .. 32 w + 31 of the block, bit b
//     = column 32 w + b) sits at position r * 32 + w;
//   * the objective keys used by the dominance kernel are the objectives
//     2..m of each point in sorted order, array-of-structs with stride m-1,
//     padded to a multiple of 1024 points with -inf;
//   * everything downstream of the peeling works in the caller's order.
#pragma once

#include <cstddef>
#include <cstdint>

#include "../../include/emo.h"

#ifndef __CUDACC__
#define __host__
#define __device__
#define __forceinline__ inline
#endif

namespace emo {

constexpr int kMaxM = EMO_MAX_OBJECTIVES;
constexpr int kMaxBatch = EMO_MAX_BATCH;
constexpr int kTileRows = 32;         // rows per row block
constexpr int kTileWords = 32;        // words per tile row
constexpr int kColBlock = 1024;       // columns per column block
constexpr int kDomRowChunk = 1024;    // row blocks per dominance work item (largest; emo_dominance)
constexpr int kDomChunkMin = 64;      // smallest row-block chunk of a selection's dominance items
constexpr int kCoopThreads = 512;     // threads of the cooperative kernels
constexpr int kOneCtaItems = 1024;    // points and references that one CTA serves alone
constexpr int kNicheBins = 4096;      // niching select: bins of the top 12 bits of a priority
constexpr int kRadixBits = 8;
constexpr int kRadix = 1 << kRadixBits;
constexpr int64_t kMaxN2 = int64_t(1) << 21;
constexpr int32_t kNotRanked = EMO_NOT_RANKED;
// Ranking without a dominance matrix (k_fronts.cu) up to this many objectives:
// with more, bounding boxes rule out too little (100,000 points of eight
// objectives: 5.9 ms by the tree, 3.3 ms by the matrix, which has since come
// down to 0.7 ms; 40,000 of five: 0.20 and 0.26 ms). Six and seven were not
// measured by the tree; 100,000 points of six on one front take 0.49 ms by the
// matrix, of five 0.50 ms by the tree.
constexpr int kTreeMaxM = 5;
constexpr int kTreeThreads = 1024;         // threads of its peeling kernel
constexpr int kFrontLeafSmem = 64 * 1024;   // leaf states up to this size are copied to shared memory once per front

enum Mode : int32_t { MODE_RANK = 1, MODE_SELECT = 2, MODE_HYPE = 3, MODE_DOM = 4 };

// What the host knows about one problem.
struct ProbIn {
    const float* F;
    const float* R;
    int32_t* survivors;
    emo_select_info* info;
    int64_t n2;
    int64_t n_keep;     // 0 = rank everything (MODE_RANK only)
    int32_t m;
    int32_t n_r;
    uint64_t seed;
    uint64_t gen;
    int32_t mode;
    int32_t niche;           // EMO_NICHE_EXACT or EMO_NICHE_ONESHOT (MODE_SELECT)
    const float* U;          // MODE_HYPE: [n_r * m] uniform numbers of the samples (n_r = samples; R = v_ref)
    double* hv_out;          // MODE_HYPE: [n2] contributions of front l (nullable)
    int32_t* rank_out;       // MODE_RANK
    int32_t* last_rank_out;  // nullable
    emo_select_debug dbg;
    uint64_t ws_off;         // byte offset of this problem's region
    // launch shapes (tuned per device, objective count and size; survivors
    // never depend on them)
    int32_t dom_chunk;       // row blocks per dominance work item: 64 .. 1024, a power of two
    int32_t cap_wide;        // most CTAs of the peeling (and TensorHypE) group; 0 = no cap
    int32_t cap_narrow;      // most CTAs of the sort / statistics / CSR / niching / survivor groups; 0 = no cap
    int32_t ranked;          // MODE_SELECT from the given ranks rank_in (no dominance matrix, no peeling)
    const int32_t* rank_in;  // [n2] caller-order ranks (EMO_NOT_RANKED beyond the last needed front)
    uint32_t* dom_out;       // MODE_DOM: [n2][dom_ld] caller-order dominance matrix
    int32_t* dom_count;      // MODE_DOM: [n2] dominator counts (nullable)
    int64_t dom_ld;          // MODE_DOM: words per row
};

__forceinline__ __host__ __device__ bool tree_ranked(const ProbIn& in)
{
    return in.m <= kTreeMaxM && !in.ranked && in.mode != MODE_DOM;
}
// Whether the points are put in lexicographic order with prefix sets (the
// dominance matrix, and the sample counts of TensorHypE).
__forceinline__ __host__ __device__ bool lex_ordered(const ProbIn& in)
{
    return !in.ranked && (in.mode == MODE_DOM || in.mode == MODE_HYPE || !tree_ranked(in));
}

// The problem whose launch shape the peeling from the matrix takes: the largest
// of those that are ranked from it (one launch serves them all; the first of
// equal ones); -1 when there is none.
inline int matrix_lead(const ProbIn* ins, int n)
{
    int lead = -1;
    for (int p = 0; p < n; ++p)
        if (!tree_ranked(ins[p]) && (lead < 0 || ins[p].n2 > ins[lead].n2)) lead = p;
    return lead;
}

// Members found per front, in three slots taken in turn. The CTAs of a group
// add to front k's slot between two barriers and read it after the second; the
// CTA of rank 0 clears the next front's slot while front k is sought. A CTA that
// leaves a barrier early therefore never adds to, or clears, a slot that one
// still behind it has to read. (A single running total would: a late reader
// sees part of the next front in it and leaves the loop alone.)
__host__ __device__ constexpr int front_slot(int k) { return (int)((unsigned)k % 3u); }

// Per-problem scalars; zeroed by the set-up kernel.
struct Scal {
    int32_t status;
    int32_t l;
    int32_t nP, nL, nS;
    int32_t nfronts;
    int32_t fallback;
    int32_t nflag;           // points associated by an FP64 scan of more than two references
    int32_t levels;
    int32_t front_new[3];    // members of front k in slot k % 3 (see front_slot)
    int32_t idx_buf;         // idx half holding the sorted order
    int32_t lbuf;            // llist half holding the sorted candidate lists
    int32_t nbad;            // points listed for the scan of every reference
    uint32_t zkey[kMaxM];
    uint32_t kor[kMaxM];     // OR of the order-preserving keys of each objective over all points
    uint32_t kinv[kMaxM];    // OR of their complements (a bit varies iff set in both)
    uint32_t asf32[kMaxM];
    unsigned long long asf64[kMaxM];
    int32_t ext[kMaxM];
    uint32_t fkey[kMaxM];    // largest order-preserving key of each objective over S
    float z[kMaxM];
    float inv_a32[kMaxM];
    double a[kMaxM];
    unsigned int bar[3];     // barrier counters of the narrow, wide and tree groups (top bit: failed)
    int32_t ncol;            // niching: keys collected from the selected histogram bin
    int32_t nsel;            // one-shot niching: references that took their nearest candidate
    int32_t longrun;         // sort: a run of equal f_1 longer than the in-place fix-up handles
    int32_t lfinal1;         // wavefront peeling: l + 1 once known, 0 before
    unsigned long long rho_sum;  // niching from a given association: sum of the given niche counts
};

struct DirGrid;  // grid of the directions (cell_order.cuh)

// Device-side descriptor with every workspace pointer of one problem.
struct ProbDev {
    ProbIn in;
    int32_t nrb, ncb;        // row blocks (32 rows), column blocks (1024 columns)
    int64_t n2p;             // n2 padded to ncb * 1024
    int64_t ntiles;
    Scal* sc;
    uint32_t* D;             // dominance tiles
    int32_t* idx;            // [2][n2p] sorted position -> caller index (ping-pong)
    float* keys;             // [n2p][m-1] objectives 2..m in sorted order
    int32_t* runstart;       // [n2p] first sorted position of the run of equal points
    int32_t* minrs;          // [ncb] min runstart of non-leading run members
    int32_t* cnt;            // [n2p] dominator counts (sorted order)
    int32_t* rank_s;         // [n2p] ranks (sorted order)
    int32_t* rank_o;         // [n2]  ranks (caller order)
    int32_t* front;          // [3][n2p] front members grouped by column block (3 buffers); the
                             // wavefront peeling keeps each block's members in front order in the first
    int32_t* front_n;        // [3][ncb] members per column block
    int32_t* wdone;          // [ncb] wavefront: fronts whose counts block cb has applied (INT32_MAX: exhausted)
    int32_t* wmaxf;          // [ncb] wavefront: last front with offsets of an exhausted block
    int32_t* wcnt;           // [n2 + 2] wavefront: members of front k
    uint16_t* wofs;          // [ncb][n2 + 2] wavefront: start of front k in block cb's member list
    int32_t* slist;          // [n2] caller indices of S = {rank <= l}
    int32_t* pi;             // [n2] associated reference
    double* d64;             // [n2] perpendicular distance (FP64)
    float* rhat;             // [n_r][m] unit reference directions (FP32)
    // references in grid-cell order, leaves of 32, nodes of 32 leaves (k_order.cu)
    int32_t rtree;           // MODE_SELECT with references
    int32_t rbits, nrcell;   // grid bits per coordinate, cells
    int32_t nrleaf, nrnode, nrleafp, nrnodep;  // (p: rounded up to 32)
    DirGrid* rgrid;          // the references' grid
    uint32_t* rcnt;          // [2][nrcell] cell counts, then offsets: references | S
    uint32_t* rcell;         // [n_r] cell of each reference
    uint32_t* rslot;         // [n_r] its slot in the cell
    int32_t* rord;           // [n_r] sorted position -> reference
    float* rsort;            // [nrleaf * 32][m rounded up to 4] unit directions in that order
    float* rball;            // [m][nrleafp] mean direction of each leaf
    float* rrad;             // [nrleafp] largest distance of a member from it
    float* rnball;           // [m][nrnodep] the same of each node
    float* rnrad;            // [nrnodep]
    int32_t* sord;           // [n2] S in the order of the references' grid cells
    uint32_t* scell;         // [n2] cell of each entry of slist
    uint32_t* sslot;         // [n2] its slot in the cell
    int32_t* flagged;        // [n2] points for the scan of every reference in FP64
    int32_t* rho;            // [n_r] niche counts of P (evolving during niching)
    int32_t* lcnt;           // [n_r] last-front members per reference (evolving)
    int32_t* loff;           // [n_r + 1] CSR offsets of the candidate lists
    int32_t* llist;          // [2][n2] last-front members (CSR order after sorting)
    int32_t* fen;            // [n2] Fenwick trees over each candidate list
    unsigned long long* ekeys;  // [max(n_r, n2)] niching keys collected from one histogram bin
    int32_t* nhist;          // niching: [kNicheBins] key histogram | [G] packed per-CTA (min, count)
    int32_t* elist;          // [n_r] references served in a level
    int32_t* flag;           // [n2] survivor flags / scan scratch
    int32_t* hist;           // [G][256] radix histograms, reused by the scans
    unsigned char* colpre;   // [ncb][K] column-block prefix sets (colprep_obj_bytes each; K = m - 1 key
                             // objectives, or all m of the caller-order columns in MODE_DOM)
    float* ckeys;            // MODE_DOM: [n2p][m] objectives in caller order (padding -inf)
    // ranking by the z-order tree (tree_ranked): points in grid-cell order,
    // leaves of 32 points, nodes of 32 leaves, state of even and odd fronts
    int32_t tree;
    int32_t zbits, ncell;    // grid bits per objective, cells
    int32_t nleaf, nnode, nleafp, nnodep;  // (p: rounded up to 32)
    uint32_t* zcell;         // [n2] cell of each point (caller order)
    uint32_t* zslot;         // [n2] its slot in the cell
    uint32_t* zcnt;          // [ncell] cell counts, then offsets
    float* zpts;             // [m][nleaf * 32] objectives in cell order
    int32_t* zidx;           // [nleaf * 32] caller index
    uint32_t* zkey;          // [nleaf * 32] cell
    int32_t* zwit;           // [nleaf * 32] witness: an unranked dominator (-1: none known)
    uint32_t* zlocal;        // [4 (nleafp + G)] bookkeeping of the leaves of large CTA shares
    float* zstate;           // [2] minima of the nodes [m][nnodep] and of the leaves [m][nleafp] (unranked
                             // points), and the leaves' masks of unranked points [nleafp]
    int32_t* spos;           // MODE_DOM: [2][n2] run of identical points of each caller index: first
                             // sorted position (-1 when alone), one past the last
};

// A population split over several GPUs (one problem per call, ranks given):
// the association of one GPU's points, or the niching from the association
// gathered from all of them.
enum SplitKind : int32_t { SPLIT_NONE = 0, SPLIT_ASSOC = 1, SPLIT_NICHE = 2 };
struct SplitArgs {
    int32_t kind;
    int32_t pad_;
    int64_t col_lo, col_hi;  // SPLIT_ASSOC: the caller indices associated
    int32_t* pi_out;         // SPLIT_ASSOC: [col_hi - col_lo] reference, -1 outside S
    double* d_out;           // SPLIT_ASSOC: [col_hi - col_lo] FP64 distance, NaN outside S
    int32_t* rho;            // SPLIT_ASSOC: output [n_r] niche counts of P in the range;
                             // SPLIT_NICHE: input [n_r] niche counts of all of P
    const int32_t* last;     // SPLIT_NICHE: [n_last] front l, ascending caller indices
    const int32_t* last_pi;  // SPLIT_NICHE: [n_last] their references
    const double* last_d;    // SPLIT_NICHE: [n_last] their FP64 distances
    int64_t n_last;
};

struct Plan {
    int32_t nprob;
    int32_t G;               // CTAs of every cooperative launch
    long long spin_budget;   // cycles a bounded wait may spin
    int32_t grp_first[kMaxBatch + 1];     // cooperative CTA groups of the peeling and TensorHypE kernels
    int32_t grpn_first[kMaxBatch + 1];    // groups of the other cooperative kernels
    int32_t grpt_first[kMaxBatch + 1];    // groups of the peeling by the z-order tree
    long long dom_item_start[kMaxBatch + 1];
    long long dom_items;
    unsigned long long dom_ctr[kMaxM + 1];  // dynamic work counters per objective count
    unsigned long long asc_next[kMaxM + 1];  // tile counters of the all-reference association, per m
    int32_t status;                       // OR of problem statuses
    int32_t pad_;
    SplitArgs split;                      // problem 0 of a one-problem call
    ProbDev p[kMaxBatch];
};

struct SetupArgs {
    int32_t nprob;
    int32_t G;
    long long spin_budget;
    ProbIn in[kMaxBatch];
};

__host__ __device__ __forceinline__ int64_t align_up(int64_t x, int64_t a) { return (x + a - 1) / a * a; }
__host__ __device__ __forceinline__ int64_t cdiv(int64_t a, int64_t b) { return (a + b - 1) / b; }

// Number of stored tiles before row block rb (tiles of row block b are the
// column blocks cb in [b / 32, ncb)).
__host__ __device__ __forceinline__ int64_t tiles_before(int64_t rb, int64_t ncb)
{
    int64_t s = rb / 32, t = rb % 32;
    return rb * ncb - 32 * (s * (s - 1) / 2) - t * s;
}
__host__ __device__ __forceinline__ int64_t tile_index(int64_t rb, int64_t cb, int64_t ncb)
{
    return tiles_before(rb, ncb) + (cb - rb / 32);
}

// Column-block prefix sets of the dominance kernels. The columns q of a
// 1024-column block with f_k(q) >= x are a prefix of the block in the order of
// f_k descending; the sets are stored so that each part of the block looks its
// own prefix up. Per key objective k:
//   fv   -- the block's 1024 values of f_k sorted descending (entry i at
//           slot i ^ ((i / 32) % 32), which spreads a binary search's
//           candidates over the shared-memory banks);
//   cum  -- how many of the first j entries of fv lie in each part of the
//           block, j = 0..1024;
//   pb   -- row c holds, for every part, the bitset of its first c columns in
//           that order (word w of a row is word w of a tile row);
//   ord  -- (halves only) each half's local column indices in that order.
// Up to kSegKeys keys: eight segments of 128 columns, every prefix stored:
//   float fv[1024] | uint8 cum[1025][8] (+pad) | uint32 pb[129][32]
// More keys (the segments' rows would not fit in shared memory): two halves of
// 512 columns, every cps-th prefix stored, the rest completed from ord:
//   float fv[1024] | uint16 cum0[1025] (+pad) | uint32 pb[512/cps + 1][32] | uint16 ord[2][512]
constexpr int kSegKeys = 7;
constexpr int kSegCols = 128, kSegs = kColBlock / kSegCols;
constexpr int kPrefCumOff = kColBlock * 4;
constexpr int kSegPbOff = kPrefCumOff + 8320;   // 1025 x 8 bytes rounded up to 128
constexpr int kPrefPbOff = kPrefCumOff + 2176;  // 1025 uint16 rounded up to 128 bytes
constexpr int kSegObjBytes = kSegPbOff + (kSegCols + 1) * 128;
__host__ __device__ constexpr int colprep_log_cps(int K) { return K <= 9 ? 3 : 4; }
__host__ __device__ constexpr int64_t colprep_ord_off(int K)
{
    return kPrefPbOff + (((kColBlock / 2) >> colprep_log_cps(K)) + 1) * 32 * 4;
}
__host__ __device__ constexpr int64_t colprep_obj_bytes(int K)
{
    return K <= kSegKeys ? (int64_t)kSegObjBytes : colprep_ord_off(K) + kColBlock * 2;
}

// Bits per coordinate of a z-order grid over n items: about two cells per
// item, at most 2^18 cells (1 MB of counters) and 256 lines per coordinate.
__host__ __device__ __forceinline__ int z_bits(int64_t n2, int m)
{
    int b = 1;
    while ((int64_t(1) << b) < n2) ++b;
    b = (b + 1 < 18 ? b + 1 : 18) / m;
    return b < 1 ? 1 : (b > 8 ? 8 : b);
}
// Bits per coordinate of the directions' grid: about four cells per reference,
// at most 2^18.
__host__ __device__ __forceinline__ int dir_bits(int64_t nr, int dims)
{
    int b = 1;
    while ((int64_t(1) << b) < nr) ++b;
    b = (b + 2 < 18 ? b + 2 : 18) / dims;
    return b < 1 ? 1 : b;
}
__host__ __device__ constexpr int64_t fronts_leaf_bytes(int64_t nleaf, int m) { return (nleaf + 31) / 32 * 32 * (m + 1) * 4; }
// Leaves of one CTA that k_fronts keeps in its shared memory (witnesses and
// objectives of 32 points each: 256 leaves of three objectives take 132 KB).
__host__ __device__ constexpr int front_local(int m) { return m <= 3 ? 256 : 128; }
// Dynamic shared memory of k_fronts for one problem: the nodes' state, the
// leaves' when it is small, and the CTA's own leaves (witness, objectives and
// four words of bookkeeping).
__host__ __device__ __forceinline__ int fronts_smem_bytes(int64_t n2, int m)
{
    const int64_t nleaf = cdiv(n2, 32), nnode = cdiv(nleaf, 32), lb = fronts_leaf_bytes(nleaf, m);
    return (int)((nnode + 31) / 32 * 32 * m * 4 + (lb <= kFrontLeafSmem ? lb : 0) +
                 (nleaf < front_local(m) ? nleaf : front_local(m)) * (4 + 32 * (m + 1)) * 4);
}

// Built-in scratch of the allocation-free selection (emo_noalloc.cu). A
// selection that fitted into 9 MiB while the references were ordered by angle
// and the prefix sets stored by halves needs up to 11.74 MiB now (the cells of
// the references' tree, 2 MB from 65,536 references on, and the sets of seven
// and eight keys).
constexpr size_t kNoallocBytes = size_t(12) << 20;

// CTA groups of the cooperative kernels: wide (peeling from the matrix,
// TensorHypE), tree (peeling by the z-order tree), narrow (the others).
enum GroupKind : int { GRP_NARROW = 0, GRP_WIDE = 1, GRP_TREE = 2 };
// Most CTAs that a problem's group gets out of G: its launch shapes' caps, and
// no more than it can use. A barrier of two CTAs costs as much as one of 152
// (1.1 us), none inside a single CTA, so small problems get one CTA: a
// selection of 500 points on 250 directions takes 199 us so and 207 with the
// narrow kernels on two CTAs; 16 leaves per CTA of the tree (ranking 600
// points, 19 leaves: 126 us by one CTA, 109 by two; 1,000 points 162 and 129).
__host__ __device__ __forceinline__ int group_cap(GroupKind kind, const ProbIn& in, int G)
{
    int64_t c = in.cap_wide > 0 && in.cap_wide < G ? in.cap_wide : G;
    if (kind == GRP_NARROW) {
        if (in.cap_narrow > 0 && in.cap_narrow < c) c = in.cap_narrow;
        const int64_t items = in.n2 + (in.mode == MODE_SELECT ? in.n_r : 0);
        const int64_t use = items <= kOneCtaItems ? 1 : cdiv(items, kCoopThreads);
        if (use < c) c = use;
    } else if (kind == GRP_TREE) {
        const int64_t nleaf = cdiv(in.n2, 32);
        const int64_t use = cdiv(nleaf, kTreeThreads / 64);
        if (use < c) c = use;
    }
    return (int)c;
}

// Byte layout of one problem region; fills `d` when base != 0. Returns the
// region size. The same function sizes the workspace on the host and carves
// it on the device.
__host__ __device__ inline int64_t layout_problem(const ProbIn& in, int G, char* base, ProbDev* d)
{
    const int64_t n2 = in.n2, m = in.m, nr = (in.mode == MODE_SELECT || in.mode == MODE_HYPE) ? in.n_r : 1;
    const int64_t nrb = cdiv(n2, 32), ncb = cdiv(n2, kColBlock), n2p = ncb * kColBlock;
    const bool tree = tree_ranked(in), lex = lex_ordered(in);
    // (the tiles' space stays in the size that callers reserve, about n2^2 / 16
    // bytes, also where the ranks come from the tree and nothing touches it: a
    // selection's workspace is stated, and tested, to be more than ten times that
    // of one from given ranks)
    const int64_t ntiles = tiles_before(nrb, ncb);
    int64_t off = 0;
    auto take = [&](int64_t bytes) { int64_t o = off; off = align_up(off + bytes, 256); return o; };
    int64_t o_sc = take(sizeof(Scal));
    int64_t o_idx = take(lex ? 2 * n2p * 4 : 0);
    int64_t o_keys = take(lex ? n2p * (m - 1) * 4 : 0);
    int64_t o_runstart = take(lex ? n2p * 4 : 0);
    int64_t o_minrs = take(lex ? ncb * 4 : 0);
    int64_t o_cnt = take(tree ? 0 : n2p * 4);
    int64_t o_rank_s = take(n2p * 4);
    int64_t o_rank_o = take(n2 * 4);
    int64_t o_front = take(tree ? 0 : 3 * n2p * 4);
    int64_t o_front_n = take(tree ? 0 : 3 * ncb * 4);
    int64_t o_wdone = take(tree ? 0 : 2 * ncb * 4);
    int64_t o_wcnt = take(tree ? 0 : (n2 + 2) * 4);
    int64_t o_wofs = (in.ranked || in.mode == MODE_DOM || tree) ? 0 : take(ncb * (n2 + 2) * 2);
    int64_t o_slist = take(n2 * 4);
    int64_t o_hist = take(int64_t(G) * kRadix * 4);
    int64_t o_flag = take((n2p + 1) * 4);
    int64_t o_pi = 0, o_d64 = 0, o_rhat = 0, o_flagged = 0, o_rho = 0, o_lcnt = 0, o_loff = 0,
            o_llist = 0, o_fen = 0, o_ekeys = 0, o_elist = 0, o_rord = 0, o_rsort = 0, o_nhist = 0, o_rgrid = 0,
            o_rcnt = 0, o_rcell = 0, o_rslot = 0, o_rball = 0, o_rrad = 0, o_rnball = 0, o_rnrad = 0, o_sord = 0,
            o_scell = 0, o_sslot = 0;
    const int64_t nrleaf = cdiv(nr, 32), nrnode = cdiv(nrleaf, 32), nrleafp = align_up(nrleaf, 32),
                  nrnodep = align_up(nrnode, 32), rdims = m <= 3 ? m - 1 : m, rbits = dir_bits(nr, (int)rdims),
                  nrcell = int64_t(1) << (rbits * rdims);
    if (in.mode == MODE_SELECT) {
        o_pi = take(n2 * 4);
        o_d64 = take(n2 * 8);
        o_rhat = take(nr * m * 4);
        o_flagged = take(n2 * 4);
        o_rho = take(nr * 4);
        o_lcnt = take(nr * 4);
        o_loff = take((nr + 1) * 4);
        o_llist = take(2 * n2 * 4);
        o_fen = take(n2 * 4);
        o_ekeys = take((nr > n2 ? nr : n2) * 8);
        o_elist = take(nr * 4);
        o_rord = take(nr * 4);
        o_rsort = take(nrleaf * 32 * align_up(m, 4) * 4);
        o_rgrid = take(2 * kMaxM * 4);
        o_rcnt = take(2 * nrcell * 4);
        o_rcell = take(nr * 4);
        o_rslot = take(nr * 4);
        o_rball = take(m * nrleafp * 4);
        o_rrad = take(nrleafp * 4);
        o_rnball = take(m * nrnodep * 4);
        o_rnrad = take(nrnodep * 4);
        o_sord = take(n2 * 4);
        o_scell = take(n2 * 4);
        o_sslot = take(n2 * 4);
        o_nhist = take(kNicheBins * 4 + int64_t(G) * 8);
    } else if (in.mode == MODE_HYPE) {
        // d64: contributions; rhat: samples; rho: their dominator counts;
        // llist: the last front and its sorted copy; ekeys: the weights alpha_c
        o_d64 = take(n2 * 8);
        o_rhat = take(nr * m * 4);
        o_rho = take(nr * 4);
        o_llist = take(2 * n2 * 4);
        o_ekeys = take((n2 + 1) * 8);
    }
    // the prefix sets, the dominance tiles and the wavefront offsets are not
    // needed when the ranks are given
    const int64_t kobj = in.mode == MODE_DOM ? m : m - 1;  // objectives with prefix sets
    int64_t o_colpre = lex ? take(ncb * kobj * colprep_obj_bytes((int)kobj)) : 0;
    int64_t o_D = (in.ranked || in.mode == MODE_DOM) ? 0 : take(ntiles * 4096);
    // the z-order tree
    const int64_t nleaf = cdiv(n2, 32), nnode = cdiv(nleaf, 32), nleafp = align_up(nleaf, 32), nnodep = align_up(nnode, 32);
    const int64_t zb = z_bits(n2, (int)m), ncell = int64_t(1) << (zb * m), zs = nleaf * 32;
    int64_t o_zcell = 0, o_zslot = 0, o_zcnt = 0, o_zpts = 0, o_zidx = 0, o_zkey = 0, o_zwit = 0, o_zlocal = 0,
            o_zstate = 0;
    if (tree) {
        o_zcell = take(n2 * 4);
        o_zslot = take(n2 * 4);
        o_zcnt = take(ncell * 4);
        o_zpts = take(m * zs * 4);
        o_zidx = take(zs * 4);
        o_zkey = take(zs * 4);
        o_zwit = take(zs * 4);
        o_zlocal = take(4 * (nleafp + G) * 4);
        o_zstate = take(2 * (m * nnodep + (m + 1) * nleafp) * 4);
    }
    int64_t o_ckeys = in.mode == MODE_DOM ? take(n2p * m * 4) : 0;
    int64_t o_spos = in.mode == MODE_DOM ? take(2 * n2 * 4) : 0;
    if (base && d) {
        d->in = in;
        d->nrb = (int32_t)nrb;
        d->ncb = (int32_t)ncb;
        d->n2p = n2p;
        d->ntiles = ntiles;
        d->sc = (Scal*)(base + o_sc);
        d->idx = (int32_t*)(base + o_idx);
        d->keys = (float*)(base + o_keys);
        d->runstart = (int32_t*)(base + o_runstart);
        d->minrs = (int32_t*)(base + o_minrs);
        d->cnt = (int32_t*)(base + o_cnt);
        d->rank_s = (int32_t*)(base + o_rank_s);
        d->rank_o = (int32_t*)(base + o_rank_o);
        d->front = (int32_t*)(base + o_front);
        d->front_n = (int32_t*)(base + o_front_n);
        d->wdone = (int32_t*)(base + o_wdone);
        d->wmaxf = d->wdone + ncb;
        d->wcnt = (int32_t*)(base + o_wcnt);
        d->wofs = (in.ranked || in.mode == MODE_DOM || tree) ? nullptr : (uint16_t*)(base + o_wofs);
        d->slist = (int32_t*)(base + o_slist);
        d->hist = (int32_t*)(base + o_hist);
        d->flag = (int32_t*)(base + o_flag);
        d->pi = in.mode == MODE_SELECT ? (int32_t*)(base + o_pi) : nullptr;
        d->d64 = (in.mode == MODE_SELECT || in.mode == MODE_HYPE) ? (double*)(base + o_d64) : nullptr;
        d->rhat = (in.mode == MODE_SELECT || in.mode == MODE_HYPE) ? (float*)(base + o_rhat) : nullptr;
        d->flagged = in.mode == MODE_SELECT ? (int32_t*)(base + o_flagged) : nullptr;
        d->rho = (in.mode == MODE_SELECT || in.mode == MODE_HYPE) ? (int32_t*)(base + o_rho) : nullptr;
        d->lcnt = in.mode == MODE_SELECT ? (int32_t*)(base + o_lcnt) : nullptr;
        d->loff = in.mode == MODE_SELECT ? (int32_t*)(base + o_loff) : nullptr;
        d->llist = (in.mode == MODE_SELECT || in.mode == MODE_HYPE) ? (int32_t*)(base + o_llist) : nullptr;
        d->fen = in.mode == MODE_SELECT ? (int32_t*)(base + o_fen) : nullptr;
        d->ekeys = (in.mode == MODE_SELECT || in.mode == MODE_HYPE) ? (unsigned long long*)(base + o_ekeys) : nullptr;
        d->elist = in.mode == MODE_SELECT ? (int32_t*)(base + o_elist) : nullptr;
        d->nhist = in.mode == MODE_SELECT ? (int32_t*)(base + o_nhist) : nullptr;
        d->rord = in.mode == MODE_SELECT ? (int32_t*)(base + o_rord) : nullptr;
        d->rsort = in.mode == MODE_SELECT ? (float*)(base + o_rsort) : nullptr;
        const bool rt = in.mode == MODE_SELECT;
        d->rtree = rt && in.R;
        d->rbits = (int32_t)rbits;
        d->nrcell = rt ? (int32_t)nrcell : 0;
        d->nrleaf = (int32_t)nrleaf;
        d->nrnode = (int32_t)nrnode;
        d->nrleafp = (int32_t)nrleafp;
        d->nrnodep = (int32_t)nrnodep;
        d->rgrid = rt ? (DirGrid*)(base + o_rgrid) : nullptr;
        d->rcnt = rt ? (uint32_t*)(base + o_rcnt) : nullptr;
        d->rcell = rt ? (uint32_t*)(base + o_rcell) : nullptr;
        d->rslot = rt ? (uint32_t*)(base + o_rslot) : nullptr;
        d->rball = rt ? (float*)(base + o_rball) : nullptr;
        d->rrad = rt ? (float*)(base + o_rrad) : nullptr;
        d->rnball = rt ? (float*)(base + o_rnball) : nullptr;
        d->rnrad = rt ? (float*)(base + o_rnrad) : nullptr;
        d->sord = rt ? (int32_t*)(base + o_sord) : nullptr;
        d->scell = rt ? (uint32_t*)(base + o_scell) : nullptr;
        d->sslot = rt ? (uint32_t*)(base + o_sslot) : nullptr;
        d->colpre = lex ? (unsigned char*)(base + o_colpre) : nullptr;
        d->D = (in.ranked || in.mode == MODE_DOM) ? nullptr : (uint32_t*)(base + o_D);
        d->tree = tree;
        d->zbits = (int32_t)zb;
        d->ncell = tree ? (int32_t)ncell : 0;
        d->nleaf = (int32_t)nleaf;
        d->nnode = (int32_t)nnode;
        d->nleafp = (int32_t)nleafp;
        d->nnodep = (int32_t)nnodep;
        d->zcell = tree ? (uint32_t*)(base + o_zcell) : nullptr;
        d->zslot = tree ? (uint32_t*)(base + o_zslot) : nullptr;
        d->zcnt = tree ? (uint32_t*)(base + o_zcnt) : nullptr;
        d->zpts = tree ? (float*)(base + o_zpts) : nullptr;
        d->zidx = tree ? (int32_t*)(base + o_zidx) : nullptr;
        d->zkey = tree ? (uint32_t*)(base + o_zkey) : nullptr;
        d->zwit = tree ? (int32_t*)(base + o_zwit) : nullptr;
        d->zlocal = tree ? (uint32_t*)(base + o_zlocal) : nullptr;
        d->zstate = tree ? (float*)(base + o_zstate) : nullptr;
        d->ckeys = in.mode == MODE_DOM ? (float*)(base + o_ckeys) : nullptr;
        d->spos = in.mode == MODE_DOM ? (int32_t*)(base + o_spos) : nullptr;
    }
    return off;
}

// Dominance work items of one problem: column block cb covers row blocks
// [0, min(nrb, 32 (cb + 1))), split into chunks of `chunk` row blocks (a
// power of two from kDomChunkMin to kDomRowChunk).
__host__ __device__ __forceinline__ int64_t dom_items_of_cb(int64_t cb, int64_t nrb, int64_t chunk)
{
    int64_t rbs = nrb < 32 * (cb + 1) ? nrb : 32 * (cb + 1);
    return cdiv(rbs, chunk);
}
// Items of column blocks 0 .. c-1 in closed form: with B = chunk / 32
// column blocks' worth of row blocks per item, block cb < nrb / 32 has
// cb / B + 1 items (its 32 (cb + 1) row blocks in chunks of `chunk`),
// every later block has cdiv(nrb, chunk).
static_assert(kDomChunkMin % 64 == 0 && kDomRowChunk % 64 == 0, "dom_items_prefix assumes an even B");
__host__ __device__ __forceinline__ int64_t dom_items_prefix(int64_t c, int64_t nrb, int64_t chunk)
{
    const int64_t B = chunk / 32;
    const int64_t A = nrb / 32, a = c < A ? c : A, q = a / B, r = a % B;
    return (q + 1) * (B / 2 * q + r) + (c > A ? (c - A) * cdiv(nrb, chunk) : 0);
}
__host__ __device__ inline int64_t dom_items_of(int64_t n2, int64_t chunk)
{
    return dom_items_prefix(cdiv(n2, kColBlock), cdiv(n2, 32), chunk);
}
__host__ __device__ inline bool dom_chunk_ok(int64_t chunk)
{
    return chunk >= kDomChunkMin && chunk <= kDomRowChunk && (chunk & (chunk - 1)) == 0;
}


}  // namespace emo

#ifdef __CUDACC__
namespace emo {

// ------------------------------------------------------------------ basics
__device__ __forceinline__ unsigned lane_id() { return threadIdx.x & 31u; }
__device__ __forceinline__ unsigned lanemask_lt()
{
    unsigned r;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(r));
    return r;
}

// Order-preserving map float -> uint32 with -0 == +0 (finite inputs).
__device__ __forceinline__ uint32_t float_key(float f)
{
    uint32_t u = __float_as_uint(f + 0.0f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float key_float(uint32_t k)
{
    uint32_t u = (k & 0x80000000u) ? (k & 0x7FFFFFFFu) : ~k;
    return __uint_as_float(u);
}

__device__ __forceinline__ unsigned ld_acquire(const unsigned* p)
{
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_release(unsigned* p, unsigned v)
{
    asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ unsigned atom_add_acq_rel(unsigned* p, unsigned v)
{
    unsigned old;
    asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], %2;" : "=r"(old) : "l"(p), "r"(v) : "memory");
    return old;
}
__device__ __forceinline__ int ld_volatile(const int* p) { return *(volatile const int*)p; }

// The first failure of a problem: its status word, and the top bit of its
// barrier counters, where the next barrier of every CTA sees it.
constexpr unsigned kBarFailed = 0x80000000u;
__device__ __forceinline__ void set_status(Scal* sc, int code)
{
    atomicCAS(&sc->status, 0, code);
    for (unsigned& b : sc->bar) atomicOr(&b, kBarFailed);
}

// Group of CTAs serving one problem inside a cooperative launch.
struct Group {
    int prob;
    int rank;       // CTA rank inside the group
    int size;       // CTAs in the group
    unsigned* bar;  // the group's barrier counter (all kernels of one assignment use the same size)
};
// The group of this CTA in one of the assignments; prob = -1 for a CTA that
// serves no problem (groups are capped by the problems' sizes and launch
// shapes), which returns at once.
__device__ __forceinline__ Group group_of(const Plan* plan, GroupKind kind)
{
    const int32_t* first = kind == GRP_WIDE ? plan->grp_first : (kind == GRP_TREE ? plan->grpt_first : plan->grpn_first);
    Group g;
    int b = blockIdx.x, p = 0;
    while (p + 1 < plan->nprob && first[p + 1] <= b) ++p;
    g.prob = b < first[plan->nprob] ? p : -1;
    g.rank = b - first[p];
    g.size = first[p + 1] - first[p];
    g.bar = &plan->p[p].sc->bar[kind];
    return g;
}

// Barrier over the CTAs of one group with a bounded spin. Returns false (in
// every thread of the CTA) when the problem has failed or the wait ran out.
// The counter only grows: an arrival adds one and waits until the count
// reaches the next multiple of the group's size, so there is no reset and no
// second word to publish, and a failure arrives in the same word. One
// barrier is one atomic plus the poll that sees the last arrival (the
// former generation barrier took an extra read, an exchange, a fence and a
// back-off: ranking 20,001 points in 46 fronts 513 -> 462 us, a selection of
// 184 points with every group at 152 CTAs 332 -> 289 us).
__device__ inline bool group_sync(const Group& g, Scal* sc, long long budget)
{
    __shared__ int s_ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        int ok = 1;
        if (g.size > 1) {
            const unsigned n = (unsigned)g.size;
            unsigned v = atom_add_acq_rel(g.bar, 1u);
            const unsigned old = v & ~kBarFailed, goal = old - old % n + n;
            if (old + 1u != goal) {
                const long long t0 = clock64();
                do {
                    v = ld_acquire(g.bar);
                    if (clock64() - t0 > budget) {
                        set_status(sc, EMO_ERR_TIMEOUT);
                        v |= kBarFailed;
                    }
                } while (!(v & kBarFailed) && (int)(v - goal) < 0);
            }
            ok = !(v & kBarFailed);
        } else {
            __threadfence();
            ok = !(ld_acquire(g.bar) & kBarFailed);
        }
        s_ok = ok;
    }
    __syncthreads();
    return s_ok != 0;
}

// ------------------------------------------------------------ Philox-4x32-10
// Salmon et al., SC'11: ten rounds of two 32x32->64 multiplies with a Weyl
// key schedule. Written from the published definition.
__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint2 k)
{
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        uint32_t hi0 = __umulhi(0xD2511F53u, c.x), lo0 = 0xD2511F53u * c.x;
        uint32_t hi1 = __umulhi(0xCD9E8D57u, c.z), lo1 = 0xCD9E8D57u * c.z;
        uint4 n;
        n.x = hi1 ^ c.y ^ k.x;
        n.y = lo1;
        n.z = hi0 ^ c.w ^ k.y;
        n.w = lo0;
        c = n;
        k.x += 0x9E3779B9u;
        k.y += 0xBB67AE85u;
    }
    return c;
}
// Niching stream: key = seed, counter = (j, 2 c + tag, generation).
__device__ __forceinline__ uint32_t niche_random(uint64_t seed, uint64_t gen, uint32_t j, uint32_t c, uint32_t tag)
{
    uint4 ctr = make_uint4(j, 2u * c + tag, (uint32_t)gen, (uint32_t)(gen >> 32));
    uint2 key = make_uint2((uint32_t)seed, (uint32_t)(seed >> 32));
    return philox4x32_10(ctr, key).x;
}

// ------------------------------------------------------------ block scans
template <int NT>
__device__ __forceinline__ int block_exclusive_scan(int v, int* s_warp, int& total)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) s_warp[warp] = x;
    __syncthreads();
    if (warp == 0) {
        int w = lane < NT / 32 ? s_warp[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            int y = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += y;
        }
        s_warp[lane] = w;
    }
    __syncthreads();
    int prefix = (warp > 0 ? s_warp[warp - 1] : 0) + x - v;
    total = s_warp[NT / 32 - 1];
    __syncthreads();
    return prefix;
}

template <int NT>
__device__ __forceinline__ int block_reduce_min(int v, int* s_warp)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = min(v, __shfl_xor_sync(0xffffffffu, v, o));
    if (lane == 0) s_warp[warp] = v;
    __syncthreads();
    if (warp == 0) {
        int w = lane < NT / 32 ? s_warp[lane] : INT32_MAX;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) w = min(w, __shfl_xor_sync(0xffffffffu, w, o));
        if (lane == 0) s_warp[32] = w;
    }
    __syncthreads();
    int r = s_warp[32];
    __syncthreads();
    return r;
}

template <int NT>
__device__ __forceinline__ int block_reduce_sum(int v, int* s_warp)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) s_warp[warp] = v;
    __syncthreads();
    if (warp == 0) {
        int w = lane < NT / 32 ? s_warp[lane] : 0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) w += __shfl_xor_sync(0xffffffffu, w, o);
        if (lane == 0) s_warp[32] = w;
    }
    __syncthreads();
    int r = s_warp[32];
    __syncthreads();
    return r;
}

// ------------------------------------------- group-wide stable compaction
// Writes the positions i in [0, n) with pred(i) true, in ascending order, to
// out[0..count). Every CTA of the group calls it; returns count. Uses
// d.hist[0..G) as scratch; needs group_sync in between (two barriers).
template <typename Pred, typename Emit>
__device__ inline int group_compact(const ProbDev& d, const Group& g, long long budget, int64_t n, Pred pred,
                                    Emit emit, bool& ok)
{
    __shared__ int s_warp[33];
    const int64_t chunk = cdiv(n, g.size);
    const int64_t lo = min(n, chunk * g.rank), hi = min(n, lo + chunk);
    int local = 0;
    for (int64_t i = lo + threadIdx.x; i < hi; i += blockDim.x) local += pred(i) ? 1 : 0;
    local = block_reduce_sum<kCoopThreads>(local, s_warp);
    if (threadIdx.x == 0) d.hist[g.rank] = local;
    ok = group_sync(g, d.sc, budget);
    if (!ok) return 0;
    int base = 0, total = 0;
    for (int c = threadIdx.x; c < g.size; c += blockDim.x) {
        int v = ld_volatile(&d.hist[c]);
        if (c < g.rank) base += v;
        total += v;
    }
    base = block_reduce_sum<kCoopThreads>(base, s_warp);
    total = block_reduce_sum<kCoopThreads>(total, s_warp);
    for (int64_t i0 = lo; i0 < hi; i0 += blockDim.x) {
        int64_t i = i0 + threadIdx.x;
        int f = (i < hi && pred(i)) ? 1 : 0;
        int tot;
        int pos = block_exclusive_scan<kCoopThreads>(f, s_warp, tot);
        if (f) emit(base + pos, i);
        base += tot;
    }
    ok = group_sync(g, d.sc, budget);
    return total;
}

}  // namespace emo
#endif
