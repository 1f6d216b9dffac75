// Pareto-dominance matrix kernels (Section III-C, Listing 1; Section IV-A;
// Algorithm S.3 first two lines).
//
// Selection path (points in lexicographic order, so for p < q only "p
// dominates q" is possible; it holds iff f_k(q) >= f_k(p) for every key
// objective k = 2..m and the points are not identical):
//   k_colprep -- for each 1024-column block and each key objective k, the
//     columns by f_k (descending): the set {q : f_k(q) >= f_k(p)} is then a
//     prefix of that order. Up to seven keys every prefix of every 128-column
//     segment is stored as a bitset.
//   k_dom_pref<M> (m = 6..8; k_dom_pref_rt for m >= 9; up to five objectives
//     are ranked without the matrix, k_fronts.cu) -- one warp per row
//     block: each lane first counts, for its row and each objective, the
//     columns of the block that are >= (binary search). Then each half-warp
//     builds one row at a time (lanes 0-15 rows 0-15, lanes 16-31 rows 16-31),
//     a lane owning 64 columns (two words): the words are the AND over the
//     objectives of the prefix bitsets, masked by q > p (diagonal blocks) and
//     by the runs of identical points. One 64-bit store per lane writes two
//     rows' 128-byte segments per warp instruction; the dominator count of
//     every column (column sums of D) is accumulated by Harley-Seal
//     bit-sliced counters per lane.
// emo_dominance (caller order, full matrix): k_dom_full compares every
//   ordered pair directly ("all <= and some <").
#include "emo_kernels.cuh"

namespace emo {

constexpr int kDomNH = 7;  // high count planes: up to 2047 rows per lane and item
static_assert(kDomRowChunk / 16 * 16 < (1 << (4 + kDomNH)), "column counter overflow");
constexpr long long kCopyWaitCycles = 1ll << 32;
constexpr int kHalf = kColBlock / 2;

// Geometry of the per-objective prefix-set blocks of halves (more than
// kSegKeys keys).
struct PrefGeom {
    int log_cps, cps, obj_bytes, ord_off;
    __device__ __forceinline__ explicit PrefGeom(int K)
        : log_cps(colprep_log_cps(K)), cps(1 << colprep_log_cps(K)), obj_bytes((int)colprep_obj_bytes(K)),
          ord_off((int)colprep_ord_off(K))
    {
    }
};

// Decode a dominance item of one problem: column blocks are served from the
// last (tallest) to the first; each is split into chunks of `rows` row
// blocks (the problem's dom_chunk). Binary search over the closed-form item
// prefix.
__device__ __forceinline__ void dom_decode(long long local, int ncb, int nrb, int rows, int& cb, int& chunk)
{
    const long long u = dom_items_prefix(ncb, nrb, rows) - local;  // in 1 .. total
    int lo = 1, hi = ncb;                                           // smallest c with prefix(c) >= u
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (dom_items_prefix(mid, nrb, rows) >= u) hi = mid;
        else lo = mid + 1;
    }
    cb = lo - 1;
    chunk = (int)(dom_items_prefix(lo, nrb, rows) - u);
}

// Flush a warp's per-lane column counters into s_cnt (column q of the block
// at index (q % 32) * 32 + q / 32, conflict free for the warp): lane l and
// lane l + 16 both count columns 64 (l % 16) .. + 63 over their own rows.
template <int NH>
__device__ __forceinline__ void flush_counts(VCount<NH>& vlo, VCount<NH>& vhi, int32_t* s_cnt, int lane)
{
    const int top = max(vlo.top_plane(), vhi.top_plane());  // planes above are zero in every lane
    if (top >= 0) {
        const int w = 2 * (lane & 15) + (lane >> 4);  // word whose columns this lane flushes
#pragma unroll 2
        for (int b = 0; b < 32; ++b) {
            int c = vlo.count_upto(b, top);
            c += __shfl_down_sync(0xffffffffu, c, 16);
            int e = vhi.count_upto(b, top);
            e += __shfl_up_sync(0xffffffffu, e, 16);
            const int v = lane < 16 ? c : e;
            if (v) atomicAdd(&s_cnt[b * 32 + w], v);
        }
    }
    vlo = VCount<NH>();
    vhi = VCount<NH>();
}

// ------------------------------------------------------------ k_colprep
// Slot of entry i of a block's descending values (bank-spreading swizzle).
__device__ __forceinline__ int fv_slot(int i) { return i ^ ((i >> 5) & 31); }

// Entries of a descending array of 512 floats that are >= x (strict: > x).
template <bool STRICT>
__device__ __forceinline__ int count_before512(const float* v, float x)
{
    int pos = 0;
#pragma unroll
    for (int step = 256; step > 0; step >>= 1) {
        const float y = v[pos + step - 1];
        if (STRICT ? y > x : y >= x) pos += step;
    }
    const float y = v[pos];
    if (STRICT ? y > x : y >= x) ++pos;
    return pos;
}

// Prefix sets of the eight 128-column segments from the block's descending
// order (values s_v, columns s_i): warp w marks where segment w's columns fall
// in the order, which gives both its share of every prefix (cum) and its own
// order; then each word of a segment's bitsets is an OR over the columns
// before, eight lanes (16 columns each) to a word.
__device__ __forceinline__ void segment_sets(unsigned char* blk, const float* s_v, const uint16_t* s_i,
                                             uint8_t* s_ord)
{
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    float* fv = reinterpret_cast<float*>(blk);
    uint8_t* cum = blk + kPrefCumOff;
    uint32_t* pb = reinterpret_cast<uint32_t*>(blk + kSegPbOff);
    for (int q = tid; q < kColBlock; q += blockDim.x) fv[fv_slot(q)] = s_v[q];
    uint8_t* ord = s_ord + warp * kSegCols;  // columns within the segment
    if (lane == 0) cum[warp] = 0;
    int before = 0;
    for (int q0 = 0; q0 < kColBlock; q0 += 32) {
        const int col = s_i[q0 + lane];
        const bool mine = col / kSegCols == warp;
        const unsigned ballot = __ballot_sync(0xffffffffu, mine);
        const int upto = before + __popc(ballot & ((2u << lane) - 1u));  // (lane 31: the mask wraps to all)
        cum[(q0 + lane + 1) * kSegs + warp] = (uint8_t)upto;
        if (mine) ord[upto - 1] = (uint8_t)(col % kSegCols);
        before += __popc(ballot);
    }
    __syncwarp();
    const int w = lane & 3, part = lane >> 2;
    uint32_t own = 0u;
#pragma unroll
    for (int e = 0; e < 16; ++e) {
        const int col = ord[part * 16 + e];
        own |= (col >> 5) == w ? 1u << (col & 31) : 0u;
    }
    uint32_t acc = own;
#pragma unroll
    for (int o = 4; o < 32; o <<= 1) {
        const uint32_t x = __shfl_up_sync(0xffffffffu, acc, o);
        if (lane >= o) acc |= x;
    }
    acc = __shfl_up_sync(0xffffffffu, acc, 4);  // the parts before
    if (part == 0) acc = 0u;
    uint32_t* row = pb + warp * 4 + w;
    if (part == 0) row[0] = 0u;
#pragma unroll
    for (int e = 0; e < 16; ++e) {
        const int col = ord[part * 16 + e];
        acc |= (col >> 5) == w ? 1u << (col & 31) : 0u;
        row[(part * 16 + e + 1) * 32] = acc;
    }
}

__global__ void __launch_bounds__(256) k_colprep(Plan* plan)
{
    __shared__ float s_v[kColBlock];
    __shared__ uint16_t s_i[kColBlock];
    __shared__ uint8_t s_mark[kColBlock];
    __shared__ uint32_t s_part[8][32];
    __shared__ int s_warp[32];
    __shared__ long long s_first[kMaxBatch + 1];  // items (column block, objective) before each problem
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // key objectives 2..m of the lexicographic order, or every objective of
    // the caller-order columns (MODE_DOM)
    auto keys_of = [&](const ProbDev& d) { return d.in.mode == MODE_DOM ? d.in.m : d.in.m - 1; };
    if (tid == 0) {
        long long acc = 0;
        for (int p = 0; p < plan->nprob; ++p) {
            s_first[p] = acc;
            const ProbDev& d = plan->p[p];
            if (d.colpre && ld_volatile(&d.sc->status) == 0) acc += (long long)d.ncb * keys_of(d);
        }
        s_first[plan->nprob] = acc;
    }
    __syncthreads();
    // the items of every problem in one sequence (a batch's small problems
    // together fill the grid)
    const long long total = s_first[plan->nprob];
    int p = 0;
    for (long long it_all = blockIdx.x; it_all < total; it_all += gridDim.x) {
        while (s_first[p + 1] <= it_all) ++p;
        const ProbDev& d = plan->p[p];
        const bool caller = d.in.mode == MODE_DOM;
        const int K = keys_of(d);
        const float* const kv = caller ? d.ckeys : d.keys;
        const PrefGeom G(K);
        const int ncp1 = kHalf >> G.log_cps;  // checkpoints after the first
        const long long it = it_all - s_first[p];
        const int cb = (int)(it / K), k = (int)(it % K);
        unsigned char* blk = d.colpre + ((int64_t)cb * K + k) * G.obj_bytes;
        for (int q = tid; q < kColBlock; q += blockDim.x) {
            s_v[q] = kv[((int64_t)cb * kColBlock + q) * K + k];
            s_i[q] = (uint16_t)q;
        }
        __syncthreads();
        // bitonic sort: value descending, then local index ascending; by halves
        // each half by itself (positions 0..511 = half 0, 512..1023 = half 1)
        const bool segs = K <= kSegKeys;
        for (int size = 2; size <= kColBlock; size <<= 1) {
            for (int stride = size >> 1; stride > 0; stride >>= 1) {
                for (int t = tid; t < kColBlock / 2; t += blockDim.x) {
                    const int i = 2 * t - (t & (stride - 1)), j = i + stride;
                    const float vi = s_v[i], vj = s_v[j];
                    const int ii = s_i[i], ij = s_i[j];
                    const int hi_ = !segs && ii >= kHalf, hj = !segs && ij >= kHalf;
                    const bool j_first = hj < hi_ || (hj == hi_ && (vj > vi || (vj == vi && ij < ii)));
                    const bool up = (i & size) == 0;
                    if (up == j_first) {
                        s_v[i] = vj; s_v[j] = vi;
                        s_i[i] = (uint16_t)ij; s_i[j] = (uint16_t)ii;
                    }
                }
                __syncthreads();
            }
        }
        if (segs) {
            segment_sets(blk, s_v, s_i, s_mark);
            __syncthreads();
            continue;
        }
        float* fv = reinterpret_cast<float*>(blk);
        uint16_t* cum0 = reinterpret_cast<uint16_t*>(blk + kPrefCumOff);
        uint32_t* pb = reinterpret_cast<uint32_t*>(blk + kPrefPbOff);
        uint16_t* so = reinterpret_cast<uint16_t*>(blk + G.ord_off);
        for (int q = tid; q < kColBlock; q += blockDim.x) so[q] = s_i[q];
        // merge of the halves into the full descending order (ties: half 0
        // first); mark the half-0 positions
        for (int q = tid; q < kColBlock; q += blockDim.x) {
            const float x = s_v[q];
            const int rank = (q & (kHalf - 1)) +
                             (q < kHalf ? count_before512<true>(s_v + kHalf, x) : count_before512<false>(s_v, x));
            fv[fv_slot(rank)] = x;
            s_mark[rank] = q < kHalf;
        }
        // interleaved prefix bitsets: lane w builds word w from the sorted
        // columns of half w / 16; warp v covers checkpoints (v*seg, (v+1)*seg]
        const int hbase = (lane >> 4) * kHalf;
        const int seg = ncp1 / 8;
        uint32_t part = 0u;
        for (int c = warp * seg; c < (warp + 1) * seg; ++c)
            for (int e = 0; e < G.cps; ++e) {
                const int col = s_i[hbase + c * G.cps + e];
                if ((col >> 5) == lane) part |= 1u << (col & 31);
            }
        s_part[warp][lane] = part;
        __syncthreads();
        uint32_t acc = 0u;
        for (int w = 0; w < warp; ++w) acc |= s_part[w][lane];
        if (warp == 0) pb[lane] = 0u;
        for (int c = warp * seg; c < (warp + 1) * seg; ++c) {
            for (int e = 0; e < G.cps; ++e) {
                const int col = s_i[hbase + c * G.cps + e];
                if ((col >> 5) == lane) acc |= 1u << (col & 31);
            }
            pb[(c + 1) * 32 + lane] = acc;
        }
        // cum0[j] = half-0 entries among the first j of the full order
        {
            const int j0 = tid * 4;  // 256 threads x 4 entries
            const int m0 = s_mark[j0], m1 = s_mark[j0 + 1], m2 = s_mark[j0 + 2], m3 = s_mark[j0 + 3];
            int tot;
            const int ex = block_exclusive_scan<256>(m0 + m1 + m2 + m3, s_warp, tot);
            if (tid == 0) cum0[0] = 0;
            cum0[j0 + 1] = (uint16_t)(ex + m0);
            cum0[j0 + 2] = (uint16_t)(ex + m0 + m1);
            cum0[j0 + 3] = (uint16_t)(ex + m0 + m1 + m2);
            cum0[j0 + 4] = (uint16_t)(ex + m0 + m1 + m2 + m3);
        }
        __syncthreads();
    }
}

// ------------------------------------------------------------ k_dom_pref
template <int K>
struct PrefSmem {
    alignas(128) unsigned char obj[K * kSegObjBytes];
    alignas(128) int32_t rs[kColBlock];
    int32_t cnt[kColBlock];
    alignas(8) unsigned char st[16][K * 128];  // each warp's staged segment counts
    uint64_t bar;
    long long item;
    int skip;
};

// How many of the block's values of one objective are >= x (binary search
// over the full descending order). Entry i of the order is stored at
// fv_slot(i): the candidates of one search level are i = c * step - 1 for
// step >= 32, all with the same low five bits, and the XOR with i / 32 puts
// them in distinct shared-memory banks.
__device__ __forceinline__ int count_ge(const unsigned char* ob, float x)
{
    const float* fv = reinterpret_cast<const float*>(ob);
    int pos = 0;
#pragma unroll
    for (int step = kColBlock / 2; step > 0; step >>= 1)
        if (fv[fv_slot(pos + step - 1)] >= x) pos += step;
    if (fv[fv_slot(pos)] >= x) ++pos;
    return pos;
}

// The count split by halves: t0 | t1 << 16.
__device__ __forceinline__ int count_ge_halves(const unsigned char* ob, float x)
{
    const int pos = count_ge(ob, x);
    const int t0 = reinterpret_cast<const uint16_t*>(ob + kPrefCumOff)[pos];
    return t0 | ((pos - t0) << 16);
}

// Segment counts of the rows g * 8 .. + 7 and 16 + g * 8 .. + 7 of a row block
// into the warp's staging area (8 bytes per objective and row): the count t[k]
// of the lane's row split over the segments.
template <int K>
__device__ __forceinline__ void stage_counts(const unsigned char* obj, unsigned char* st, const int (&t)[K], int g, int lane)
{
    __syncwarp();  // the rows before are read
    if (((lane >> 3) & 1) == g) {
        const int row = (lane & 7) + (lane >> 4) * 8;
#pragma unroll
        for (int k = 0; k < K; ++k)
            *reinterpret_cast<unsigned long long*>(st + k * 128 + row * 8) =
                *reinterpret_cast<const unsigned long long*>(obj + k * kSegObjBytes + kPrefCumOff + t[k] * kSegs);
    }
    __syncwarp();
}

// Two words (columns 64 l .. 64 l + 63, l = lane % 16) of the AND of the
// objectives' prefix sets for the staged row jj (of the lane's half-warp): the
// segment's share of each prefix, then that row of its bitsets. The 16 lanes
// read one 8-byte entry and then 16 different bank pairs. (A shuffle of the
// row's count and a look-up of its share instead of the staged bytes: one more
// dependent access per objective, 575 us instead of 543 at 100,000 points of
// eight objectives.)
template <int K>
__device__ __forceinline__ unsigned long long row_words(const unsigned char* obj_l, const unsigned char* st_l, int jj)
{
    unsigned long long word = ~0ull;
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const int c = st_l[k * 128 + jj * 8];
        word &= *reinterpret_cast<const unsigned long long*>(obj_l + k * kSegObjBytes + kSegPbOff + c * 128);
    }
    return word;
}

// First column of the block (0 .. 1024) that row p may dominate: past p itself
// (diagonal blocks) and past the points identical to p, which follow it in the
// order -- the columns whose run starts at p or before. nv: the block's points.
template <bool DUP>
__device__ __forceinline__ int first_column(const int32_t* rs, int64_t p, int64_t cbase, int nv)
{
    int lo = (int)min((int64_t)kColBlock, max((int64_t)0, p + 1 - cbase));
    if (DUP) {
        int hi = nv;  // run starts ascend: the first one beyond p
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if ((int64_t)rs[mid] <= p) lo = mid + 1;
            else hi = mid;
        }
    }
    return lo;
}

// Keep the columns from `first` on of the lane's 64. (With the run starts tested
// column by column in every row, the few blocks of rows beside the diagonal
// left one SM busy while the others had finished: 543 us instead of 462 at
// 100,000 points of eight objectives on a grid.)
__device__ __forceinline__ unsigned long long keep_from(unsigned long long word, int first, int l)
{
    const int off = first - 64 * l;
    return off >= 64 ? 0ull : (off > 0 ? word & (~0ull << off) : word);
}

// The 32 rows of row block rb in column block cb; t[k] is the count of
// objective k for the lane's row.
// EDGE: rows keep only the columns from `first` (of the lane's row) on.
template <int K, bool EDGE>
__device__ __forceinline__ void pref_rows(const unsigned char* __restrict__ obj, unsigned char* st,
                                          const int (&t)[K], int first, uint32_t* tile, VCount<kDomNH>& vlo, VCount<kDomNH>& vhi, int lane)
{
    const int l = lane & 15, h = lane >> 4;
    unsigned long long* dst = reinterpret_cast<unsigned long long*>(tile + h * 16 * 32) + l;
    const unsigned char* const obj_l = obj + l * 8;
    const unsigned char* const st_l = st + h * 64 + (l >> 1);
#pragma unroll 1
    for (int g = 0; g < 2; ++g) {
        stage_counts<K>(obj, st, t, g, lane);
        uint32_t xl[8], xh[8];
#pragma unroll
        for (int jj = 0; jj < 8; ++jj) {
            const int j = g * 8 + jj, i = j + 16 * h;
            unsigned long long word = row_words<K>(obj_l, st_l, jj);
            if (EDGE) word = keep_from(word, __shfl_sync(0xffffffffu, first, i), l);
            __stcs(dst + j * 16, word);
            xl[jj] = (uint32_t)word;
            xh[jj] = (uint32_t)(word >> 32);
        }
        vlo.add8_warp(xl);
        vhi.add8_warp(xh);
    }
}

// Stage the prefix sets of column block cb (and its run starts); returns
// false when the problem is skipped or the copy timed out.
__device__ __forceinline__ bool dom_stage(const ProbDev& d, int cb, int K, int obj_bytes, unsigned char* obj,
                                          int32_t* rs, int32_t* cnt, uint64_t* bar, int* s_skip, uint32_t& parity,
                                          bool& fatal)
{
    const int tid = threadIdx.x;
    const uint32_t ob = (uint32_t)(K * obj_bytes);
    if (tid == 0) {
        *s_skip = ld_volatile(&d.sc->status) != 0 || d.in.m - 1 != K;
        if (!*s_skip) {
            fence_proxy_async_smem();
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
                         "r"(ob + (uint32_t)(kColBlock * 4))
                         : "memory");
            asm volatile(
                "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                    smem_u32(obj)),
                "l"(d.colpre + (int64_t)cb * ob), "r"(ob), "r"(smem_u32(bar))
                : "memory");
            asm volatile(
                "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                    smem_u32(rs)),
                "l"(d.runstart + (int64_t)cb * kColBlock), "r"((uint32_t)(kColBlock * 4)), "r"(smem_u32(bar))
                : "memory");
        }
    }
    for (int i = tid; i < kColBlock; i += blockDim.x) cnt[i] = 0;
    __syncthreads();
    if (*s_skip) return false;
    // The copy is a local load that always completes; the bound only guards
    // against a lost completion. On timeout the status is set and the CTA
    // still waits (bounded) so that no copy is in flight at exit.
    if (!mbar_wait(bar, parity, kCopyWaitCycles)) {
        if (tid == 0) set_status(d.sc, EMO_ERR_TIMEOUT);
        mbar_wait(bar, parity, kCopyWaitCycles);
        fatal = true;
        return false;
    }
    parity ^= 1u;
    return true;
}

// Column counts of the item: smem reduction, one global atomic per column.
__device__ __forceinline__ void dom_flush_item(const ProbDev& d, int64_t cbase, VCount<kDomNH>& vlo,
                                               VCount<kDomNH>& vhi, int32_t* cnt, int lane)
{
    flush_counts(vlo, vhi, cnt, lane);
    __syncthreads();
    for (int q = threadIdx.x; q < kColBlock; q += blockDim.x) {
        const int c = cnt[(q & 31) * 32 + (q >> 5)];
        if (c) atomicAdd(&d.cnt[cbase + q], c);
    }
    __syncthreads();
}

template <int M>
__global__ void __launch_bounds__(512, 1) k_dom_pref(Plan* plan, long long item_lo, long long item_hi,
                                                     unsigned long long* counter)
{
    constexpr int K = M - 1, NW = 16;
    extern __shared__ __align__(128) unsigned char smraw[];
    PrefSmem<K>& sm = *reinterpret_cast<PrefSmem<K>*>(smraw);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) mbar_init(&sm.bar, 1);
    __syncthreads();
    uint32_t parity = 0;

    while (true) {
        if (tid == 0) sm.item = item_lo + (long long)atomicAdd(counter, 1ull);
        __syncthreads();
        const long long item = sm.item;
        if (item >= item_hi) break;
        int p = 0;
        while (p + 1 < plan->nprob && plan->dom_item_start[p + 1] <= item) ++p;
        const ProbDev& d = plan->p[p];
        int cb, chunk;
        const int rows = d.in.dom_chunk;
        dom_decode(item - plan->dom_item_start[p], d.ncb, d.nrb, rows, cb, chunk);
        bool fatal = false;
        if (!dom_stage(d, cb, K, kSegObjBytes, sm.obj, sm.rs, sm.cnt, &sm.bar, &sm.skip, parity, fatal)) {
            if (fatal) break;
            continue;
        }
        const int64_t n2 = d.in.n2;
        const int rbmax = min(d.nrb, 32 * (cb + 1));
        const int rb_lo = chunk * rows, rb_hi = min(rbmax, rb_lo + rows);
        const int dupcut = d.minrs[cb];
        const int64_t cbase = (int64_t)cb * kColBlock;
        const int nv = (int)min((int64_t)kColBlock, n2 - cbase);
        // in registers: the tile stores could alias the plan, which would
        // otherwise reload these after every row block
        uint32_t* const Dm = d.D;
        const float* const keys = d.keys;
        const int ncb = d.ncb;
        VCount<kDomNH> vlo, vhi;

        // keys of the lane's row in the warp's next row block (prefetched)
        float key[K];
        {
            const int64_t pl = (int64_t)(rb_lo + warp) * kTileRows + lane;
#pragma unroll
            for (int k = 0; k < K; ++k) key[k] = (rb_lo + warp < rb_hi && pl < n2) ? __ldg(&keys[pl * K + k]) : 0.0f;
        }
        for (int rb = rb_lo + warp; rb < rb_hi; rb += NW) {
            const int64_t pl = (int64_t)rb * kTileRows + lane;
            int t[K];
#pragma unroll
            for (int k = 0; k < K; ++k) t[k] = pl < n2 ? count_ge(sm.obj + k * kSegObjBytes, key[k]) : 0;
            {
                const int rbn = rb + NW;
                const int64_t pn = (int64_t)rbn * kTileRows + lane;
#pragma unroll
                for (int k = 0; k < K; ++k) key[k] = (rbn < rb_hi && pn < n2) ? __ldg(&keys[pn * K + k]) : 0.0f;
            }
            const bool diag = (int64_t)rb * kTileRows + 31 >= cbase;
            const bool dup = rb * kTileRows + 31 >= dupcut;
            uint32_t* tile = Dm + tile_index(rb, cb, ncb) * (int64_t)(kTileRows * kTileWords);
            if (dup) pref_rows<K, true>(sm.obj, sm.st[warp], t, first_column<true>(sm.rs, pl, cbase, nv), tile, vlo, vhi, lane);
            else if (diag) pref_rows<K, true>(sm.obj, sm.st[warp], t, first_column<false>(sm.rs, pl, cbase, nv), tile, vlo, vhi, lane);
            else pref_rows<K, false>(sm.obj, sm.st[warp], t, 0, tile, vlo, vhi, lane);
        }
        dom_flush_item(d, cbase, vlo, vhi, sm.cnt, lane);
    }
}

// ------------------------------------------------------------ k_dom_caller
// The full dominance matrix in the caller's order (emo_dominance_ws) by the
// same prefix sets, built over caller-order column blocks for all K = m
// objectives: the set {q : f_k(q) >= f_k(p) for every k} is the AND of K
// prefix sets, and p dominates q iff q is in that set and is not identical to
// p (all equal: p itself and its exact duplicates, found as the runs of the
// lexicographic sort). Items: (column block, chunk of row blocks) over the
// whole square; a warp builds one 1024-column row segment at a time (a lane
// owns 32 columns), written into row p of D; column counts as in k_dom_pref.
// m <= 5 (the blocks' prefix data must fit in shared memory).
// Set-up of the caller-order matrix after the sort: the objectives in the
// caller's order padded with -inf to whole column blocks (the prefix sets of
// every objective are built on them), and each point's run of identical
// points in sorted positions (first, one past the last; first = -1 when the
// point has no duplicate).
__global__ void k_dom_keys(Plan* plan)
{
    const ProbDev& d = plan->p[0];
    if (d.in.mode != MODE_DOM || ld_volatile(&d.sc->status) != 0) return;
    const int m = d.in.m;
    const int64_t n2 = d.in.n2;
    const int32_t* idx = d.idx + (int64_t)ld_volatile(&d.sc->idx_buf) * d.n2p;
    const int32_t* rs = d.runstart;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < d.n2p * m; e += stride)
        d.ckeys[e] = e / m < n2 ? d.in.F[e] + 0.0f : -INFINITY;
    for (int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; s < n2; s += stride) {
        const int r0 = rs[s];
        int r1 = (int)s + 1;
        while (r1 < n2 && rs[r1] == r0) ++r1;
        const int q = idx[s];
        d.spos[q] = (r1 - r0 > 1) ? r0 : -1;
        d.spos[n2 + q] = r1;
    }
}

// A row of D starts at any word (its stride is the caller's, by default
// ceil(n2 / 32) words), so the segment of a row that a column block covers
// shares its first and last 32-byte sectors with the blocks beside it. A lane
// therefore owns one word and a warp stores 128 contiguous bytes of one row;
// the items run along the rows, so that neighbouring blocks write at about the
// same time, and the stores are kept in L2 like any other, where the shared
// sectors meet. 100,000 points of three objectives (1.25 GB, a stride of 3125
// words): 885 us with two words per lane stored one by one, 761 so, 816 with
// stores that leave L2 first.
// (up to three objectives two CTAs fit on an SM)
constexpr int kCallerNH = 8;  // high count planes: up to 4095 rows per lane and item
template <int K>
struct CallerShape {
    static constexpr int NT = K <= 3 ? 512 : 1024, NW = NT / 32;
    static_assert((kDomRowChunk + NW - 1) / NW * 32 < (1 << (4 + kCallerNH)), "column counter overflow");
};
template <int K>
struct CallerSmem {
    alignas(128) unsigned char obj[K * kSegObjBytes];
    int32_t cnt[kColBlock];
    alignas(8) unsigned char st[CallerShape<K>::NW][K * 256];  // each warp's segment counts: 8 bytes per objective and row
    uint64_t bar;
    long long item;
    int skip;
};

// The 32 rows of one row block in one column block; the lane's word of the
// first row goes to row0, w0 is its index within a row. PLAIN: none of the
// checks below can apply.
template <int K, bool PLAIN>
__device__ __forceinline__ void caller_rows(const unsigned char* obj, const unsigned char* st, int64_t rowbase,
                                            int64_t cbase, int64_t n2, uint32_t* row0, int64_t w0, int64_t ld,
                                            const int32_t* idx, int dup_lo, int dup_hi, VCount<kCallerNH>& vc, int lane)
{
    const unsigned char* const obj_l = obj + kSegPbOff + lane * 4;
    const unsigned char* const st_l = st + (lane >> 2);
#pragma unroll 1
    for (int g = 0; g < 4; ++g) {
        uint32_t x[8];
#pragma unroll
        for (int jj = 0; jj < 8; ++jj) {
            const int i = g * 8 + jj;
            uint32_t word = ~0u;
#pragma unroll
            for (int k = 0; k < K; ++k) {
                const int c = st_l[k * 256 + i * 8];
                word &= *reinterpret_cast<const uint32_t*>(obj_l + k * kSegObjBytes + c * 128);
            }
            if (!PLAIN) {
                // not identical to p: p itself, and its duplicates
                const int64_t p = rowbase + i;
                const int dlo = __shfl_sync(0xffffffffu, dup_lo, i), dhi = __shfl_sync(0xffffffffu, dup_hi, i);
                if (dhi > dlo) {
                    for (int r = dlo; r < dhi; ++r) {
                        const int64_t off = (int64_t)__ldg(&idx[r]) - cbase - 32 * lane;
                        if (off >= 0 && off < 32) word &= ~(1u << off);
                    }
                } else {
                    const int64_t off = p - cbase - 32 * lane;
                    if (off >= 0 && off < 32) word &= ~(1u << off);
                }
                if (p >= n2) word = 0u;
                if (p < n2 && w0 < ld) row0[i * ld] = word;  // words past ld (a short last block) are not stored
            } else {
                row0[i * ld] = word;
            }
            x[jj] = word;
        }
        vc.add8_warp(x);
    }
}

template <int K>
__global__ void __launch_bounds__(CallerShape<K>::NT, K <= 3 ? 2 : 1) k_dom_caller(Plan* plan, long long nitems,
                                                                                 unsigned long long* counter)
{
    constexpr int NW = CallerShape<K>::NW;
    extern __shared__ __align__(128) unsigned char smraw[];
    CallerSmem<K>& sm = *reinterpret_cast<CallerSmem<K>*>(smraw);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) mbar_init(&sm.bar, 1);
    __syncthreads();
    uint32_t parity = 0;
    const ProbDev& d = plan->p[0];
    const int64_t n2 = d.in.n2, ld = d.in.dom_ld;
    const int nrb = d.nrb, ncb = d.ncb;
    const int rows = d.in.dom_chunk;
    const int32_t* const idx = d.idx + (int64_t)ld_volatile(&d.sc->idx_buf) * d.n2p;
    const int32_t* const spos = d.spos;
    const float* const ck = d.ckeys;
    uint32_t* const Dout = d.in.dom_out;
    while (true) {
        if (tid == 0) sm.item = (long long)atomicAdd(counter, 1ull);
        __syncthreads();
        const long long item = sm.item;
        if (item >= nitems) break;
        const int cb = (int)(item % ncb), chunk = (int)(item / ncb);
        if (tid == 0) {
            sm.skip = ld_volatile(&d.sc->status) != 0;
            if (!sm.skip) {
                fence_proxy_async_smem();
                bulk_load(sm.obj, d.colpre + (int64_t)cb * (K * kSegObjBytes), (uint32_t)(K * kSegObjBytes), &sm.bar);
            }
        }
        for (int i = tid; i < kColBlock; i += blockDim.x) sm.cnt[i] = 0;
        __syncthreads();
        if (sm.skip) break;
        if (!mbar_wait(&sm.bar, parity, kCopyWaitCycles)) {
            if (tid == 0) set_status(d.sc, EMO_ERR_TIMEOUT);
            mbar_wait(&sm.bar, parity, kCopyWaitCycles);
            break;
        }
        parity ^= 1u;
        const int64_t cbase = (int64_t)cb * kColBlock;
        const int rb_lo = chunk * rows, rb_hi = min(nrb, rb_lo + rows);
        VCount<kCallerNH> vc;
        unsigned char* const st = sm.st[warp];
        for (int rb = rb_lo + warp; rb < rb_hi; rb += NW) {
            const int64_t rowbase = (int64_t)rb * kTileRows, pl = rowbase + lane;  // the lane's row (search)
            __syncwarp();  // the counts before are read
#pragma unroll
            for (int k = 0; k < K; ++k) {
                const unsigned char* const ob = sm.obj + k * kSegObjBytes;
                const int pos = pl < n2 ? count_ge(ob, __ldg(&ck[pl * K + k])) : 0;
                *reinterpret_cast<unsigned long long*>(st + k * 256 + lane * 8) =
                    *reinterpret_cast<const unsigned long long*>(ob + kPrefCumOff + pos * kSegs);
            }
            // duplicates of the lane's row: sorted positions [dup_lo, dup_hi) when it has any
            const int dup_lo = pl < n2 ? __ldg(&spos[pl]) : -1, dup_hi = dup_lo >= 0 ? __ldg(&spos[n2 + pl]) : -1;
            __syncwarp();
            // (the usual block of rows: all there, none with a duplicate, none
            // among the block's columns, whole words to store)
            const bool plain = rowbase + kTileRows <= n2 && cb * 32 + 32 <= ld &&
                               (rowbase + kTileRows <= cbase || rowbase >= cbase + kColBlock) &&
                               !__any_sync(0xffffffffu, dup_hi > dup_lo);
            const int64_t w0 = (int64_t)cb * 32 + lane;
            uint32_t* const row0 = Dout + rowbase * ld + w0;
            if (plain) caller_rows<K, true>(sm.obj, st, rowbase, cbase, n2, row0, w0, ld, idx, dup_lo, dup_hi, vc, lane);
            else caller_rows<K, false>(sm.obj, st, rowbase, cbase, n2, row0, w0, ld, idx, dup_lo, dup_hi, vc, lane);
        }
        // column counts of the item: shared-memory reduction, one global atomic per column
        if (d.in.dom_count) {
            const int top = vc.top_plane();
            if (top >= 0) {
#pragma unroll 4
                for (int b = 0; b < 32; ++b) {
                    const int c = vc.count_upto(b, top);
                    if (c) atomicAdd(&sm.cnt[b * 32 + lane], c);
                }
            }
            __syncthreads();
            for (int q = tid; q < kColBlock; q += blockDim.x) {
                const int c = sm.cnt[(q & 31) * 32 + (q >> 5)];
                if (c && cbase + q < n2) atomicAdd(&d.in.dom_count[cbase + q], c);
            }
        }
        __syncthreads();
    }
}

// Runtime-K variant for m >= 9, prefix sets by halves (compact code: loops over the key objectives
// are not unrolled; the packed half counts of a row block are staged in
// shared memory).
__global__ void __launch_bounds__(512, 1) k_dom_pref_rt(Plan* plan, long long item_lo, long long item_hi,
                                                        unsigned long long* counter, int K)
{
    constexpr int NW = 16;
    const PrefGeom G(K);
    extern __shared__ __align__(128) unsigned char smraw[];
    const int obj_total = K * G.obj_bytes;
    unsigned char* obj = smraw;
    int32_t* rs = reinterpret_cast<int32_t*>(smraw + ((obj_total + 127) & ~127));
    int32_t* cnt = rs + kColBlock;
    int32_t* st = cnt + kColBlock;  // [NW][K][32] packed half counts of the warp's row block
    uint64_t* bar = reinterpret_cast<uint64_t*>(st + NW * K * 32);
    long long* s_item = reinterpret_cast<long long*>(bar + 1);
    int* s_skip = reinterpret_cast<int*>(s_item + 1);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int32_t* myst = st + warp * K * 32;
    const int l = lane & 15, h = lane >> 4, half = l >> 3, hs = half * 16;
    if (tid == 0) mbar_init(bar, 1);
    __syncthreads();
    uint32_t parity = 0;

    while (true) {
        if (tid == 0) *s_item = item_lo + (long long)atomicAdd(counter, 1ull);
        __syncthreads();
        const long long item = *s_item;
        if (item >= item_hi) break;
        int p = 0;
        while (p + 1 < plan->nprob && plan->dom_item_start[p + 1] <= item) ++p;
        const ProbDev& d = plan->p[p];
        int cb, chunk;
        const int rows = d.in.dom_chunk;
        dom_decode(item - plan->dom_item_start[p], d.ncb, d.nrb, rows, cb, chunk);
        bool fatal = false;
        if (!dom_stage(d, cb, K, G.obj_bytes, obj, rs, cnt, bar, s_skip, parity, fatal)) {
            if (fatal) break;
            continue;
        }
        const int64_t n2 = d.in.n2;
        const int rbmax = min(d.nrb, 32 * (cb + 1));
        const int rb_lo = chunk * rows, rb_hi = min(rbmax, rb_lo + rows);
        const int dupcut = d.minrs[cb];
        const int64_t cbase = (int64_t)cb * kColBlock;
        const int nv = (int)min((int64_t)kColBlock, n2 - cbase);
        uint32_t* const Dm = d.D;
        const float* const keys = d.keys;
        const int ncb = d.ncb;
        VCount<kDomNH> vlo, vhi;
        for (int rb = rb_lo + warp; rb < rb_hi; rb += NW) {
            const int64_t pl = (int64_t)rb * kTileRows + lane;
            for (int k = 0; k < K; ++k)
                myst[k * 32 + lane] = pl < n2 ? count_ge_halves(obj + k * G.obj_bytes, __ldg(&keys[pl * K + k])) : 0;
            __syncwarp();
            const bool diag = (int64_t)rb * kTileRows + 31 >= cbase;
            const bool dup = rb * kTileRows + 31 >= dupcut;
            const int first = dup ? first_column<true>(rs, pl, cbase, nv) : (diag ? first_column<false>(rs, pl, cbase, nv) : 0);
            uint32_t* tile = Dm + tile_index(rb, cb, ncb) * (int64_t)(kTileRows * kTileWords);
            unsigned long long* dst = reinterpret_cast<unsigned long long*>(tile + h * 16 * 32) + l;
#pragma unroll 1
            for (int g = 0; g < 2; ++g) {
                uint32_t xl[8], xh[8];
#pragma unroll
                for (int jj = 0; jj < 8; ++jj) {
                    const int j = g * 8 + jj, i = j + 16 * h;
                    unsigned long long word = ~0ull;
#pragma unroll 1
                    for (int k = 0; k < K; ++k) {
                        const unsigned char* ob = obj + k * G.obj_bytes;
                        const int t = (myst[k * 32 + i] >> hs) & 0xFFFF;
                        const int c = t >> G.log_cps;
                        unsigned long long wk =
                            *reinterpret_cast<const unsigned long long*>(ob + kPrefPbOff + c * 128 + l * 8);
                        const int rem = t & (G.cps - 1);
                        const uint16_t* so =
                            reinterpret_cast<const uint16_t*>(ob + G.ord_off) + half * kHalf + (c << G.log_cps);
                        for (int e = 0; e < rem; ++e) {
                            const int col = so[e];
                            if ((col >> 6) == l) wk |= 1ull << (col & 63);
                        }
                        word &= wk;
                    }
                    if (diag | dup) word = keep_from(word, __shfl_sync(0xffffffffu, first, i), l);
                    __stcs(dst + j * 16, word);
                    xl[jj] = (uint32_t)word;
                    xh[jj] = (uint32_t)(word >> 32);
                }
                vlo.add8_warp(xl);
                vhi.add8_warp(xh);
            }
            __syncwarp();
        }
        dom_flush_item(d, cbase, vlo, vhi, cnt, lane);
    }
}

// Full matrix in caller order: D_ij = all(F_i <= F_j) and any(F_i < F_j).
constexpr int kFullNH = 8;  // up to 4095 rows per lane and item
template <int M>
struct FullSmem {
    alignas(16) float ck[kColBlock * M];
    alignas(16) uint32_t tiles[8][2][kTileRows * kTileWords];
    int32_t cnt[kColBlock];
    long long item;
};

// Columns [col_lo, col_hi) (col_lo a multiple of 1024); D word w of a row
// holds columns col_lo + 32 w .. + 31, dom_count[j - col_lo] their sums.
template <int M>
__global__ void __launch_bounds__(256, 1) k_dom_full(const float* __restrict__ F, int64_t n2, int64_t col_lo,
                                                     int64_t col_hi, uint32_t* D, int64_t ld, int32_t* cnt,
                                                     long long nitems)
{
    constexpr int R = 2, NW = 8;
    extern __shared__ __align__(128) unsigned char smraw[];
    FullSmem<M>& sm = *reinterpret_cast<FullSmem<M>*>(smraw);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int nrb = (int)cdiv(n2, 32);
    const long long per_cb = cdiv(nrb, kDomRowChunk);
    const int cb_lo = (int)(col_lo / kColBlock);
    for (long long item = blockIdx.x; item < nitems; item += gridDim.x) {
        const int cb = cb_lo + (int)(item / per_cb), chunk = (int)(item % per_cb);
        const int64_t cbase = (int64_t)cb * kColBlock;
        for (int i = tid; i < kColBlock * M; i += blockDim.x) {
            const int64_t q = cbase + i / M;
            sm.ck[i] = q < col_hi ? F[q * M + i % M] + 0.0f : -INFINITY;
        }
        for (int i = tid; i < kColBlock; i += blockDim.x) sm.cnt[i] = 0;
        __syncthreads();
        const int rb_lo = chunk * kDomRowChunk, rb_hi = min(nrb, rb_lo + kDomRowChunk);
        VCount<kFullNH> vc;
        for (int rbg = rb_lo + warp * R; rbg < rb_hi; rbg += NW * R) {
            float rk[R][M];
            int64_t prow[R];
            bool rvalid[R];
#pragma unroll
            for (int r = 0; r < R; ++r) {
                rvalid[r] = rbg + r < rb_hi;
                prow[r] = (int64_t)(rbg + r) * kTileRows + lane;
                const bool live = rvalid[r] && prow[r] < n2;
#pragma unroll
                for (int k = 0; k < M; ++k) rk[r][k] = live ? F[prow[r] * M + k] + 0.0f : INFINITY;
            }
            for (int w = 0; w < kTileWords; ++w) {
                uint32_t wd[R];
#pragma unroll
                for (int r = 0; r < R; ++r) wd[r] = 0u;
#pragma unroll 4
                for (int b = 0; b < 32; ++b) {
                    const float* c = sm.ck + (w * 32 + b) * M;
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        bool le = true, lt = false;
#pragma unroll
                        for (int k = 0; k < M; ++k) {
                            le = le & (rk[r][k] <= c[k]);
                            lt = lt | (rk[r][k] < c[k]);
                        }
                        if (le & lt) wd[r] |= 1u << b;
                    }
                }
#pragma unroll
                for (int r = 0; r < R; ++r) sm.tiles[warp][r][lane * 32 + (w ^ lane)] = wd[r];
            }
            __syncwarp();
#pragma unroll
            for (int r = 0; r < R; ++r) {
                if (!rvalid[r]) continue;
                uint32_t x[32];
#pragma unroll
                for (int row = 0; row < 32; ++row) x[row] = sm.tiles[warp][r][row * 32 + (lane ^ row)];
                vc.add16(x);
                vc.add16(x + 16);
                const int64_t wcol = (int64_t)(cb - cb_lo) * 32 + lane;
                if (wcol < ld) {
#pragma unroll 4
                    for (int row = 0; row < 32; ++row) {
                        const int64_t pr = (int64_t)(rbg + r) * kTileRows + row;
                        if (pr < n2) D[pr * ld + wcol] = x[row];
                    }
                }
            }
            __syncwarp();
        }
        if (cnt) {
            if (__any_sync(0xffffffffu, vc.any())) {
#pragma unroll 4
                for (int b = 0; b < 32; ++b) {
                    const int c = vc.count(b);
                    if (c) atomicAdd(&sm.cnt[b * 32 + lane], c);
                }
            }
            __syncthreads();
            for (int q = tid; q < kColBlock; q += blockDim.x) {
                const int c = sm.cnt[(q & 31) * 32 + (q >> 5)];
                if (c && cbase + q < col_hi) atomicAdd(&cnt[cbase + q - col_lo], c);
            }
        }
        __syncthreads();
    }
}

// ------------------------------------------------------------ launchers
template <int M>
static cudaError_t launch_tri_m(Plan* plan, int sms, cudaStream_t s, long long lo, long long hi,
                                unsigned long long* counter)
{
    const size_t smem = sizeof(PrefSmem<M - 1>);
    cudaError_t e = cudaFuncSetAttribute(k_dom_pref<M>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int occ = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_dom_pref<M>, 512, smem);
    if (e != cudaSuccess) return e;
    long long grid = (long long)sms * (occ > 0 ? occ : 1);
    if (grid > hi - lo) grid = hi - lo;
    if (grid < 1) return cudaSuccess;
    k_dom_pref<M><<<(unsigned)grid, 512, smem, s>>>(plan, lo, hi, counter);
    return cudaGetLastError();
}

static cudaError_t launch_tri_rt(int K, Plan* plan, int sms, cudaStream_t s, long long lo, long long hi,
                                 unsigned long long* counter)
{
    const int obj_total = K * (int)colprep_obj_bytes(K);
    const size_t smem = (size_t)((obj_total + 127) & ~127) + 2 * kColBlock * 4 + 16 * K * 32 * 4 + 64;
    cudaError_t e = cudaFuncSetAttribute(k_dom_pref_rt, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int occ = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_dom_pref_rt, 512, smem);
    if (e != cudaSuccess) return e;
    long long grid = (long long)sms * (occ > 0 ? occ : 1);
    if (grid > hi - lo) grid = hi - lo;
    if (grid < 1) return cudaSuccess;
    k_dom_pref_rt<<<(unsigned)grid, 512, smem, s>>>(plan, lo, hi, counter, K);
    return cudaGetLastError();
}

template <int M>
static cudaError_t launch_full_m(const float* F, int64_t n2, int64_t col_lo, int64_t col_hi, uint32_t* D, int64_t ld,
                                 int32_t* cnt, int sms, cudaStream_t s)
{
    const size_t smem = sizeof(FullSmem<M>);
    cudaError_t e = cudaFuncSetAttribute(k_dom_full<M>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int occ = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_dom_full<M>, 256, smem);
    if (e != cudaSuccess) return e;
    const long long nitems = cdiv(col_hi - col_lo, kColBlock) * cdiv(cdiv(n2, 32), kDomRowChunk);
    long long grid = (long long)sms * (occ > 0 ? occ : 1);
    if (grid > nitems) grid = nitems;
    k_dom_full<M><<<(unsigned)grid, 256, smem, s>>>(F, n2, col_lo, col_hi, D, ld, cnt, nitems);
    return cudaGetLastError();
}

template <int K>
static cudaError_t launch_caller_k(Plan* plan, int sms, cudaStream_t s, long long nitems, unsigned long long* counter)
{
    const size_t smem = sizeof(CallerSmem<K>);
    cudaError_t e = cudaFuncSetAttribute(k_dom_caller<K>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int occ = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_dom_caller<K>, CallerShape<K>::NT, smem);
    if (e != cudaSuccess) return e;
    long long grid = (long long)sms * (occ > 0 ? occ : 1);
    if (grid > nitems) grid = nitems;
    if (grid < 1) return cudaSuccess;
    k_dom_caller<K><<<(unsigned)grid, CallerShape<K>::NT, smem, s>>>(plan, nitems, counter);
    return cudaGetLastError();
}

cudaError_t launch_dominance_caller(int m, Plan* plan, int sms, cudaStream_t s, long long nitems,
                                    unsigned long long* counter)
{
    k_dom_keys<<<sms * 2, 256, 0, s>>>(plan);
    cudaError_t e0 = cudaGetLastError();
    if (e0 != cudaSuccess) return e0;
    e0 = launch_colprep(plan, sms, s);
    if (e0 != cudaSuccess) return e0;
    switch (m) {
    case 2: return launch_caller_k<2>(plan, sms, s, nitems, counter);
    case 3: return launch_caller_k<3>(plan, sms, s, nitems, counter);
    case 4: return launch_caller_k<4>(plan, sms, s, nitems, counter);
    case 5: return launch_caller_k<5>(plan, sms, s, nitems, counter);
    default: return cudaErrorInvalidValue;
    }
}

#define EMO_FOR_EACH_M(X) X(2) X(3) X(4) X(5) X(6) X(7) X(8) X(9) X(10) X(11) X(12) X(13) X(14) X(15) X(16)

// The plan's problems are ordered by m; items of objective count m form one
// contiguous range served by the m-instantiation.
cudaError_t launch_colprep(Plan* plan, int sms, cudaStream_t s)
{
    k_colprep<<<sms * 4, 256, 0, s>>>(plan);
    return cudaGetLastError();
}

cudaError_t launch_dominance_tri_range(int m, Plan* plan, int sms, cudaStream_t s, long long lo, long long hi,
                                       unsigned long long* counter)
{
    switch (m) {
    case 6: return launch_tri_m<6>(plan, sms, s, lo, hi, counter);
    case 7: return launch_tri_m<7>(plan, sms, s, lo, hi, counter);
    case 8: return launch_tri_m<8>(plan, sms, s, lo, hi, counter);
    default:
        if (m <= kTreeMaxM || m > kMaxM) return cudaErrorInvalidValue;  // (fewer objectives need no matrix)
        return launch_tri_rt(m - 1, plan, sms, s, lo, hi, counter);
    }
}

cudaError_t launch_dominance_full_c(const float* F, int64_t n2, int64_t col_lo, int64_t col_hi, int m, uint32_t* D,
                                    int64_t ld, int32_t* cnt, int sms, cudaStream_t s)
{
    switch (m) {
#define X(MM) \
    case MM: return launch_full_m<MM>(F, n2, col_lo, col_hi, D, ld, cnt, sms, s);
        EMO_FOR_EACH_M(X)
#undef X
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace emo
