// Nondominated ranks without a dominance matrix (Section IV-A "Nondominated
// Sorting", Algorithm S.3: front k is the set of points that no unranked
// point dominates), for problems of few objectives.
//
// The paper's peel needs every bit of D (n^2 / 2 of them, written once and
// read once per ranked row). Front membership alone needs much less: a point
// stays out of front k as long as ONE unranked point that dominates it (its
// witness) is known, and a new witness is sought only when the old one has
// been ranked -- about two searches per point in all. A search is a walk over a
// two-level tree of bounding boxes:
//   * k_order puts the points in the order of the Morton (z-order) cells of a
//     grid whose lines are sample quantiles of each objective. 32 consecutive
//     points form a leaf, 32 leaves a node. Dominance never points backwards
//     along this order (p <= q in every objective puts p's cell no later).
//   * k_fronts peels. Per leaf and node: the componentwise minimum of its
//     unranked points (a leaf also holds their bit mask), kept twice, for the
//     even and the odd fronts, so that one group barrier per front is enough:
//     everyone reads the state of front k while the owners write the state of
//     front k + 1 (a node's minimum is one front behind its leaves': still a
//     lower bound, since points only leave). One warp owns a leaf, a lane a
//     point. A box can hold a dominator of q only if its minimum is <= q and
//     differs from q; the leaves that pass are compared point by point, the
//     leaf's 32 points at once against one searching point after the other.
//     Boxes are visited from the point's own leaf downwards, which finds
//     witnesses of high rank (they live long).
// Ranks do not depend on the order of any of this.
//
// Bound: latency -- a front costs one barrier (1.1 us), the state's way through
// L2 and the longest search of any warp. Measured against the tiles of the
// dominance matrix (set-up, matrix and peel): 400,000 points of three
// objectives to their 37th front 0.88 ms (3.36 ms), 20,001 points, all 46
// fronts 0.30 ms (0.43 ms), 40,000 points of five objectives 0.20 ms (0.26 ms).
// Also tried: one warp walking for all searching points of a leaf together
// (their union of boxes makes the slowest warp 2-4 times slower); the boxes of
// four nodes and the points of four leaves loaded at once (more instructions
// than latency hidden). A search that goes on where the point's last witness
// was, instead of from its own leaf, took 0.96 ms to 0.82.
#include "emo_kernels.cuh"

namespace emo {

// ------------------------------------------------------------ k_fronts
// Leaves of a CTA looked at before their searches run (a round ends with its
// longest search: 400,000 points, 82 leaves per CTA, 1.63 ms with 64, 1.44 with 128).
constexpr int kFrontRound = 128;
constexpr int kFrontQueue = kFrontRound * 32;  // searches of a round

struct FrontSmem {
    int warp[33];
    int count, base;  // new members; list base
    int qn, qnext;    // queued searches, next one
    int32_t queue[kFrontQueue];
};

__device__ __forceinline__ void front_copy16(void* dst, const void* src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}

// Peels one problem. SHARED: the leaves' state is copied to shared memory too.
template <int M, bool SHARED>
__device__ __noinline__ bool peel_tree(const ProbDev& d, const Group& g, long long budget, float* s_dyn,
                                          FrontSmem& sm)
{
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr int NW = kTreeThreads / 32;
    const int64_t n2 = d.in.n2;
    const int nleaf = d.nleaf, nnode = d.nnode, ls = d.nleafp, ns = d.nnodep;
    const int64_t zs = (int64_t)nleaf * 32;
    const int target = (int)(d.in.n_keep > 0 ? d.in.n_keep : n2);
    Scal* const sc = d.sc;
    const float* const zp = d.zpts;
    int32_t* const rank_s = d.rank_s;
    // state of one parity: nodes' minima [M][ns] | leaves' minima [M][ls] | masks [ls]
    const int64_t state_n = (int64_t)M * ns + (int64_t)(M + 1) * ls;
    const int copied = M * ns + (SHARED ? (M + 1) * ls : 0);  // floats copied to shared memory per front
    float* const zstate = d.zstate;
    const float* const s_nlo = s_dyn;
    // leaves dealt round-robin over the CTAs (neighbours search together: spread
    // them); what only their CTA reads is kept in shared memory when it fits:
    // per leaf the unranked points, those found for this front, whether the other
    // parity's state is out of date and the limit of searches; per point the
    // witness and the objectives
    const int nloc = (nleaf - g.rank + g.size - 1) / g.size;
    const bool local = nloc <= front_local(M);
    const int cap = local ? min(front_local(M), nleaf) : (int)cdiv(nleaf, g.size);
    uint32_t* const own = local ? reinterpret_cast<uint32_t*>(s_dyn + copied) : d.zlocal + (int64_t)g.rank * 4 * cap;
    uint32_t* const fresh = own + cap;
    uint32_t* const late = fresh + cap;
    int32_t* const lims = reinterpret_cast<int32_t*>(late + cap);
    int32_t* const wit = local ? lims + cap : d.zwit + g.rank * 32;
    const float* const qs = local ? reinterpret_cast<const float*>(lims + cap + cap * 32) : zp + g.rank * 32;
    const int64_t qk = local ? cap * 32 : zs;               // stride of an objective
    const int64_t qi = local ? 32 : (int64_t)g.size * 32;   // stride of a leaf (witnesses too)

    // minima of the points of `mask` (NaN when there is none: never <=)
    auto leaf_box = [&](int leaf, unsigned mask, const float (&q)[M], float* state) {
#pragma unroll
        for (int k = 0; k < M; ++k) {
            const uint32_t v = __reduce_min_sync(0xffffffffu, (mask >> lane) & 1u ? float_key(q[k]) : 0xffffffffu);
            if (lane == k) state[M * ns + k * ls + leaf] = key_float(v);
        }
        if (lane == 0) reinterpret_cast<uint32_t*>(state)[M * ns + M * ls + leaf] = mask;
    };
    // ---- the tree of all points (state 0), the limit of each leaf's searches:
    // the last leaf that starts in a cell no later than the leaf's last point
    for (int i = warp; i < nloc; i += NW) {
        const int leaf = g.rank + i * g.size;
        const int64_t s = (int64_t)leaf * 32 + lane;
        float q[M];
#pragma unroll
        for (int k = 0; k < M; ++k) {
            q[k] = s < n2 ? __ldg(&zp[k * zs + s]) : 0.0f;
            if (local) const_cast<float*>(qs)[k * qk + i * qi + lane] = q[k];
        }
        const unsigned mask = __ballot_sync(0xffffffffu, s < n2);
        leaf_box(leaf, mask, q, zstate);
        wit[i * qi + lane] = -1;
        rank_s[s] = kNotRanked;
        const uint32_t mine = __ldg(&d.zkey[min(n2, (int64_t)leaf * 32 + 32) - 1]);
        int lo = leaf, hi = nleaf - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (__ldg(&d.zkey[(int64_t)mid * 32]) <= mine) lo = mid;
            else hi = mid - 1;
        }
        if (lane == 0) {
            lims[i] = lo;
            own[i] = mask;
            fresh[i] = 0u;
            late[i] = 1u;
        }
    }
    if (!group_sync(g, sc, budget)) return false;
    auto node_box = [&](int a, const float* from, float* to) {
        const int c = a * 32 + lane;
        float l[M];
#pragma unroll
        for (int k = 0; k < M; ++k) l[k] = c < nleaf ? __ldcg(&from[M * ns + k * ls + c]) : NAN;
#pragma unroll
        for (int k = 0; k < M; ++k) {
            const uint32_t v = __reduce_min_sync(0xffffffffu, l[k] == l[k] ? float_key(l[k]) : 0xffffffffu);
            if (lane == k) to[k * ns + a] = key_float(v);
        }
    };
    const int gw = warp * g.size + g.rank, nw = g.size * NW;
    for (int a = gw; a < nnode; a += nw) node_box(a, zstate, zstate);
    if (!group_sync(g, sc, budget)) return false;

    int k_front = 0, found = 0, total = 0;  // members of the front before, points ranked
    for (;; ++k_front) {
        float* const cur = zstate + (k_front & 1) * state_n;
        float* const nxt = zstate + (~k_front & 1) * state_n;
        // ---- this front's state
        for (int i = tid * 4; i < copied; i += kTreeThreads * 4) front_copy16(s_dyn + i, cur + i);
        if (k_front > 0) found = ld_volatile(&sc->front_new[front_slot(k_front - 1)]);
        total += found;
        if (g.rank == 0 && tid == 0) sc->front_new[front_slot(k_front + 1)] = 0;
        if (tid == 0) sm.count = sm.qn = sm.qnext = 0;
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();
        if (total >= target) break;
        if ((k_front > 0 && found == 0) || k_front >= n2) {  // an empty front before the target: inconsistent
            if (tid == 0) set_status(sc, EMO_ERR_INVALID_ARG);
            return false;
        }
        // the leaves' state (in global memory: read past L1)
        const float* const llo = (SHARED ? s_dyn : cur) + M * ns;
        const uint32_t* const lmask = reinterpret_cast<const uint32_t*>(llo + M * ls);
        auto leaf_lo = [&](int k, int c) { return SHARED ? llo[k * ls + c] : __ldcg(&llo[k * ls + c]); };
        auto leaf_mask = [&](int c) { return SHARED ? lmask[c] : __ldcg(&lmask[c]); };

        for (int r0 = 0; r0 < nloc; r0 += kFrontRound) {
            const int rn = min(nloc, r0 + kFrontRound);
            if (r0 > 0) {
                __syncthreads();
                if (tid == 0) sm.qn = sm.qnext = 0;
                __syncthreads();
            }
            // ---- (A) points whose witness has gone: their own leaf, else queued
            for (int i = r0 + warp; i < rn; i += NW) {
                const unsigned mask = own[i];
                if (!mask) continue;
                const int w = (mask >> lane) & 1u ? wit[i * qi + lane] : -1;
                const bool held = w >= 0 && ((leaf_mask(w >> 5) >> (w & 31)) & 1u);
                unsigned need = __ballot_sync(0xffffffffu, ((mask >> lane) & 1u) && !held);
                if (!need) continue;
                const int leaf = g.rank + i * g.size;
                float q[M];
#pragma unroll
                for (int k = 0; k < M; ++k) q[k] = qs[k * qk + i * qi + lane];
                int wnew = -1;
                // (a witness outside the leaf: the leaf held no dominator)
                for (unsigned sub = __ballot_sync(0xffffffffu, w < 0 || w >> 5 == leaf) & need; sub;) {
                    const int j = 31 - __clz(sub);
                    sub ^= 1u << j;
                    bool le = (mask >> lane) & 1u, lt = false;
#pragma unroll
                    for (int k = 0; k < M; ++k) {
                        const float x = __shfl_sync(0xffffffffu, q[k], j);
                        le = le && q[k] <= x;
                        lt = lt || q[k] < x;
                    }
                    const unsigned dom = __ballot_sync(0xffffffffu, le && lt);
                    if (dom) {
                        need ^= 1u << j;
                        if (lane == j) wnew = leaf * 32 + 31 - __clz(dom);
                    }
                }
                if (wnew >= 0) wit[i * qi + lane] = wnew;
                if (need) {
                    int at = 0;
                    if (lane == 0) at = atomicAdd(&sm.qn, __popc(need));
                    at = __shfl_sync(0xffffffffu, at, 0);
                    if ((need >> lane) & 1u) sm.queue[at + __popc(need & lanemask_lt())] = i * 32 + lane;
                }
            }
            __syncthreads();

            // ---- (B) the queued searches, one warp each: the minima of 32 nodes,
            // of a node's 32 leaves and the 32 points of a leaf at a time; the own
            // node first, then the ones before it, then those after it
            const int qn = sm.qn;
            for (;;) {
                int at = 0;
                if (lane == 0) at = atomicAdd(&sm.qnext, 1);
                at = __shfl_sync(0xffffffffu, at, 0);
                if (at >= qn) break;
                const int item = sm.queue[at], i = item >> 5, leaf = g.rank + i * g.size;
                const int lim = lims[i], a0 = leaf >> 5, a1 = lim >> 5;
                float q[M];
#pragma unroll
                for (int k = 0; k < M; ++k) q[k] = qs[k * qk + i * qi + (item & 31)];
                // Points only leave, so what an earlier search of this point passed
                // without a find stays empty: go on at the last witness's leaf.
                const int w = wit[i * qi + (item & 31)];
                const bool fresh_start = w < 0 || w >> 5 == leaf;
                const int aw = fresh_start ? a0 : w >> 10;
                int found = -1, last = fresh_start ? lim : w >> 5;  // leaves of the first node up to here
                int b0 = aw, dir = aw > a0 ? 1 : -1, hop = 1;
                for (unsigned nodes = 1u;;) {
                    if (!nodes) {  // the next 32 nodes
                        b0 += dir * hop;
                        hop = 32;
                        last = lim;
                        if (dir < 0 && b0 < 0) {
                            dir = 1;
                            b0 = a0 + 1;
                        }
                        if (dir > 0 && b0 > a1) break;  // no dominator left
                        const int a = b0 + dir * lane;
                        bool le = a >= 0 && a <= a1;
#pragma unroll
                        for (int k = 0; k < M; ++k) le = le && s_nlo[k * ns + (le ? a : 0)] <= q[k];
                        nodes = __ballot_sync(0xffffffffu, le);
                        continue;
                    }
                    const int a = b0 + dir * (__ffs(nodes) - 1), c = a * 32 + lane;
                    nodes &= nodes - 1;
                    bool le = c <= last && c != leaf, lt = false;
#pragma unroll
                    for (int k = 0; k < M; ++k) {
                        const float l = leaf_lo(k, min(c, lim));
                        le = le && l <= q[k];
                        lt = lt || l < q[k];
                    }
                    unsigned bits = __ballot_sync(0xffffffffu, le && lt);
                    while (bits) {
                        const int t = a * 32 + 31 - __clz(bits);
                        bits ^= 1u << (t & 31);
                        // the next leaf that passes is read with it
                        const int t2 = bits ? a * 32 + 31 - __clz(bits) : t;
                        bits &= ~(1u << (t2 & 31));
                        const uint32_t m1 = leaf_mask(t), m2 = leaf_mask(t2);
                        float o1[M], o2[M];
#pragma unroll
                        for (int k = 0; k < M; ++k) {
                            o1[k] = __ldg(&zp[k * zs + t * 32 + lane]);
                            o2[k] = __ldg(&zp[k * zs + t2 * 32 + lane]);
                        }
                        bool le1 = (m1 >> lane) & 1u, lt1 = false, le2 = (m2 >> lane) & 1u, lt2 = false;
#pragma unroll
                        for (int k = 0; k < M; ++k) {
                            le1 = le1 && o1[k] <= q[k];
                            lt1 = lt1 || o1[k] < q[k];
                            le2 = le2 && o2[k] <= q[k];
                            lt2 = lt2 || o2[k] < q[k];
                        }
                        const unsigned d1 = __ballot_sync(0xffffffffu, le1 && lt1);
                        const unsigned d2 = __ballot_sync(0xffffffffu, le2 && lt2);
                        if (d1 | d2) {
                            found = d1 ? t * 32 + 31 - __clz(d1) : t2 * 32 + 31 - __clz(d2);
                            break;
                        }
                    }
                    if (found >= 0) break;
                }
                if (lane == 0) {
                    if (found >= 0) {
                        wit[i * qi + (item & 31)] = found;
                    } else {  // a member of this front
                        rank_s[leaf * 32 + (item & 31)] = k_front;
                        atomicOr(&fresh[i], 1u << (item & 31));
                        atomicAdd(&sm.count, 1);
                    }
                }
            }
        }
        __syncthreads();

        // ---- (C) the state of the next front: leaves that lost points, and
        // those whose other parity is a front behind
        if (tid == 0 && sm.count) atomicAdd(&sc->front_new[front_slot(k_front)], sm.count);
        for (int i = warp; i < nloc; i += NW) {
            const unsigned gone = *(volatile uint32_t*)&fresh[i], behind = *(volatile uint32_t*)&late[i];
            if (!(gone | behind)) continue;
            const int leaf = g.rank + i * g.size;
            const unsigned mask = own[i];
            if (gone) {
                float q[M];
#pragma unroll
                for (int k = 0; k < M; ++k) q[k] = qs[k * qk + i * qi + lane];
                leaf_box(leaf, mask & ~gone, q, nxt);
            } else {
                if (lane < M) nxt[M * ns + lane * ls + leaf] = leaf_lo(lane, leaf);
                if (lane == 0) reinterpret_cast<uint32_t*>(nxt)[M * ns + M * ls + leaf] = mask;
            }
            __syncwarp();
            if (lane == 0) {
                own[i] = mask & ~gone;
                fresh[i] = 0u;
                late[i] = gone ? 1u : 0u;
            }
        }
        for (int a = nw - 1 - gw; a < nnode; a += nw) node_box(a, cur, nxt);
        if (!group_sync(g, sc, budget)) return false;
    }
    // l, |P|, |L|
    if (g.rank == 0 && tid == 0) {
        const int l = k_front - 1;
        sc->l = l;
        sc->nP = total - found;
        sc->nL = found;
        sc->nfronts = l + 1;
        if (d.in.last_rank_out) *d.in.last_rank_out = l;
    }
    return true;
}

__global__ void __launch_bounds__(kTreeThreads, 1) k_fronts(Plan* plan)
{
    extern __shared__ __align__(16) float s_dynf[];
    __shared__ FrontSmem sm;
    const Group g = group_of(plan, GRP_TREE);
    if (g.prob < 0) return;  // a CTA beyond every problem's group
    const ProbDev& d = plan->p[g.prob];
    const long long budget = plan->spin_budget;
    if (!d.tree || ld_volatile(&d.sc->status) != 0) return;
    bool ok = false;
    switch (d.in.m) {
#define X(MM) \
    case MM: \
        ok = fronts_leaf_bytes(d.nleaf, MM) <= kFrontLeafSmem ? peel_tree<MM, true>(d, g, budget, s_dynf, sm) \
                                                              : peel_tree<MM, false>(d, g, budget, s_dynf, sm); \
        break;
        X(2) X(3) X(4) X(5)
#undef X
    }
    if (!ok) return;
    // ranks in the caller's order; the list of S (leaf by leaf, so neighbours
    // stay together)
    const int64_t n2 = d.in.n2;
    const int64_t stride = (int64_t)g.size * kTreeThreads;
    for (int64_t s0 = (int64_t)g.rank * kTreeThreads; s0 < n2; s0 += stride) {
        const int64_t s = s0 + threadIdx.x;
        int r = kNotRanked;
        int32_t v = 0;
        if (s < n2) {
            r = __ldcg(&d.rank_s[s]);
            v = __ldcg(&d.zidx[s]);
            d.rank_o[v] = r;
            if (d.in.mode == MODE_RANK && d.in.rank_out) d.in.rank_out[v] = r;
        }
        const bool inS = r != kNotRanked;
        int tot;
        const int pos = block_exclusive_scan<kTreeThreads>(inS ? 1 : 0, sm.warp, tot);
        if (threadIdx.x == 0) sm.base = tot ? atomicAdd(&d.sc->nS, tot) : 0;
        __syncthreads();
        if (inS) d.slist[sm.base + pos] = v;
        __syncthreads();
    }
}

}  // namespace emo
