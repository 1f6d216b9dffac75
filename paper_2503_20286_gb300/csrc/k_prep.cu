// Set-up, input validation and the lexicographic ordering of the points.
//
// The points are put in lexicographic order of (f_1, ..., f_m) by a stable
// LSD radix sort (8-bit digits of the varying bits of order-preserving uint32
// keys, objective m first, objective 1 last) where the dominance matrix or the
// prefix sets are built (lex_ordered). In that order a point can only be dominated
// by points before it (Section IV-A: p dominates q implies f(p) <= f(q)
// componentwise, hence f(p) <=_lex f(q)), which is what lets the dominance
// kernel compute and store only the upper triangle of D. Runs of identical
// objective vectors (which never dominate each other) are recorded so the
// dominance kernel can clear them.
#include "emo_kernels.cuh"
#include "group_radix.cuh"

namespace emo {

// One thread per problem carves its workspace, the warps zero the scalars, a
// warp per kind splits the cooperative grid into CTA groups, and one more thread
// counts the work items.
__global__ void k_setup(SetupArgs a, SplitArgs sp, Plan* plan, char* ws)
{
    const int t = threadIdx.x;
    if (t < a.nprob) {
        ProbDev d;
        layout_problem(a.in[t], a.G, ws + a.in[t].ws_off, &d);
        plan->p[t] = d;
    }
    for (int p = t >> 5; p < a.nprob; p += blockDim.x >> 5) {  // (the scalars open the region)
        uint32_t* sc = reinterpret_cast<uint32_t*>(ws + a.in[p].ws_off);
        for (int i = t & 31; i < (int)(sizeof(Scal) / 4); i += 32) sc[i] = 0u;
    }
    // CTA groups of each kind (one warp per kind, a lane per problem): shares of
    // the grid in proportion to the work, at least one CTA for every problem that
    // the kind serves and at most the problem's cap. Wide groups by n2^2
    // (dominance tiles read per front), narrow ones by n2, tree groups by the CTA
    // time to expect: 0.13 us per point of two objectives (many fronts), 0.09 of
    // three, 0.19 of five. A tree group gets the CTAs that hold its leaves in shared memory
    // before the rest is shared out, where the grid suffices for that (38,524
    // points of two objectives: 18 us a front with the leaves in global memory,
    // 13 in shared). CTAs beyond the groups serve no problem.
    if (t < 96) {
        __shared__ int s_cnt[3][kMaxBatch];
        const GroupKind kind = (GroupKind)(t >> 5);
        const int lane = t & 31;
        int* const cnt = s_cnt[kind];
        auto weight = [&](int p) -> float {
            const ProbIn& in = a.in[p];
            const float n = (float)in.n2;
            if (kind == GRP_WIDE) return tree_ranked(in) && in.mode != MODE_HYPE ? 0.0f : n * n;
            if (kind == GRP_TREE) return tree_ranked(in) ? n * (in.m == 2 ? 3.0f : (float)max(2, in.m - 1)) : 0.0f;
            return n;
        };
        auto cap = [&](int p) { return group_cap(kind, a.in[p], a.G); };
        auto least = [&](int p, bool held) -> int {
            if (!held || kind != GRP_TREE) return 1;
            return min(cap(p), (int)cdiv(cdiv(a.in[p].n2, 32), front_local(a.in[p].m)));
        };
        int32_t* first = kind == GRP_WIDE ? plan->grp_first : (kind == GRP_TREE ? plan->grpt_first : plan->grpn_first);
        if (a.nprob == 1) {
            if (lane == 0) {
                first[0] = 0;
                first[1] = weight(0) > 0.0f ? cap(0) : 0;
            }
        } else {
            float tot = 0.0f;
            int sum = 0;  // of the least numbers
            for (int p = lane; p < a.nprob; p += 32) {
                const float w = weight(p);
                tot += w;
                if (w > 0.0f) sum += least(p, true);
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) tot += __shfl_xor_sync(0xffffffffu, tot, o);
            sum = __reduce_add_sync(0xffffffffu, sum);
            const bool held = sum <= a.G;
            // what a proportional share exceeds the least number by, scaled to a
            // little less than what is left (so that no rounding takes it above)
            const float unit = tot > 0.0f ? (float)a.G / tot : 0.0f;
            float over = 0.0f;
            sum = 0;
            for (int p = lane; p < a.nprob; p += 32) {
                const float w = weight(p);
                if (w > 0.0f) {
                    const int l = least(p, held);
                    over += fmaxf(0.0f, w * unit - l);
                    sum += l;
                }
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) over += __shfl_xor_sync(0xffffffffu, over, o);
            sum = __reduce_add_sync(0xffffffffu, sum);
            const float scale = over > 0.0f ? (float)(a.G - sum) / over * 0.9999f : 0.0f;
            int given = 0;
            for (int p = lane; p < a.nprob; p += 32) {
                const float w = weight(p);
                cnt[p] = 0;
                if (w > 0.0f) {
                    const int l = least(p, held);
                    cnt[p] = min(cap(p), l + (int)(fmaxf(0.0f, w * unit - l) * scale));
                }
                given += cnt[p];
            }
            given = __reduce_add_sync(0xffffffffu, given);
            __syncwarp();
            // the rest: one CTA each in turn to those below their cap
            for (bool grew = true; given < a.G && grew;) {
                grew = false;
                for (int p0 = 0; p0 < a.nprob && given < a.G; p0 += 32) {
                    const int p = p0 + lane;
                    const bool can = p < a.nprob && cnt[p] > 0 && cnt[p] < cap(p);
                    const unsigned ask = __ballot_sync(0xffffffffu, can);
                    if (can && __popc(ask & ((1u << lane) - 1u)) < a.G - given) cnt[p]++;
                    grew |= ask != 0u;
                    given += min(__popc(ask), a.G - given);
                }
            }
            __syncwarp();
            int acc = 0;
            for (int p0 = 0; p0 < a.nprob; p0 += 32) {
                const int p = p0 + lane, c = p < a.nprob ? cnt[p] : 0;
                int run = c;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int x = __shfl_up_sync(0xffffffffu, run, o);
                    if (lane >= o) run += x;
                }
                if (p < a.nprob) first[p] = acc + run - c;
                acc += __shfl_sync(0xffffffffu, run, 31);
            }
            if (lane == 0) first[a.nprob] = acc;
        }
    }
    if (t == 96) {
        plan->nprob = a.nprob;
        plan->G = a.G;
        plan->spin_budget = a.spin_budget;
        plan->split = sp;
        for (int i = 0; i <= kMaxM; ++i) plan->dom_ctr[i] = 0;
        for (int i = 0; i <= kMaxM; ++i) plan->asc_next[i] = 0;
        plan->status = 0;
        long long di = 0;
        for (int p = 0; p < a.nprob; ++p) {
            plan->dom_item_start[p] = di;
            if (!tree_ranked(a.in[p])) di += dom_items_of(a.in[p].n2, a.in[p].dom_chunk);
        }
        plan->dom_item_start[a.nprob] = di;
        plan->dom_items = di;
    }
}

// Validation and initialisation: as many CTAs per problem (a grid row each) as
// its items need.
__global__ void k_prep(Plan* plan)
{
    const ProbDev& d = plan->p[blockIdx.y];
    const ProbIn& in = d.in;
    const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t items = max(max(d.n2p, (int64_t)d.ncell), max((int64_t)in.n_r, 2 * (int64_t)d.nrcell));
    const int64_t ctas = min((int64_t)gridDim.x, cdiv(items, blockDim.x)), stride = ctas * blockDim.x;
    if ((int64_t)blockIdx.x >= ctas) return;
    const int64_t n2 = in.n2, m = in.m;
    bool bad = false;
    if (in.F && !lex_ordered(in)) {
        for (int64_t e = tid; e < n2 * m; e += stride) bad |= !isfinite(in.F[e]);
    } else if (in.F) {  // null only for the niching from a given association
        // finiteness, and which bits of each objective's sort key vary (a
        // radix pass over a byte that no point changes is skipped)
        uint32_t kor[kMaxM], kinv[kMaxM];
#pragma unroll
        for (int k = 0; k < kMaxM; ++k) kor[k] = kinv[k] = 0u;
        for (int64_t i = tid; i < n2; i += stride) {
#pragma unroll
            for (int k = 0; k < kMaxM; ++k) {
                if (k >= m) break;
                const float f = in.F[i * m + k];
                if (!isfinite(f)) bad = true;
                const uint32_t key = float_key(f);
                kor[k] |= key;
                kinv[k] |= ~key;
            }
        }
#pragma unroll
        for (int k = 0; k < kMaxM; ++k) {
            if (k >= m) break;
            uint32_t a = kor[k], b = kinv[k];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                a |= __shfl_xor_sync(0xffffffffu, a, o);
                b |= __shfl_xor_sync(0xffffffffu, b, o);
            }
            if ((threadIdx.x & 31) == 0) {
                if (a) atomicOr(&d.sc->kor[k], a);
                if (b) atomicOr(&d.sc->kinv[k], b);
            }
        }
    }
    for (int64_t s = tid; s < d.n2p; s += stride) {
        if (lex_ordered(in)) d.idx[s] = (int32_t)s;
        if (!d.tree) d.cnt[s] = 0;
        d.rank_s[s] = kNotRanked;
        d.flag[s] = 0;
    }
    for (int64_t c = tid; c < d.ncell; c += stride) d.zcnt[c] = 0u;
    for (int64_t c = tid; c < 2 * (int64_t)d.nrcell; c += stride) d.rcnt[c] = 0u;
    for (int64_t i = tid; i < n2; i += stride) d.rank_o[i] = kNotRanked;
    if (!d.tree) {
        for (int64_t c = tid; c < 3 * (int64_t)d.ncb; c += stride) d.front_n[c] = 0;
        for (int64_t c = tid; c < n2 + 2; c += stride) d.wcnt[c] = 0;  // front sizes of the wavefront peeling
    }
    if (lex_ordered(in))
        for (int64_t c = tid; c < d.ncb; c += stride) d.minrs[c] = INT32_MAX;
    if (in.mode == MODE_SELECT && !in.R) {
        for (int64_t j = tid; j < in.n_r; j += stride) {
            d.rho[j] = 0;
            d.lcnt[j] = 0;
        }
    } else if (in.mode == MODE_SELECT) {
        for (int64_t j = tid; j < in.n_r; j += stride) {
            double rr = 0.0;
            bool fin = true, neg = false;
            for (int k = 0; k < m; ++k) {
                float r = in.R[j * m + k];
                fin = fin && isfinite(r);
                neg = neg || r < 0.0f;
                rr += (double)r * (double)r;
            }
            if (!fin || !(rr > 0.0)) bad = true;
            if (neg) set_status(d.sc, EMO_ERR_INVALID_ARG);  // directions lie in the non-negative orthant
            double inv = fin && rr > 0.0 ? 1.0 / sqrt(rr) : 0.0;
            for (int k = 0; k < m; ++k) d.rhat[j * m + k] = (float)((double)in.R[j * m + k] * inv);
            d.rho[j] = 0;
            d.lcnt[j] = 0;
        }
    }
    if (bad) set_status(d.sc, EMO_ERR_NONFINITE);
}

// Lexicographic order, sorted objective keys and runs of equal points.
__global__ void __launch_bounds__(kCoopThreads, 1) k_sort(Plan* plan)
{
    const Group g = group_of(plan, GRP_NARROW);
    if (g.prob < 0) return;  // a CTA beyond every problem's group
    const ProbDev& d = plan->p[g.prob];
    const ProbIn& in = d.in;
    const long long budget = plan->spin_budget;
    if (ld_volatile(&d.sc->status) != 0) return;
    const int64_t n2 = in.n2;
    const int m = in.m;
    const int gs = radix_ctas(g, n2);
    const float* F = in.F;
    __shared__ RadixSmem rsm;
    if (!lex_ordered(in)) return;  // ranks given, or ranked by the z-order tree

    // Lexicographic order of (f_1, ..., f_m), ties by index. First a stable
    // radix sort by f_1; then every run of equal f_1 (almost always short for
    // continuous objectives) is put in (f_2, ..., f_m, index) order in place
    // by one thread. If some run is longer than kShortRun, the full stable
    // LSD sort over all objectives runs instead (from the index order).
    int buf = 0;
    // A stable sort by the objectives [ka, kb) takes the bits between the lowest
    // and the highest that vary over the points (k_prep), objective kb - 1
    // lowest, as one string of digits: on a grid of 64 values eight objectives
    // need 10 passes instead of 18 (100,000 points: 354 us, 517 by whole bytes).
    __shared__ uint32_t s_lo[kMaxM], s_width[kMaxM];
    __shared__ int s_at[kMaxM];
    auto sort_by = [&](int ka, int kb) -> bool {
        __syncthreads();
        int bits = 0;
        for (int k = kb - 1; k >= ka; --k) {
            const uint32_t varies = __ldcg(&d.sc->kor[k]) & __ldcg(&d.sc->kinv[k]);
            const int lo = varies ? __ffs(varies) - 1 : 0, width = varies ? 32 - __clz(varies) - lo : 0;
            if (threadIdx.x == 0) {
                s_lo[k] = lo;
                s_width[k] = width;
                s_at[k] = bits;
            }
            bits += width;
        }
        __syncthreads();
        for (int at = 0; at < bits; at += kRadixBits) {
            int k1 = kb - 1, k0 = ka;  // the objectives with bits in this digit
            while (k1 > ka && s_at[k1] + (int)s_width[k1] <= at) --k1;
            while (k0 < k1 && s_at[k0] >= at + kRadixBits) ++k0;
            const int32_t* src = d.idx + (int64_t)buf * d.n2p;
            int32_t* dst = d.idx + (int64_t)(buf ^ 1) * d.n2p;
            bool skipped = false;
            auto key = [&](int32_t v) {
                uint32_t digit = 0u;
                for (int k = k0; k <= k1; ++k) {
                    const uint32_t w = s_width[k], x = float_key(__ldg(&F[(int64_t)v * m + k])) >> s_lo[k];
                    const uint32_t val = w < 32 ? x & ((1u << w) - 1u) : x;
                    const int rel = s_at[k] - at;
                    digit |= rel >= 0 ? val << rel : val >> -rel;
                }
                return digit;
            };
            if (!radix_pass(d, g, gs, budget, n2, src, dst, 0, key, skipped, rsm)) return false;
            if (!skipped) buf ^= 1;
        }
        return true;
    };
    if (!sort_by(0, 1)) return;
    {
        constexpr int kShortRun = 32;
        int32_t* cur = d.idx + (int64_t)buf * d.n2p;
        auto key0 = [&](int64_t s) { return float_key(__ldg(&F[(int64_t)__ldcg(&cur[s]) * m])); };
        // (f_2, ..., f_m, index) order of two points
        auto before = [&](int32_t a, int32_t b) {
            for (int k = 1; k < m; ++k) {
                const uint32_t ka = float_key(__ldg(&F[(int64_t)a * m + k]));
                const uint32_t kb = float_key(__ldg(&F[(int64_t)b * m + k]));
                if (ka != kb) return ka < kb;
            }
            return a < b;
        };
        // a run's f_1 is the same at every one of its positions, so the
        // neighbours' reads below see the same keys while other threads
        // permute their own runs
        const int64_t stride = (int64_t)g.size * blockDim.x;
        for (int64_t s = (int64_t)g.rank * blockDim.x + threadIdx.x; s + 1 < n2; s += stride) {
            const uint32_t k0 = key0(s);
            if ((s > 0 && key0(s - 1) == k0) || key0(s + 1) != k0) continue;  // not the start of a run
            int64_t e = s + 2;
            while (e < n2 && e - s <= kShortRun && key0(e) == k0) ++e;
            if (e - s > kShortRun) {
                d.sc->longrun = 1;
                continue;
            }
            for (int64_t i = s + 1; i < e; ++i) {  // insertion sort, stable (reads bypass L1)
                const int32_t v = __ldcg(&cur[i]);
                int64_t j = i;
                while (j > s) {
                    const int32_t u = __ldcg(&cur[j - 1]);
                    if (!before(v, u)) break;
                    cur[j] = u;
                    --j;
                }
                cur[j] = v;
            }
        }
        if (!group_sync(g, d.sc, budget)) return;
        if (ld_volatile(&d.sc->longrun)) {  // full stable LSD sort from the index order
            int32_t* id = d.idx + (int64_t)(buf ^ 1) * d.n2p;
            for (int64_t s = (int64_t)g.rank * blockDim.x + threadIdx.x; s < n2; s += stride) id[s] = (int32_t)s;
            buf ^= 1;
            if (!group_sync(g, d.sc, budget)) return;
            if (!sort_by(0, m)) return;
        }
    }
    if (g.rank == 0 && threadIdx.x == 0) d.sc->idx_buf = buf;
    const int32_t* idx = d.idx + (int64_t)buf * d.n2p;

    // objective keys 2..m in sorted order (padding = -inf), run starts
    const int64_t chunk = cdiv(d.n2p, g.size);
    const int64_t lo = min(d.n2p, chunk * g.rank), hi = min(d.n2p, lo + chunk);
    const int mk = m - 1;
    for (int64_t s = lo + threadIdx.x; s < hi; s += blockDim.x) {
        if (s < n2) {
            const int64_t v = __ldcg(&idx[s]);
            for (int k = 1; k < m; ++k) d.keys[s * mk + k - 1] = F[v * m + k] + 0.0f;
        } else {
            for (int k = 1; k < m; ++k) d.keys[s * mk + k - 1] = -INFINITY;
        }
    }
    auto is_start = [&](int64_t s) -> bool {
        if (s == 0 || s >= n2) return true;
        const int64_t a = __ldcg(&idx[s]), b = __ldcg(&idx[s - 1]);
        for (int k = 0; k < m; ++k)
            if (F[a * m + k] != F[b * m + k]) return true;
        return false;
    };
    // inclusive max-scan of (start ? s : 0) across the group
    __shared__ int s_warp[33];
    int local = -1;
    for (int64_t s = lo + threadIdx.x; s < hi; s += blockDim.x)
        if (is_start(s)) local = max(local, (int)s);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) local = max(local, __shfl_xor_sync(0xffffffffu, local, o));
    if ((threadIdx.x & 31) == 0) s_warp[threadIdx.x >> 5] = local;
    __syncthreads();
    if (threadIdx.x == 0) {
        int mx = -1;
        for (int w = 0; w < kCoopThreads / 32; ++w) mx = max(mx, s_warp[w]);
        d.hist[g.rank] = mx;
    }
    if (!group_sync(g, d.sc, budget)) return;
    int carry = 0;  // the last run start before this CTA's share
    for (int r = threadIdx.x; r < g.rank; r += blockDim.x) carry = max(carry, __ldcg(&d.hist[r]));
    carry = __reduce_max_sync(0xffffffffu, carry);
    if ((threadIdx.x & 31) == 0) s_warp[threadIdx.x >> 5] = carry;
    __syncthreads();
    for (int w = 0; w < kCoopThreads / 32; ++w) carry = max(carry, s_warp[w]);
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int64_t base = lo; base < hi; base += blockDim.x) {
        const int64_t s = base + threadIdx.x;
        int v = (s < hi && is_start(s)) ? (int)s : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            int y = __shfl_up_sync(0xffffffffu, v, o);
            if (lane >= o) v = max(v, y);
        }
        if (lane == 31) s_warp[warp] = v;
        __syncthreads();
        int pre = carry;
        for (int w = 0; w < warp; ++w) pre = max(pre, s_warp[w]);
        int rs = max(pre, v);
        if (s < hi) {
            d.runstart[s] = rs;
            if (rs < s) atomicMin(&d.minrs[s / kColBlock], rs);
        }
        __syncthreads();
        int tmax = carry;
        for (int w = 0; w < kCoopThreads / 32; ++w) tmax = max(tmax, s_warp[w]);
        carry = tmax;
        __syncthreads();
    }
}

}  // namespace emo
