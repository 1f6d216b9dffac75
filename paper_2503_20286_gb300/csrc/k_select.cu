// Normalisation, association, niche counts, niching and survivor extraction
// (Algorithm S.1 with Algorithm S.5; Section IV-A "Normalization",
// "Association", "Niche Count Calculation", "Niche Selection").
//
// Precision: everything that decides an index is taken in the same FP64
// arithmetic, operation order and rounding as the FP64 reference statement
// of the method (no fused multiply-add: explicit __d*_rn intrinsics):
//   * ideal point z = min over S (exact in float);
//   * ASF extreme points: an FP32 pass bounds the minimum, points within the
//     FP32 error band are re-evaluated in FP64;
//   * hyperplane intercepts: Gaussian elimination with partial pivoting in
//     FP64 on one warp, a lane per row (m <= 16), nadir fallback;
//   * association: an FP32 search keeps the three smallest distances; references
//     whose distance lies within a rigorous error band of the best are
//     re-evaluated with the FP64 perpendicular distance d^2 = sum (f_k - t r_k)^2,
//     t = f.r / r.r.
#include "emo_kernels.cuh"
#include "emo_launch.cuh"
#include "cell_order.cuh"

namespace emo {

// ------------------------------------------------------------ FP64 helpers
__device__ __forceinline__ double fnorm64(float F, float z, double a)
{
    return __ddiv_rn(__dsub_rn((double)F, (double)z), a);
}

// Perpendicular distance^2 of normalised point fn[0..m) to the line of r.
__device__ inline double perp_d2(const double* fn, const float* r, int m)
{
    double rr = 0.0, fr = 0.0;
    for (int k = 0; k < m; ++k) rr = __dadd_rn(rr, __dmul_rn((double)r[k], (double)r[k]));
    for (int k = 0; k < m; ++k) fr = __dadd_rn(fr, __dmul_rn(fn[k], (double)r[k]));
    const double t = __ddiv_rn(fr, rr);
    double d2 = 0.0;
    for (int k = 0; k < m; ++k) {
        const double e = __dsub_rn(fn[k], __dmul_rn(t, (double)r[k]));
        d2 = __dadd_rn(d2, __dmul_rn(e, e));
    }
    return d2;
}

__device__ __forceinline__ unsigned long long dbits(double x) { return (unsigned long long)__double_as_longlong(x); }

// ------------------------------------------------------------ k_stats
// Ideal point, ASF extreme points, nadir point, intercepts (Algorithm S.5).
// Minima and maxima are kept per thread, reduced per warp, then per CTA; the
// FP64 elimination runs on one warp, a lane per row, every element by the
// operations of the plain loops in their order.
struct StatsSmem {
    uint32_t u[2][kMaxM];
    unsigned long long best[kMaxM];
    float z[kMaxM], lim[kMaxM];
    double A[kMaxM][kMaxM + 1], b[kMaxM];  // column m: right-hand side
    int warp[33];
};

// FP32 achievement scalarising function of axis j: max of dev_j and
// 1e6 dev_k, k != j (top: the largest 1e6 dev_k, at `arg`; second: the next).
struct AsfTop {
    float top = 0.0f, second = 0.0f;
    int arg = -1;
    __device__ __forceinline__ void add(float a, int k)
    {
        if (a > top) {
            second = top;
            top = a;
            arg = k;
        } else {
            second = fmaxf(second, a);
        }
    }
    __device__ __forceinline__ float asf(float dev, int j) const { return fmaxf(dev, j == arg ? second : top); }
};

// MM: objectives at compile time, or kMaxM for any m.
template <int MM>
__device__ __noinline__ bool stats_body(const ProbDev& d, const Group& g, long long budget, StatsSmem& sm)
{
    const ProbIn& in = d.in;
    Scal* sc = d.sc;
    const int m = MM == kMaxM ? in.m : MM, tid = threadIdx.x, lane = tid & 31;
    const int nS = ld_volatile(&sc->nS);
    const float* F = in.F;
    const int64_t stride = (int64_t)g.size * blockDim.x;
    const int64_t t0 = (int64_t)g.rank * blockDim.x + tid;

    // 1. ideal point and largest objectives (~key and key maxima; Scal is zero-initialised)
    if (tid < kMaxM) sm.u[0][tid] = sm.u[1][tid] = 0u;
    __syncthreads();
    {
        uint32_t lo[MM], hi[MM];
#pragma unroll
        for (int k = 0; k < MM; ++k) lo[k] = hi[k] = 0u;
        for (int64_t i = t0; i < nS; i += stride) {
            const int64_t v = d.slist[i];
#pragma unroll
            for (int k = 0; k < MM; ++k)
                if (k < m) {
                    const uint32_t key = float_key(F[v * m + k]);
                    lo[k] = max(lo[k], ~key);
                    hi[k] = max(hi[k], key);
                }
        }
#pragma unroll
        for (int k = 0; k < MM; ++k)
            if (k < m) {
                const uint32_t a = __reduce_max_sync(0xffffffffu, lo[k]), b = __reduce_max_sync(0xffffffffu, hi[k]);
                if (lane == 0 && b) {
                    atomicMax(&sm.u[0][k], a);
                    atomicMax(&sm.u[1][k], b);
                }
            }
    }
    __syncthreads();
    if (tid < m && sm.u[1][tid]) {
        atomicMax(&sc->zkey[tid], sm.u[0][tid]);
        atomicMax(&sc->fkey[tid], sm.u[1][tid]);
    }
    if (!group_sync(g, sc, budget)) return false;
    if (tid < m) sm.z[tid] = key_float(~__ldcg(&sc->zkey[tid]));
    if (tid < kMaxM) sm.u[0][tid] = 0u;
    __syncthreads();
    float z[MM];
#pragma unroll
    for (int k = 0; k < MM; ++k) z[k] = k < m ? sm.z[k] : 0.0f;
    auto devs = [&](int64_t v, float (&dev)[MM]) {
        AsfTop t;
#pragma unroll
        for (int k = 0; k < MM; ++k) {
            dev[k] = k < m ? F[v * m + k] - z[k] : 0.0f;
            if (k < m) t.add(dev[k] * 1.0e6f, k);
        }
        return t;
    };

    // 2. FP32 ASF minima per axis (stored as ~bits maxima)
    {
        float best[MM];
#pragma unroll
        for (int k = 0; k < MM; ++k) best[k] = INFINITY;
        for (int64_t i = t0; i < nS; i += stride) {
            float dev[MM];
            const AsfTop t = devs(d.slist[i], dev);
#pragma unroll
            for (int k = 0; k < MM; ++k) best[k] = fminf(best[k], t.asf(dev[k], k));
        }
#pragma unroll
        for (int k = 0; k < MM; ++k)
            if (k < m) {
                const uint32_t b = __reduce_max_sync(0xffffffffu, ~__float_as_uint(best[k]));
                if (lane == 0) atomicMax(&sm.u[0][k], b);
            }
    }
    __syncthreads();
    if (tid < m) atomicMax(&sc->asf32[tid], sm.u[0][tid]);
    if (!group_sync(g, sc, budget)) return false;

    // 3. exact FP64 ASF of the candidates within the FP32 error band
    if (tid < kMaxM) sm.best[tid] = 0ull;
    if (tid < m) {
        const float mn = __uint_as_float(~__ldcg(&sc->asf32[tid]));
        sm.lim[tid] = mn * (1.0f + 0x1p-18f) + 1e-30f;
    }
    __syncthreads();
    auto asf64 = [&](int64_t v, int j) {
        double mx = -INFINITY;
        for (int k = 0; k < m; ++k) {
            const double w = k == j ? 1.0 : 1e-6;
            const double t = __ddiv_rn(__dsub_rn((double)F[v * m + k], (double)sm.z[k]), w);
            if (t > mx) mx = t;
        }
        return mx;
    };
    for (int64_t i = t0; i < nS; i += stride) {
        const int64_t v = d.slist[i];
        float dev[MM];
        const AsfTop t = devs(v, dev);
#pragma unroll
        for (int k = 0; k < MM; ++k)
            if (k < m && t.asf(dev[k], k) <= sm.lim[k]) atomicMax(&sm.best[k], ~dbits(asf64(v, k)));
    }
    __syncthreads();
    if (tid < m && sm.best[tid]) atomicMax(&sc->asf64[tid], sm.best[tid]);
    if (!group_sync(g, sc, budget)) return false;

    // 4. lowest index attaining the FP64 minimum (stored as INT32_MAX - i maxima)
    if (tid < m) sm.best[tid] = ~__ldcg(&sc->asf64[tid]);
    __syncthreads();
    for (int64_t i = t0; i < nS; i += stride) {
        const int64_t v = d.slist[i];
        float dev[MM];
        const AsfTop t = devs(v, dev);
#pragma unroll
        for (int k = 0; k < MM; ++k)
            if (k < m && t.asf(dev[k], k) <= sm.lim[k] && dbits(asf64(v, k)) == sm.best[k])
                atomicMax(&sc->ext[k], INT32_MAX - (int)v);
    }
    if (!group_sync(g, sc, budget)) return false;

    // 5. intercepts by Gaussian elimination with partial pivoting (FP64)
    if (g.rank == 0 && tid < 32) {
        const int e = lane < m ? ld_volatile(&sc->ext[lane]) : 1;
        if (__any_sync(0xffffffffu, e <= 0)) {  // no candidate attained the minimum (non-finite values)
            if (lane == 0) set_status(sc, EMO_ERR_NONFINITE);
        } else {
            const int ext = INT32_MAX - e;
            double maxabs = 0.0;
            if (lane < m) {
                for (int k = 0; k < m; ++k) {
                    const double x = __dsub_rn((double)F[(int64_t)ext * m + k], (double)sm.z[k]);
                    sm.A[lane][k] = x;
                    maxabs = fmax(maxabs, fabs(x));
                }
                sm.A[lane][m] = 1.0;
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) maxabs = fmax(maxabs, __shfl_xor_sync(0xffffffffu, maxabs, o));
            __syncwarp();
            bool singular = false;
            for (int col = 0; col < m; ++col) {
                int piv = col;
                for (int r = col + 1; r < m; ++r)
                    if (fabs(sm.A[r][col]) > fabs(sm.A[piv][col])) piv = r;
                if (!(fabs(sm.A[piv][col]) > __dmul_rn(1e-12, maxabs))) {
                    singular = true;
                    break;
                }
                __syncwarp();
                if (piv != col && lane <= m) {
                    const double t = sm.A[col][lane];
                    sm.A[col][lane] = sm.A[piv][lane];
                    sm.A[piv][lane] = t;
                }
                __syncwarp();
                if (lane > col && lane < m) {
                    const double f = __ddiv_rn(sm.A[lane][col], sm.A[col][col]);
                    for (int c = col; c <= m; ++c)
                        sm.A[lane][c] = __dsub_rn(sm.A[lane][c], __dmul_rn(f, sm.A[col][c]));
                }
                __syncwarp();
            }
            double a = 1.0;
            bool fallback = singular;
            if (!singular) {
                for (int col = m - 1; col >= 0; --col) {
                    double s = sm.A[col][m];
                    for (int c = col + 1; c < m; ++c) s = __dsub_rn(s, __dmul_rn(sm.A[col][c], sm.b[c]));
                    s = __ddiv_rn(s, sm.A[col][col]);
                    __syncwarp();
                    if (lane == 0) sm.b[col] = s;
                    __syncwarp();
                }
                if (lane < m) a = __ddiv_rn(1.0, sm.b[lane]);
                fallback = __any_sync(0xffffffffu, lane < m && (!isfinite(a) || a <= 1e-10));
            }
            if (lane < m) {
                if (fallback) {  // the nadir point: the largest F_k - z_k of S
                    a = __dsub_rn((double)key_float(__ldcg(&sc->fkey[lane])), (double)sm.z[lane]);
                    if (a <= 1e-10) a = 1.0;
                }
                sc->a[lane] = a;
                sc->inv_a32[lane] = (float)__ddiv_rn(1.0, a);
                sc->z[lane] = sm.z[lane];
                sc->ext[lane] = ext;
            }
            if (lane == 0) sc->fallback = fallback;
        }
    }

    // 6. S in the order of the references' grid cells (direction of the
    // normalised point), so that the points of an association warp look at the
    // same references. Any order of S gives the same result.
    if (!group_sync(g, sc, budget)) return false;
    __shared__ DirGrid s_grid;
    if (tid < kMaxM) {
        s_grid.lo[tid] = d.rgrid->lo[tid];
        s_grid.scale[tid] = d.rgrid->scale[tid];
    }
    float ia[MM];
#pragma unroll
    for (int k = 0; k < MM; ++k) ia[k] = k < m ? __ldcg(&sc->inv_a32[k]) : 0.0f;
    __syncthreads();
    const CellSort cs{nS, d.nrcell, d.rcnt + d.nrcell, d.scell, d.sslot};
    cell_count(cs, g, [&](int64_t i) {
        const int64_t v = d.slist[i];
        float f[MM], n2 = 0.0f;
#pragma unroll
        for (int k = 0; k < MM; ++k) {
            f[k] = k < m ? (F[v * m + k] - z[k]) * ia[k] : 0.0f;
            n2 = fmaf(f[k], f[k], n2);
        }
        const float inv = rsqrtf(n2);
        return dir_cell(s_grid, m, d.rbits, [&](int k) { return f[k] * inv; });
    });
    if (!group_sync(g, sc, budget)) return false;
    cell_total(cs, g, d.hist, sm.warp);
    if (!group_sync(g, sc, budget)) return false;
    cell_offsets(cs, g, d.hist, sm.warp);
    if (!group_sync(g, sc, budget)) return false;
    cell_place(cs, g, [&](int64_t i, uint32_t, int64_t pos) { d.sord[pos] = d.slist[i]; });
    return true;
}

__global__ void __launch_bounds__(kCoopThreads, 1) k_stats(Plan* plan)
{
    __shared__ StatsSmem sm;
    const Group g = group_of(plan, GRP_NARROW);
    if (g.prob < 0) return;  // a CTA beyond every problem's group
    const ProbDev& d = plan->p[g.prob];
    if (d.in.mode != MODE_SELECT || ld_volatile(&d.sc->status) != 0) return;
    switch (d.in.m) {
    case 2: stats_body<2>(d, g, plan->spin_budget, sm); break;
    case 3: stats_body<3>(d, g, plan->spin_budget, sm); break;
    case 4: stats_body<4>(d, g, plan->spin_budget, sm); break;
    case 5: stats_body<5>(d, g, plan->spin_budget, sm); break;
    default: stats_body<kMaxM>(d, g, plan->spin_budget, sm);
    }
}

// ------------------------------------------------------------ association
// FP32 scan: the perpendicular distance is computed in the cancellation-free
// form d^2 = sum_k (f_k - g u_k)^2, g = f.u, u = r/|r| (linear in the angle
// near the optimum, so its error band is narrow). References are visited
// through the two-level tree of balls that k_order built over the unit
// directions: a warp takes neighbouring points of S (any objective count; the
// fewer points there are, the more lanes share one), finds the leaf nearest to
// their mean direction, then every leaf whose ball may hold a reference nearer
// than the best so far to one of them: |p - c| <= R + b, with p the point's
// unit direction, c and R the ball and b the chord of the best angle (plus a
// margin). A leaf's 32 references pass through shared memory.
// Bound by issue and the latency of the leaves' tests. Measured (association
// and decision together): 200,864 points on 200,028 references, m = 3, 0.27 ms
// (0.43 ms by a scan outward from each point's polar angle); 22,170 points on
// 20,475 references, m = 5, 0.23 ms (0.79 ms visiting every reference); 10,056
// on 10,011, m = 3, 53 us (92 us).
//
// Error band of the FP32 distance (relative to |f|), two evaluations:
// |delta d| <= (sqrt(m)(m + 10) + (m + 1)/2) u |f| each.
__device__ __forceinline__ float assoc_band(int m)
{
    return (2.0f * sqrtf((float)m) * (float)(m + 10) + (float)(m + 8)) * 1.05f * 0x1p-24f;
}
// Extra margin of the search: covers the rounding of the directions, balls
// and chords and keeps every unvisited reference farther than the band from
// the best.
__device__ __forceinline__ float assoc_margin(int m) { return 1e-5f + 8.0f * assoc_band(m); }

template <int M>
__device__ __forceinline__ float d2_f32(const float* f, const float* u)
{
    float g = f[0] * u[0];
#pragma unroll
    for (int k = 1; k < M; ++k) g = fmaf(f[k], u[k], g);
    float d2 = 0.0f;
#pragma unroll
    for (int k = 0; k < M; ++k) {
        const float e = fmaf(-g, u[k], f[k]);
        d2 = fmaf(e, e, d2);
    }
    return d2;
}

// The three smallest FP32 squared distances, sorted positions of the two smallest.
struct Top3 {
    float c1, c2, c3;
    int s1, s2;
    __device__ __forceinline__ void init() { c1 = c2 = c3 = INFINITY; s1 = s2 = -1; }
    __device__ __forceinline__ void add(float dd, int j)
    {
        if (dd < c3) {
            const bool b1 = dd < c1, b2 = dd < c2;
            c3 = b2 ? c2 : dd;
            s2 = b1 ? s1 : (b2 ? j : s2);
            c2 = b1 ? c1 : (b2 ? dd : c2);
            s1 = b1 ? j : s1;
            c1 = b1 ? dd : c1;
        }
    }
};

// Chord up to which references have to be visited, given the best d and |f|
// (infinite beyond an angle of pi / 4).
template <int M>
__device__ __forceinline__ float assoc_chord(float c1, float nrm)
{
    const float sn = sqrtf(c1) / nrm * 1.00001f + 2.0f * assoc_band(M);
    if (!(sn < 0.70710678f)) return INFINITY;
    const float cs = sqrtf(1.0f - sn * sn);
    return sn * sqrtf(2.0f / (1.0f + cs)) * 1.00001f + assoc_margin(M);
}

constexpr int kAssocWarps = 8;
constexpr int kAssocFill = 2432;   // warps that keep the GPU busy: 16 per SM (up to five objectives 24 fit, 2% more)
// Tasks are uneven (a warp whose points lie apart visits several times the
// leaves of another), so up to kAssocShare lanes per point there are four for
// each of those warps where the references fill more than one node; with more
// lanes per point the search itself loses (10,056 points: 16 lanes each 18 us
// longer), and a few leaves make tasks too short to split (156 references: 43 us,
// 70 with more tasks). With one task per warp 22,170 points of five objectives
// and 20,475 references kept the SMs active for half of 258 us; 247 -> 206 us,
// 200,864 points of three objectives and 200,028 references 282 -> 223 us.
constexpr int kAssocTasks = 9728;
constexpr int kAssocShare = 8;
constexpr int kAssocMany = 6;     // balls within the warp's reach from which each point is asked

template <int M>
__global__ void __launch_bounds__(kAssocWarps * 32, M <= kTreeMaxM ? 3 : 2) k_assoc(Plan* plan, int pfirst, int plast)
{
    constexpr int MP = (M + 3) / 4 * 4, V = MP / 4;
    __shared__ float4 s_u[kAssocWarps][32 * V];
    __shared__ float s_pt[kAssocWarps][M + 1][32];  // unit directions and bounds of the warp's points
    __shared__ int s_first[kMaxBatch + 1];
    __shared__ int s_share;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // lanes per point: enough tasks for the GPU, at most a warp per point;
    // tasks (warps' worth of points) before each problem
    if (tid == 0) {
        long long tot = 0;
        auto count = [&](int p) {
            const ProbDev& d = plan->p[p];
            return d.in.mode == MODE_SELECT && d.in.m == M && ld_volatile(&d.sc->status) == 0 ? ld_volatile(&d.sc->nS) : 0;
        };
        bool large = false;
        for (int p = pfirst; p < plast; ++p) {
            const int c = count(p);
            tot += c;
            large |= c > 0 && plan->p[p].nrnode > 1;
        }
        int share = 1;
        while (share < 32 && tot * share < 32ll * (large && share < kAssocShare ? kAssocTasks : kAssocFill)) share *= 2;
        int acc = 0;
        for (int p = pfirst; p < plast; ++p) {
            s_first[p - pfirst] = acc;
            acc += (int)cdiv(count(p), 32 / share);
        }
        s_first[plast - pfirst] = acc;
        s_share = share;
    }
    __syncthreads();
    const int share = s_share, ppw = 32 / share, sub = lane & (share - 1), ntask = s_first[plast - pfirst];
    float4* const su = s_u[warp];
    float (*const sp)[32] = s_pt[warp];
    // a population split over GPUs associates only its own points
    const bool ranged = plan->split.kind == SPLIT_ASSOC;
    int p = pfirst;
    for (;;) {
        int task = 0;
        if (lane == 0) task = (int)atomicAdd(&plan->asc_next[M], 1ull);
        task = __shfl_sync(0xffffffffu, task, 0);
        if (task >= ntask) break;
        while (s_first[p + 1 - pfirst] <= task) ++p;
        const ProbDev& d = plan->p[p];
        Scal* const sc = d.sc;
        const int nS = ld_volatile(&sc->nS), nr = d.in.n_r, nleaf = d.nrleaf, nnode = d.nrnode;
        const int ls = d.nrleafp, ns = d.nrnodep;
        const float* __restrict__ lball = d.rball;
        const float* __restrict__ lrad = d.rrad;
        const float* __restrict__ nball = d.rnball;
        const float* __restrict__ nrad = d.rnrad;
        const float4* __restrict__ rs = reinterpret_cast<const float4*>(d.rsort);
        const int32_t* __restrict__ ro = d.rord;
        const int64_t lo = ranged ? plan->split.col_lo : 0, hi = ranged ? plan->split.col_hi : d.in.n2;
        const int s = (task - s_first[p - pfirst]) * ppw + lane / share;
        const int64_t v = s < nS ? (int64_t)d.sord[s] : -1;
        const bool act = v >= lo && v < hi && s < nS;
        if (sub == 0 && s < nS) d.scell[s] = 0xffffffffu;  // candidates: none yet
        float f[M], n2 = 0.0f;
#pragma unroll
        for (int k = 0; k < M; ++k) {
            f[k] = act ? (d.in.F[v * M + k] - sc->z[k]) * sc->inv_a32[k] : 0.0f;
            n2 = fmaf(f[k], f[k], n2);
        }
        // next to the ideal point: scaled by a power of two (which changes no
        // angle), so that no square underflows and the error band holds
        float least = 0.0f;
        if (n2 < 0x1p-80f) {
            n2 = 0.0f;
#pragma unroll
            for (int k = 0; k < M; ++k) {
                f[k] *= 0x1p96f;
                n2 = fmaf(f[k], f[k], n2);
            }
            least = 0x1p-24f;  // (below, the rounding of denormal components counts)
        }
        const float nrm = sqrtf(n2);
        const bool bad = act && (!(nrm > least) || !isfinite(nrm));
        if (bad && sub == 0) {  // at the ideal point (or overflow): every reference in FP64
            atomicAdd(&sc->nflag, 1);
            d.flagged[atomicAdd(&sc->nbad, 1)] = (int32_t)v;
        }
        const bool seek = act && !bad;
        const unsigned seekers = __ballot_sync(0xffffffffu, seek);
        if (!seekers) continue;
        // unit directions, their mean and the ball around it
        float u[M], wc[M];
        const float inv = seek ? 1.0f / nrm : 0.0f, part = 1.0f / (float)__popc(seekers);
        float wr = 0.0f;
#pragma unroll
        for (int k = 0; k < M; ++k) {
            u[k] = f[k] * inv;
            float t = u[k];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
            wc[k] = t * part;
            const float e = u[k] - wc[k];
            wr = fmaf(e, e, wr);
        }
        __syncwarp();
#pragma unroll
        for (int k = 0; k < M; ++k) sp[k][lane] = u[k];
        wr = sqrtf(__uint_as_float(__reduce_max_sync(0xffffffffu, seek ? __float_as_uint(wr) : 0u))) * 1.00001f + 1e-6f;

        Top3 top;
        top.init();
        float chord = INFINITY, reach = INFINITY;  // the lane's bound; the warp's largest
        auto stage = [&](int t) {                  // the 32 references of leaf t into shared memory
            __syncwarp();
#pragma unroll
            for (int e = 0; e < V; ++e) su[e * 32 + lane] = __ldg(&rs[(int64_t)t * 32 * V + e * 32 + lane]);
            __syncwarp();
        };
        auto member = [&](int j, float (&r)[MP]) {
#pragma unroll
            for (int e = 0; e < V; ++e) {
                const float4 x = su[j * V + e];
                r[4 * e] = x.x; r[4 * e + 1] = x.y; r[4 * e + 2] = x.z; r[4 * e + 3] = x.w;
            }
        };
        // distance of a ball from the warp's, less both radii: at most the
        // distance of any member from any of the points
        auto gap = [&](const float* ball, const float* rad, int stride, int at) {
            float d2 = 0.0f;
#pragma unroll
            for (int k = 0; k < M; ++k) {
                const float e = __ldg(&ball[k * stride + at]) - wc[k];
                d2 = fmaf(e, e, d2);
            }
            return sqrtf(d2) * (1.0f - 1e-5f) - __ldg(&rad[at]) - wr;
        };
        auto nearest = [&](const float* ball, const float* rad, int stride, int from, int to) {  // by gap
            float bg = INFINITY;
            int bi = from;
            for (int a = from + lane; a < to; a += 32) {
                const float x = gap(ball, rad, stride, a);
                if (x < bg) { bg = x; bi = a; }
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const float og = __shfl_xor_sync(0xffffffffu, bg, o);
                const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
                if (og < bg || (og == bg && oi < bi)) { bg = og; bi = oi; }
            }
            return bi;
        };
        // whether one of the points may need ball `at` (a lane per ball, one
        // point after the other)
        auto wanted = [&](const float* ball, const float* rad, int stride, int at) {
            float c[M];
#pragma unroll
            for (int k = 0; k < M; ++k) c[k] = __ldg(&ball[k * stride + at]);
            const float r = __ldg(&rad[at]);
            bool any = false;
            for (unsigned left = seekers; left; left &= left - 1) {
                const int i = __ffs(left) - 1;
                if (i & (share - 1)) continue;
                float d2 = 0.0f;
#pragma unroll
                for (int k = 0; k < M; ++k) {
                    const float e = c[k] - sp[k][i];
                    d2 = fmaf(e, e, d2);
                }
                const float lim = r + sp[M][i];
                any = any || !(d2 > lim * lim);
            }
            return any;
        };
        const int an = nearest(nball, nrad, ns, 0, nnode);
        const int first = nearest(lball, lrad, ls, an * 32, min(nleaf, an * 32 + 32));
        // first leaf, then the nodes and leaves within reach
        int b0 = -32, a = 0;
        unsigned nodes = 0u, leaves = 0u;
        for (int t = first;;) {
            stage(t);
            const int cnt = min(32, nr - t * 32);
            for (int j = sub; j < cnt; j += share) {
                float r[MP];
                member(j, r);
                top.add(d2_f32<M>(f, r), t * 32 + j);
            }
            float c = top.c1;
            for (int o = 1; o < share; o <<= 1) c = fminf(c, __shfl_xor_sync(0xffffffffu, c, o));
            chord = seek ? assoc_chord<M>(c, nrm) : 0.0f;
            reach = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(chord)));
            sp[M][lane] = chord;
            __syncwarp();
            // the next leaf that one of the points may need
            t = -1;
            while (t < 0) {
                if (leaves) {
                    const int c0 = a * 32 + __ffs(leaves) - 1;
                    leaves &= leaves - 1;
                    if (c0 == first) continue;
                    float d2 = 0.0f;
#pragma unroll
                    for (int k = 0; k < M; ++k) {
                        const float e = __ldg(&lball[k * ls + c0]) - u[k];
                        d2 = fmaf(e, e, d2);
                    }
                    const float lim = __ldg(&lrad[c0]) + chord;
                    if (__any_sync(0xffffffffu, seek && !(d2 > lim * lim))) t = c0;
                } else if (nodes) {
                    a = b0 + __ffs(nodes) - 1;
                    nodes &= nodes - 1;
                    const int c0 = a * 32 + lane;
                    bool in = c0 < nleaf && !(gap(lball, lrad, ls, min(c0, nleaf - 1)) > reach);
                    leaves = __ballot_sync(0xffffffffu, in);
                    if (__popc(leaves) >= kAssocMany) {
                        in = in && wanted(lball, lrad, ls, min(c0, nleaf - 1));
                        leaves = __ballot_sync(0xffffffffu, in);
                    }
                } else {
                    b0 += 32;
                    if (b0 >= nnode) break;
                    const int a0 = min(b0 + lane, nnode - 1);
                    bool in = b0 + lane < nnode && !(gap(nball, nrad, ns, a0) > reach);
                    nodes = __ballot_sync(0xffffffffu, in);
                    if (__popc(nodes) >= kAssocMany) {
                        in = in && wanted(nball, nrad, ns, a0);
                        nodes = __ballot_sync(0xffffffffu, in);
                    }
                }
            }
            if (t < 0) break;
        }
        // the lanes that share a point merge their lists
        for (int o = 1; o < share; o <<= 1) {
            const float e1 = __shfl_xor_sync(0xffffffffu, top.c1, o), e2 = __shfl_xor_sync(0xffffffffu, top.c2, o),
                        e3 = __shfl_xor_sync(0xffffffffu, top.c3, o);
            const int i1 = __shfl_xor_sync(0xffffffffu, top.s1, o), i2 = __shfl_xor_sync(0xffffffffu, top.s2, o);
            top.add(e1, i1);
            top.add(e2, i2);
            top.add(e3, -1);
        }
        const float lim = sqrtf(top.c1) + assoc_band(M) * nrm;
        const bool mine = seek && sub == 0;
        const bool three = mine && sqrtf(top.c3) <= lim;  // three or more references inside the band
        if (mine && !three) {  // one or two candidates for the FP64 decision
            d.scell[s] = (uint32_t)__ldg(&ro[top.s1]);
            d.sslot[s] = top.s2 >= 0 && sqrtf(top.c2) <= lim ? (uint32_t)__ldg(&ro[top.s2]) : 0xffffffffu;
        }
        // those points, one after the other: a lane per reference, the ones
        // inside the band in FP64
        for (unsigned left = __ballot_sync(0xffffffffu, three); left; left &= left - 1) {
            const int src = __ffs(left) - 1;
            const int64_t pv = __shfl_sync(0xffffffffu, (int)v, src);
            const float plim = __shfl_sync(0xffffffffu, lim, src);
            const float pchord = __shfl_sync(0xffffffffu, assoc_chord<M>(top.c1, nrm), src);
            float pf[M], pu[M];
            double fn[M];
#pragma unroll
            for (int k = 0; k < M; ++k) {
                pf[k] = __shfl_sync(0xffffffffu, f[k], src);
                pu[k] = __shfl_sync(0xffffffffu, u[k], src);
                fn[k] = fnorm64(d.in.F[pv * M + k], sc->z[k], sc->a[k]);
            }
            double bd2 = INFINITY;
            int bj = INT32_MAX;
            auto near = [&](const float* ball, const float* rad, int stride, int at) {
                float d2 = 0.0f;
#pragma unroll
                for (int k = 0; k < M; ++k) {
                    const float e = __ldg(&ball[k * stride + at]) - pu[k];
                    d2 = fmaf(e, e, d2);
                }
                const float r = __ldg(&rad[at]) + pchord;
                return !(d2 > r * r);
            };
            for (int a0 = 0; a0 < nnode; a0 += 32) {
                unsigned an2 = __ballot_sync(0xffffffffu, a0 + lane < nnode && near(nball, nrad, ns, min(a0 + lane, nnode - 1)));
                for (; an2; an2 &= an2 - 1) {
                    const int c0 = (a0 + __ffs(an2) - 1) * 32;
                    unsigned lf = __ballot_sync(0xffffffffu, c0 + lane < nleaf && near(lball, lrad, ls, min(c0 + lane, nleaf - 1)));
                    for (; lf; lf &= lf - 1) {
                        const int t = c0 + __ffs(lf) - 1;
                        stage(t);
                        float r[MP];
                        member(lane, r);
                        if (t * 32 + lane < nr && sqrtf(d2_f32<M>(pf, r)) <= plim) {
                            const int j = __ldg(&ro[t * 32 + lane]);
                            const double d2 = perp_d2(fn, d.in.R + (int64_t)j * M, M);
                            if (d2 < bd2 || (d2 == bd2 && j < bj)) { bd2 = d2; bj = j; }
                        }
                    }
                }
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const double od = __shfl_xor_sync(0xffffffffu, bd2, o);
                const int oj = __shfl_xor_sync(0xffffffffu, bj, o);
                if (od < bd2 || (od == bd2 && oj < bj)) { bd2 = od; bj = oj; }
            }
            if (lane == 0) {
                atomicAdd(&sc->nflag, 1);
                if (bj == INT32_MAX) {  // every distance was NaN
                    set_status(sc, EMO_ERR_NONFINITE);
                    bj = 0;
                }
                d.pi[pv] = bj;
                d.d64[pv] = __dsqrt_rn(bd2);
            }
        }
    }
}

// The FP64 decision between the candidates of each point (a thread per point:
// with several lanes to a point in the search, FP64 there would run mostly
// empty warps), and the points at the ideal point or whose normalised
// objectives overflow, where a warp evaluates every reference. Bound by FP64:
// four divisions and a square root per point.
template <int MM>
__device__ __forceinline__ void decide_points(const ProbDev& d, int64_t first, int64_t stride)
{
    Scal* const sc = d.sc;
    const int m = MM == kMaxM ? d.in.m : MM;
    const int nS = ld_volatile(&sc->nS);
    double z[MM], a[MM];
#pragma unroll
    for (int k = 0; k < MM; ++k)
        if (k < m) { z[k] = (double)sc->z[k]; a[k] = sc->a[k]; }
    for (int64_t s = first; s < nS; s += stride) {
        const int j1 = (int)d.scell[s];
        if (j1 < 0) continue;  // associated by the search, or listed
        const int j2 = (int)d.sslot[s];
        const int64_t v = d.sord[s];
        double fn[MM];
#pragma unroll
        for (int k = 0; k < MM; ++k)
            if (k < m) fn[k] = __ddiv_rn(__dsub_rn((double)d.in.F[v * m + k], z[k]), a[k]);
        int bj = j1;
        double bd2 = perp_d2(fn, d.in.R + (int64_t)j1 * m, m);
        if (j2 >= 0) {
            const double d2 = perp_d2(fn, d.in.R + (int64_t)j2 * m, m);
            if (d2 < bd2 || (d2 == bd2 && j2 < bj)) { bd2 = d2; bj = j2; }
        }
        d.pi[v] = bj;
        d.d64[v] = __dsqrt_rn(bd2);
    }
}

__global__ void __launch_bounds__(256) k_decide(Plan* plan)
{
    const int lane = threadIdx.x & 31;
    const int64_t t0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, stride = (int64_t)gridDim.x * blockDim.x;
    const ProbDev& d = plan->p[blockIdx.y];
    Scal* sc = d.sc;
    if (d.in.mode != MODE_SELECT || ld_volatile(&sc->status) != 0) return;
    const int m = d.in.m, nr = d.in.n_r;
    switch (m) {
    case 2: decide_points<2>(d, t0, stride); break;
    case 3: decide_points<3>(d, t0, stride); break;
    default: decide_points<kMaxM>(d, t0, stride);
    }
    const int nbad = ld_volatile(&sc->nbad);
    for (int64_t w = t0 >> 5; w < nbad; w += stride >> 5) {
        const int64_t v = d.flagged[w];
        double fn[kMaxM];
        for (int k = 0; k < m; ++k) fn[k] = fnorm64(d.in.F[v * m + k], sc->z[k], sc->a[k]);
        double bd2 = INFINITY;
        int bj = INT32_MAX;
        for (int j = lane; j < nr; j += 32) {
            const double d2 = perp_d2(fn, d.in.R + (int64_t)j * m, m);
            if (d2 < bd2 || (d2 == bd2 && j < bj)) { bd2 = d2; bj = j; }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const double od = __shfl_xor_sync(0xffffffffu, bd2, o);
            const int oj = __shfl_xor_sync(0xffffffffu, bj, o);
            if (od < bd2 || (od == bd2 && oj < bj)) { bd2 = od; bj = oj; }
        }
        if (lane == 0) {
            if (bj == INT32_MAX) {  // every distance was NaN
                set_status(sc, EMO_ERR_NONFINITE);
                bj = 0;
            }
            d.pi[v] = bj;
            d.d64[v] = __dsqrt_rn(bd2);
        }
    }
}

// Host launcher: one instantiation per objective count.
cudaError_t launch_assoc(Plan* plan, int nprob, const int* m_of, int sms, int blocks_per_sm, cudaStream_t s)
{
    for (int p = 0; p < nprob;) {
        int q = p;
        while (q < nprob && m_of[q] == m_of[p]) ++q;
        const unsigned grid = (unsigned)sms * (unsigned)(blocks_per_sm > 0 ? blocks_per_sm : 8);
        switch (m_of[p]) {
#define X(MM) \
    case MM: k_assoc<MM><<<grid, kAssocWarps * 32, 0, s>>>(plan, p, q); break;
            X(2) X(3) X(4) X(5) X(6) X(7) X(8) X(9) X(10) X(11) X(12) X(13) X(14) X(15) X(16)
#undef X
        default: return cudaErrorInvalidValue;
        }
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        p = q;
    }
    return cudaSuccess;
}

}  // namespace emo
