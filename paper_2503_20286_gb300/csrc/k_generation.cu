// One generation around the selection: random mating, simulated binary
// crossover and polynomial mutation (Appendix S.I), the stand-in objective
// evaluation, the row gather that forms the next population, and IGD.
//
// Random numbers: Philox-4x32-10 keyed by the seed, counter (row,
// 0x80000000 | tag << 24 | slot, generation lo, generation hi); tag 1 the
// two parents of a pair (slot 0 / 1; word 1 of slot 0 decides crossover),
// tag 2 the SBX spread of a variable, tag 3 the mutation of a child's
// variable (word 0 decides, word 1 is mu). A word x is the uniform x 2^-32
// and the index (x n) >> 32.
// Arithmetic is FP64 with explicitly rounded operations in the order of the
// operator definitions; pow is CUDA's, so children can differ from another
// implementation's in the last bit of the FP64 value.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <type_traits>

#include "emo_internal.cuh"
#include "emo_launch.cuh"

namespace emo {
namespace {

constexpr int kGenThreads = 256;

__device__ __forceinline__ uint4 gen_random(uint64_t seed, uint64_t gen, int64_t row, uint32_t tag, int64_t slot)
{
    const uint4 c = make_uint4((uint32_t)row, 0x80000000u | (tag << 24) | ((uint32_t)slot & 0x00FFFFFFu),
                               (uint32_t)gen, (uint32_t)(gen >> 32));
    return philox4x32_10(c, make_uint2((uint32_t)seed, (uint32_t)(seed >> 32)));
}
__device__ __forceinline__ double unit_of(uint32_t x) { return (double)x * 2.3283064365386962890625e-10; }
__device__ __forceinline__ int64_t index_of(uint32_t x, int64_t n)
{
    return (int64_t)(((unsigned long long)x * (unsigned long long)n) >> 32);
}
__device__ __forceinline__ bool hit(uint32_t x, double p)
{
    if (p >= 1.0) return true;
    if (!(p > 0.0)) return false;
    return (double)x < p * 4294967296.0;
}
__device__ __forceinline__ double clip(double v, double lo, double hi) { return v < lo ? lo : (v > hi ? hi : v); }

// SBX of one variable: beta from mu, children 0.5[(1 +- beta) x1 + (1 -+ beta) x2].
// (One pow for both halves of mu: a warp holds both.)
__device__ __forceinline__ void sbx(double x1, double x2, double mu, double eta_c, double& c1, double& c2)
{
    const double e = __ddiv_rn(1.0, __dadd_rn(eta_c, 1.0)), mu2 = __dmul_rn(2.0, mu);
    const double beta = pow(mu <= 0.5 ? mu2 : __ddiv_rn(1.0, __dsub_rn(2.0, mu2)), e);
    const double bp = __dadd_rn(1.0, beta), bm = __dsub_rn(1.0, beta);
    c1 = __dmul_rn(0.5, __dadd_rn(__dmul_rn(bp, x1), __dmul_rn(bm, x2)));
    c2 = __dmul_rn(0.5, __dadd_rn(__dmul_rn(bm, x1), __dmul_rn(bp, x2)));
}

// Polynomial mutation of one variable (original form, eta = eta_m + 1):
// mu <= 0.5: t = 2 mu + (1 - 2 mu)(1 - (x - lo) / w)^eta, step t^(1/eta) - 1;
// otherwise:  t = 2 - 2 mu + (2 mu - 1)(1 - (hi - x) / w)^eta, step 1 - t^(1/eta).
__device__ __forceinline__ double pm(double x, double lo, double hi, double mu, double eta_m)
{
    const double eta = __dadd_rn(eta_m, 1.0);
    const double width = __dsub_rn(hi, lo);
    const double inv = __ddiv_rn(1.0, eta);
    const double mu2 = __dmul_rn(2.0, mu);
    const bool low = mu <= 0.5;
    const double delta = __ddiv_rn(low ? __dsub_rn(x, lo) : __dsub_rn(hi, x), width);
    const double q = pow(__dsub_rn(1.0, delta), eta);
    const double t = low ? __dadd_rn(mu2, __dmul_rn(__dsub_rn(1.0, mu2), q))
                         : __dadd_rn(__dsub_rn(2.0, mu2), __dmul_rn(__dsub_rn(mu2, 1.0), q));
    const double r = pow(t, inv);
    const double step = low ? __dsub_rn(r, 1.0) : __dsub_rn(1.0, r);
    return __dadd_rn(x, __dmul_rn(step, width));
}

// One thread per (pair, variable): both children of that variable. Variables
// to be mutated (one in d by default) are collected in shared memory and
// mutated by full warps: done in place, nearly every warp held one and ran both
// FP64 powers of the mutation for it, twice per child. Bound by FP64 (a pow per
// crossover and two per mutation): 500 us before, 120 with the queue (50,000
// offspring of 12 variables).
constexpr int kPmQueue = 4 * kGenThreads;

__global__ void __launch_bounds__(kGenThreads) k_variation(VariationArgs a)
{
    __shared__ double s_v[kPmQueue];      // the child's value before the mutation
    __shared__ int64_t s_at[kPmQueue];    // its place in X_off
    __shared__ uint32_t s_mu[kPmQueue];
    __shared__ int s_n;
    const int lane = threadIdx.x & 31;
    const int64_t pairs = (a.n_off + 1) / 2;
    const int64_t work = pairs * a.d;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    if (threadIdx.x == 0) s_n = 0;
    __syncthreads();
    for (int64_t e0 = (int64_t)blockIdx.x * blockDim.x; e0 < work; e0 += stride) {
        const int64_t e = e0 + threadIdx.x;
        const bool has = e < work;
        int64_t p = 0, k = 0;
        double c[2] = {0.0, 0.0}, lo = 0.0, hi = 1.0;
        if (has) {
            p = work <= INT32_MAX ? (int64_t)((uint32_t)e / (uint32_t)a.d) : e / a.d;
            k = e - p * a.d;
            const uint4 r0 = gen_random(a.seed, a.gen, p, 1u, 0), r1 = gen_random(a.seed, a.gen, p, 1u, 1);
            const int64_t pa = index_of(r0.x, a.n), pb = index_of(r1.x, a.n);
            if (k == 0 && a.parents) {
                a.parents[2 * p] = (int32_t)pa;
                a.parents[2 * p + 1] = (int32_t)pb;
            }
            const double x1 = (double)a.X[pa * a.d + k], x2 = (double)a.X[pb * a.d + k];
            if (a.lo) lo = (double)a.lo[k];
            if (a.hi) hi = (double)a.hi[k];
            c[0] = x1;
            c[1] = x2;
            if (hit(r0.y, a.p_c)) {
                const uint4 rs = gen_random(a.seed, a.gen, p, 2u, k);
                sbx(x1, x2, unit_of(rs.x), a.eta_c, c[0], c[1]);
            }
        }
#pragma unroll
        for (int child = 0; child < 2; ++child) {
            const int64_t row = child == 0 ? p : pairs + p;
            bool mutate = false;
            uint32_t mu = 0u;
            const double v = clip(c[child], lo, hi);
            if (has && row < a.n_off) {
                const uint4 rm = gen_random(a.seed, a.gen, row, 3u, k);
                // PM is defined over (x - lo) / (hi - lo): a variable without a
                // positive width (outside the contract) is left unmutated.
                mutate = hit(rm.x, a.p_m) && hi > lo;
                mu = rm.y;
                if (!mutate) a.Xoff[row * a.d + k] = (float)v;
            }
            const unsigned mask = __ballot_sync(0xffffffffu, mutate);
            if (mask) {
                int at = 0;
                if (lane == 0) at = atomicAdd(&s_n, __popc(mask));
                at = __shfl_sync(0xffffffffu, at, 0);
                if (mutate) {
                    at += __popc(mask & lanemask_lt());
                    s_v[at] = v;
                    s_at[at] = row * a.d + k;
                    s_mu[at] = mu;
                }
            }
        }
        __syncthreads();
        const int n = s_n;
        if (n > (e0 + stride < work ? kPmQueue - 2 * kGenThreads : 0)) {  // the next round may not fit
            for (int q = threadIdx.x; q < n; q += blockDim.x) {
                const int64_t at = s_at[q], kk = at % a.d;
                const double l = a.lo ? (double)a.lo[kk] : 0.0, h = a.hi ? (double)a.hi[kk] : 1.0;
                a.Xoff[at] = (float)clip(pm(s_v[q], l, h, unit_of(s_mu[q]), a.eta_m), l, h);
            }
            __syncthreads();
            if (threadIdx.x == 0) s_n = 0;
        }
        __syncthreads();
    }
}

// Stand-in objectives: g = sum_{i >= m-1} (x_i - 0.5)^2; sphere: (1 + g)
// times the unit vector of angles x_i pi/2; linear: 0.5 (1 + 100 g) times
// the stick-breaking simplex point of x_0 .. x_{m-2}.
__global__ void __launch_bounds__(kGenThreads) k_standin(const float* __restrict__ X, int64_t n, int64_t d, int m,
                                                          int shape, float* __restrict__ F)
{
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
        const float* x = X + i * d;
        double g = 0.0;
        for (int64_t v = m - 1; v < d; ++v) {
            const double t = __dsub_rn((double)x[v], 0.5);
            g = __dadd_rn(g, __dmul_rn(t, t));
        }
        double s[kMaxM];
        if (shape == EMO_SHAPE_SPHERE) {
            double prod = 1.0;
            for (int k = 0; k < m - 1; ++k) {
                const double ang = (double)x[k] * 1.5707963267948966;
                s[m - 1 - k] = __dmul_rn(prod, sin(ang));
                prod = __dmul_rn(prod, cos(ang));
            }
            s[0] = prod;
            for (int k = 0; k < m; ++k) F[i * m + k] = (float)__dmul_rn(__dadd_rn(1.0, g), s[k]);
        } else {
            double rest = 1.0;
            for (int k = 0; k < m - 1; ++k) {
                s[k] = __dmul_rn(rest, (double)x[k]);
                rest = __dmul_rn(rest, __dsub_rn(1.0, (double)x[k]));
            }
            s[m - 1] = rest;
            const double scale = __dmul_rn(0.5, __dadd_rn(1.0, __dmul_rn(100.0, g)));
            for (int k = 0; k < m; ++k) F[i * m + k] = (float)__dmul_rn(scale, s[k]);
        }
    }
}

// dst[j] = src[idx[j]] for rows of `width` floats, one warp per row.
__global__ void __launch_bounds__(kGenThreads) k_gather_rows(const float* __restrict__ src, const int32_t* idx,
                                                              int64_t rows, int64_t width, float* __restrict__ dst)
{
    const int lane = threadIdx.x & 31;
    const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t j = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); j < rows; j += warps) {
        const int64_t s = idx[j];
        for (int64_t k = lane; k < width; k += 32) dst[j * width + k] = src[s * width + k];
    }
}

// ------------------------------------------------------------------ IGD
// Squared distances are formed in float32 in one order everywhere (k
// ascending, fused multiply-add), so every route below returns the same
// minimum of every reference point.
//
// Two routes to the nearest population point of every reference point:
//   * direct: every pair (k_igd_direct). Two reference points per thread, the
//     population staged in shared memory and read as float4 (for m <= 5), and
//     the population cut into slices when there are too few reference points to
//     fill the GPU (minima combined by an atomic minimum on the float bits).
//     Bound by FP32 issue.
//   * grouped: reference points ordered by Hilbert cell and cut into groups of
//     128. A sample of the population gives an upper bound d_c of the distance
//     from a group's centre to its nearest population point; with all of the
//     group within rad of the centre, the nearest point of any of its members
//     lies within d_c + 2 rad of the centre. So each population point needs one
//     distance per GROUP (n n_ref / 128 instead of n n_ref), and only the few
//     that pass are compared with the group's members. The sample (every 8th
//     point) loosens d_c by about eight points of the distance order, which is
//     far less than what 2 rad lets in.
// Measured at n = 200,000, n_ref = 200,028, m = 3: 66.5 ms for a thread per
// reference point over every pair with runtime m (the former kernel),
// grouped 0.30 in a warm loop: near 0.22 (the groups that straddle two patches
// of the front are its tail), centre 0.034, ordering 0.05.
constexpr int kIgdGroup = 128;     // reference points per group
constexpr int kIgdGroups = 8;      // groups per block
constexpr int kIgdSample = 8;      // every kIgdSample-th point bounds d_c
constexpr int kIgdCellBits = 15;   // Hilbert cells of the ordering
constexpr int kIgdCells = 1 << kIgdCellBits;
constexpr int kIgdCand = 768;      // candidate buffer of a group
constexpr int kIgdNear = 2048;     // points near a block's groups
constexpr int kIgdStage = 128;     // candidates compared at once

// The grouped route costs about 75 us before the first comparison; the direct
// one grows with n n_ref. Measured (direct / grouped, us): n = 65,536, n_ref =
// 8,192 (5.4e8 pairs) 96 / 105 at m = 2, 131 / 117 at m = 3, 235 / 296 at m = 5,
// 1623 / 1300 at m = 8; n = n_ref = 8,192 (6.7e7 pairs) 33 / 84 at m = 3. One
// line for every m: that of m = 3, for m = 8 it would lie lower. Where the skipping
// rules nothing out (every point about equally far from a group's members) the
// grouped route loses instead: n = n_ref = 200,000, m = 3, 9.9 / 14.3 ms (9.9 /
// 0.5 near the front), n = n_ref = 50,000 0.56 / 1.00 ms (0.56 / 0.19).
constexpr int64_t kIgdMinRefs = 1024;
constexpr double kIgdMinPairs = 7e8;

struct IgdLayout {
    int64_t perm, hist, box, dcen, total;
    int64_t ngroups;
};
// best [n_ref] (float bits) | perm [n_ref] (also the partial sums) | cell
// counters | bounding box | bound of each group's centre distance.
IgdLayout igd_layout(int64_t n_ref)
{
    IgdLayout L;
    L.ngroups = (n_ref + kIgdGroup - 1) / kIgdGroup;
    L.perm = 4 * n_ref;
    L.hist = L.perm + 4 * n_ref;
    L.box = L.hist + 4 * (int64_t)kIgdCells;
    L.dcen = L.box + 4 * 2 * kMaxM;
    L.total = (L.dcen + 4 * L.ngroups + 7) / 8 * 8;
    return L;
}

__device__ __forceinline__ float igd_d2(const float* q, const float* f, int m)
{
    float s = 0.0f;
#pragma unroll
    for (int k = 0; k < m; ++k) {
        const float t = q[k] - f[k];
        s = fmaf(t, t, s);
    }
    return s;
}

__global__ void __launch_bounds__(kGenThreads) k_igd_init(uint32_t* best, int64_t n_ref, uint32_t* hist, uint32_t* box,
                                                           uint32_t* dcen, int64_t ngroups)
{
    const int64_t stride = (int64_t)gridDim.x * blockDim.x, t0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    for (int64_t i = t0; i < n_ref; i += stride) best[i] = __float_as_uint(INFINITY);
    if (!hist) return;
    for (int64_t i = t0; i < kIgdCells; i += stride) hist[i] = 0u;
    for (int64_t i = t0; i < 2 * kMaxM; i += stride) box[i] = 0xFFFFFFFFu;
    for (int64_t i = t0; i < ngroups; i += stride) dcen[i] = __float_as_uint(INFINITY);
}

// Per-coordinate minima of the order-preserving key and of its complement.
__global__ void __launch_bounds__(kGenThreads) k_igd_box(const float* __restrict__ Ref, int64_t n_ref, int m,
                                                          uint32_t* box)
{
    uint32_t lo[kMaxM], hi[kMaxM];
#pragma unroll
    for (int k = 0; k < kMaxM; ++k) lo[k] = hi[k] = 0xFFFFFFFFu;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < n_ref; r += stride) {
#pragma unroll
        for (int k = 0; k < kMaxM; ++k) {
            if (k >= m) break;
            const uint32_t key = float_key(Ref[r * m + k]);
            lo[k] = min(lo[k], key);
            hi[k] = min(hi[k], ~key);
        }
    }
#pragma unroll
    for (int k = 0; k < kMaxM; ++k) {
        if (k >= m) break;
        const uint32_t a = __reduce_min_sync(0xffffffffu, lo[k]), b = __reduce_min_sync(0xffffffffu, hi[k]);
        if ((threadIdx.x & 31) == 0) {
            atomicMin(&box[k], a);
            atomicMin(&box[kMaxM + k], b);
        }
    }
}

// Cell of a reference point on a Hilbert curve through the bounding box (the
// leading bits of its first min(m, 15) coordinates, transformed by Skilling's
// "Programming the Hilbert curve", 2004); in range for any input. Consecutive
// cells touch, so the groups stay compact: along a Morton curve some span
// distant patches of the front and let in up to 130,000 of 200,000 points
// (27,000 here; 352 and 113 on average).
struct IgdCells {
    float lo[kIgdCellBits], scale[kIgdCellBits];
    int nd, nb;
    __device__ IgdCells(const uint32_t* box, int m)
    {
        nd = min(m, kIgdCellBits);
        nb = kIgdCellBits / nd;
        for (int k = 0; k < nd; ++k) {
            lo[k] = key_float(__ldg(&box[k]));
            const float w = key_float(~__ldg(&box[kMaxM + k])) - lo[k];
            scale[k] = w > 0.0f && w < INFINITY ? (float)(1 << nb) / w : 0.0f;
        }
    }
    __device__ uint32_t cell(const float* r) const
    {
        uint32_t c[kIgdCellBits], key = 0u;
        for (int k = 0; k < nd; ++k) c[k] = (uint32_t)min(max(__float2int_rz((r[k] - lo[k]) * scale[k]), 0), (1 << nb) - 1);
        for (uint32_t q = 1u << (nb - 1); q > 1u; q >>= 1)  // undo the rotations of the coarser levels
            for (int k = 0; k < nd; ++k) {
                const uint32_t t = (c[k] & q) ? q - 1u : (c[0] ^ c[k]) & (q - 1u);
                c[0] ^= t;
                if (!(c[k] & q)) c[k] ^= t;
            }
        for (int k = 1; k < nd; ++k) c[k] ^= c[k - 1];  // Gray code
        uint32_t t = 0u;
        for (uint32_t q = 1u << (nb - 1); q > 1u; q >>= 1)
            if (c[nd - 1] & q) t ^= q - 1u;
        for (int b = nb - 1; b >= 0; --b)
            for (int k = 0; k < nd; ++k) key = key << 1 | (((c[k] ^ t) >> b) & 1u);
        return key;
    }
};

// Counts (perm null) or places (perm given, hist = running offsets) the
// reference points by cell. The order inside a cell depends on the run; it
// only changes which points share a group, never a result.
__global__ void __launch_bounds__(kGenThreads) k_igd_cells(const float* __restrict__ Ref, int64_t n_ref, int m,
                                                            const uint32_t* __restrict__ box, uint32_t* hist,
                                                            int32_t* perm)
{
    const IgdCells cells(box, m);
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < n_ref; r += stride) {
        const uint32_t pos = atomicAdd(&hist[cells.cell(Ref + r * m)], 1u);
        if (perm) perm[pos] = (int32_t)r;
    }
}

// Exclusive scan of the cell counters (one block; a warp takes 1024
// consecutive cells, 32 at a time).
__global__ void __launch_bounds__(1024) k_igd_scan(uint32_t* hist)
{
    static_assert(kIgdCells == 32 * 1024, "one warp per 1024 cells");
    __shared__ int s_warp[32];
    const int lane = threadIdx.x & 31;
    uint32_t* h = hist + (threadIdx.x >> 5) * 1024;
    int v[32], sum = 0;
#pragma unroll
    for (int e = 0; e < 32; ++e) {
        v[e] = (int)h[e * 32 + lane];
        sum += v[e];
    }
    // offset of the warp's first cell: scan of the warps' totals
    int tot, run = block_exclusive_scan<1024>(sum, s_warp, tot);
    run = __shfl_sync(0xffffffffu, run, 0);
#pragma unroll
    for (int e = 0; e < 32; ++e) {
        int x = v[e];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        h[e * 32 + lane] = (uint32_t)(run + x - v[e]);
        run += __shfl_sync(0xffffffffu, x, 31);
    }
}

// Centre and radius of each of the block's groups, one warp per group.
template <int MM>
__device__ __forceinline__ void igd_centres(const float* __restrict__ Ref, const int32_t* __restrict__ perm,
                                            int64_t n_ref, int m, float (*s_c)[kMaxM], float* s_rad)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t r0 = ((int64_t)blockIdx.x * kIgdGroups + warp) * kIgdGroup;
    const int cnt = (int)max((int64_t)0, min((int64_t)kIgdGroup, n_ref - r0));
    float lo[MM ? MM : kMaxM], hi[MM ? MM : kMaxM];
#pragma unroll
    for (int k = 0; k < (MM ? MM : kMaxM); ++k) { lo[k] = INFINITY; hi[k] = -INFINITY; }
    const int mk = MM ? MM : m;
    for (int i = lane; i < cnt; i += 32) {
        const float* r = Ref + (int64_t)perm[r0 + i] * mk;
#pragma unroll
        for (int k = 0; k < (MM ? MM : kMaxM); ++k)
            if (k < mk) { lo[k] = fminf(lo[k], r[k]); hi[k] = fmaxf(hi[k], r[k]); }
    }
    float c[MM ? MM : kMaxM];
#pragma unroll
    for (int k = 0; k < (MM ? MM : kMaxM); ++k) {
        c[k] = 0.0f;
        if (k < mk) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                lo[k] = fminf(lo[k], __shfl_xor_sync(0xffffffffu, lo[k], o));
                hi[k] = fmaxf(hi[k], __shfl_xor_sync(0xffffffffu, hi[k], o));
            }
            c[k] = 0.5f * lo[k] + 0.5f * hi[k];
            if (lane == 0) s_c[warp][k] = c[k];
        }
    }
    float r2 = 0.0f;
    for (int i = lane; i < cnt; i += 32) r2 = fmaxf(r2, igd_d2(c, Ref + (int64_t)perm[r0 + i] * mk, mk));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) r2 = fmaxf(r2, __shfl_xor_sync(0xffffffffu, r2, o));
    if (lane == 0) s_rad[warp] = sqrtf(r2);
}

// Upper bound of each group's centre distance over a sample of the points.
template <int MM>
__global__ void __launch_bounds__(kGenThreads) k_igd_centre(const float* __restrict__ F, int64_t n, int m_,
                                                             const float* __restrict__ Ref,
                                                             const int32_t* __restrict__ perm, int64_t n_ref,
                                                             int64_t ngroups, uint32_t* dcen)
{
    __shared__ float s_c[kIgdGroups][kMaxM];
    __shared__ float s_rad[kIgdGroups];
    const int m = MM ? MM : m_;
    igd_centres<MM>(Ref, perm, n_ref, m, s_c, s_rad);
    __syncthreads();
    float best[kIgdGroups];
#pragma unroll
    for (int g = 0; g < kIgdGroups; ++g) best[g] = INFINITY;
    const int64_t ns = (n + kIgdSample - 1) / kIgdSample;
    for (int64_t i = (int64_t)blockIdx.y * blockDim.x + threadIdx.x; i < ns; i += (int64_t)gridDim.y * blockDim.x) {
        float f[MM ? MM : kMaxM];
#pragma unroll
        for (int k = 0; k < (MM ? MM : kMaxM); ++k)
            if (k < m) f[k] = __ldg(&F[i * kIgdSample * m + k]);
#pragma unroll
        for (int g = 0; g < kIgdGroups; ++g) best[g] = fminf(best[g], igd_d2(s_c[g], f, m));
    }
#pragma unroll
    for (int g = 0; g < kIgdGroups; ++g) {
        const uint32_t b = __reduce_min_sync(0xffffffffu, __float_as_uint(best[g]));
        const int64_t gg = (int64_t)blockIdx.x * kIgdGroups + g;
        if ((threadIdx.x & 31) == 0 && gg < ngroups) atomicMin(&dcen[gg], b);
    }
}

// The points near each group, compared with its members. A point that cannot
// be ruled out (NaN included) is compared. The block's groups are neighbours
// in the ordering, so a first test against one ball around all of them
// (centre C, every group's limit plus its centre's distance from C) leaves
// few points for the tests of the groups.
template <int MM>
__global__ void __launch_bounds__(kGenThreads) k_igd_near(const float* __restrict__ F, int64_t n, int m_,
                                                           const float* __restrict__ Ref,
                                                           const int32_t* __restrict__ perm, int64_t n_ref,
                                                           int64_t ngroups, const uint32_t* __restrict__ dcen,
                                                           uint32_t* best)
{
    static_assert(kGenThreads == 256 && kIgdGroups == kGenThreads / 32 && kIgdGroup == 128, "thread layout");
    constexpr int MA = MM ? MM : kMaxM, PPT = 4;
    constexpr int kTile = PPT * kGenThreads;
    __shared__ float s_c[kIgdGroups][kMaxM], s_ball[kMaxM];
    __shared__ float s_rad[kIgdGroups], s_lim[kIgdGroups], s_blim;
    __shared__ int s_n[kIgdGroups], s_near_n;
    __shared__ int32_t s_near[kIgdNear];
    __shared__ int32_t s_cand[kIgdGroups][kIgdCand];
    __shared__ float s_f[kIgdStage * MA];
    const int m = MM ? MM : m_;
    const int tid = threadIdx.x, lane = tid & 31;
    igd_centres<MM>(Ref, perm, n_ref, m, s_c, s_rad);
    __syncthreads();
    const int ng = (int)min((int64_t)kIgdGroups, ngroups - (int64_t)blockIdx.x * kIgdGroups);
    if (tid < m) {
        float c = 0.0f;
        for (int g = 0; g < ng; ++g) c += s_c[g][tid];
        s_ball[tid] = c / (float)ng;
    }
    if (tid < kIgdGroups) s_n[tid] = 0;
    if (tid == 0) s_near_n = 0;
    __syncthreads();
    if (tid == 0) {
        // d_c + 2 rad, with room for the rounding of the float distances
        float ball = 0.0f;
        for (int g = 0; g < ng; ++g) {
            const float lim = (sqrtf(__uint_as_float(dcen[(int64_t)blockIdx.x * kIgdGroups + g])) + 2.0f * s_rad[g]) *
                                  (1.0f + 4e-5f) + 1e-18f;
            const float reach = (lim + sqrtf(igd_d2(s_ball, s_c[g], m))) * (1.0f + 4e-5f);
            ball = reach <= ball ? ball : reach;  // NaN: every point passes
            s_lim[g] = lim * lim;
        }
        s_blim = ball * ball;
    }
    __syncthreads();
    auto flush = [&](int g) {
        const int cnt = s_n[g];
        const int64_t r0 = ((int64_t)blockIdx.x * kIgdGroups + g) * kIgdGroup;
        const int a = tid & 63, slice = tid >> 6;
        const bool ha = r0 + a < n_ref, hb = r0 + a + 64 < n_ref;
        const int32_t ra = ha ? perm[r0 + a] : 0, rb = hb ? perm[r0 + a + 64] : 0;
        float qa[MA], qb[MA], va = INFINITY, vb = INFINITY;
#pragma unroll
        for (int k = 0; k < MA; ++k)
            if (k < m) { qa[k] = __ldg(&Ref[(int64_t)ra * m + k]); qb[k] = __ldg(&Ref[(int64_t)rb * m + k]); }
        for (int base = 0; base < cnt; base += kIgdStage) {
            const int nc = min(kIgdStage, cnt - base);
            for (int e = tid; e < nc * m; e += kGenThreads) {
                const int i = e / m;
                s_f[e] = __ldg(&F[(int64_t)s_cand[g][base + i] * m + (e - i * m)]);
            }
            __syncthreads();
            for (int i = slice; i < nc; i += kGenThreads / 64) {
                va = fminf(va, igd_d2(qa, s_f + i * m, m));
                vb = fminf(vb, igd_d2(qb, s_f + i * m, m));
            }
            __syncthreads();
        }
        if (ha) atomicMin(&best[ra], __float_as_uint(va));
        if (hb) atomicMin(&best[rb], __float_as_uint(vb));
    };
    auto append = [&](bool in, int* count, auto* list, int value) {
        const unsigned mask = __ballot_sync(0xffffffffu, in);
        if (!mask) return;
        int at = 0;
        if (lane == 0) at = atomicAdd(count, __popc(mask));
        at = __shfl_sync(0xffffffffu, at, 0);
        if (in) list[at + __popc(mask & lanemask_lt())] = (std::remove_reference_t<decltype(list[0])>)value;
    };
    const float blim = s_blim;
    for (int64_t i0 = (int64_t)blockIdx.y * kTile; i0 < n; i0 += (int64_t)gridDim.y * kTile) {
#pragma unroll
        for (int u = 0; u < PPT; ++u) {
            const int64_t id = i0 + u * kGenThreads + tid, src = id < n ? id : n - 1;
            float f[MA];
#pragma unroll
            for (int k = 0; k < MA; ++k)
                if (k < m) f[k] = __ldg(&F[src * m + k]);
            append(id < n && !(igd_d2(s_ball, f, m) > blim), &s_near_n, s_near, (int)id);
        }
        __syncthreads();
        const bool last = i0 + (int64_t)gridDim.y * kTile >= n;
        const int nn = s_near_n;
        __syncthreads();  // every warp has read the count before the next tile adds to it
        if (nn <= (last ? 0 : kIgdNear - kTile)) continue;  // room for the next tile
        for (int j0 = 0; j0 < nn; j0 += kGenThreads) {
            const int j = j0 + tid;
            const int32_t id = s_near[j < nn ? j : 0];
            float f[MA];
#pragma unroll
            for (int k = 0; k < MA; ++k)
                if (k < m) f[k] = __ldg(&F[(int64_t)id * m + k]);
            for (int g = 0; g < ng; ++g) append(j < nn && !(igd_d2(s_c[g], f, m) > s_lim[g]), &s_n[g], s_cand[g], id);
            __syncthreads();
            const bool done = last && j0 + kGenThreads >= nn;
            for (int g = 0; g < ng; ++g)
                if (s_n[g] > (done ? 0 : kIgdCand - kGenThreads)) {  // the next round may not fit
                    flush(g);
                    __syncthreads();
                    if (tid == 0) s_n[g] = 0;
                }
            __syncthreads();
        }
        if (tid == 0) s_near_n = 0;
        __syncthreads();
    }
    // (the last tile's points may all have failed the first test)
    for (int g = 0; g < ng; ++g)
        if (s_n[g] > 0) flush(g);
}

// Every pair: reference points 2 t and 2 t + 1 of a block's 256 per thread.
template <int MM>
__global__ void __launch_bounds__(128) k_igd_direct(const float* __restrict__ F, int64_t n, int m_,
                                                     const float* __restrict__ Ref, int64_t n_ref, uint32_t* best)
{
    constexpr int MA = MM ? MM : kMaxM, TILE = MM ? 1024 : 512;
    __shared__ __align__(16) float s_f[TILE * MA];
    const int m = MM ? MM : m_;
    const int tid = threadIdx.x;
    const int64_t per = ((n + gridDim.y - 1) / gridDim.y + 3) / 4 * 4;
    const int64_t lo = min(n, blockIdx.y * per), hi = min(n, lo + per);
    for (int64_t r0 = (int64_t)blockIdx.x * 256; r0 < n_ref; r0 += (int64_t)gridDim.x * 256) {
        const int64_t ra = r0 + tid, rb = ra + 128;
        float qa[MA], qb[MA], va = INFINITY, vb = INFINITY;
#pragma unroll
        for (int k = 0; k < MA; ++k)
            if (k < m) {
                qa[k] = ra < n_ref ? __ldg(&Ref[ra * m + k]) : 0.0f;
                qb[k] = rb < n_ref ? __ldg(&Ref[rb * m + k]) : 0.0f;
            }
        for (int64_t base = lo; base < hi; base += TILE) {
            const int cnt = (int)min((int64_t)TILE, hi - base), pad = (cnt + 3) / 4 * 4;
            __syncthreads();
            for (int e = tid; e < pad * m; e += 128) s_f[e] = e < cnt * m ? __ldg(&F[base * m + e]) : INFINITY;
            __syncthreads();
            if constexpr (MM > 0) {
                const float4* s4 = reinterpret_cast<const float4*>(s_f);
                for (int i = 0; i < pad / 4; ++i) {
                    float x[4 * MA];
#pragma unroll
                    for (int k = 0; k < MA; ++k) {
                        const float4 v = s4[i * MA + k];
                        x[4 * k] = v.x; x[4 * k + 1] = v.y; x[4 * k + 2] = v.z; x[4 * k + 3] = v.w;
                    }
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        va = fminf(va, igd_d2(qa, x + u * MA, MA));
                        vb = fminf(vb, igd_d2(qb, x + u * MA, MA));
                    }
                }
            } else {
                for (int i = 0; i < cnt; ++i) {
                    va = fminf(va, igd_d2(qa, s_f + i * m, m));
                    vb = fminf(vb, igd_d2(qb, s_f + i * m, m));
                }
            }
        }
        if (ra < n_ref) atomicMin(&best[ra], __float_as_uint(va));
        if (rb < n_ref) atomicMin(&best[rb], __float_as_uint(vb));
    }
}

// Sum of the distances (square roots in FP64) over a fixed split of the
// reference points: block b sums range b, the last step adds the ranges in
// order. One block alone finishes the mean itself. (One block for everything
// was bound by a single SM's FP64 rate.)
__global__ void __launch_bounds__(kGenThreads) k_igd_sum(const uint32_t* __restrict__ best, int64_t n_ref,
                                                          double* partial, double* out)
{
    __shared__ double s_w[kGenThreads / 32];
    const int64_t chunk = (n_ref + gridDim.x - 1) / gridDim.x;
    const int64_t lo = blockIdx.x * chunk, hi = min(n_ref, lo + chunk);
    double s = 0.0;
    for (int64_t r = lo + threadIdx.x; r < hi; r += blockDim.x) s += sqrt((double)__uint_as_float(best[r]));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) s_w[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < kGenThreads / 32; ++w) t += s_w[w];
        if (gridDim.x == 1) *out = t / (double)n_ref;
        else partial[blockIdx.x] = t;
    }
}
__global__ void __launch_bounds__(kGenThreads) k_igd_mean(const double* __restrict__ partial, int nparts,
                                                           int64_t n_ref, double* out)
{
    __shared__ double s_p[kGenThreads];
    double s = 0.0;
    for (int i = threadIdx.x; i < nparts; i += blockDim.x) s += partial[i];
    s_p[threadIdx.x] = s;
    __syncthreads();
    for (int o = kGenThreads / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) s_p[threadIdx.x] += s_p[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) *out = s_p[0] / (double)n_ref;
}

template <int MM>
void igd_grouped(const float* F, int64_t n, int m, const float* Ref, int64_t n_ref, char* ws, int sms, cudaStream_t s)
{
    const IgdLayout L = igd_layout(n_ref);
    uint32_t *best = (uint32_t*)ws, *hist = (uint32_t*)(ws + L.hist), *box = (uint32_t*)(ws + L.box),
             *dcen = (uint32_t*)(ws + L.dcen);
    int32_t* perm = (int32_t*)(ws + L.perm);
    const unsigned gr = (unsigned)std::max<int64_t>(1, std::min<int64_t>((n_ref + 255) / 256, 2 * sms));
    k_igd_init<<<gr, kGenThreads, 0, s>>>(best, n_ref, hist, box, dcen, L.ngroups);
    k_igd_box<<<gr, kGenThreads, 0, s>>>(Ref, n_ref, m, box);
    k_igd_cells<<<gr, kGenThreads, 0, s>>>(Ref, n_ref, m, box, hist, nullptr);
    k_igd_scan<<<1, 1024, 0, s>>>(hist);
    k_igd_cells<<<gr, kGenThreads, 0, s>>>(Ref, n_ref, m, box, hist, perm);
    const int64_t gx = (L.ngroups + kIgdGroups - 1) / kIgdGroups;
    auto slices = [&](int64_t tiles) { return (unsigned)std::max<int64_t>(1, std::min<int64_t>({tiles, 8ll * sms / gx, 65535})); };
    const dim3 gc((unsigned)gx, slices((n / kIgdSample + kGenThreads - 1) / kGenThreads));
    k_igd_centre<MM><<<gc, kGenThreads, 0, s>>>(F, n, m, Ref, perm, n_ref, L.ngroups, dcen);
    const dim3 gn((unsigned)gx, slices((n + 4 * kGenThreads - 1) / (4 * kGenThreads)));
    k_igd_near<MM><<<gn, kGenThreads, 0, s>>>(F, n, m, Ref, perm, n_ref, L.ngroups, dcen, best);
}

template <int MM>
void igd_direct(const float* F, int64_t n, int m, const float* Ref, int64_t n_ref, char* ws, int sms, cudaStream_t s)
{
    uint32_t* best = (uint32_t*)ws;
    const unsigned gr = (unsigned)std::max<int64_t>(1, std::min<int64_t>((n_ref + 255) / 256, 2 * sms));
    k_igd_init<<<gr, kGenThreads, 0, s>>>(best, n_ref, nullptr, nullptr, nullptr, 0);
    const int64_t gx = std::min<int64_t>((n_ref + 255) / 256, 1 << 20);
    // slices of at least 256 points, about eight blocks per SM
    const int64_t sl = std::max<int64_t>(1, std::min<int64_t>({(n + 255) / 256, 8ll * sms / gx, 65535}));
    k_igd_direct<MM><<<dim3((unsigned)gx, (unsigned)sl), 128, 0, s>>>(F, n, m, Ref, n_ref, best);
}

template <int MM>
void igd_nearest(bool grouped, const float* F, int64_t n, int m, const float* Ref, int64_t n_ref, char* ws, int sms,
                 cudaStream_t s)
{
    if (grouped) igd_grouped<MM>(F, n, m, Ref, n_ref, ws, sms, s);
    else igd_direct<MM>(F, n, m, Ref, n_ref, ws, sms, s);
}

unsigned grid_for(int64_t work, int per_block, int sms, int max_per_sm)
{
    const int64_t need = (work + per_block - 1) / per_block;
    return (unsigned)std::max<int64_t>(1, std::min<int64_t>(need, (int64_t)sms * max_per_sm));
}

}  // namespace

cudaError_t launch_variation(const VariationArgs& a, int sms, cudaStream_t s)
{
    const int64_t work = (a.n_off + 1) / 2 * a.d;
    k_variation<<<grid_for(work, kGenThreads, sms, 16), kGenThreads, 0, s>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_standin(const float* X, int64_t n, int64_t d, int m, int shape, float* F, int sms, cudaStream_t s)
{
    k_standin<<<grid_for(n, kGenThreads, sms, 8), kGenThreads, 0, s>>>(X, n, d, m, shape, F);
    return cudaGetLastError();
}

cudaError_t launch_gather_rows(const float* src, const int32_t* idx, int64_t rows, int64_t width, float* dst, int sms,
                               cudaStream_t s)
{
    k_gather_rows<<<grid_for(rows, kGenThreads / 32, sms, 16), kGenThreads, 0, s>>>(src, idx, rows, width, dst);
    return cudaGetLastError();
}

int64_t igd_workspace(int64_t n_ref)
{
    return n_ref < kIgdMinRefs ? n_ref * 8 : igd_layout(n_ref).total;
}

cudaError_t launch_igd(const float* F, int64_t n, int m, const float* Ref, int64_t n_ref, void* ws, int64_t ws_bytes,
                       double* out, int sms, cudaStream_t s)
{
    const bool grouped = n_ref >= kIgdMinRefs && n_ref <= INT32_MAX && n <= INT32_MAX &&
                         (double)n * (double)n_ref >= kIgdMinPairs && ws_bytes >= igd_layout(n_ref).total;
    switch (m) {
    case 2: igd_nearest<2>(grouped, F, n, m, Ref, n_ref, (char*)ws, sms, s); break;
    case 3: igd_nearest<3>(grouped, F, n, m, Ref, n_ref, (char*)ws, sms, s); break;
    case 4: igd_nearest<4>(grouped, F, n, m, Ref, n_ref, (char*)ws, sms, s); break;
    case 5: igd_nearest<5>(grouped, F, n, m, Ref, n_ref, (char*)ws, sms, s); break;
    default: igd_nearest<0>(grouped, F, n, m, Ref, n_ref, (char*)ws, sms, s);
    }
    const int parts = (int)std::min<int64_t>(512, (n_ref + 511) / 512);
    double* partial = (double*)((char*)ws + (4 * n_ref + 7) / 8 * 8);  // where perm was
    k_igd_sum<<<parts, kGenThreads, 0, s>>>((const uint32_t*)ws, n_ref, partial, out);
    if (parts > 1) k_igd_mean<<<1, kGenThreads, 0, s>>>(partial, parts, n_ref, out);
    return cudaGetLastError();
}

}  // namespace emo
