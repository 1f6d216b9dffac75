// TensorMOEA/D environmental selection (Algorithm S.8) with the PBI
// aggregation of Section IV-B.
//
// The paper materialises I_new (n x n) and takes one argmin per column. Only
// the n*T (offspring, neighbour) pairs can be marked (the offspring's value
// does not exceed the neighbour's own, H(0) = 1), so a pair lowers the
// neighbour's best marked value with a 64-bit atomicMin on the bits of the
// (non-negative) double, and a second pass finds the lowest offspring index at
// that value. The column argmin of the paper then resolves per subproblem j
// without the n x n tensor:
//   * no marked pair               -> j keeps its solution;
//   * best marked value <  g_old_j -> the lowest offspring at that value;
//   * best marked value == g_old_j -> every marked value equals g_old_j, the
//     first position holding g_old_j is 0 (unmarked unless offspring 0 is
//     marked), so offspring 0 wins exactly when it is the lowest marked one.
// Each PBI value is computed in FP64 from the float32 inputs with k
// ascending and explicitly rounded operations (no contraction), so every
// decision equals that of the same arithmetic done on a CPU. What depends
// only on the subproblem -- ||w||, the unit weights w / ||w|| and the
// subproblem's own value g_old -- is computed once per subproblem, and pairs
// that a float value with its error bound rules out are not evaluated in FP64.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "emo_internal.cuh"
#include "emo_launch.cuh"

namespace emo {
namespace {

constexpr int kMoeadThreads = 256;
// From this many pairs on they are filtered in float first (one launch more):
// 20 neighbours, m = 3: 133,400 pairs 54.0 us filtered and 51.2 not, 260,820
// pairs 57.6 and 65.8.
constexpr int64_t kMoeadFilterPairs = 3 << 16;
constexpr unsigned long long kNoMark = 0x7FF0000000000000ull;  // +inf: above every PBI value

// Order-preserving map of a float to uint32 (-0 and +0 map alike).
__device__ __forceinline__ uint32_t fkey(float v)
{
    uint32_t b = __float_as_uint(v);
    if (b == 0x80000000u) b = 0u;
    return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}
__device__ __forceinline__ float fkey_inv(uint32_t k)
{
    return __uint_as_float((k & 0x80000000u) ? (k & 0x7FFFFFFFu) : ~k);
}

__device__ __forceinline__ void set_status(int32_t* st, int32_t code) { atomicCAS(st, 0, code); }

// PBI of an offspring, d1 = |(f - z).w| / ||w||, d2 = ||(f - z) - d1 w / ||w||||,
// g = d1 + theta d2, with the subproblem's ||w|| and unit weights taken from
// `sub` (k_moead_prep).
__device__ double pbi_pre(const float* __restrict__ f, const float* __restrict__ w, const double* __restrict__ sub,
                          const float* z, int m, double theta)
{
    const double nw = __ldg(sub);
    double fw = 0.0, dd = 0.0;
    for (int k = 0; k < m; ++k)
        fw = __dadd_rn(fw, __dmul_rn(__dsub_rn((double)__ldg(f + k), (double)z[k]), (double)__ldg(w + k)));
    const double d1 = __ddiv_rn(fabs(fw), nw);
    for (int k = 0; k < m; ++k) {
        const double r = __dsub_rn(__dsub_rn((double)__ldg(f + k), (double)z[k]), __dmul_rn(d1, __ldg(sub + 2 + k)));
        dd = __dadd_rn(dd, __dmul_rn(r, r));
    }
    return __dadd_rn(d1, __dmul_rn(theta, __dsqrt_rn(dd)));
}

// The same value in float, and a bound of its error: every float operation is
// off by at most u = 2^-24 of its result, the unit weights by u each, so with
// |e| = sum |f_k - z_k|: |delta d1| <= (m + 3) u |e|, and each component of
// (f - z) - d1 w / ||w|| is off by at most (m + 6) u |e|, their norm by sqrt(m)
// times that plus (m + 2) u |e| from its own sum and root; a quarter on top. Squares that underflow
// take at most sqrt(16 2^-149) = 1.5e-22 off the norm. (Overflow, of a square or of the penalty, gives
// inf or NaN: the pair is then decided in FP64.)
template <int MM>
__device__ __forceinline__ void pbi_float(const float* __restrict__ f, const float* __restrict__ wh, const float* z, int m,
                                          float theta, float& g, float& err)
{
    float e[MM], d1 = 0.0f, sum = 0.0f, dd = 0.0f;
#pragma unroll
    for (int k = 0; k < MM; ++k)
        if (k < m) {
            e[k] = f[k] - z[k];
            d1 = fmaf(e[k], wh[k], d1);
            sum += fabsf(e[k]);
        }
    d1 = fabsf(d1);
#pragma unroll
    for (int k = 0; k < MM; ++k)
        if (k < m) {
            const float r = fmaf(-d1, wh[k], e[k]);
            dd = fmaf(r, r, dd);
        }
    g = fmaf(theta, sqrtf(dd), d1);
    const float fm = (float)m;
    err = sum * 1.25f * 0x1p-24f * (fm + 5.0f + theta * (sqrtf(fm) * (fm + 6.0f) + 0.5f * fm + 4.0f)) + 1e-30f +
          theta * 2e-22f;
}

__device__ __forceinline__ void load_zmin(const uint32_t* zkey, int m, float* z)
{
    for (int k = 0; k < m; ++k) z[k] = fkey_inv(zkey[k]);
}

__global__ void __launch_bounds__(kMoeadThreads) k_moead_init(MoeadArgs a)
{
    const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t j = tid; j < a.n; j += stride) {
        a.gmin[j] = kNoMark;
        a.tie[j] = INT32_MAX;
    }
    if (tid == 0) {
        *a.status = 0;
        *a.nexact = 0ull;
    }
    if (tid < a.m) {
        const float zk = a.z[tid];
        if (!isfinite(zk)) set_status(a.status, EMO_ERR_NONFINITE);
        a.zkey[tid] = fkey(zk);
    }
}

// z_min = min(z, column minima of F2); F2 must be finite.
__global__ void __launch_bounds__(kMoeadThreads) k_moead_zmin(MoeadArgs a)
{
    uint32_t lk[kMaxM];
    for (int k = 0; k < kMaxM; ++k) lk[k] = 0xFFFFFFFFu;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    bool bad = false;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < a.n; i += stride)
        for (int k = 0; k < a.m; ++k) {
            const float v = __ldg(a.F2 + i * a.m + k);
            bad |= !isfinite(v);
            lk[k] = min(lk[k], fkey(v));
        }
    if (bad) set_status(a.status, EMO_ERR_NONFINITE);
    const int lane = threadIdx.x & 31;
    for (int k = 0; k < a.m; ++k) {
        const uint32_t v = __reduce_min_sync(0xFFFFFFFFu, lk[k]);
        if (lane == 0 && v != 0xFFFFFFFFu) atomicMin(a.zkey + k, v);
    }
}

// Per subproblem j: sub[j] = (||w_j||, g_old_j = PBI(F1_j | w_j, z_min),
// w_j0 / ||w_j||, ..., w_j,m-1 / ||w_j||), in the operation order of pbi_pre(),
// and the float record of the filter: the unit weights and g_old rounded up.
// F1 and W must be finite, W non-zero.
__global__ void __launch_bounds__(kMoeadThreads) k_moead_prep(MoeadArgs a)
{
    float z[kMaxM];
    load_zmin(a.zkey, a.m, z);
    const int mp = moead_rec(a.m);
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < a.n; j += stride) {
        const float* w = a.W + j * a.m;
        const float* f = a.F1 + j * a.m;
        double* sub = a.sub + j * (a.m + 2);
        float* rec = a.rec + j * mp;
        double ww = 0.0, fw = 0.0, dd = 0.0;
        bool bad = false;
        for (int k = 0; k < a.m; ++k) {
            const float wv = __ldg(w + k), fv = __ldg(f + k);
            bad |= !isfinite(wv) || !isfinite(fv);
            const double wk = (double)wv;
            ww = __dadd_rn(ww, __dmul_rn(wk, wk));
            fw = __dadd_rn(fw, __dmul_rn(__dsub_rn((double)fv, (double)z[k]), wk));
        }
        if (bad || !(ww > 0.0)) set_status(a.status, EMO_ERR_NONFINITE);
        const double nw = __dsqrt_rn(ww);
        sub[0] = nw;
        const double d1 = __ddiv_rn(fabs(fw), nw);
        for (int k = 0; k < a.m; ++k) {
            const double wh = __ddiv_rn((double)__ldg(w + k), nw);
            sub[2 + k] = wh;
            if (a.rec) rec[k] = (float)wh;
            const double r = __dsub_rn(__dsub_rn((double)__ldg(f + k), (double)z[k]), __dmul_rn(d1, wh));
            dd = __dadd_rn(dd, __dmul_rn(r, r));
        }
        const double g = __dadd_rn(d1, __dmul_rn(a.theta, __dsqrt_rn(dd)));
        sub[1] = g;
        if (a.rec) rec[a.m] = __double2float_ru(g);
    }
}

// The pairs (offspring i, neighbour slot t) in float. An offspring can lower
// subproblem j only if its value does not exceed g_old_j, and can be the one
// that j takes only if no other's upper bound lies below its lower bound; so
// the first pass lowers gmin[j] to the least upper bound of j's offspring, the
// second lists the pairs whose lower bound does not exceed it -- one or two per
// subproblem instead of T -- and k_moead_exact decides those in FP64, a full
// warp at a time; those that mark j lower gmin[j] to their exact value. (With
// any mark gmin ends at the least
// marked value: an offspring that does not mark lies above g_old, so above it.
// A neighbour listed twice marks with the same value and offspring: no effect.)
// Both passes are bound by the gather of the neighbours' records; FP64 for
// every pair took 455 us at 200,028 subproblems, T = 20, m = 3 (with a search
// for repeated neighbours before each), the two passes and the exact pairs 96 us;
// the whole selection went from 676 to 205 us.
template <int MM, bool LIST>
__global__ void __launch_bounds__(kMoeadThreads) k_moead_pairs(MoeadArgs a)
{
    const int m = MM == kMaxM ? a.m : MM, mp = moead_rec(m);
    float z[MM];
#pragma unroll
    for (int k = 0; k < MM; ++k)
        if (k < m) z[k] = fkey_inv(a.zkey[k]);
    const float theta = (float)a.theta;
    const int64_t pairs = a.n * (int64_t)a.T;  // below 2^32 - 1 on this route
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t p0 = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); p0 < pairs; p0 += stride) {
        const int64_t p = p0 + (threadIdx.x & 31);
        bool exact = false;
        int64_t i = 0;
        int32_t j = 0;
        if (p < pairs) {
            i = (int64_t)((uint32_t)p / (uint32_t)a.T);
            j = __ldg(a.I_nb + p);
            if (j < 0 || j >= a.n) {
                if (!LIST) set_status(a.status, EMO_ERR_INVALID_ARG);
            } else {
                float f[MM], r[MM + 1], g, err;
                const float* rec = a.rec + (int64_t)j * mp;
#pragma unroll
                for (int k = 0; k < MM; ++k)
                    if (k < m) f[k] = __ldg(a.F2 + i * m + k);
                if constexpr (MM <= 3) {
                    const float4 x = __ldg(reinterpret_cast<const float4*>(rec));
                    r[0] = x.x;
                    r[1] = x.y;
                    r[2] = x.z;
                    if constexpr (MM == 3) r[3] = x.w;
                } else {
#pragma unroll
                    for (int k = 0; k < MM; ++k)
                        if (k < m) r[k] = __ldg(rec + k);
                    r[MM] = __ldg(rec + m);
                }
                pbi_float<MM>(f, r, z, m, theta, g, err);
                const float low = g < INFINITY ? g - err : -INFINITY;  // (-inf, NaN: undecided)
                if (!(low > r[MM])) {
                    if (LIST)
                        exact = !((double)low > __longlong_as_double((long long)__ldcg(a.gmin + j)));
                    else if (g + err < INFINITY)
                        atomicMin(a.gmin + j, (unsigned long long)__double_as_longlong((double)(g + err)));
                }
            }
        }
        if (LIST) {
            const unsigned mask = __ballot_sync(0xffffffffu, exact);
            if (mask) {
                unsigned long long at = 0;
                if ((threadIdx.x & 31) == 0) at = atomicAdd(a.nexact, (unsigned long long)__popc(mask));
                at = __shfl_sync(0xffffffffu, at, 0);
                if (exact) a.exact[at + __popc(mask & lanemask_lt())] = (uint32_t)p;
            }
        }
    }
}

// The listed pairs in FP64; the ones that do not mark their subproblem leave
// the list.
__global__ void __launch_bounds__(kMoeadThreads) k_moead_exact(MoeadArgs a)
{
    float z[kMaxM];
    load_zmin(a.zkey, a.m, z);
    const int64_t listed = (int64_t)*a.nexact;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < listed; e += stride) {
        const int64_t p = a.exact[e], i = p / a.T;
        const int32_t j = __ldg(a.I_nb + p);
        const double* sub = a.sub + (int64_t)j * (a.m + 2);
        const double g = pbi_pre(a.F2 + i * a.m, a.W + (int64_t)j * a.m, sub, z, a.m, a.theta);
        if (__dsub_rn(__ldg(sub + 1), g) >= 0.0) atomicMin(a.gmin + j, (unsigned long long)__double_as_longlong(g));
        else a.exact[e] = UINT32_MAX;
    }
}

// The lowest offspring index whose marked value equals gmin[j], over the
// listed pairs (their values again: the same operations, the same bits).
__global__ void __launch_bounds__(kMoeadThreads) k_moead_tie(MoeadArgs a)
{
    float z[kMaxM];
    load_zmin(a.zkey, a.m, z);
    const int64_t listed = (int64_t)*a.nexact;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < listed; e += stride) {
        const int64_t p = a.exact[e], i = p / a.T;
        if (p == UINT32_MAX) continue;
        const int32_t j = __ldg(a.I_nb + p);
        const double g = pbi_pre(a.F2 + i * a.m, a.W + (int64_t)j * a.m, a.sub + (int64_t)j * (a.m + 2), z, a.m, a.theta);
        if ((unsigned long long)__double_as_longlong(g) == a.gmin[j]) atomicMin(a.tie + j, (int32_t)i);
    }
}

// Few pairs, or no room for the float records beside the list (fewer neighbours
// than floats of a record, or 2^32 pairs): FP64 for every pair, the marked value
// kept per pair, -1 when unmarked.
__global__ void __launch_bounds__(kMoeadThreads) k_moead_compare(MoeadArgs a)
{
    float z[kMaxM];
    load_zmin(a.zkey, a.m, z);
    const int64_t pairs = a.n * (int64_t)a.T;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < pairs; p += stride) {
        const int64_t i = p / a.T;
        const int32_t j = __ldg(a.I_nb + p);
        double g = -1.0;
        if (j < 0 || j >= a.n) {
            set_status(a.status, EMO_ERR_INVALID_ARG);
        } else {
            const double* sub = a.sub + (int64_t)j * (a.m + 2);
            const double g_new = pbi_pre(a.F2 + i * a.m, a.W + (int64_t)j * a.m, sub, z, a.m, a.theta);
            if (__dsub_rn(__ldg(sub + 1), g_new) >= 0.0) {
                g = g_new;
                atomicMin(a.gmin + j, (unsigned long long)__double_as_longlong(g_new));
            }
        }
        a.gpair[p] = g;
    }
}
__global__ void __launch_bounds__(kMoeadThreads) k_moead_tie_all(MoeadArgs a)
{
    const int64_t pairs = a.n * (int64_t)a.T;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < pairs; p += stride) {
        const double g = a.gpair[p];
        if (!(g >= 0.0)) continue;
        const int32_t j = __ldg(a.I_nb + p);
        if ((unsigned long long)__double_as_longlong(g) == a.gmin[j]) atomicMin(a.tie + j, (int32_t)(p / a.T));
    }
}

// The offspring that subproblem j takes, -1 when it keeps its solution.
__device__ __forceinline__ int32_t moead_winner(const MoeadArgs& a, int64_t j)
{
    const int32_t tie = a.tie[j];
    if (tie == INT32_MAX) return -1;  // no marked pair
    const double g_old = a.sub[j * (a.m + 2) + 1], best = __longlong_as_double((long long)a.gmin[j]);
    return best < g_old ? tie : (tie == 0 ? 0 : -1);
}

// Rows of X or O and of F1 or F2: one thread per element (a warp per row of 12
// floats left 20 lanes idle: 102 us at 200,028 subproblems). Each element is
// read and written by one thread, so X_next may be X and F_next may be F1.
__global__ void __launch_bounds__(kMoeadThreads) k_moead_gather(MoeadArgs a)
{
    const int64_t w = a.d + a.m, total = a.n * w;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    if (blockIdx.x == 0) {  // z_min and the status, final since the pairs were decided
        if (threadIdx.x < a.m) a.z[threadIdx.x] = fkey_inv(a.zkey[threadIdx.x]);
        if (threadIdx.x == 0) {
            const int32_t st = *a.status;
            if (a.status_out) *a.status_out = st;
            if (st != 0) atomicCAS(a.sticky, 0, st);
        }
    }
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += stride) {
        const int64_t j = total <= INT32_MAX ? (int64_t)((uint32_t)e / (uint32_t)w) : e / w, k = e - j * w;
        const int32_t win = moead_winner(a, j);
        if (k < a.d) {
            a.X_next[j * a.d + k] = win >= 0 ? a.O[(int64_t)win * a.d + k] : a.X[j * a.d + k];
        } else {
            const int64_t q = k - a.d;
            a.F_next[j * a.m + q] = win >= 0 ? a.F2[(int64_t)win * a.m + q] : a.F1[j * a.m + q];
            if (q == 0 && a.winner) a.winner[j] = win;
        }
    }
}

}  // namespace

int64_t moead_layout(int64_t n, int32_t m, int32_t T, char* ws, MoeadArgs* a)
{
    auto up = [](int64_t b) { return (b + 255) / 256 * 256; };
    const int64_t off_gmin = 256;                       // status word at 0, list length at 8, z_min keys at 64
    const int64_t off_tie = up(off_gmin + 8 * n);
    const int64_t off_pair = up(off_tie + 4 * n);
    const int64_t off_sub = up(off_pair + 8 * n * (int64_t)T);
    const int64_t total = up(off_sub + 8 * n * (int64_t)(m + 2));
    if (ws && a) {
        a->status = (int32_t*)ws;
        a->nexact = (unsigned long long*)(ws + 8);
        a->zkey = (uint32_t*)(ws + 64);
        a->gmin = (unsigned long long*)(ws + off_gmin);
        a->tie = (int32_t*)(ws + off_tie);
        a->gpair = (double*)(ws + off_pair);
        a->sub = (double*)(ws + off_sub);
        // the pair region holds the list and the records, or every pair's value
        const int64_t list = (4 * n * (int64_t)T + 15) / 16 * 16;
        const bool fits = list + 4 * n * moead_rec(m) <= 8 * n * (int64_t)T && n * (int64_t)T < UINT32_MAX &&
                          n * (int64_t)T >= kMoeadFilterPairs;
        a->exact = fits ? (uint32_t*)(ws + off_pair) : nullptr;
        a->rec = fits ? (float*)(ws + off_pair + list) : nullptr;
    }
    return total;
}

namespace {
template <int MM>
void moead_pairs(const MoeadArgs& a, unsigned grid, cudaStream_t s)
{
    k_moead_pairs<MM, false><<<grid, kMoeadThreads, 0, s>>>(a);
    k_moead_pairs<MM, true><<<grid, kMoeadThreads, 0, s>>>(a);
}
}  // namespace

cudaError_t launch_moead_select(const MoeadArgs& a, int sms, cudaStream_t s)
{
    auto grid_for = [&](int64_t work, int per_block, int max_per_sm) {
        const int64_t need = (work + per_block - 1) / per_block;
        return (unsigned)std::max<int64_t>(1, std::min<int64_t>(need, (int64_t)sms * max_per_sm));
    };
    const int64_t pairs = a.n * (int64_t)a.T;
    k_moead_init<<<grid_for(a.n, kMoeadThreads, 8), kMoeadThreads, 0, s>>>(a);
    k_moead_zmin<<<grid_for(a.n, kMoeadThreads, 4), kMoeadThreads, 0, s>>>(a);
    k_moead_prep<<<grid_for(a.n, kMoeadThreads, 8), kMoeadThreads, 0, s>>>(a);
    const unsigned gp = grid_for(pairs, kMoeadThreads, 16);
    if (a.rec) {
        switch (a.m) {
        case 2: moead_pairs<2>(a, gp, s); break;
        case 3: moead_pairs<3>(a, gp, s); break;
        default: moead_pairs<kMaxM>(a, gp, s);
        }
        k_moead_exact<<<grid_for(2 * a.n, kMoeadThreads, 8), kMoeadThreads, 0, s>>>(a);
        k_moead_tie<<<grid_for(2 * a.n, kMoeadThreads, 8), kMoeadThreads, 0, s>>>(a);
    } else {
        k_moead_compare<<<gp, kMoeadThreads, 0, s>>>(a);
        k_moead_tie_all<<<gp, kMoeadThreads, 0, s>>>(a);
    }
    k_moead_gather<<<grid_for(a.n * (a.d + a.m), kMoeadThreads, 16), kMoeadThreads, 0, s>>>(a);
    return cudaGetLastError();
}

}  // namespace emo
