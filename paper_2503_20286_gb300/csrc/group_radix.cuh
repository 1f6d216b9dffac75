// Group-wide stable LSD radix pass shared by the ordering and CSR stages.
#pragma once

#include "emo_kernels.cuh"

namespace emo {

// ------------------------------------------------ group-wide stable radix sort
// One LSD pass over idx_src[0..n) -> idx_dst, digit = (key(v) >> shift) & 255.
// Returns false when the group failed. Sets `skipped` when every element has
// the same digit (the pass would not move anything).
// Shared-memory scratch of radix_pass; declared once by the calling kernel
// (a function-scope __shared__ array in a template would be duplicated per
// key function).
struct RadixSmem {
    int hist[kRadix];
    int off[kRadix];
    int wc[kCoopThreads / 32][kRadix];
    int tot[kRadix / 32];
    int skip;
};

// CTAs that a pass over n items is spread over.
// (100,000 points of eight objectives: 1,533 us with 2,048, 1,499 with 1,024)
constexpr int kRadixItems = 1024;
__device__ __forceinline__ int radix_ctas(const Group& g, int64_t n)
{
    return (int)max((int64_t)1, min((int64_t)g.size, cdiv(n, kRadixItems)));
}

template <typename KeyFn>
__device__ bool radix_pass(const ProbDev& d, const Group& g, int gs, long long budget, int64_t n,
                           const int32_t* src, int32_t* dst, int shift, KeyFn key, bool& skipped, RadixSmem& rsm)
{
    int* s_hist = rsm.hist;
    int* s_off = rsm.off;
    int (*s_wc)[kRadix] = rsm.wc;
    int* s_tot = rsm.tot;
    int& s_skip = rsm.skip;
    static_assert(kCoopThreads == 2 * kRadix, "thread layout");
    const int tid = threadIdx.x, warp = tid >> 5;
    const bool active = g.rank < gs;
    const int64_t chunk = cdiv(n, gs);
    const int64_t lo = active ? min(n, chunk * g.rank) : n, hi = active ? min(n, lo + chunk) : n;

    for (int i = tid; i < kRadix; i += blockDim.x) s_hist[i] = 0;
    __syncthreads();
    for (int64_t i = lo + tid; i < hi; i += blockDim.x)
        atomicAdd(&s_hist[(key(__ldcg(&src[i])) >> shift) & (kRadix - 1)], 1);
    __syncthreads();
    if (active)
        for (int i = tid; i < kRadix; i += blockDim.x) d.hist[g.rank * kRadix + i] = s_hist[i];
    if (!group_sync(g, d.sc, budget)) return false;

    // digit offsets of this CTA: all earlier digits + same digit of earlier CTAs
    // (two threads per digit, each over half of the CTAs, then a scan by warps:
    // with one thread adding up the 256 totals a pass over 100,000 points took
    // 8 us longer)
    if (tid == 0) s_skip = 0;
    {
        const int dg = tid & (kRadix - 1), half = tid >> kRadixBits, mid = (gs + 1) / 2;
        const int end = half ? gs : mid;
        int col = 0, pre = 0;
#pragma unroll 8
        for (int c = half ? mid : 0; c < end; ++c) {
            const int v = __ldcg(&d.hist[c * kRadix + dg]);
            col += v;
            if (c < g.rank) pre += v;
        }
        s_wc[half][dg] = col;
        s_wc[2 + half][dg] = pre;
    }
    __syncthreads();
    int col = 0, incl = 0;
    if (tid < kRadix) {
        col = s_wc[0][tid] + s_wc[1][tid];
        s_off[tid] = s_wc[2][tid] + s_wc[3][tid];
        if ((int64_t)col == n) s_skip = 1;
        incl = col;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int x = __shfl_up_sync(0xffffffffu, incl, o);
            if ((tid & 31) >= o) incl += x;
        }
        if ((tid & 31) == 31) s_tot[warp] = incl;
    }
    __syncthreads();
    skipped = s_skip != 0;
    if (!skipped) {
        if (tid < kRadix) {
            int before = incl - col;
            for (int w = 0; w < warp; ++w) before += s_tot[w];
            s_off[tid] += before;
        }
        for (int i = tid; i < (kCoopThreads / 32) * kRadix; i += blockDim.x) (&s_wc[0][0])[i] = 0;
        __syncthreads();
        // stable scatter, one tile of blockDim elements at a time
        for (int64_t base = lo; base < hi; base += blockDim.x) {
            int64_t i = base + tid;
            bool valid = i < hi;
            int32_t v = valid ? __ldcg(&src[i]) : 0;
            int dg = valid ? (int)((key(v) >> shift) & (kRadix - 1)) : kRadix;
            unsigned peers = __match_any_sync(0xffffffffu, dg);
            int r = __popc(peers & lanemask_lt());
            if (valid && r == 0) s_wc[warp][dg] = __popc(peers);
            __syncthreads();
            for (int dd = tid; dd < kRadix; dd += blockDim.x) {
                int run = 0;
                for (int w = 0; w < kCoopThreads / 32; ++w) { int c = s_wc[w][dd]; s_wc[w][dd] = run; run += c; }
                s_hist[dd] = run;  // tile count of digit dd
            }
            __syncthreads();
            if (valid) dst[s_off[dg] + s_wc[warp][dg] + r] = v;
            __syncthreads();
            for (int dd = tid; dd < kRadix; dd += blockDim.x) {
                s_off[dd] += s_hist[dd];
                for (int w = 0; w < kCoopThreads / 32; ++w) s_wc[w][dd] = 0;
            }
            __syncthreads();
        }
    }
    return group_sync(g, d.sc, budget);
}

}  // namespace emo
