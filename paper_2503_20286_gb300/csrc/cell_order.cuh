// Counting sort by grid cell: the order of the points (k_order.cu) and of the
// references that the tree searches walk over, and of S for the association.
// Points are ordered by the z-order cells of a grid whose lines are sample
// quantiles of each objective, so any distribution fills them about evenly;
// directions (references and S) by a Hilbert curve through an even grid.
// The order inside a cell depends on the run; nothing downstream depends on it.
#pragma once

#include "emo_kernels.cuh"

namespace emo {

constexpr int kZSample = 512;  // items whose quantiles set the grid lines
static_assert(kCoopThreads == kZSample, "one sample per thread");

// Grid lines of one grid, 2^bits slots per coordinate (m 2^bits <= 512).
constexpr int kZLines = 512;

// Lines from a strided sample of coord(i, k), i < n: two coordinates sorted at
// once by a bitonic network. Every CTA computes the same lines.
template <class Coord>
__device__ __forceinline__ void z_lines(float (*s_smp)[kZSample], float* line, int64_t n, int m, int bits, Coord coord)
{
    const int tid = threadIdx.x, ns = (int)min((int64_t)kZSample, n);
    for (int k0 = 0; k0 < m; k0 += 2) {
        const int64_t src = (int64_t)tid * n / ns;
        for (int h = 0; h < 2; ++h) s_smp[h][tid] = tid < ns && k0 + h < m ? coord(src, k0 + h) : INFINITY;
        __syncthreads();
        const int t = tid & (kZSample / 2 - 1);
        float* v = s_smp[tid / (kZSample / 2)];
        for (int size = 2; size <= kZSample; size <<= 1)
            for (int stride = size >> 1; stride > 0; stride >>= 1) {
                const int i = 2 * t - (t & (stride - 1)), j = i + stride;
                const float a = v[i], b = v[j];
                if ((a > b) == ((i & size) == 0)) { v[i] = b; v[j] = a; }
                __syncthreads();
            }
        for (int e = tid; e < 2 << bits; e += blockDim.x) {
            const int h = e >> bits, b = e & ((1 << bits) - 1);
            if (k0 + h < m && b < (1 << bits) - 1) line[((k0 + h) << bits) + b] = s_smp[h][(int64_t)(b + 1) * ns >> bits];
        }
        __syncthreads();
    }
}

// Z-order cell of an item: leading bits first, coordinates interleaved.
template <class Coord>
__device__ __forceinline__ uint32_t z_cell(const float* line, int m, int bits, Coord f)
{
    uint32_t key = 0u;
    for (int k = 0; k < m; ++k) {
        const float x = f(k);
        uint32_t c = 0u;
        for (int step = 1 << (bits - 1); step > 0; step >>= 1)
            if (line[(k << bits) + c + step - 1] <= x) c += step;
        for (int b = 0; b < bits; ++b) key |= ((c >> b) & 1u) << (b * m + m - 1 - k);
    }
    return key;
}

// Grid of the directions: the references' extent (of a sample) cut evenly, in
// simplex coordinates u_k / sum u, k < m - 1, for up to three objectives, in
// the m components of the unit direction beyond. (Measured on leaves of 32
// references: 200,028 directions of three objectives, points of 32 neighbours
// need 9 leaves; with all three components 50, with lines at quantiles 13.)
struct DirGrid {
    float lo[kMaxM], scale[kMaxM];
};
__host__ __device__ constexpr int dir_dims(int m) { return m <= 3 ? m - 1 : m; }

// Coordinate k of direction u(0), ..., u(m - 1); inv: 1 / sum u (m <= 3).
// Cell of a direction by its place on a Hilbert curve through the grid
// (Skilling, "Programming the Hilbert curve", 2004): consecutive cells touch,
// so runs of items stay compact.
template <class Coord>
__device__ __forceinline__ uint32_t dir_cell(const DirGrid& grid, int m, int bits, Coord u)
{
    const int nd = dir_dims(m);
    float inv = 1.0f;
    if (m <= 3) {
        float s = 0.0f;
        for (int k = 0; k < m; ++k) s += u(k);
        inv = 1.0f / s;
    }
    uint32_t c[kMaxM], key = 0u;
    for (int k = 0; k < nd; ++k)
        c[k] = (uint32_t)min(max(__float2int_rz((u(k) * inv - grid.lo[k]) * grid.scale[k]), 0), (1 << bits) - 1);
    for (uint32_t q = 1u << (bits - 1); q > 1u; q >>= 1)
        for (int k = 0; k < nd; ++k) {
            const uint32_t t = (c[k] & q) ? q - 1u : (c[0] ^ c[k]) & (q - 1u);
            c[0] ^= t;
            if (!(c[k] & q)) c[k] ^= t;
        }
    for (int k = 1; k < nd; ++k) c[k] ^= c[k - 1];
    uint32_t t = 0u;
    for (uint32_t q = 1u << (bits - 1); q > 1u; q >>= 1)
        if (c[nd - 1] & q) t ^= q - 1u;
    for (int b = bits - 1; b >= 0; --b)
        for (int k = 0; k < nd; ++k) key = key << 1 | (((c[k] ^ t) >> b) & 1u);
    return key;
}

// One array of items being ordered: cell counts (zero before), then per item
// its cell and its slot in it (the old value of the cell's counter).
struct CellSort {
    int64_t n, ncell;
    uint32_t* cnt;
    uint32_t* cell;
    uint32_t* slot;
};
template <class CellOf>
__device__ __forceinline__ void cell_count(const CellSort& c, const Group& g, CellOf cell_of)
{
    for (int64_t i = (int64_t)g.rank * blockDim.x + threadIdx.x; i < c.n; i += (int64_t)g.size * blockDim.x) {
        const uint32_t key = cell_of(i);
        c.cell[i] = key;
        c.slot[i] = atomicAdd(&c.cnt[key], 1u);
    }
}
// The CTA's share of the cells.
__device__ __forceinline__ void cell_share(const CellSort& c, const Group& g, int64_t& lo, int64_t& hi)
{
    const int64_t chunk = cdiv(c.ncell, g.size);
    lo = min(c.ncell, chunk * g.rank);
    hi = min(c.ncell, lo + chunk);
}
// After a barrier: the share's total into part[rank].
__device__ __forceinline__ void cell_total(const CellSort& c, const Group& g, int32_t* part, int* s_warp)
{
    int64_t lo, hi;
    cell_share(c, g, lo, hi);
    int sum = 0;
    for (int64_t i = lo + threadIdx.x; i < hi; i += blockDim.x) sum += (int)__ldcg(&c.cnt[i]);
    sum = block_reduce_sum<kCoopThreads>(sum, s_warp);
    if (threadIdx.x == 0) part[g.rank] = sum;
}
// After a barrier: counts to offsets (exclusive).
__device__ __forceinline__ void cell_offsets(const CellSort& c, const Group& g, const int32_t* part, int* s_warp)
{
    constexpr int PER = 4;
    int64_t lo, hi;
    cell_share(c, g, lo, hi);
    int base = 0;
    for (int r = threadIdx.x; r < g.rank; r += blockDim.x) base += __ldcg(&part[r]);
    base = block_reduce_sum<kCoopThreads>(base, s_warp);
    for (int64_t c0 = lo; c0 < hi; c0 += (int64_t)PER * blockDim.x) {
        int v[PER], s = 0;
#pragma unroll
        for (int e = 0; e < PER; ++e) {
            const int64_t i = c0 + (int64_t)threadIdx.x * PER + e;
            v[e] = i < hi ? (int)__ldcg(&c.cnt[i]) : 0;
            s += v[e];
        }
        int tot, run = base + block_exclusive_scan<kCoopThreads>(s, s_warp, tot);
#pragma unroll
        for (int e = 0; e < PER; ++e) {
            const int64_t i = c0 + (int64_t)threadIdx.x * PER + e;
            if (i < hi) c.cnt[i] = (uint32_t)run;
            run += v[e];
        }
        base += tot;
    }
}
// After a barrier: place(i, cell, position) of every item.
template <class Place>
__device__ __forceinline__ void cell_place(const CellSort& c, const Group& g, Place place)
{
    for (int64_t i = (int64_t)g.rank * blockDim.x + threadIdx.x; i < c.n; i += (int64_t)g.size * blockDim.x) {
        const uint32_t key = c.cell[i];  // this thread's own
        place(i, key, (int64_t)__ldcg(&c.cnt[key]) + c.slot[i]);
    }
}

}  // namespace emo
