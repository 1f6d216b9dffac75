// The orders that the tree searches walk over: the points of a problem ranked
// by k_fronts, and the reference directions of the association.
//
// References: unit directions along a Hilbert curve through their grid, 32 to a leaf,
// 32 leaves to a node; per leaf and node the mean direction and the largest
// distance of a member from it. A reference's angle decides the association
// and grows with the distance of the unit directions, so a leaf whose ball is
// farther from a point's direction than the nearest reference found so far
// (plus the ball's radius) holds nothing nearer (k_select.cu).
#include "cell_order.cuh"

namespace emo {

// Mean direction and radius of the references [r0, r0 + cnt) (sorted
// positions) by one warp, into column `at` of ball[m][stride] and rad[at].
__device__ __forceinline__ void ref_ball(const float* rsort, int mp, int m, int64_t r0, int cnt, float* ball, int stride,
                                         float* rad, int at)
{
    const int lane = threadIdx.x & 31;
    float mine = 0.0f;  // coordinate `lane` of the centre
    for (int k = 0; k < m; ++k) {
        float s = 0.0f;
        for (int i = lane; i < cnt; i += 32) s += __ldcg(&rsort[(r0 + i) * mp + k]);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        s /= (float)cnt;
        if (lane == k) mine = s;
    }
    float far = 0.0f;
    for (int i0 = 0; i0 < cnt; i0 += 32) {
        const int i = i0 + lane;
        float d2 = 0.0f;
        for (int k = 0; k < m; ++k) {
            const float c = __shfl_sync(0xffffffffu, mine, k);
            const float e = i < cnt ? __ldcg(&rsort[(r0 + i) * mp + k]) - c : 0.0f;
            d2 = fmaf(e, e, d2);
        }
        far = fmaxf(far, d2);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) far = fmaxf(far, __shfl_xor_sync(0xffffffffu, far, o));
    if (lane < m) ball[lane * stride + at] = mine;
    if (lane == 0) rad[at] = sqrtf(far) * (1.0f + 1e-5f) + 1e-6f;  // (covers the rounding of both sums)
}

__global__ void __launch_bounds__(kCoopThreads, 1) k_order(Plan* plan)
{
    const Group g = group_of(plan, GRP_NARROW);
    if (g.prob < 0) return;  // a CTA beyond every problem's group
    const ProbDev& d = plan->p[g.prob];
    const ProbIn& in = d.in;
    const long long budget = plan->spin_budget;
    const bool pts = d.tree, refs = d.rtree;
    if (!(pts || refs) || ld_volatile(&d.sc->status) != 0) return;
    __shared__ float s_smp[2][kZSample];
    __shared__ float s_pline[kZLines];
    __shared__ DirGrid s_grid;
    __shared__ int s_warp[33];
    const int m = in.m, tid = threadIdx.x;
    const int64_t n2 = in.n2, nr = in.n_r;
    const float* F = in.F;
    const float* rhat = d.rhat;
    auto fcoord = [&](int64_t i, int k) { return F[i * m + k] + 0.0f; };
    if (pts) z_lines(s_smp, s_pline, n2, m, d.zbits, fcoord);
    if (refs) {  // extent of a sample of the references (a warp per coordinate)
        const int ns = (int)min((int64_t)kZSample, nr), nd = dir_dims(m);
        for (int k = tid >> 5; k < nd; k += kCoopThreads / 32) {
            float lo = INFINITY, hi = -INFINITY;
            for (int e = tid & 31; e < ns; e += 32) {
                const float* u = rhat + (int64_t)e * nr / ns * m;
                float t = 1.0f;
                if (m <= 3) {
                    t = 0.0f;
                    for (int q = 0; q < m; ++q) t += u[q];
                }
                const float x = u[k] / t;
                lo = fminf(lo, x);
                hi = fmaxf(hi, x);
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
                hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
            }
            if ((tid & 31) == 0) {
                s_grid.lo[k] = lo;
                s_grid.scale[k] = hi > lo ? (float)(1 << d.rbits) / (hi - lo) : 0.0f;
                if (g.rank == 0) {  // S is put in the same cells later
                    d.rgrid->lo[k] = s_grid.lo[k];
                    d.rgrid->scale[k] = s_grid.scale[k];
                }
            }
        }
        __syncthreads();
    }
    const CellSort cp{n2, d.ncell, d.zcnt, d.zcell, d.zslot};
    const CellSort cr{nr, d.nrcell, d.rcnt, d.rcell, d.rslot};
    int32_t* const ppart = d.hist;
    int32_t* const rpart = d.hist + g.size;
    if (pts) cell_count(cp, g, [&](int64_t i) { return z_cell(s_pline, m, d.zbits, [&](int k) { return fcoord(i, k); }); });
    if (refs) cell_count(cr, g, [&](int64_t j) { return dir_cell(s_grid, m, d.rbits, [&](int k) { return rhat[j * m + k]; }); });
    if (!group_sync(g, d.sc, budget)) return;
    if (pts) cell_total(cp, g, ppart, s_warp);
    if (refs) cell_total(cr, g, rpart, s_warp);
    if (!group_sync(g, d.sc, budget)) return;
    if (pts) cell_offsets(cp, g, ppart, s_warp);
    if (refs) cell_offsets(cr, g, rpart, s_warp);
    if (!group_sync(g, d.sc, budget)) return;
    if (pts) {
        const int64_t zs = (int64_t)d.nleaf * 32;
        cell_place(cp, g, [&](int64_t i, uint32_t key, int64_t pos) {
            for (int k = 0; k < m; ++k) d.zpts[k * zs + pos] = fcoord(i, k);
            d.zidx[pos] = (int32_t)i;
            d.zkey[pos] = key;
        });
    }
    if (!refs) return;
    const int mp = (m + 3) / 4 * 4;
    cell_place(cr, g, [&](int64_t j, uint32_t, int64_t pos) {
        for (int k = 0; k < mp; ++k) d.rsort[pos * mp + k] = k < m ? rhat[j * m + k] : 0.0f;
        d.rord[pos] = (int32_t)j;
    });
    if (!group_sync(g, d.sc, budget)) return;
    const int nw = g.size * (kCoopThreads / 32), gw = (tid >> 5) * g.size + g.rank;
    for (int t = gw; t < d.nrleaf; t += nw)
        ref_ball(d.rsort, mp, m, (int64_t)t * 32, (int)min((int64_t)32, nr - (int64_t)t * 32), d.rball, d.nrleafp, d.rrad, t);
    for (int a = nw - 1 - gw; a < d.nrnode; a += nw)
        ref_ball(d.rsort, mp, m, (int64_t)a * 1024, (int)min((int64_t)1024, nr - (int64_t)a * 1024), d.rnball, d.nrnodep,
                 d.rnrad, a);
}

}  // namespace emo
