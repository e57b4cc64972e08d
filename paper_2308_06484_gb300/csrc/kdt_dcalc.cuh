// d-calculation (Section III "Notation and definitions"; Section IV, the sub-algorithm
// d-calculation): for a constant N, every point's distance to its N-th nearest
// neighbour, its minimum per block and over all blocks (mindistance), and the block
// N-spread that follows from it.
//
// The N-th nearest neighbour is found on the triangulation itself.  Order the other
// points by squared distance to p (equal ones in any order).  The k-th of them, q, is a
// Delaunay neighbour of p or of one of the k-1 before it: grow a circle through q with its
// centre moving from q towards p; the first point it meets lies strictly inside the disk
// of radius |pq| around p, hence before q, and the empty circle through q and that point
// makes them adjacent (when several points are met at once, q is adjacent to one of them in
// every triangulation of that Delaunay face).  So taking the k nearest one at a time,
// each time from the neighbours of p and of the points already taken (the expansion of
// Dickerson, Drysdale and Sack for k nearest neighbours), is exact, and a candidate
// list of N entries suffices.  Distances are exact int64 squares.
#pragma once

#include "kdt_kernels.cuh"

namespace kd {

constexpr int DC_MAX_N = 16;  // largest N a call may ask for

__device__ __forceinline__ long long dist2_of(int2 a, int2 b)
{
    long long dx = (long long)a.x - b.x, dy = (long long)a.y - b.y;
    return dx * dx + dy * dy;
}

// One thread per point: the N <= CAP nearest, one at a time, each time from the stars of p
// and of the points already taken (see the header).  A star is walked on the triangulation
// itself; neighbouring threads take neighbouring points (order: the build's Hilbert order,
// or null: ids), so the triangles and positions of one warp's walks come from the same few
// sectors of L1 and L2.  bd / bi hold the best candidates by distance, in registers (every
// loop over them is unrolled); the N in use are the last ones, so that a candidate is compared with
// the worst of them at a fixed place, and most are dropped there.  Which of several
// points at one distance comes first does not matter: the header's argument finds a
// neighbour strictly nearer.
// Bound by the chain of a star's triangles, and beyond N = 8 by the insertions into bd.  The
// next triangle is loaded before a vertex is looked at, for N <= 4 from both ends of the
// star.  1e6 points, us a call (neighbour lists, which the walk replaced / now): N = 1
// 250 / 119, 4 438 / 216, 8 846 / 454, 9 995 / 738, 16 2132 / 1726; one point of degree
// 4,000: 852 / 808 (N = 4; 1,185 from one end), 886 / 1011 (N = 9).
// Writes dist2[p] (if asked), the minimum of its partition (cell_min, if asked) and of all
// points (gmin); the largest degree met goes to max_deg.
template <int CAP>
__global__ void __launch_bounds__(128) k_nth_nn(const int2 *xy, const int *pt_tri, TriHalf tv, TriHalf tn,
                                                const int *order, int n, int N, Inst I, int bits, long long *dist2,
                                                unsigned long long *cell_min, unsigned long long *gmin, int *max_deg)
{
    constexpr bool TWO = CAP <= 4;  // walk a star from both ends
    long long best = LLONG_MAX;
    int mdeg = 0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const int p = order ? __ldg(order + i) : i;
        const int2 pp = __ldg(xy + p);
        long long bd[CAP];
        int bi[CAP];
#pragma unroll
        for (int j = 0; j < CAP; ++j) {
            bd[j] = j < CAP - N ? LLONG_MIN : LLONG_MAX;
            bi[j] = j < CAP - N ? -1 : INT_MAX;
        }
        // a neighbour w at x (w < 0: the vertex at infinity)
        int deg = 0;
        auto take = [&](int w, int2 x) {
            if (w < 0) return;
            ++deg;
            long long cd = dist2_of(pp, x);
            if (w == p || cd >= bd[CAP - 1]) return;
            bool seen = false;
#pragma unroll
            for (int j = 0; j < CAP; ++j) seen = seen || bi[j] == w;
            if (seen) return;
#pragma unroll
            for (int j = 0; j < CAP; ++j)
                if (cd < bd[j]) {
                    const long long td = bd[j];
                    const int tj = bi[j];
                    bd[j] = cd;
                    bi[j] = w;
                    cd = td;
                    w = tj;
                }
        };
        int src = p;
        for (int e = 0; e < N; ++e) {
            // add the neighbours of src (p, then the point taken last)
            const int t0 = __ldg(pt_tri + src);
            int4 v = __ldg(tv + t0), nb = __ldg(tn + t0);
            int tb = (v.x == src ? nb.z : (v.y == src ? nb.x : nb.y)) >> 2;
            int4 bv = v, bn = nb;
            if (TWO) {
                bv = __ldg(tv + tb);
                bn = __ldg(tn + tb);
            }
            int steps = 0;
            bool more = true, both = TWO;
            deg = 0;
            while (more) {
                const int k = v.x == src ? 0 : (v.y == src ? 1 : 2), kb = bv.x == src ? 0 : (bv.y == src ? 1 : 2);
                int w = k == 0 ? v.y : (k == 1 ? v.z : v.x), wb = kb == 0 ? bv.y : (kb == 1 ? bv.z : bv.x);
                const int t = (k == 0 ? nb.y : (k == 1 ? nb.z : nb.x)) >> 2;
                const int u = (kb == 0 ? bn.z : (kb == 1 ? bn.x : bn.y)) >> 2;
                if (!both) wb = -1;
                more = (TWO ? both && t != tb : t != t0) && ++steps <= n;  // (a star has at most n triangles)
                both = TWO && more && t != u;
                tb = u;
                // (the next triangles on their way before these ones' vertices are looked at)
                int2 x = __ldg(xy + max(w, 0));
                const int2 xb = TWO ? __ldg(xy + max(wb, 0)) : x;
                if (more) {
                    v = __ldg(tv + t);
                    nb = __ldg(tn + t);
                }
                if (TWO && both) {
                    bv = __ldg(tv + u);
                    bn = __ldg(tn + u);
                }
#pragma unroll 1
                for (int s = 0; s < (TWO ? 2 : 1); ++s, w = wb, x = xb) take(w, x);
            }
            mdeg = max(mdeg, deg);
#pragma unroll
            for (int j = 0; j < CAP; ++j)
                if (j == CAP - N + e) src = bi[j];  // the (e+1)-th nearest: expand it next
            if (src == INT_MAX) break;  // fewer than N other points reachable (cannot happen for n > N)
        }
        const long long v = bd[CAP - 1];
        if (dist2) dist2[p] = v;
        if (cell_min) {
            const int inst = I.ninst > 1 ? csr_find(I.pofs, I.ninst + 1, p) : 0;
            atomicMin(cell_min + partition_of(I, inst, bits, pp), (unsigned long long)v);
        }
        best = min(best, v);
    }
    for (int o = 16; o > 0; o >>= 1) {
        best = min(best, (long long)__shfl_xor_sync(FULL, (unsigned long long)best, o));
        mdeg = max(mdeg, __shfl_xor_sync(FULL, mdeg, o));
    }
    if ((threadIdx.x & 31) == 0) {
        atomicMin(gmin, (unsigned long long)best);
        atomicMax(max_deg, mdeg);
    }
}

// run[c] = min(run[c], cur[c]) (or cur[c] when restart): the running per-partition
// d_local^2 of the displacement rule
__global__ void k_merge_min_u64(unsigned long long *run, const unsigned long long *cur, long long n, int restart)
{
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        run[i] = restart ? cur[i] : min(run[i], cur[i]);
}

__global__ void k_fill_u64(unsigned long long *a, long long n, unsigned long long v)
{
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        a[i] = v;
}

}  // namespace kd
