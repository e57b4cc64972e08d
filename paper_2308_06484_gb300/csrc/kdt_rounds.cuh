// Rounds of operations on the whole triangulation: a group of lanes plans one operation on
// the triangulation as it stands (region_plan), the operations that do not meet are
// committed together, the others are planned again in the next round.
//
//   k_round_plan    plans the round's operations and claims their triangles: the owner
//                   word of every triangle of the region takes the largest priority
//                   (atomicMax), nothing else is written;
//   k_round_commit  an operation wins when it owns its whole region and no triangle
//                   next to its region belongs to a higher priority; winners write their
//                   triangles, losers go to the next round's list;
//   k_round_clear   after the last round of a step: every claimed owner word zero again,
//                   and what is still not done to the list of the warp-wide path.
//
// Why a round's result is the Delaunay triangulation of the new positions: let A be the
// triangles an operation destroys.  Two winners' regions share no triangle and no edge
// (the higher priority owns its region; the lower one, next to it, loses).  An edge inside
// a new region, or between it and the unchanged triangle across its border, is locally
// Delaunay because it is in the triangulation after that operation alone; every other
// edge is unchanged, and no unchanged triangle has a moved vertex, for the star of a moved
// point is in its region.  All edges locally Delaunay: the whole is Delaunay.  So nothing
// is certified after a round, no read is ever of a half-written triangle, and no
// operation waits for another.
//
// What it replaced, and what it measured (GB300, times of a kdt_step / kdt_rebuild): one warp
// per move or insertion, claiming star and ring by compare-and-swap, re-reading them under
// the claims and certifying afterwards took about 6,500 warp instructions an operation
// in code too large for the instruction caches ("no instruction" 10-15 stalled cycles per
// issue).  The plan takes 1,970 with a warp to itself (12 of 32 lanes active), 1,460 where two
// share a warp.
//   step, 1e6 uniform points, 4096 moves          125 -> 77 us
//   step, 16e6 clustered points, 140,000 moves   2.75 -> 1.25 ms (median)
//   step, 512 instances, 212,000 moves            2.6 -> 0.8 ms
//   step, 2e5 points, 1,950 moves that leave their star   390 -> 180 us
//   rebuild, 1e6 uniform points                  28.8 -> 9.6 ms
//   rebuild, 128 instances, 1.5e6 points         37   -> 9.6 ms
// Bound now: the latency of the plan's chain (12-27 us a round of a few thousand operations,
// 42 % of the issue slots used) times the number of rounds; with 1e5 operations or more,
// the issue slots and the spread of the loads over L2.
//
// Owner words keep the claims of earlier rounds until the end (a priority starts with
// the round's number, so older ones always lose); only k_round_clear or k_clear_owner
// zero them, before any kernel that takes claims by compare-and-swap runs.
#pragma once
#include "kdt_kernels.cuh"
#include "kdt_region.cuh"

namespace kd {

constexpr int ROUND_BITS = 18;
constexpr int ROUND_OPS = 1 << ROUND_BITS;  // operations of one round at most
constexpr int ROUND_MAX = 4095;             // rounds between two clears of the owner words
constexpr int ROUND_THREADS = 64;           // of k_round_plan
constexpr int ROUND_BLOCKS = 16;            // ... its blocks per SM: 64 registers a thread, a few spills.
                                            // 140,000 moves: 8 blocks (120 registers) 1.75, 12 1.65,
                                            // 16 1.55, 20 1.75 ms a step
constexpr int ROUND_LANES = 8;              // lanes of k_round_commit per operation

// What one round works on: the losers of the round before (lost[b & 1]), then fresh items
// of the queue.  Counters have one entry per round, written by the rounds before, so a
// round's kernels read constants: one 16-byte load a thread, for every warp of the GPU reads
// the same words (a word more cost 4 us in each kernel of thousands of blocks).
struct Rounds {
    int4 *cnt;      // [rounds + 1] next fresh item, losers of the round before, refused items (in a
                    // step's last round), operations planned before the round
    int *lost[2];   // item ids
    int4 *hdr;      // per operation of the round: item, triangles (0: plan again, -1: left to the
                    // other path), priority, k | ncav << 8 | edge << 24 | ghost << 25 | prop << 26
    int4 *rec;      // per operation of the round: RT triangles (region_plan's out)
    int *slots;     // moves only, per operation since the step's start: RT slots (-1: none)
    int *left;      // items for the warp-wide path
    int *left_count;
    int *refused;   // items 16 lanes could not plan, for a round of 32 lanes
    int *refused_count;
    const int *wide;  // this round takes nwide of these (once refused): > 0 (builds) instead of fresh
    int nwide;        // items, < 0 (a step's last round) all of them before fresh items
    int *pending;   // moves only: moves not done after the last round
    int div;        // builds: operations up to the points inserted or up to `few`, and 1 / div of
                    // them beyond (0: no such limit)
    int few;
    int base;       // points inserted before the first round (div > 0)
    int ops;        // room for operations of one round
};

// items of the refused list that a round with nwide < 0 and counters c takes after its losers
__device__ __forceinline__ int round_all_refused(const Rounds &R, const int4 &c)
{
    return min(c.z, max(0, R.ops - c.y));
}

__device__ __forceinline__ int *round_word(const Rounds &R, int b, int i)
{
    return reinterpret_cast<int *>(R.cnt + b) + i;
}

// the round's operations: losers, nw items of the wide list, fresh items from `head` (total:
// length of the queue)
__device__ __forceinline__ void round_window(const Rounds &R, int b, int total, int &nlost, int &nw, int &head,
                                             int &count, int &off)
{
    const int4 c = __ldcg(R.cnt + b);
    head = c.x;
    nlost = c.y;
    off = c.w;
    nw = R.nwide >= 0 ? R.nwide : round_all_refused(R, c);
    int lim = R.ops;
    if (R.div > 0) {
        const int in = R.base + head - nlost;
        lim = min(lim, max(max(64, in / R.div), min(in, R.few)));
    }
    count = nlost + nw + (R.nwide > 0 ? 0 : max(0, min(lim - nlost - nw, total - head)));
}

// priority of operation x of round b: the round first, then a different order of the
// operations in every round (an odd multiplier permutes the 18-bit numbers)
__device__ __forceinline__ int round_priority(int b, int x)
{
    const unsigned h = (((unsigned)x ^ ((unsigned)(b + 1) * 40503u)) * 0x9E375u) & (ROUND_OPS - 1);
    return ((b + 1) << ROUND_BITS) | (int)h;
}

struct RoundMoves {
    const int3 *gmoves;  // (point, x, y) per move
};

struct RoundBuild {
    const int *queue;   // position in `order` per queue entry
    const int *order;   // points in Hilbert order, instance by instance
    const int *third;   // per instance: local position of the third point of its first triangle
    const int *pofs, *tofs;
    int ninst;
    int total;          // length of the queue
    int n;              // one instance: its points (0: pofs has them)
};

// The point of the inserted ones among the 16 before and after position j of the order, in
// steps of its level's stride, that is nearest to q: the start of the walk (a triangle of
// it), or -1.  (Neighbours along the Hilbert curve are near in the plane; the nearest of
// several saves walk steps, and the long walks along thin triangles near the hull.)
template <int RL>
__device__ __forceinline__ int near_start(const Dev &d, const int *order, int n, int j, int2 q, int l, unsigned gm)
{
    const int lev = __ffs(j) - 1, c = (l & 15) - 8;
    const long long a = j + ((long long)(c < 0 ? c : c + 1) << lev);
    int t = -1;
    long long best = LLONG_MAX;
    if (a >= 0 && a < n) {
        const int v = __ldg(order + a);
        t = __ldcg(d.pt_tri + v);
        const int2 x = __ldcg(d.xy + v);
        const long long dx = (long long)x.x - q.x, dy = (long long)x.y - q.y;
        if (t >= 0) best = dx * dx + dy * dy;
    }
#pragma unroll
    for (int o = RL / 2; o; o >>= 1) {
        const long long ob = __shfl_xor_sync(gm, best, o, RL);
        const int ot = __shfl_xor_sync(gm, t, o, RL);
        if (ob < best || (ob == best && ot > t)) {
            best = ob;
            t = ot;
        }
    }
    return best == LLONG_MAX ? -1 : t;
}

// RL lanes per operation.  With fewer operations than warps every operation has a warp to
// itself, so no warp is as long as the union of two operations' paths.  An operation
// outside RL's limits goes to the list of the warp-wide path when `last` is set, otherwise to
// the refused list: the triangulation changes little from round to round, so the same lanes
// would refuse it again.  A move whose walk is too long goes to the warp-wide path at once.
//
// round_plan: `tid` of `nthreads` threads (whole warps), shared: one RegionShared per group of
// the block.
template <int MODE, int RL>
__device__ __forceinline__ void round_plan(const Dev &d, const Rounds &R, int b, const RoundMoves &M,
                                           const RoundBuild &B, int total, int last, RegionShared<RL> *shared, int tid,
                                           int nthreads)
{
    constexpr bool MOVE = MODE != REGION_INSERT;
    int nlost, nw, head, count, off;  // (nw > 0 in rounds of 32 lanes only)
    round_window(R, b, total, nlost, nw, head, count, off);
    if (tid == 0) {
        *round_word(R, b + 1, 0) = head + count - nlost - nw;
        *round_word(R, b + 1, 3) = off + count;
    }
    constexpr int PER_WARP = 32 / RL;
    const int l = threadIdx.x & (RL - 1), g0 = threadIdx.x & 31 & ~(RL - 1);
    const unsigned gm = (FULL >> (32 - RL)) << g0;
    const int warps = nthreads / 32;
    const bool alone = count <= warps;
    if (alone && g0) return;
    RegionShared<RL> &sh = shared[threadIdx.x / RL];
    unsigned ex = 0, ti = 0, steps = 0;
    const int groups = alone ? warps : warps * PER_WARP;
    for (int x = alone ? tid / 32 : tid / RL; x < count; x += groups) {
        int item;
        if (x < nlost) {
            item = __ldcg(R.lost[b & 1] + x);
        } else if (RL == 32 && x < nlost + nw) {
            item = __ldcg(R.wide + x - nlost);
        } else {
            item = head + x - nlost - (RL == 32 ? nw : 0);
            if (!MOVE) item = __ldcg(B.queue + item);
        }
        RegionOut o;
        int4 *rec = R.rec + (size_t)x * (2 * RT);
        int rc, p;
        if constexpr (MOVE) {
            const int3 mv = M.gmoves[item];
            p = mv.x;
            rc = region_plan<MODE, RL>(d, sh, l, gm, g0, p, make_int2(mv.y, mv.z), -1, -1, -1, rec, o);
        } else {
            const int inst = B.ninst > 1 ? csr_find(B.pofs, B.ninst + 1, item) : 0;
            const int p0 = __ldg(B.pofs + inst), j = item - p0;
            p = __ldg(B.order + item);
            if (__ldcg(d.pt_tri + p) >= 0) {  // a point of the first triangle
                if (l == 0) R.hdr[x] = make_int4(item, -1, 0, 0);
                continue;
            }
            const int2 q = __ldcg(d.xy + p);
            // its two slots: every instance's slots in the order of its points
            const int s = __ldg(B.tofs + inst) + 4 + 2 * (j - 2 - (j > __ldg(B.third + inst)));
            // the walk starts at a point near by, else at the nearest one before it in the
            // levels' tree that is in already (position 0 always is)
            int start = near_start<RL>(d, B.order + p0, B.n > 0 ? B.n : __ldg(B.pofs + inst + 1) - p0, j, q, l, gm);
            for (int a = j; start < 0 && a > 0;) {
                a &= a - 1;
                start = __ldcg(d.pt_tri + __ldg(B.order + p0 + a));
            }
            rc = region_plan<REGION_INSERT, RL>(d, sh, l, gm, g0, p, q, start, s, s + 1, rec, o);
        }
        ex += o.ex;
        ti += o.ti;
        int nt = rc == RG_OK ? o.nt : -1;
        if (rc == RG_VERTEX) {
            // q lies on a point: one that moves in this step may have left by the next round
            if (!MOVE) atomicCAS(d.status, 0, DEV_DUPLICATE);
            else nt = __ldcg(d.pt_stamp + o.vtx) == d.stamp ? 0 : -1;
        }
        const int pr = round_priority(b, x);
        for (int i = l; i < RT; i += RL) {
            const int s = i < nt ? sh.pool[i] : -1;
            if (s >= 0) atomicMax(&d.tn[s].w, pr);
            if (MOVE) R.slots[(size_t)(off + x) * RT + i] = s;
        }
        if (l == 0) {
            steps += o.steps;
            if (nt < 0) {
                if (last || (MOVE && rc != RG_BAIL)) R.left[atomicAdd(R.left_count, 1)] = item;
                else R.refused[atomicAdd(R.refused_count, 1)] = item;
            }
            R.hdr[x] = make_int4(item, nt, pr, o.k | o.ncav << 8 | o.edge << 24 | o.ghost << 25 | o.prop << 26);
        }
        __syncwarp(gm);
    }
    if (!d.counters) return;
    ex = __reduce_add_sync(gm, ex);
    ti = __reduce_add_sync(gm, ti);
    if (l != 0) return;
    if (ex) atomicAdd(d.counters + C_EXACT, (unsigned long long)ex);
    if (ti) atomicAdd(d.counters + C_TIES, (unsigned long long)ti);
    if (steps) atomicAdd(d.counters + C_WALK_STEPS, (unsigned long long)steps);
}

template <int MODE, int RL>
__global__ void __launch_bounds__(ROUND_THREADS, ROUND_BLOCKS) k_round_plan(Dev d, Rounds R, int b, RoundMoves M,
                                                                            RoundBuild B, int last)
{
    if (__ldcg(d.status)) return;
    __shared__ RegionShared<RL> shared[ROUND_THREADS / RL];
    int total = B.total;
    if (MODE != REGION_INSERT && d.ctl) {
        total = __ldcg(d.ctl);
        d.stamp = __ldcg(d.ctl + 1);
    }
    round_plan<MODE, RL>(d, R, b, M, B, total, last, shared, blockIdx.x * blockDim.x + threadIdx.x,
                         gridDim.x * ROUND_THREADS);
}

// ROUND_LANES lanes per operation, lane l its triangles l, l + 8, ...  The owner
// words keep the priorities (a neighbour that checks its own border meanwhile must still
// see them).
template <bool MOVE>
__device__ __forceinline__ void round_commit(const Dev &d, const Rounds &R, int b, const RoundMoves &M, int total,
                                             int *sum, int tid, int nthreads)
{
    int nlost, nw, head, count, off;
    round_window(R, b, total, nlost, nw, head, count, off);
    const int lane = threadIdx.x & (ROUND_LANES - 1);
    const unsigned gm = 0xffu << (threadIdx.x & 24);  // this operation's lanes
    int nwin = 0, nlose = 0, degs = 0, flips = 0, edges = 0, ghosts = 0, props = 0, hits = 0;
    const int groups = nthreads / ROUND_LANES;
    // (whole warps take part in the ballots: the loop ends for a warp at once)
    for (int x0 = (tid & ~31) / ROUND_LANES; x0 < count; x0 += groups) {
        const int x = x0 + ((threadIdx.x & 31) / ROUND_LANES);
        int4 h = make_int4(-1, -1, 0, 0);
        if (x < count) h = __ldcg(R.hdr + x);
        const int nt = h.y;
        const int4 *rec = R.rec + (size_t)x * (2 * RT);
        int4 v = make_int4(0, 0, 0, 0), n = v;
        bool ok = nt > 0;
        // (from the last triangle down, so that the lane's first one stays in registers)
        for (int j = lane + (nt > lane ? (nt - 1 - lane) / ROUND_LANES * ROUND_LANES : 0); j >= 0 && j < nt;
             j -= ROUND_LANES) {
            v = __ldcg(rec + 2 * j);
            n = __ldcg(rec + 2 * j + 1);
            ok = ok && __ldcg(&d.tn[n.w].w) == h.z;
            if (n.x < 0) ok = ok && __ldcg(&d.tn[(~n.x) >> 2].w) < h.z;
            if (n.y < 0) ok = ok && __ldcg(&d.tn[(~n.y) >> 2].w) < h.z;
            if (n.z < 0) ok = ok && __ldcg(&d.tn[(~n.z) >> 2].w) < h.z;
        }
        const bool win = (__ballot_sync(FULL, ok) & gm) == gm;
        if (win) {
            for (int j = lane; j < nt; j += ROUND_LANES) {
                if (j != lane) {
                    v = __ldcg(rec + 2 * j);
                    n = __ldcg(rec + 2 * j + 1);
                }
                const int s = n.w;
                if (n.x < 0) backptr(d, n.x = ~n.x, s << 2);
                if (n.y < 0) backptr(d, n.y = ~n.y, s << 2 | 1);
                if (n.z < 0) backptr(d, n.z = ~n.z, s << 2 | 2);
                n.w = h.z;
                d.tv[s] = v;
                d.tn[s] = n;
                if (v.x >= 0) d.pt_tri[v.x] = s;
                if (v.y >= 0) d.pt_tri[v.y] = s;
                if (v.z >= 0) d.pt_tri[v.z] = s;
            }
        }
        if (lane == 0 && nt >= 0) {
            if (win) {
                if (MOVE) {
                    const int3 mv = M.gmoves[h.x];
                    d.xy[mv.x] = make_int2(mv.y, mv.z);
                }
                ++nwin;
                degs += h.w & 0xff;
                flips += ((h.w >> 8) & 0xffff) - 1;
                edges += (h.w >> 24) & 1;
                ghosts += (h.w >> 25) & 1;
                props += (h.w >> 26) & 1;
                hits += (h.w >> 27) & 1;
            } else {
                ++nlose;
                R.lost[(b + 1) & 1][atomicAdd(round_word(R, b + 1, 1), 1)] = h.x;
            }
        }
    }
    if (!d.counters) return;
    if (threadIdx.x < 8) sum[threadIdx.x] = 0;
    __syncthreads();
    const int part[8] = {nwin, nlose, degs, flips, edges, ghosts, props, hits};
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int s = __reduce_add_sync(FULL, part[i]);
        if ((threadIdx.x & 31) == 0 && s) atomicAdd(sum + i, s);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        const int slot[8] = {C_INSERTS,    C_RETRIES,     C_DEG_DEL,    C_FLIPS,
                             C_SPLIT_EDGE, C_SPLIT_GHOST, C_PROP_MOVES, C_PROP_HITS};
        for (int i = 0; i < 8; ++i)
            if (sum[i]) atomicAdd(d.counters + slot[i], (unsigned long long)sum[i]);
        if (MOVE && sum[0]) atomicAdd(d.counters + C_DELETES, (unsigned long long)sum[0]);
    }
}

template <bool MOVE>
__global__ void __launch_bounds__(256) k_round_commit(Dev d, Rounds R, int b, RoundMoves M, RoundBuild B)
{
    if (__ldcg(d.status)) return;
    __shared__ int sum[8];
    round_commit<MOVE>(d, R, b, M, MOVE && d.ctl ? __ldcg(d.ctl) : B.total, sum, blockIdx.x * blockDim.x + threadIdx.x,
                       gridDim.x * blockDim.x);
}

// After the last of `rounds` rounds of a step: the owner words of every operation's
// slots zero, and the moves not done (left out, losers of the last round, refused and fresh ones
// never taken) to the kinetic kernel: few of them as a list, more on the lists of their
// partitions, whose moves run one after another, so that moves that meet do not compete
// (all 3,000 points of one partition moving at once filled the list of moves left for
// later when every warp took one; 85,000 partitions' empty lists cost 100 us to look at).
__device__ __forceinline__ void round_clear(const Dev &d, const Rounds &R, int rounds, int m, const Inst &I, int bits,
                                            const int3 *gmoves, const int2 *old_xy, int *head, int *next, int tid,
                                            int nthreads)
{
    const int4 end = __ldcg(R.cnt + rounds), last = __ldcg(R.cnt + rounds - 1);
    const long long words = (long long)end.w * RT;
    for (long long i = 4ll * tid; i < words; i += 4ll * nthreads) {
        const int4 s = __ldcg(reinterpret_cast<const int4 *>(R.slots + i));
        if (s.x >= 0) d.tn[s.x].w = 0;
        if (s.y >= 0) d.tn[s.y].w = 0;
        if (s.z >= 0) d.tn[s.z].w = 0;
        if (s.w >= 0) d.tn[s.w].w = 0;
    }
    const int nleft = __ldcg(R.left_count), nlost = end.y, fresh = end.x;
    const int ref0 = round_all_refused(R, last), nref = last.z - ref0;
    const int pending = nleft + nlost + nref + m - fresh;
    if (tid == 0) *R.pending = pending;
    for (int i = tid; i < pending; i += nthreads) {
        const int j = i - nleft, k = j - nlost, f = k - nref;
        int item = fresh + f;
        if (j < 0) item = __ldcg(R.left + i);
        else if (k < 0) item = __ldcg(R.lost[rounds & 1] + j);
        else if (f < 0) item = __ldcg(R.refused + ref0 + k);
        const int inst = I.ninst > 1 ? csr_find(I.pofs, I.ninst + 1, gmoves[item].x) : 0;
        if (pending <= I.few_left) R.left[i] = item;
        else next[item] = atomicExch(head + partition_of(I, inst, bits, old_xy[item]), item);
    }
}

__global__ void k_round_clear(Dev d, Rounds R, int rounds, int m, Inst I, int bits, const int3 *gmoves,
                              const int2 *old_xy, int *head, int *next)
{
    if (__ldcg(d.status)) return;
    round_clear(d, R, rounds, d.ctl ? __ldcg(d.ctl) : m, I, bits, gmoves, old_xy, head, next,
                blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x);
}

// A whole small step in one block: clearing, intake, rounds until every move is done (or a
// round does none), and what is left to the kinetic kernel.  The kernels it replaces take
// 2 to 4 us each whatever they do, and a step of a few moves is three rounds of them; but one
// block plans 16 moves at a time and the whole GPU all of them.  us a step with a wait after
// each, one block / whole GPU:
//   moves                                     4      16      32      40      48      64
//   1e6 points, short moves               39 / 48  38 / 51  47 / 51  54 / 54  51 / 51  63 / 51
//   1,000 points, one unit                38 / 49  51 / 62  56 / 61  67 / 65  74 / 71  97 / 99
//   2e5 points, jumps of two spacings     39 / 52  42 / 53  54 / 56  63 / 57  69 / 59  84 / 65
constexpr int SMALL_MOVES = 32;      // two moves a warp, one after the other
constexpr int SMALL_THREADS = 512;
constexpr int SMALL_ROUNDS = 16;
constexpr int SMALL_CELLS = 8192;    // partitions one block clears in passing

__global__ void __launch_bounds__(SMALL_THREADS) k_step_small(Dev d, const int3 *moves, int m, Inst I, int bits,
                                                              int *scal, int nscal, int *head, int ncells, int *next,
                                                              int4 *deferred, int ndef, int2 *old_xy, int3 *gmoves,
                                                              const unsigned long long *dloc2, double far2, Rounds R,
                                                              int *counters, int ncounters)
{
    __shared__ RegionShared<32> shared[SMALL_THREADS / 32];
    __shared__ int sum[8];
    const int tid = threadIdx.x;
    if (d.ctl) {
        m = __ldcg(d.ctl);
        d.stamp = __ldcg(d.ctl + 1);
    }
    // (every phase's writes are seen by the next one's: one block, a fence, a barrier)
    auto phase = [] {
        __threadfence();
        __syncthreads();
    };
    step_clear(scal, nscal, head, ncells, deferred, ndef, counters, ncounters, tid, SMALL_THREADS);
    phase();
    intake(d, step_moves(d, moves), m, I, bits, nullptr, next, old_xy, gmoves, dloc2, far2, tid, SMALL_THREADS);
    phase();
    if (__ldcg(d.status)) return;
    const RoundMoves M{gmoves};
    const RoundBuild B{};
    int b = 0;
    for (int pending = m; b < SMALL_ROUNDS;) {
        round_plan<REGION_MOVE, 32>(d, R, b, M, B, m, 1, shared, tid, SMALL_THREADS);
        phase();
        round_commit<true>(d, R, b, M, m, sum, tid, SMALL_THREADS);
        phase();
        ++b;
        const int4 c = __ldcg(R.cnt + b);
        const int now = c.y + m - c.x;
        if (now == 0 || now == pending) break;
        pending = now;
    }
    round_clear(d, R, b, m, I, bits, gmoves, old_xy, head, next, tid, SMALL_THREADS);
}

// the owner words of slots [s0, s0 + n) zero (after the rounds of a build)
__global__ void k_clear_owner(TriHalf tn, int s0, int n)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) tn[s0 + i].w = 0;
}

// The build's queue: the levels from the coarsest (positions (2j + 1) 2^level of every
// instance), each level's items in a scattered order (a stride coprime with their number,
// near the golden ratio of it), so that the points of one round lie far apart along the
// Hilbert curve.  lvoff: ninst + 1 offsets of this level's items.
__global__ void k_build_queue(RoundBuild B, const int *lvoff, int level, int items, int stride, int *queue)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < items; i += gridDim.x * blockDim.x) {
        const int g = (int)(((long long)i * stride) % items);
        const int inst = B.ninst > 1 ? csr_find(lvoff, B.ninst + 1, g) : 0;
        const int j = g - __ldg(lvoff + inst);
        queue[i] = __ldg(B.pofs + inst) + (int)((2ll * j + 1) << level);
    }
}

// what is still to insert before round b, `nref` refused items included, to the list of the
// warp-wide path
__global__ void k_build_rest(Rounds R, int b, RoundBuild B, const int *refused, int nref)
{
    const int4 c = __ldcg(R.cnt + b);
    const int nlost = c.y, head = c.x, n = nlost + B.total - head;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n + nref; i += gridDim.x * blockDim.x)
        R.left[atomicAdd(R.left_count, 1)] =
            i < nlost ? __ldcg(R.lost[b & 1] + i)
                      : (i < n ? __ldg(B.queue + head + i - nlost) : __ldcg(refused + i - n));
}

// Insertions by one warp each: the staged Bowyer-Watson insertion, else split and flips, with
// claims by compare-and-swap.  The points are those the rounds left out (a cavity above
// their limits; left: the list), or one level of every instance (left null: positions
// (2j + 1) 2^level, lvoff: its item offsets), for which the coarser levels are in already.
// Each warp takes a contiguous run.
__global__ void __launch_bounds__(WPB * 32) k_insert_warps(Dev dp, const int *left, int items, RoundBuild B, int level,
                                                           const int *lvoff)
{
    KD_BLOCK_DEV(dp);
    __shared__ WarpShared shs[WPB];
    int wib = threadIdx.x >> 5;
    int gw = blockIdx.x * (blockDim.x >> 5) + wib;
    int nw = gridDim.x * (blockDim.x >> 5);
    Warp w = make_warp(&shs[wib], gw + 1, gw * 7 + (level + 1) * 1315423911u, d);
    const int per = (items + nw - 1) / nw;
    const int jend = min(items, (gw + 1) * per);
    for (int g = gw * per; g < jend; ++g) {
        if (read_status(d)) break;
        int inst = 0, item;
        if (left) {
            item = __ldcg(left + g);
            if (B.ninst > 1) inst = csr_find(B.pofs, B.ninst + 1, item);
        } else {
            if (B.ninst > 1) inst = csr_find(lvoff, B.ninst + 1, g);
            const int k = B.ninst > 1 ? g - __ldg(lvoff + inst) : g;
            item = __ldg(B.pofs + inst) + (int)((2ll * k + 1) << level);
        }
        const int p0 = __ldg(B.pofs + inst), j = item - p0;
        const int v = __ldg(B.order + item);
        if (B.ninst > 1) set_instance(w, p0, __ldg(B.pofs + inst + 1) - p0);
        if (__shfl_sync(FULL, __ldcg(d.pt_tri + v), 0) >= 0) continue;  // a point of the first triangle
        const int s = __ldg(B.tofs + inst) + 4 + 2 * (j - 2 - (j > __ldg(B.third + inst)));
        int start = -1;
        for (int a = j; start < 0 && a > 0;) {
            a &= a - 1;
            start = __shfl_sync(FULL, __ldcg(d.pt_tri + __ldg(B.order + p0 + a)), 0);
        }
        const int2 q = d.xy[v];
        int rc = insert_staged(w, d, v, q, start, s, s + 1, false);
        if (rc == INS_GLOBAL) rc = insert_point(w, d, v, q, start, s, s + 1, false);
        if (rc) {
            if (rc > 0) set_status(d, rc);
            break;
        }
    }
    flush_counters(w, d);
}

}  // namespace kd
