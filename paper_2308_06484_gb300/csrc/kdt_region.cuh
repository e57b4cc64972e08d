// One operation planned by a group of RL = 16 or 32 lanes on a triangulation that nothing writes
// meanwhile: insert a point (a build), or delete a moved point and insert it at its new
// position (Fig. 4: Delete, Update, Insert; Section IV).  region_plan reads the store,
// computes the triangles the operation destroys and those that replace them, and returns
// them as a list; it changes nothing.  k_round_plan (kdt_rounds.cuh) runs it for many
// operations at once and k_round_commit writes the results of those that do not meet.
//
// One lane holds one item of each kind, in registers: link vertex l of the moved point with
// the ring triangle behind link edge l, and one triangle of the hole the deletion leaves.
//   deletion   Delaunay ears of the link polygon (the simple deletion Section IV prefers):
//              lane l tests the ear that starts at vertex l against every other vertex; all
//              valid ears of a round are clipped (each is a triangle of the hole's unique
//              triangulation, so no two of them share an edge of the polygon, except the
//              two of a quadrilateral).  An ear's triangle belongs to the lane of the vertex
//              it cuts off, so nothing is ever compacted: the polygon is a bit mask.
//   locate     q against every hole triangle at once, else a walk from the ring.
//   insertion  Bowyer-Watson (the insertion Section IV names): the hole and ring
//              triangles in conflict with q at once; when the cavity is the whole hole, the
//              fan around q stands on the link polygon and the lanes already know their
//              neighbours.  Otherwise the cavity grows level by level in shared memory, an
//              edge per lane, and the fan's neighbours are found by their end points.
// A reference is (slot << 2) | edge for a triangle of the store, the complement of (lane
// << 2) | edge for one of the hole.  Ghost triangles (and hull points) need no special
// case: conflict() knows them.
//
// The result is exact (the predicates and their tie-breaking are those of the whole
// library), so it is the unique Delaunay triangulation after this one operation.  An
// operation outside the limits (a degree above RL, a cavity or its border above RL) is
// left to the warp-wide path.
//
// What bounds it: latency.  An operation is a chain of dependent loads (the star two
// triangles at a time, coordinates, ring, or the walk's steps and the cavity's levels) and
// of predicates; the groups of a warp and the warps of an SM overlap theirs.
#pragma once
#include "kdt_predicates.cuh"

namespace kd {

constexpr int RT = 32;     // most triangles an operation writes
constexpr int RWALK = 1 << 12;  // steps of a walk before the operation is left to the other path

enum RegionMode : int { REGION_INSERT = 0, REGION_MOVE = 1, REGION_GUESS = 2 };
// RG_BAIL: outside the limits of RL lanes, RG_LEFT: of any number of lanes
enum RegionResult : int { RG_OK = 0, RG_BAIL = 1, RG_VERTEX = 2, RG_LEFT = 3 };

// What the RL lanes of an operation share (RL: also the largest degree, cavity and border).
template <int RL>
struct RegionShared {
    int pool[RT];                           // the region's slots
    int ba[RL], bb[RL], bc[RL];             // border edges: start, end, reference across
    int gs[RL], gv[RL][3], gn[RL][3];       // cavity triangles of the store
    int2 gx[RL][3];
    int star[RL];                           // star triangles' slots
    unsigned char lnode[RL], hfan[4 * RL];  // hole edge behind each link edge, fan triangle across each hole edge
};

struct RegionOut {
    int nt;           // triangles written (and destroyed, the insertion's two fresh slots included)
    int k;            // degree of the deleted point
    int ncav;         // cavity size
    int edge, ghost;  // q lay on an edge / outside the hull
    int vtx;          // RG_VERTEX: the point q coincides with
    unsigned ex, ti;  // exact predicate calls, ties (this lane's)
    int steps;        // triangles walked through
    int prop;         // the learned proposal: 0 none, 1 a guess, 3 a guess whose triangle holds q
};

__device__ __forceinline__ int rcomp(const int4 &v, int i) { return i == 0 ? v.x : (i == 1 ? v.y : v.z); }
__device__ __forceinline__ int rnext(int e) { return e == 2 ? 0 : e + 1; }
__device__ __forceinline__ int rprev(int e) { return e == 0 ? 2 : e - 1; }
// the set bit of m after / before bit i, round the end
__device__ __forceinline__ int bit_next(unsigned m, int i)
{
    const unsigned a = m & ~((2u << i) - 1u);
    return __ffs((int)(a ? a : m)) - 1;
}
__device__ __forceinline__ int bit_prev(unsigned m, int i)
{
    const unsigned a = m & ((1u << i) - 1u);
    return 31 - __clz((int)(a ? a : m));
}

// MODE REGION_MOVE: delete p (its position is still the old one in d.xy) and insert it at q;
// REGION_GUESS: the same with the learned proposal's guess as the locate's first candidate.
// REGION_INSERT: insert p at q, walking from slot `start`, with the dead slots spare0, spare1.
// All RL lanes of the group (lane l, member mask gm, first lane g0 of the warp) call with
// the same arguments.  out[2 r], out[2 r + 1] receive triangle r < nt: (v0, v1, v2, alive
// flag 1) and (n0, n1, n2, slot); a neighbour outside the region is stored as the
// complement of its reference (its back reference has to follow).  sh.pool holds the slots.
template <int MODE, int RL, class D>
__device__ __forceinline__ int region_plan(const D &d, RegionShared<RL> &sh, int l, unsigned gm, int g0, int p, int2 q,
                                           int start, int spare0, int spare1, int4 *out, RegionOut &o)
{
    constexpr bool MOVE = MODE != REGION_INSERT;
    const int2 zero = make_int2(0, 0);
    auto sh1 = [&](int v, int src) { return __shfl_sync(gm, v, src, RL); };
    auto sh2 = [&](int2 v, int src) { return make_int2(__shfl_sync(gm, v.x, src, RL), __shfl_sync(gm, v.y, src, RL)); };
    auto votes = [&](bool b) { return (__ballot_sync(gm, b) >> g0) & (0xffffffffu >> (32 - RL)); };
    const unsigned below = (1u << l) - 1u;
    o.nt = 0;
    o.k = 0;
    o.ncav = 0;
    o.edge = 0;
    o.ghost = 0;
    o.vtx = -1;
    o.ex = 0;
    o.ti = 0;
    o.steps = 0;
    o.prop = 0;
    int k = 0;
    // this lane's link vertex, its successor, its star triangle, the ring behind its link edge
    int id = -1, idn = -1, S = -1, O = 0, A = -1;
    int2 x = zero, xn = zero, AX = zero;
    // this lane's hole triangle: vertices' lanes, what lies across its edges (0x80 | link edge,
    // or lane << 2 | edge of another), ids and coordinates
    unsigned HM = 0, CH = 0, CR = 0;
    int n0 = 0, n1 = 0, n2 = 0, ia = -1, ib = -1, ic = -1;
    int2 xa = zero, xb = zero, xc = zero;
    bool inhole = false;
    if (MOVE) {
        // ---- the star, walked in both directions at once
        const int t0 = __ldcg(d.pt_tri + p);
        if (t0 < 0 || t0 >= d.cap) return RG_BAIL;
        int nf = 0, nbk = 0, tf = t0, tb = -1;
        while (true) {
            int4 fv, fn, bv = make_int4(0, 0, 0, 0), bn = bv;
            fv = __ldcg(d.tv + tf);
            fn = __ldcg(d.tn + tf);
            if (tb >= 0) {
                bv = __ldcg(d.tv + tb);
                bn = __ldcg(d.tn + tb);
            }
            const int If = fv.x == p ? 0 : (fv.y == p ? 1 : (fv.z == p ? 2 : -1));
            if (!(fv.w & 1) || If < 0 || nf + nbk + 1 > RL) return RG_BAIL;
            if (l == nf) {
                S = tf;
                id = rcomp(fv, rnext(If));
                O = rcomp(fn, If);
            }
            ++nf;
            const int fnx = rcomp(fn, rnext(If)) >> 2;
            if (tb < 0) {
                const int fpv = rcomp(fn, rprev(If)) >> 2;
                if (fnx < 0 || fnx >= d.cap || fpv < 0 || fpv >= d.cap || fnx == t0 || fnx == fpv) return RG_BAIL;
                tf = fnx;
                tb = fpv;
                continue;
            }
            if (tb == tf) break;  // both directions reached the same triangle
            const int Ib = bv.x == p ? 0 : (bv.y == p ? 1 : (bv.z == p ? 2 : -1));
            if (!(bv.w & 1) || Ib < 0 || nf + nbk + 1 > RL) return RG_BAIL;
            if (l == RL - 1 - nbk) {  // (kept at the top until the degree is known)
                S = tb;
                id = rcomp(bv, rnext(Ib));
                O = rcomp(bn, Ib);
            }
            ++nbk;
            const int bpv = rcomp(bn, rprev(Ib)) >> 2;
            if (fnx == tb) break;
            if (fnx < 0 || fnx >= d.cap || bpv < 0 || bpv >= d.cap) return RG_BAIL;
            tf = fnx;
            tb = bpv;
        }
        k = nf + nbk;
        if (k < 3) return RG_BAIL;
        {
            const int src = l < nf ? l : (l < k ? RL - k + l : l);
            S = sh1(S, src);
            id = sh1(id, src);
            O = sh1(O, src);
        }
        const bool inl = l < k;
        if (inl) {
            if ((O >> 2) < 0 || (O >> 2) >= d.cap) O = 0;
            if (id >= 0) x = __ldcg(d.xy + id);
            A = __ldcg(reinterpret_cast<const int *>(d.tv + (O >> 2)) + (O & 3));
            if (A >= 0) AX = __ldcg(d.xy + A);
        }
        const int ln = l + 1 < k ? l + 1 : 0;
        idn = sh1(id, ln);
        xn = sh2(x, ln);
        const unsigned gh = votes(inl && id < 0);
        if (gh) {
            // a hull point whose other link vertices lie on one line: its deletion may leave
            // nothing but that line (the other path decides)
            const int g = __ffs((int)gh) - 1, f0 = g + 1 < k ? g + 1 : 0, f1 = f0 + 1 < k ? f0 + 1 : 0;
            const int2 x0 = sh2(x, f0), x1 = sh2(x, f1);
            if (!votes(inl && id >= 0 && orient2d(x0, x1, x) != 0)) return RG_LEFT;
        }
        // ---- 1. delete: ears
        unsigned alive = 0xffffffffu >> (32 - k);
        int m = k, eo = 0x80 | l, ta = 0, tb3 = 0, tc = 0;
        bool has = false, pend = false;  // has a triangle; its last edge's neighbour still open
        while (m > 3) {
            const int i1 = bit_next(alive, l), i2 = bit_next(alive, i1);
            const int id1 = sh1(id, i1), id2 = sh1(id, i2);
            const int2 x1 = sh2(x, i1), x2 = sh2(x, i2);
            bool ok = (alive >> l) & 1u;
            if (ok && id >= 0 && id1 >= 0 && id2 >= 0) ok = orient2d(x, x1, x2) > 0;
            int c = i2;
            for (int t = 3; t < m; ++t) {
                c = bit_next(alive, c);
                const int idc = sh1(id, c);
                const int2 xcc = sh2(x, c);
                if (ok) ok = !conflict(id, id1, id2, x, x1, x2, idc, xcc, d.use_filter, &o.ex, &o.ti);
            }
            unsigned sel = votes(ok);
            if (m == 4) sel &= 0u - sel;
            if (sel == 0 || __popc(sel) > m - 3) return RG_BAIL;
            // the vertex after an ear's first goes; its lane takes the ear
            const int pv = bit_prev(alive, l);
            const bool rem = ((alive >> l) & 1u) && ((sel >> pv) & 1u);
            const unsigned removed = votes(rem);
            const int eop = sh1(eo, pv);
            if (pend) {
                // the polygon edge that starts at vertex ta was this triangle's: used now?
                if ((removed >> ta) & 1u) {
                    n1 = ta << 2;
                    pend = false;
                } else if ((sel >> ta) & 1u) {
                    n1 = bit_next(alive, ta) << 2 | 2;
                    pend = false;
                }
            }
            if (rem) {
                ta = pv;
                tb3 = l;
                tc = i1;
                n0 = eo;
                n2 = eop;
                has = true;
                pend = true;
            }
            if ((sel >> l) & 1u) eo = i1 << 2 | 1;
            alive &= ~removed;
            m -= __popc(removed);
        }
        {
            const int f = __ffs((int)alive) - 1, f1 = bit_next(alive, f), f2 = bit_next(alive, f1);
            const int e1 = sh1(eo, f1), e2 = sh1(eo, f2);
            if (pend) n1 = f << 2 | (ta == f ? 2 : (ta == f1 ? 0 : 1));
            if (l == f) {
                ta = f;
                tb3 = f1;
                tc = f2;
                n0 = e1;
                n1 = e2;
                n2 = eo;
                has = true;
            }
        }
        HM = votes(has);
        ia = sh1(id, ta);
        ib = sh1(id, tb3);
        ic = sh1(id, tc);
        xa = sh2(x, ta);
        xb = sh2(x, tb3);
        xc = sh2(x, tc);
        // the learned proposal's guess (made by the step planner for this move): the rank of
        // the hole triangle it names, as hole_rank and move_wedge define it.  (1e6 points,
        // 4096 moves, planner on the tensor cores: 190 us a step with one warp a move, 121 so.)
        int rank = -1, guess = -2;
        if constexpr (MODE == REGION_GUESS) if (!gh) {
            const int2 po = __ldcg(d.xy + p);
            const long long dx = (long long)q.x - po.x, dy = (long long)q.y - po.y;
            const long long ax = (long long)x.x - po.x, ay = (long long)x.y - po.y;
            const long long bx = (long long)xn.x - po.x, by = (long long)xn.y - po.y;
            const unsigned wm = votes(inl && ax * dy - ay * dx >= 0 && dx * by - dy * bx > 0);
            if (__popc(wm) == 1) {
                const int j0 = __ffs((int)wm) - 1;
                const int ra = ta - j0 < 0 ? ta - j0 + k : ta - j0, rb = tb3 - j0 < 0 ? tb3 - j0 + k : tb3 - j0,
                          rc = tc - j0 < 0 ? tc - j0 + k : tc - j0;
                const int lo = min(ra, min(rb, rc)), hi = max(ra, max(rb, rc)), mid = ra + rb + rc - lo - hi;
                const int key = lo << 12 | mid << 6 | hi;
                rank = 0;
                for (unsigned b = HM; b; b &= b - 1u) rank += sh1(key, __ffs((int)b) - 1) < key;
                if (!has) rank = -1;
                guess = (int)__ldcg(d.pguess + p);
                o.prop = 1;
            }
        }
        // ---- 2. locate q in the hole (first the triangle the proposal names)
        {
            bool in = false, out_ = false;
            int zeros = 0, vt = -1;
            if (has) {
                if (ia >= 0 && ib >= 0 && ic >= 0) {
                    const int o0 = orient2d(xb, xc, q), o1 = orient2d(xc, xa, q), o2 = orient2d(xa, xb, q);
                    in = o0 >= 0 && o1 >= 0 && o2 >= 0;
                    zeros = (o0 == 0) + (o1 == 0) + (o2 == 0);
                    vt = o0 != 0 ? ia : (o1 != 0 ? ib : ic);
                } else {
                    out_ = orient2d(ia < 0 ? xb : (ib < 0 ? xc : xa), ia < 0 ? xc : (ib < 0 ? xa : xb), q) > 0;
                }
            }
            unsigned inm = votes(in);
            const unsigned om = votes(out_), pm = o.prop ? votes(in && zeros < 2 && rank == guess) : 0u;
            if (pm) {
                inm = pm;
                o.prop = 3;
            }
            if (inm) {
                const int src = __ffs((int)inm) - 1;
                zeros = sh1(zeros, src);
                vt = sh1(vt, src);
                if (zeros >= 2) {
                    o.vtx = vt;
                    return RG_VERTEX;
                }
                o.edge = zeros;
                inhole = true;
            } else if (om) {
                o.ghost = 1;
                inhole = true;
            } else {
                // outside the link polygon: walk from the ring triangle across an edge q is beyond
                const unsigned bm = votes(inl && id >= 0 && idn >= 0 && orient2d(x, xn, q) < 0);
                start = sh1(O, bm ? __ffs((int)bm) - 1 : 0) >> 2;
            }
        }
        o.k = k;
    }
    int ng = 0, nb = 0;
    if (!inhole) {
        // ---- visibility walk (exact orientations; the triangulation is Delaunay, so it ends)
        int t = start;
        while (true) {
            if (t < 0 || t >= d.cap) return RG_BAIL;
            if (++o.steps > RWALK) return RG_LEFT;
            const int4 v = __ldcg(d.tv + t), n = __ldcg(d.tn + t);
            if (!(v.w & 1)) return RG_BAIL;
            const int2 a = v.x >= 0 ? __ldcg(d.xy + v.x) : zero, b = v.y >= 0 ? __ldcg(d.xy + v.y) : zero,
                       c = v.z >= 0 ? __ldcg(d.xy + v.z) : zero;
            const int g = v.x < 0 ? 0 : (v.y < 0 ? 1 : (v.z < 0 ? 2 : -1));
            int go = -1;
            if (g >= 0) {
                if (orient2d(g == 0 ? b : (g == 1 ? c : a), g == 0 ? c : (g == 1 ? a : b), q) > 0) o.ghost = 1;
                else go = g;  // across the finite edge
            } else {
                const int o0 = orient2d(b, c, q), o1 = orient2d(c, a, q), o2 = orient2d(a, b, q);
                // the edge tried first changes from step to step
                const int r = o.steps % 3;
                if (r == 0) go = o0 < 0 ? 0 : (o1 < 0 ? 1 : (o2 < 0 ? 2 : -1));
                else if (r == 1) go = o1 < 0 ? 1 : (o2 < 0 ? 2 : (o0 < 0 ? 0 : -1));
                else go = o2 < 0 ? 2 : (o0 < 0 ? 0 : (o1 < 0 ? 1 : -1));
                if (go < 0) {
                    const int zeros = (o0 == 0) + (o1 == 0) + (o2 == 0);
                    if (zeros >= 2) {
                        o.vtx = o0 != 0 ? v.x : (o1 != 0 ? v.y : v.z);
                        return RG_VERTEX;
                    }
                    o.edge = zeros;
                }
            }
            if (go < 0) {
                if (l == 0) {
                    sh.gs[0] = t;
                    sh.gv[0][0] = v.x;
                    sh.gv[0][1] = v.y;
                    sh.gv[0][2] = v.z;
                    sh.gn[0][0] = n.x;
                    sh.gn[0][1] = n.y;
                    sh.gn[0][2] = n.z;
                    sh.gx[0][0] = a;
                    sh.gx[0][1] = b;
                    sh.gx[0][2] = c;
                }
                ng = 1;
                break;
            }
            t = rcomp(n, go) >> 2;
        }
        if (MOVE && votes(l < k && S == t)) return RG_BAIL;  // (q is outside the star)
    }
    // ---- 3. the cavity: the hole and ring triangles in conflict with q
    if (MOVE) {
        CH = votes(((HM >> l) & 1u) && conflict(ia, ib, ic, xa, xb, xc, p, q, d.use_filter, &o.ex, &o.ti));
        CR = votes(l < k && conflict(A, idn, id, AX, xn, x, p, q, d.use_filter, &o.ex, &o.ti));
    }
    if (MOVE && inhole && CH == HM && CR == 0) {
        // the whole hole and no more: the fan stands on the link polygon, triangle l in the
        // star's slot l
        const int Sn = sh1(S, l + 1 < k ? l + 1 : 0), Sp = sh1(S, l > 0 ? l - 1 : k - 1);
        if (l < k) {
            sh.pool[l] = S;
            out[2 * l] = make_int4(p, id, idn, 1);
            out[2 * l + 1] = make_int4(~O, (Sn << 2) | 2, (Sp << 2) | 1, S);
        }
        o.nt = k;
        o.ncav = k - 2;
        __syncwarp(gm);
        return RG_OK;
    }
    // what lies across edge f of this lane's hole triangle
    if (MOVE) {
        // the ring triangles in conflict (each once) join the cavity
        if (l < k) sh.star[l] = S;
        if ((HM >> l) & 1u) {
            if (n0 & 0x80) sh.lnode[n0 & 0x7f] = (unsigned char)(l << 2);
            if (n1 & 0x80) sh.lnode[n1 & 0x7f] = (unsigned char)(l << 2 | 1);
            if (n2 & 0x80) sh.lnode[n2 & 0x7f] = (unsigned char)(l << 2 | 2);
        }
        __syncwarp(gm);
        if (CR) {
            bool add = (CR >> l) & 1u;
            for (unsigned r = CR; r; r &= r - 1u) {
                const int i = __ffs((int)r) - 1, o2 = sh1(O, i);
                if (i < l && (o2 >> 2) == (O >> 2)) add = false;
            }
            if (ng && sh.gs[0] == (O >> 2)) add = false;
            const unsigned am = votes(add);
            if (ng + __popc(am) > RL) return RG_BAIL;
            if (add) {
                const int at = ng + __popc(am & below), f = O & 3;
                const int4 n = __ldcg(d.tn + (O >> 2));
                sh.gs[at] = O >> 2;
                sh.gn[at][0] = n.x;
                sh.gn[at][1] = n.y;
                sh.gn[at][2] = n.z;
                sh.gv[at][f] = A;
                sh.gv[at][rnext(f)] = idn;
                sh.gv[at][rprev(f)] = id;
                sh.gx[at][f] = AX;
                sh.gx[at][rnext(f)] = xn;
                sh.gx[at][rprev(f)] = x;
            }
            ng += __popc(am);
        }
        // border edges of the hole triangles in the cavity
#pragma unroll
        for (int f = 0; f < 3; ++f) {
            const int nc = f == 0 ? n0 : (f == 1 ? n1 : n2);
            const bool link = (nc & 0x80) != 0;
            const int Oi = sh1(O, link ? nc & 0x7f : l);
            const bool bd = ((CH >> l) & 1u) && (link ? !((CR >> (nc & 0x7f)) & 1u) : !((CH >> (nc >> 2)) & 1u));
            const unsigned bm = votes(bd);
            if (nb + __popc(bm) > RL) return RG_BAIL;
            if (bd) {
                const int at = nb + __popc(bm & below);
                sh.ba[at] = f == 0 ? ib : (f == 1 ? ic : ia);
                sh.bb[at] = f == 0 ? ic : (f == 1 ? ia : ib);
                sh.bc[at] = link ? Oi : ~nc;
            }
            nb += __popc(bm);
        }
    }
    __syncwarp(gm);
    // the cavity triangles of the store, level by level: an edge per lane; a triangle across
    // one in conflict joins, otherwise the edge is on the border
    for (int done = 0; done < ng;) {
        const int end = ng;
        for (int c0 = 3 * done; c0 < 3 * end; c0 += RL) {
            const int c = c0 + l, j = c / 3, e = c - 3 * j;
            bool act = c < 3 * end;
            int ref = 0, hole = -1, a = -1, b = -1, ap = -1;
            int2 pa = zero, pb = zero, px = zero;
            int4 n = make_int4(0, 0, 0, 0);
            bool cf = false;
            if (act) {
                ref = sh.gn[j][e];
                a = sh.gv[j][rnext(e)];
                b = sh.gv[j][rprev(e)];
                pa = sh.gx[j][rnext(e)];
                pb = sh.gx[j][rprev(e)];
                for (int t = 0; t < ng; ++t)
                    if (sh.gs[t] == (ref >> 2)) act = false;  // an edge inside the cavity
                if (MOVE)
                    for (int t = 0; t < k; ++t)
                        if (sh.star[t] == (ref >> 2)) hole = sh.lnode[t];
            }
            if (act && ((ref >> 2) < 0 || (ref >> 2) >= d.cap)) act = false;  // (never: the border check fails)
            if (act && hole < 0) {
                ap = __ldcg(reinterpret_cast<const int *>(d.tv + (ref >> 2)) + (ref & 3));
                n = __ldcg(d.tn + (ref >> 2));
                if (ap >= 0) px = __ldcg(d.xy + ap);
                cf = conflict(ap, b, a, px, pb, pa, p, q, d.use_filter, &o.ex, &o.ti);
            }
            // (two edges can lead to the same triangle when the search began at several)
            const unsigned same = __match_any_sync(gm, cf ? (ref >> 2) : -1 - l) >> g0;
            const unsigned addm = votes(cf && !(same & below));
            const bool bd = act && (hole >= 0 ? !((CH >> (hole >> 2)) & 1u) : !cf);
            const unsigned bm = votes(bd);
            if (ng + __popc(addm) > RL || nb + __popc(bm) > RL) return RG_BAIL;
            if ((addm >> l) & 1u) {
                const int at = ng + __popc(addm & below), f = ref & 3;
                sh.gs[at] = ref >> 2;
                sh.gn[at][0] = n.x;
                sh.gn[at][1] = n.y;
                sh.gn[at][2] = n.z;
                sh.gv[at][f] = ap;
                sh.gv[at][rnext(f)] = b;
                sh.gv[at][rprev(f)] = a;
                sh.gx[at][f] = px;
                sh.gx[at][rnext(f)] = pb;
                sh.gx[at][rprev(f)] = pa;
            }
            if (bd) {
                const int at = nb + __popc(bm & below);
                sh.ba[at] = a;
                sh.bb[at] = b;
                sh.bc[at] = hole >= 0 ? ~hole : ref;
            }
            ng += __popc(addm);
            nb += __popc(bm);
            __syncwarp(gm);
        }
        done = end;
    }
    const int ncav = __popc(CH) + ng, nt = MOVE ? k + ng : ng + 2;
    // (a disk: two more border edges than triangles)
    if (nb != ncav + 2 || nt > RT) return RG_BAIL;
    // ---- 4. the new triangles: the fan around q in slots 0 .. nb-1 of the region, then the
    // hole triangles outside the cavity
    if (MOVE) {
        if (l < k) sh.pool[l] = S;
        if (l < ng) sh.pool[k + l] = sh.gs[l];
    } else {
        if (l < ng) sh.pool[l] = sh.gs[l];
        if (l < 2) sh.pool[ng + l] = l ? spare1 : spare0;
    }
    const unsigned surv = HM & ~CH;
    int bcl = 0, al = -1, bl = -1, nx = -1, pv = -1;
    if (l < nb) {
        al = sh.ba[l];
        bl = sh.bb[l];
        bcl = sh.bc[l];
        if (bcl < 0) sh.hfan[~bcl] = (unsigned char)l;  // the hole triangle there gets fan triangle l across
        for (int t = 0; t < nb; ++t) {
            if (sh.ba[t] == bl) nx = t;
            if (sh.bb[t] == al) pv = t;
        }
    }
    if (votes(l < nb && (nx < 0 || pv < 0))) return RG_BAIL;
    __syncwarp(gm);
    if (l < nb) {
        const int s = sh.pool[l];
        int r0 = ~bcl;
        if (bcl < 0) {
            const int h = (~bcl) >> 2;
            r0 = sh.pool[nb + __popc(surv & ((1u << h) - 1u))] << 2 | ((~bcl) & 3);
        }
        out[2 * l] = make_int4(p, al, bl, 1);
        out[2 * l + 1] = make_int4(r0, (sh.pool[nx] << 2) | 2, (sh.pool[pv] << 2) | 1, s);
    }
    if (MOVE) {
        const bool sv = (surv >> l) & 1u;
        const int at = nb + __popc(surv & below);
        int r[3];
#pragma unroll
        for (int f = 0; f < 3; ++f) {
            const int nc = f == 0 ? n0 : (f == 1 ? n1 : n2);
            const bool link = (nc & 0x80) != 0;
            const int Oi = sh1(O, link ? nc & 0x7f : l);
            r[f] = 0;
            if (sv) {
                const bool cav = link ? ((CR >> (nc & 0x7f)) & 1u) != 0 : ((CH >> (nc >> 2)) & 1u) != 0;
                if (cav) r[f] = sh.pool[sh.hfan[l << 2 | f]] << 2;
                else if (link) r[f] = ~Oi;
                else r[f] = sh.pool[nb + __popc(surv & ((1u << (nc >> 2)) - 1u))] << 2 | (nc & 3);
            }
        }
        if (sv) {
            out[2 * at] = make_int4(ia, ib, ic, 1);
            out[2 * at + 1] = make_int4(r[0], r[1], r[2], sh.pool[at]);
        }
    }
    o.nt = nt;
    o.ncav = ncav;
    __syncwarp(gm);
    return RG_OK;
}

}  // namespace kd
