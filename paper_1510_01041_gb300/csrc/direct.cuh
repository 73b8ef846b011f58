// direct.cuh -- one-kernel exact branch-and-bound over slopes (sm_103a).
//
// The LMS value is min over slopes s of w(s), the narrowest vertical window
// holding h of the projections z_k(s) = y_k - s x_k, attained at a pairwise
// slope (Sec. 3.1, 3.3).  A team of CTAs (one CTA, or one thread-block
// cluster) keeps a stack of slope intervals.  Groups of G threads take the
// leftmost ones and answer one question each:
//
//   can some slope of [A, B] have a window no wider than U?
//
// For s in [A, B] point k projects into [lo_k, hi_k], the hull of its
// projections at A and B.  If w(s) <= U, the window [t, t + U] meets at least
// h of those hulls, so t lies in at least h of the intervals
// [lo_k - U, hi_k].  The group builds the histogram of interval starts and
// ends over bins of t (starts rounded down, ends up), takes the running sum
// and drops the interval when no bin reaches depth h: nothing is sorted.
// When some bins do, the same pass is repeated on the hull of those bins with
// finer bins, until the answer is no, the bins are exact or fine enough.
// (Sorting the hull ends, which the tree of bnb.cu did before, asks for the
// same bound: it cost 990 instructions a point at n = 8192, a histogram pass
// about 25.)  A surviving interval's midpoint gives an upper bound of the
// optimum the same way (ub_at); the interval is then cut at sampled pair
// slopes or into equal parts.  The upper bounds of each level sit near the
// best of the level, so the number of tests hardly grows with n: ordinary sets
// (lines, random points, curves, lattices, digitised lines) of 300 to 4096
// points take 7 to 20 phases, 130 to 1300 interval tests and score at most 10
// slopes.
//
// Intervals expected to hold few pair slopes are leaves.  The pairs of a leaf
// [A, B) are found by hashing the points into cells of z(A) as wide as a pair
// of the leaf can be apart, X (B - A): only points in one cell or neighbouring
// cells can form such a pair.  (Narrow leaves are tried by reduced fractions,
// see list_pairs.)  The distinct slopes found, each with a dx that it has, are
// sorted and go through the same interval test as runs of slopes; single
// slopes that survive are scored exactly, from histograms of the exact
// integers down to single values (all projections sorted where those stay
// wide, and kept sorted from slope to slope where many survive).  The smallest
// index pair is looked for at the best slope alone (line_pair).  Ties: an interval right of the best slope
// so far only survives if it can be strictly narrower (widths at pair slopes
// are rationals with denominators below 2^16, so two different ones differ by
// more than 2^-32, one unit), so the lexicographic minimum over (w, theta1,
// theta2, pair) is the one of every other path.
//
// The stack is taken from the left and each node has at most NODE_F children, so
// it holds a few levels' worth of siblings (a fit whose stack would overflow
// is reported, never answered wrongly); leaves that hold more distinct slopes
// than the list are cut until they fit.  No thread waits on memory: teams of several CTAs meet at the
// hardware cluster barrier.
#pragma once

#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "kernels.cuh"
#include "lms.h"

// Counters of the host build that the tests make of this file (one thread a
// group, T = G = 1): phases by mode and what each works on.
#ifndef LMS_DIRECT_COUNT
#define LMS_DIRECT_COUNT(what, n)
#endif

namespace lms {
namespace direct {

constexpr long long D_MAX = 0x7fffffffffffffffLL;
constexpr long long D_GUARD = 1LL << 46;   // slope keys beyond it are used in units of 2^-26 (no overflow)
constexpr int F_YS = 29;                   // float sets: units of 2^-29 of a grid step, slope keys of 2^-29
constexpr int F_BITS = 29;                 // .. grid coordinates below 2^F_BITS
constexpr long long F_KMAX = 1LL << 32;    // .. and slopes (of the scaled axes) below 8: projections below 2^62
constexpr int STEEP = 6;                   // .. that is, without their last bits
constexpr int NODE_F = 4;                  // children of an interval
constexpr int EV_F = 8;                    // children of a run of slopes
constexpr int TABLE = 2048;                // slots of a CTA's slope table
constexpr float LEAF_FRACTIONS = 32.0f;      // an interval with this few possible slopes is a leaf
constexpr float FRACTIONS = 1000.0f;         // expected fractions of a leaf up to which they are tried one by one
constexpr int REGROW = 3;                    // .. times that leaves are cut instead when they hold more
constexpr float LIST_HOPE = 4.0f;            // .. leaves are listed together up to so many lists of expected slopes
constexpr int CELLS_MAX = 8192;             // cells of the pair search
constexpr float DENSE = 16384.0f;            // candidates up to which a leaf's pairs are searched in the cells ..
constexpr float DENSE_PER_POINT = 64.0f;     // .. and so many more for each point (ordinary sets: at most 30 a point)
constexpr float F_DENSE = 8388608.0f;        // .. of a float set, which is left to the sweep beyond (no fractions there)
constexpr int WIDE_ITEMS = 2;              // up to so many questions a CTA, the whole CTA works on each
constexpr int DEPTH_MAX = 28;              // levels: 2^49 keys come down to one in at most 28 cuts (tails included)
// A float set is left to the sweep beyond these (ordinary sets: at most 13 phases, 1 cut, 130 slopes scored).
constexpr int F_SCORES = 256;              // slopes scored
constexpr int F_PHASES = 48;
constexpr int F_CUTS = 6;                  // lists that did not hold their leaves' slopes
constexpr int PHASES_MAX = 1 << 20;        // phases of one fit before it is reported as failed
constexpr int RUN_MIN = 12;                // slopes a CTA scores from which it keeps the points sorted between them
constexpr int EXCHANGES = 16;              // passes that repair their order, else they are sorted again
// A small set of a batch is left to the per-slope kernel beyond these (ordinary
// sets up to 256 points: at most 16 phases and 12 slopes scored).
constexpr int SMALL_PHASES = 20;
constexpr int SMALL_SCORES = 64;
constexpr int EV_DEPTH = 6;                // levels of a run of at most EV_F^EV_DEPTH slopes

struct DNode {
    long long a, b;     // slope keys [a, b), or a run of sorted slopes [a, b)
    long long t0, t1;   // where a narrow enough window can start (t0 > t1: not known yet)
    float est;          // expected pairs
    int force;          // levels to cut whatever is expected
};

enum Mode { M_TREE, M_PAIRS, M_EVENT, M_EXACT, M_DONE };

// What the CTAs of a team share, in global memory.
struct TeamState {
    long long ub;                // upper bound of the LMS value, units of 2^-32
    int nlist[2], over[2];       // distinct slopes listed (by turns); 1: too many, 2: too many candidates
    int bad;                     // a consistency check failed
    unsigned pair[2];            // smallest index pair of a slope (by turns)
};

// Answer to an interval test.
struct Answer {
    long long t0, t1;
    int keep, dense;   // dense: the pair search of a leaf was left out
};

// Best float candidate: lexicographic (w, theta1, theta2, pair).
struct CandD {
    double w, s, t;
    unsigned pair;
    int valid;
};

// Sizes of one team's memory; the same on the host and the device.
struct TeamShape {
    int PM;      // work items of a phase, leaves held
    int LC;
    int HC;      // slopes listed at a time (power of two)
    int Q;       // root intervals
    float leaf;  // expected pairs of a leaf
    long long ptsn;   // points kept in global memory (0: in shared memory)
    long long dupw;   // words of one bit a point
    long long sortw;  // bytes of global sort scratch per CTA
    int C;       // CTAs of a team
};

__host__ __device__ inline long long d_up(long long v) { return (v + 255) & ~255LL; }
__host__ __device__ inline int stack_cap(const TeamShape &s) { return s.Q + 2 + s.LC + s.PM * NODE_F * DEPTH_MAX; }
__host__ __device__ inline int estack_cap(const TeamShape &s) { return s.PM * EV_F * EV_DEPTH; }

struct TeamMem {
    TeamState *st;
    DNode *stack, *estack;
    Answer *ans;
    long long *lkey;      // listed slopes and their dx, as found
    unsigned *lden;
    long long *ev;        // the same by ascending slope
    unsigned *evd;
    Cand *xres;
    int *pts;
    unsigned *dup;        // points that repeat an earlier one (marked when asked for)
    unsigned char *sort;
};

__host__ __device__ inline long long team_bytes(const TeamShape &s)
{
    return d_up(sizeof(TeamState)) + d_up(sizeof(DNode) * (long long)stack_cap(s)) +
           d_up(sizeof(DNode) * (long long)estack_cap(s)) + d_up(2 * sizeof(Answer) * (long long)s.PM) +
           2 * d_up(8LL * s.HC) +
           2 * d_up(4LL * s.HC) + d_up(sizeof(CandD) * (long long)s.PM) + d_up(4LL * s.ptsn) + d_up(4LL * s.dupw) +
           d_up(s.sortw) * s.C;
}

__device__ inline TeamMem team_carve(unsigned char *p, const TeamShape &s)
{
    TeamMem m;
    auto take = [&](long long b) { unsigned char *r = p; p += d_up(b); return r; };
    m.st = reinterpret_cast<TeamState *>(take(sizeof(TeamState)));
    m.stack = reinterpret_cast<DNode *>(take(sizeof(DNode) * (long long)stack_cap(s)));
    m.estack = reinterpret_cast<DNode *>(take(sizeof(DNode) * (long long)estack_cap(s)));
    m.ans = reinterpret_cast<Answer *>(take(2 * sizeof(Answer) * (long long)s.PM));
    m.lkey = reinterpret_cast<long long *>(take(8LL * s.HC));
    m.lden = reinterpret_cast<unsigned *>(take(4LL * s.HC));
    m.ev = reinterpret_cast<long long *>(take(8LL * s.HC));
    m.evd = reinterpret_cast<unsigned *>(take(4LL * s.HC));
    m.xres = reinterpret_cast<Cand *>(take(sizeof(CandD) * (long long)s.PM));   // or CandD
    m.pts = reinterpret_cast<int *>(take(4LL * s.ptsn));
    m.dup = reinterpret_cast<unsigned *>(take(4LL * s.dupw));
    m.sort = p;
    return m;
}

// Bounding box of the centred points.
struct Box {
    int xc, yc;                  // centre taken off every point
    int xlo, xhi, ylo, yhi;      // centred extremes
    int dh;                      // any h points span at least this in x
};

// ------------------------------------------------------------------ hardware
__device__ __forceinline__ unsigned cluster_ctas()
{
    unsigned v;
    asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(v));
    return v;
}
__device__ __forceinline__ unsigned cluster_rank()
{
    unsigned v;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(v));
    return v;
}
__device__ __forceinline__ unsigned smem_size()
{
    unsigned v;
    asm("mov.u32 %0, %%dynamic_smem_size;" : "=r"(v));
    return v;
}
// every thread of the cluster; global writes before it are seen after it
__device__ __forceinline__ void cluster_meet()
{
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
template <int G>
__device__ __forceinline__ void group_meet(int id)
{
    asm volatile("bar.sync %0, %1;" ::"r"(1 + id), "n"(G) : "memory");
}
__device__ __forceinline__ Cand ld_cand(const Cand *p)
{
    const longlong2 a = __ldcg(reinterpret_cast<const longlong2 *>(p));
    const int4 b = __ldcg(reinterpret_cast<const int4 *>(p) + 1);
    Cand c;
    c.w = a.x;
    c.t = a.y;
    c.dy = b.x;
    c.dx = b.y;
    c.i = b.z;
    c.j = b.w;
    return c;
}

// nodes written by another CTA: read past this SM's L1
__device__ __forceinline__ DNode ld_node(const DNode *p)
{
    DNode d;
    d.a = __ldcg(&p->a);
    d.b = __ldcg(&p->b);
    d.t0 = __ldcg(&p->t0);
    d.t1 = __ldcg(&p->t1);
    d.est = __ldcg(&p->est);
    d.force = __ldcg(&p->force);
    return d;
}

// ------------------------------------------------------------------ groups
// G threads that work on one question.  G = 32: a warp; larger groups meet at
// a named barrier of their own.
template <int G>
struct Group {
    static constexpr int SIZE = G;
    int id, lane;
    long long *red;   // 4 words per warp of the group, shared memory
    __device__ __forceinline__ void sync() const
    {
        if constexpr (G <= 32) __syncwarp();
        else group_meet<G>(id);
    }
    __device__ __forceinline__ long long min_ll(long long v) const
    {
        if constexpr (G >= 32) {
#pragma unroll
            for (int s = 16; s >= 1; s >>= 1) v = min(v, __shfl_xor_sync(FULL, v, s));
            if constexpr (G > 32) {
                if ((lane & 31) == 0) red[lane >> 5] = v;
                sync();
                v = red[(lane & 31) % (G / 32)];
#pragma unroll
                for (int s = 16; s >= 1; s >>= 1) v = min(v, __shfl_xor_sync(FULL, v, s));
                sync();
            }
        }
        return v;
    }
    // lane 0's value
    __device__ __forceinline__ long long first(long long v) const
    {
        if constexpr (G >= 32) {
            v = __shfl_sync(FULL, v, 0);
            if constexpr (G > 32) {
                if (lane == 0) red[0] = v;
                sync();
                v = red[0];
                sync();
            }
        }
        return v;
    }
    // minima of two ints and maxima of two ints
    __device__ __forceinline__ void min2_max2(int &a, int &b, int &c, int &d) const
    {
        if constexpr (G >= 32) {
            a = __reduce_min_sync(FULL, a);
            b = __reduce_min_sync(FULL, b);
            c = __reduce_max_sync(FULL, c);
            d = __reduce_max_sync(FULL, d);
            if constexpr (G > 32) {
                int4 *r = reinterpret_cast<int4 *>(red);
                if ((lane & 31) == 0) r[lane >> 5] = make_int4(a, b, c, d);
                sync();
                const int4 v = r[(lane & 31) % (G / 32)];
                a = __reduce_min_sync(FULL, v.x);
                b = __reduce_min_sync(FULL, v.y);
                c = __reduce_max_sync(FULL, v.z);
                d = __reduce_max_sync(FULL, v.w);
                sync();
            }
        }
    }
    // exclusive prefix sum over the group
    __device__ __forceinline__ int scan_ex(int v) const
    {
        if constexpr (G >= 32) {
            int x = v;
            const int l = lane & 31;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const int o = __shfl_up_sync(FULL, x, d);
                if (l >= d) x += o;
            }
            if constexpr (G > 32) {
                int *r = reinterpret_cast<int *>(red);
                if (l == 31) r[lane >> 5] = x;
                sync();
                const int base = (int)__reduce_add_sync(FULL, l < (lane >> 5) ? (unsigned)r[l] : 0u);
                sync();
                return base + x - v;
            }
            return x - v;
        }
        return 0;
    }
};

// Histogram slot of bin b.  Threads walk their own runs of PER = NB / G bins;
// with long runs the index is XORed with the row inside each row of 32 bins,
// so the lanes of a warp never meet on a bank.
template <int PER>
__device__ __forceinline__ int slot_of(int b)
{
    if constexpr (PER <= 8) return b;
    return (b & ~31) | ((b ^ (b >> 5)) & 31);
}

// Float points are quantised to a grid of 2^30 steps a side (int2, see
// k_direct); every other set is packed in 16-bit halves.
using ::lms::px;
using ::lms::py;
__device__ __forceinline__ int px(int2 p) { return p.x; }
__device__ __forceinline__ int py(int2 p) { return p.y; }

__device__ __forceinline__ int packed_of(int p) { return p; }
__device__ __forceinline__ int packed_of(int2) { return 0; }

// z at slope K 2^-ys, in units of 2^-ys.
template <class P>
__device__ __forceinline__ long long z_at(P p, long long K, int ys)
{
    return ((long long)py(p) << ys) - (long long)px(p) * K;
}

// Extremes of z over the box at slope key K.
__device__ __forceinline__ void box_range(const Box &bx, long long K, int ys, long long &lo, long long &hi)
{
    const long long u = (long long)bx.xlo * K, v = (long long)bx.xhi * K;
    lo = ((long long)bx.ylo << ys) - max(u, v);
    hi = ((long long)bx.yhi << ys) - min(u, v);
}

// Smallest shift that brings v (>= 0) below lim.
__device__ __forceinline__ int shift_below(long long v, int lim)
{
    int sh = 0;
    if (v >= lim) {
        sh = max(0, 63 - __clzll(v) - (31 - __clz(lim)));
        while ((v >> sh) >= lim) ++sh;
    }
    return sh;
}

__device__ __forceinline__ float pow2f(int e) { return __int_as_float((127 + e) << 23); }

// Nearest integer of f (|f| < 2^21) by one addition.
__device__ __forceinline__ int round_int(float f) { return __float_as_int(f + 12582912.0f) - 0x4b400000; }

template <int G, int NB>
__device__ __forceinline__ void hist_zero(const Group<G> &g, int *hist)
{
    for (int b = g.lane; b < NB; b += G) hist[b] = 0;
    g.sync();
}

// ------------------------------------------------------------------ interval test
// Whether some slope key in [A, B] can have a window of at most U units
// (false only when none can).  tol: bins this fine are fine enough.
// Intervals that reach beyond D_GUARD are rounded outwards to units of 2^-26
// and leave no T0, T1.
//
// [T0, T1]: where such a window can start, when known from an interval around
// this one (hulls over a part of an interval lie inside the hulls over all of
// it, so a start that was out stays out); narrowed on return.
//
// Without it the first pass covers the box and works in float: bins of 2^sh units, positions
// p = (z - zlo) 2^-sh < NB, each term rounded to 2^-24 of at most NB, five
// roundings in all, so |error| < NB 2^-20 = eps, which widens every interval.
// Later passes are exact in 64-bit integers; they only look at [T0, T1], the
// hull of the bins that reached depth h.
template <int G, int NB, class P>
__device__ __noinline__ bool may_hold_at(const Group<G> &g, const P *pts, int n, int h, long long A, long long B,
                                         long long U, long long tol, const Box &bx, int *hist, long long &T0,
                                         long long &T1, int ys)
{
    constexpr int PER = NB / G;
    long long la, ha, lb, hb;
    box_range(bx, A, ys, la, ha);
    box_range(bx, B, ys, lb, hb);
    const long long zlo = min(la, lb), zhi = max(ha, hb);
    if (U >= zhi - zlo) {
        if (T0 > T1) { T0 = zlo; T1 = zhi; }
        return true;
    }
    const bool known = T0 <= T1;
    if (!known) { T0 = zlo; T1 = zhi; }
    // depth of the bins after the starts and ends are in: the first and last bin of depth h
    auto scan = [&](int &b0, int &b1) {
        g.sync();
        int sum = 0;
        const int base = g.lane * PER;
#pragma unroll 8
        for (int r = 0; r < PER; ++r) sum += hist[slot_of<NB / G>(base + r)];
        int run = g.scan_ex(sum);
        b0 = 0x7fffffff;
        b1 = -1;
#pragma unroll 8
        for (int r = 0; r < PER; ++r) {
            run += hist[slot_of<NB / G>(base + r)];
            if (run >= h) {
                b0 = min(b0, base + r);
                b1 = base + r;
            }
        }
        int d0 = 0, d1 = 0;
        g.min2_max2(b0, d0, b1, d1);
    };
    {
        const int sh = shift_below(zhi - zlo, NB - 2);
        if (!known && sh >= 16) {
            constexpr float eps = NB * (1.0f / (1 << 20));
            const float sc = pow2f(ys - sh), dn = pow2f(-sh);
            const float fa = (float)A * dn, fb = (float)B * dn;
            const float c0 = -((float)zlo * dn);
            const float fu = __fmul_ru(__ll2float_ru(U), dn);
            const float off = fu + eps + 0.5f, up = eps - 0.5f;
            hist_zero<G, NB>(g, hist);
#pragma unroll 4
            for (int k = g.lane; k < n; k += G) {
                const P p = pts[k];
                const float x = (float)px(p), y = (float)py(p);
                const float base = fmaf(y, sc, c0);
                const float pa = fmaf(-x, fa, base), pb = fmaf(-x, fb, base);
                const float s = fmaxf(fminf(pa, pb) - off, 0.0f);
                const float e = fminf(fmaxf(fmaxf(pa, pb) + up, 0.0f), (float)(NB - 2));
                atomicAdd(&hist[slot_of<NB / G>(min(round_int(s), NB - 2))], 1);
                atomicAdd(&hist[slot_of<NB / G>(round_int(e) + 1)], -1);
            }
            int b0, b1;
            scan(b0, b1);
            if (b1 < 0) return false;
            T0 = zlo + ((long long)max(b0 - 1, 0) << sh);
            T1 = zlo + ((long long)(b1 + 2) << sh) - 1;
            if ((1LL << sh) <= tol) return true;
        }
    }
    for (int pass = 0; pass < 5; ++pass) {
        const int sh = shift_below(T1 - T0, NB - 1);
        g.sync();
        hist_zero<G, NB>(g, hist);
        // Short pass: positions relative to T0 in units of 2^(17 - ys) as 32-bit
        // integers (the products may wrap; the differences that matter do
        // not, and a point that wraps into the region only adds depth), the
        // low 17 bits of the slope by a float product (below 2 of y).  The
        // positions of interest lie within reach = (T1 - T0) + U + X (B - A)
        // + 2 of T0, so each of the five roundings is below 2^-24 reach.
        const long long reach = (T1 - T0) + U + (long long)(bx.xhi - bx.xlo) * (B - A) + (1LL << 33);
        bool packed = false;
        if constexpr (sizeof(P) == 4) {
        if (B - A < (1LL << 40) && reach < (1LL << 46) && (reach >> sh) < NB * 64) {
            packed = true;
            const unsigned ta = (unsigned)(T0 >> 17), ah = (unsigned)(A >> 17), bh = (unsigned)(B >> 17);
            const float sc = pow2f(17 - sh), dn = pow2f(-sh);
            const float al = (float)(int)(A & 0x1ffff) * dn, bl = (float)(int)(B & 0x1ffff) * dn;
            const float c0 = -(float)(int)(T0 & 0x1ffff) * dn;
            const float eps = (float)(reach >> sh) * (1.0f / (1 << 21)) + 1.0f / 1024;
            const float off = __fmul_ru(__ll2float_ru(U), dn) + eps + 0.5f, up = eps - 0.5f;
            const float last = (float)(int)((T1 - T0) >> sh);
#pragma unroll 4
            for (int k = g.lane; k < n; k += G) {
                const int p = packed_of(pts[k]);
                const int xi = px(p);
                const unsigned yb = (unsigned)((int)(p & 0xffff0000) >> (33 - ys)) - ta;
                const float xf = -(float)xi;
                const float pa = fmaf(xf, al, fmaf((float)(int)(yb - (unsigned)xi * ah), sc, c0));
                const float pb = fmaf(xf, bl, fmaf((float)(int)(yb - (unsigned)xi * bh), sc, c0));
                const float s = fminf(pa, pb) - off, e = fmaxf(pa, pb) + up;
                if (e < -0.5f || s > last + 0.5f) continue;
                atomicAdd(&hist[slot_of<NB / G>(round_int(fminf(fmaxf(s, 0.0f), last)))], 1);
                atomicAdd(&hist[slot_of<NB / G>(round_int(fminf(fmaxf(e, 0.0f), last)) + 1)], -1);
            }
        }
        }
        if (!packed)
#pragma unroll 2
        for (int k = g.lane; k < n; k += G) {
            const P p = pts[k];
            const long long u = z_at(p, A, ys), v = z_at(p, B, ys);
            const long long s = min(u, v) - U, e = max(u, v);
            if (e < T0 || s > T1) continue;
            const int bs = s <= T0 ? 0 : (int)((s - T0) >> sh);
            const int be = (int)((min(e, T1) - T0) >> sh);
            atomicAdd(&hist[slot_of<NB / G>(bs)], 1);
            atomicAdd(&hist[slot_of<NB / G>(be + 1)], -1);
        }
        int b0, b1;
        scan(b0, b1);
        if (b1 < 0) return false;
        T1 = min(T1, T0 + ((long long)(b1 + 1) << sh) - 1);
        T0 = T0 + ((long long)b0 << sh);
        if (sh == 0 || (1LL << sh) <= tol || b1 - b0 + 1 > NB / 2) return true;
    }
    return true;
}

template <int G, int NB, class P>
__device__ bool may_hold(const Group<G> &g, const P *pts, int n, int h, long long A, long long B, long long U,
                                      long long tol, const Box &bx, int *hist, long long &T0, long long &T1)
{
    if (U < 0) return false;
    if constexpr (sizeof(P) == 8) return may_hold_at<G, NB>(g, pts, n, h, A, B, U, tol, bx, hist, T0, T1, F_YS);
    int ys = 32;
    if (A <= -D_GUARD || B >= D_GUARD) {
        ys = 32 - STEEP;
        A >>= STEEP;
        B = (B + (1 << STEEP) - 1) >> STEEP;
        U = (U >> STEEP) + 1;
        long long s0 = 1, s1 = 0;
        const bool keep = may_hold_at<G, NB>(g, pts, n, h, A, B, U, tol >> STEEP, bx, hist, s0, s1, ys);
        T0 = 1;
        T1 = 0;
        return keep;
    }
    return may_hold_at<G, NB>(g, pts, n, h, A, B, U, tol, bx, hist, T0, T1, ys);
}

// ------------------------------------------------------------------ upper bound
// Narrowest window of h points over the bins of a histogram whose running sum
// is in hist, among those no wider than lim.  Start bins b < nstart; ends
// anywhere.  Bins lie at lo1 + b 2^sh for b < half - 1, bin half - 1 holds
// everything between the two regions and bins from half on lie at
// lo2 + (b - half) 2^sh (one region: half = 0).  Returns the width from the
// start bin's left edge to the end bin's right edge, less one unit (D_MAX:
// none), the hull of the start bins of the windows that may be narrower than
// it, the first of their end bins, and the first start bin of that width.
template <int G, int NB>
__device__ long long window_search(const Group<G> &g, const int *cum, int nstart, int h, long long lim, long long lo1,
                                   long long lo2, int half, int sh, int &b0, int &b1, int &e0, int &bm)
{
    constexpr int ROWS = NB / G, U4 = ROWS < 4 ? ROWS : 4;
    const int total = cum[slot_of<NB / G>(NB - 1)];
    const long long two = 2LL << sh;
    long long mn = D_MAX;
    lim = min(lim, D_MAX / 4);
    b0 = e0 = bm = 0x7fffffff;
    b1 = -1;
    // thread by thread over consecutive start bins, U4 searches side by side
    for (int r = 0; r < ROWS && r * G < nstart; r += U4) {
        // a window within two bins of the limit that starts in bin b ends by bin b + off
        const long long reach = min(lim, mn) + two + 1 + (half ? lo1 - lo2 : 0);
        const int off = (int)max((long long)-NB, min((long long)NB, reach >> sh)) + half;
        int target[U4], pos[U4];
        bool any = false;
#pragma unroll
        for (int u = 0; u < U4; ++u) {
            const int b = (r + u) * G + g.lane;
            const int before = b ? cum[slot_of<NB / G>(b - 1)] : 0;
            const int em = min(b + off, NB - 1);
            // starts at a point, and can be narrow enough
            const bool ok = b < nstart && em >= 0 && before + h <= total && cum[slot_of<NB / G>(em)] >= before + h &&
                            cum[slot_of<NB / G>(b)] != before;
            target[u] = ok ? before + h : 0;
            any |= ok;
            pos[u] = 0;
        }
        if (!__any_sync(FULL, any)) continue;
#pragma unroll
        for (int d = NB / 2; d >= 1; d >>= 1) {   // first bin whose running sum reaches the target
#pragma unroll
            for (int u = 0; u < U4; ++u) pos[u] += cum[slot_of<NB / G>(pos[u] + d - 1)] < target[u] ? d : 0;
        }
#pragma unroll
        for (int u = 0; u < U4; ++u) {
            if (target[u] == 0) continue;
            const int b = (r + u) * G + g.lane, e = pos[u];
            long long right;
            if (half == 0 || e < half - 1) right = lo1 + ((long long)(e + 1) << sh);
            else if (e == half - 1) right = lo2;
            else right = lo2 + ((long long)(e - half + 1) << sh);
            const long long w = right - (lo1 + ((long long)b << sh)) - 1;
            if (w - two > min(mn, lim)) continue;
            if (w < mn - two) { b0 = e0 = 0x7fffffff; b1 = -1; }
            if (w < mn || (w == mn && b < bm)) bm = b;
            mn = min(mn, w);
            b0 = min(b0, b);
            b1 = max(b1, b);
            e0 = min(e0, e);
        }
    }
    const long long gm = g.min_ll(mn);
    if (mn > gm) bm = 0x7fffffff;
    if (mn - two > gm) { b0 = e0 = 0x7fffffff; b1 = -1; }
    int nbm = bm == 0x7fffffff ? -0x7fffffff : -bm;   // minimum of bm as a maximum
    g.min2_max2(b0, e0, b1, nbm);
    bm = -nbm;
    return gm;
}

template <int G, int NB>
__device__ __forceinline__ void hist_cumulate(const Group<G> &g, int *hist)
{
    constexpr int PER = NB / G;
    g.sync();
    const int base = g.lane * PER;
    int sum = 0;
#pragma unroll 8
    for (int r = 0; r < PER; ++r) sum += hist[slot_of<NB / G>(base + r)];
    int run = g.scan_ex(sum);
#pragma unroll 8
    for (int r = 0; r < PER; ++r) {
        run += hist[slot_of<NB / G>(base + r)];
        hist[slot_of<NB / G>(base + r)] = run;
    }
    g.sync();
}

// An upper bound of w at slope key K (units of 2^-32), within a few 2^-20 of
// it where the windows that could be narrowest are few.  Gives up early
// (returning what it has) once the slope cannot beat cur.  [T0, T1]: where a
// window that beats cur must start, when known.  The same two kinds of pass
// as may_hold: float bins of the whole range (with `coarse` only that pass), then integer bins of
// the regions where the narrowest windows start and end.
template <int G, int NB, class P>
__device__ __noinline__ long long ub_at(const Group<G> &g, const P *pts, int n, int h, long long K, long long cur,
                                        const Box &bx, int *hist, long long T0, long long T1,
                                        bool coarse = false)
{
    const bool steep = K <= -D_GUARD || K >= D_GUARD;
    const int ys = sizeof(P) == 8 ? F_YS : steep ? 32 - STEEP : 32;
    if (steep) {
        K >>= STEEP;   // some slope beside it
        cur = (cur >> STEEP) + 1;
    }
    auto result = [&](long long w) { return !steep || w == D_MAX ? w : w > D_MAX >> STEEP ? D_MAX : w << STEEP; };
    long long zlo, zhi;
    box_range(bx, K, ys, zlo, zhi);
    long long best = D_MAX;
    int sh = shift_below(zhi - zlo, NB - 2);
    int b0, b1, e0, bm;
    // windows start in [lo1, sl) and end in [lo2, hi2)
    long long lo1 = zlo, hi1 = zhi + 1, lo2 = zlo, hi2 = zhi + 1, sl = zhi + 1;
    int margin = 0;
    bool two = false;
    if (T0 <= T1 && !steep) {
        // only windows starting in [T0, T1] and no wider than cur are wanted
        lo1 = lo2 = T0;
        sl = T1 + 1;
        hi1 = hi2 = (cur > zhi - T1 ? max(zhi, T1) : T1 + cur) + 1;
        sh = 62;
    } else if (sh >= 16) {
        const float sc = pow2f(ys - sh), dn = pow2f(-sh);
        const float fk = (float)K * dn;
        const float c0 = -((float)zlo * dn) - 0.5f;
        g.sync();
        hist_zero<G, NB>(g, hist);
#pragma unroll 4
        for (int k = g.lane; k < n; k += G) {
            const P p = pts[k];
            const float f = fmaf(-(float)px(p), fk, fmaf((float)py(p), sc, c0));
            atomicAdd(&hist[slot_of<NB / G>(round_int(fminf(fmaxf(f, 0.0f), (float)(NB - 1))))], 1);
        }
        hist_cumulate<G, NB>(g, hist);
        const long long w = window_search<G, NB>(g, hist, NB, h, cur, zlo, zlo, 0, sh, b0, b1, e0, bm);
        if (w == D_MAX) return D_MAX;
        best = w + (1LL << sh);   // the rounding of the float positions, below 1/32 of a bin
        if (coarse || w - (4LL << sh) >= cur) return result(best);
        margin = 1;
        lo1 = zlo + ((long long)(b0 - margin) << sh);
        hi1 = zlo + ((long long)(b1 + 1 + margin) << sh);
        lo2 = zlo + ((long long)(e0 - margin) << sh);
        hi2 = min(zhi + 1, hi1 + best + 1);   // later points of a start bin end later than its first
        sl = hi1;
        two = lo2 > hi1;
    } else {
        sh = 62;
    }
    for (int pass = 0; pass < 4; ++pass) {
        int s2;
        if (two) {
            s2 = shift_below(max(hi1 - lo1, hi2 - lo2) - 1, NB / 2 - 1);
        } else {
            hi2 = max(hi1, hi2);
            lo1 = min(lo1, lo2);
            s2 = shift_below(hi2 - lo1 - 1, NB);
        }
        if (s2 >= sh) break;
        sh = s2;
        g.sync();
        hist_zero<G, NB>(g, hist);
        int mid = 0;
        long long slack = 0;
        // Short pass, as in may_hold, but no point may wrap (it would count
        // where it is not): units of 2^(q - ys) with q as large as the box
        // asks for.  Positions err by less than eps bins, so windows are
        // widened by a quarter of a bin.
        const long long reach = max(zhi, hi2) - min(zlo, lo1);
        int q = 17;
        while (q < 24 && (reach >> (q + 30)) != 0) ++q;
        const long long span = hi2 - lo1 + (1LL << (q + 16));
        bool packed = false;
        if constexpr (sizeof(P) == 4) {
        if ((reach >> (q + 30)) == 0 && (span >> sh) < (1 << 18) && sh >= 4) {
            packed = true;
            const unsigned tl = (unsigned)(lo1 >> q), kh = (unsigned)(K >> q);
            const float sc = pow2f(q - sh), dn = pow2f(-sh);
            const int low = (1 << q) - 1;
            const float kl = (float)(int)(K & low) * dn;
            const float c0 = -(float)(int)(lo1 & low) * dn - 0.5f;
            const float len1 = (float)((two ? hi1 : hi2) - lo1) * dn - 0.5f;
            const float beg2 = (float)(lo2 - lo1) * dn, end2 = (float)(hi2 - lo1) * dn - 0.5f;
            const float lim1 = two ? (float)(NB / 2 - 2) : (float)(NB - 1);
            slack = 1LL << (sh - 2);
#pragma unroll 4
            for (int k = g.lane; k < n; k += G) {
                const int p = packed_of(pts[k]);
                const int xi = px(p);
                const unsigned d = ((unsigned)((int)(p & 0xffff0000) >> 16) << (ys - q)) - tl - (unsigned)xi * kh;
                const float f = fmaf(-(float)xi, kl, fmaf((float)(int)d, sc, c0));
                if (f < -0.5f || f > end2) continue;
                if (f < len1) atomicAdd(&hist[slot_of<NB / G>(round_int(fminf(fmaxf(f, 0.0f), lim1)))], 1);
                else if (!two) continue;
                else if (f < beg2 - 0.5f) ++mid;
                else atomicAdd(&hist[slot_of<NB / G>(NB / 2 + round_int(fminf(fmaxf(f - beg2, 0.0f), (float)(NB / 2 - 1))))], 1);
            }
        }
        }
        if (!packed)
#pragma unroll 2
        for (int k = g.lane; k < n; k += G) {
            const long long z = z_at(pts[k], K, ys);
            if (z < lo1 || z >= hi2) continue;
            if (!two) atomicAdd(&hist[slot_of<NB / G>((int)((z - lo1) >> sh))], 1);
            else if (z < hi1) atomicAdd(&hist[slot_of<NB / G>((int)((z - lo1) >> sh))], 1);
            else if (z < lo2) ++mid;
            else atomicAdd(&hist[slot_of<NB / G>(NB / 2 + (int)((z - lo2) >> sh))], 1);
        }
        if (two) {
            if constexpr (G >= 32) {
                mid = __reduce_add_sync(FULL, mid);
                if ((g.lane & 31) == 0) atomicAdd(&hist[slot_of<NB / G>(NB / 2 - 1)], mid);
            } else {
                atomicAdd(&hist[slot_of<NB / G>(NB / 2 - 1)], mid);
            }
        }
        hist_cumulate<G, NB>(g, hist);
        const int half = two ? NB / 2 : 0;
        const int nst = (int)min((long long)(two ? NB / 2 - 1 : NB), ((sl - 1 - lo1) >> sh) + 2);
        const long long w = window_search<G, NB>(g, hist, nst, h, cur, lo1, lo2, half, sh, b0, b1, e0, bm);
        if (w == D_MAX) break;
        best = min(best, w + slack);
        if (w - (4LL << sh) >= cur || sh == 0 || (1LL << sh) <= (w >> 20)) break;
        const long long o1 = lo1, o2 = lo2;
        auto left = [&](int b) {
            return half == 0 || b < half ? o1 + ((long long)b << sh) : o2 + ((long long)(b - half) << sh);
        };
        lo1 = left(b0);
        hi1 = left(b1) + (1LL << sh);
        lo2 = left(e0);
        hi2 = min(hi2, hi1 + best + 1);
        sl = hi1;
        two = lo2 > hi1;
    }
    g.sync();
    return result(best);
}

// Lower bound of w over slope keys [A, B] on one side of 0: h points span at
// least dh in x and at most yr in y, so w >= |s| dh - yr (units of 2^-32).
__device__ __forceinline__ bool steep_above(long long A, long long B, int dh, int yr, long long U)
{
    long long K;
    if (B <= 0 && B > -D_MAX) K = -B;
    else if (A >= 0 && A < D_MAX) K = A;
    else return false;
    const __int128 v = (__int128)K * dh - ((__int128)yr << 32);
    return v > (__int128)U;
}

// The same for every slope beyond F_KMAX of a float set (dh less one step, yr
// more one step: the grid).
__device__ __forceinline__ bool steep_above_at(long long K, int dh, int yr, long long U)
{
    const __int128 v = (__int128)K * (dh - 1) - ((__int128)(yr + 1) << F_YS);
    return v > (__int128)U;
}

// ------------------------------------------------------------------ CTA helpers
template <int T>
__device__ __forceinline__ int cta_scan_ex(int v, int *s_warp, int &total)
{
    if constexpr (T >= 32) {
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
        int x = v;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int o = __shfl_up_sync(FULL, x, d);
            if (lane >= d) x += o;
        }
        if (lane == 31) s_warp[warp] = x;
        __syncthreads();
        const unsigned c = lane < T / 32 ? (unsigned)s_warp[lane] : 0u;
        const int base = (int)__reduce_add_sync(FULL, lane < warp ? c : 0u);
        total = (int)__reduce_add_sync(FULL, c);
        __syncthreads();
        return base + x - v;
    } else {
        total = v;
        return 0;
    }
}

// Whether the threads' values add up to more than limit (the same in every thread).
template <int T>
__device__ __forceinline__ bool candidates_above(float v, float limit, int *s_warp)
{
    if constexpr (T >= 32) {
#pragma unroll
        for (int d = 16; d >= 1; d >>= 1) v += __shfl_xor_sync(FULL, v, d);
        if ((threadIdx.x & 31) == 0) s_warp[threadIdx.x >> 5] = __float_as_int(v);
        __syncthreads();
        const int lane = threadIdx.x & 31;
        v = lane < T / 32 ? __int_as_float(s_warp[lane]) : 0.0f;
#pragma unroll
        for (int d = 16; d >= 1; d >>= 1) v += __shfl_xor_sync(FULL, v, d);
        __syncthreads();
    }
    return v > limit;
}

template <int T>
__device__ __forceinline__ void cta_min_max_i(int &lo, int &hi, int *s_a, int *s_b)
{
    if constexpr (T >= 32) {
        lo = __reduce_min_sync(FULL, lo);
        hi = __reduce_max_sync(FULL, hi);
        if ((threadIdx.x & 31) == 0) { s_a[threadIdx.x >> 5] = lo; s_b[threadIdx.x >> 5] = hi; }
        __syncthreads();
        lo = __reduce_min_sync(FULL, s_a[(threadIdx.x & 31) % (T / 32)]);
        hi = __reduce_max_sync(FULL, s_b[(threadIdx.x & 31) % (T / 32)]);
        __syncthreads();
    }
}

__device__ __forceinline__ unsigned mix32(unsigned v)
{
    v ^= v >> 16;
    v *= 0x7feb352du;
    v ^= v >> 15;
    v *= 0x846ca68bu;
    return v ^ (v >> 16);
}

__device__ __forceinline__ unsigned key_hash(long long k)
{
    return mix32((unsigned)k ^ mix32((unsigned)(k >> 32) + 0x9e3779b9u));
}

// Distinct slope keys of one leaf, each with the dx of a pair that has it: an
// open-addressing table in shared memory.
struct SlopeTable {
    unsigned long long *key;   // TABLE, empty slots ~0
    unsigned *den;             // TABLE
    int *count;                // keys held; above TABLE * 3 / 4 the leaf does not fit
};

__device__ __forceinline__ void table_put(const SlopeTable &t, long long key, int dx)
{
    const unsigned long long k = (unsigned long long)key;
    unsigned s = key_hash(key) & (TABLE - 1);
    for (int probe = 0; probe < TABLE; ++probe, s = (s + 1) & (TABLE - 1)) {
        unsigned long long cur = *reinterpret_cast<volatile unsigned long long *>(&t.key[s]);
        if (cur == k) return;
        if (cur == ~0ull) {
            if (*reinterpret_cast<volatile int *>(t.count) > TABLE * 3 / 4) return;
            cur = atomicCAS(&t.key[s], ~0ull, k);
            if (cur == ~0ull) {
                atomicAdd(t.count, 1);
                t.den[s] = (unsigned)dx;
                return;
            }
            if (cur == k) return;
        }
    }
}

template <int T>
__device__ __forceinline__ SlopeTable table_clear(unsigned char *wk)
{
    SlopeTable t;
    t.key = reinterpret_cast<unsigned long long *>(wk);
    t.den = reinterpret_cast<unsigned *>(t.key + TABLE);
    t.count = reinterpret_cast<int *>(t.den + TABLE);
    for (int k = threadIdx.x; k < TABLE; k += T) t.key[k] = ~0ull;
    if (threadIdx.x == 0) *t.count = 0;
    return t;
}

// The table's slopes go to the end of the team's list; *over when they do not fit.
template <int T>
__device__ __forceinline__ void table_append(const SlopeTable &tab, const TeamMem &m, int *nlist, int *over, int HC,
                                             int *s_warp)
{
    const int held = *tab.count;
    __shared__ int s_at;
    if (threadIdx.x == 0) {
        s_at = held > TABLE * 3 / 4 ? HC : atomicAdd(nlist, held);
        if (s_at + held > HC) atomicMax(over, 1);
    }
    __syncthreads();
    int at = s_at;
    if (at + held <= HC) {
        const int per = TABLE / T;
        int c = 0, total;
        for (int r = 0; r < per; ++r) c += tab.key[threadIdx.x * per + r] != ~0ull;
        at += cta_scan_ex<T>(c, s_warp, total);
        for (int r = 0; r < per; ++r) {
            const unsigned long long k = tab.key[threadIdx.x * per + r];
            if (k != ~0ull) {
                m.lkey[at] = (long long)k;
                m.lden[at++] = tab.den[threadIdx.x * per + r];
            }
        }
    }
    __syncthreads();
}

// The dy of the slope with this key and dx: key <= dy 2^32 / dx < key + 1.
__device__ __forceinline__ int dy_of(long long key, int dx)
{
    return (int)((key * dx + 0xffffffffLL) >> 32);
}

__device__ __forceinline__ unsigned gcd32(unsigned a, unsigned b)
{
    while (b) { const unsigned r = a % b; a = b; b = r; }
    return a;
}

// Largest q of a fraction p / q with key in [A, B), q <= X and |p| <= Y.
__device__ __forceinline__ int fraction_q(long long A, long long B, int xr, int yr)
{
    const long long nearest = A > 0 ? A : B < 0 ? -B : 0;
    return nearest ? (int)min((long long)xr, (((long long)yr + 1) << 32) / nearest + 1) : xr;
}

// Expected reduced fractions p / q of such a leaf: about 0.31 q^2 times its width.
__device__ __forceinline__ float fractions(long long A, long long B, int xr, int yr)
{
    // (fraction_q in float: it is asked for every interval)
    const float nearest = A > 0 ? (float)A : B < 0 ? -(float)B : 0.0f;
    const float q = nearest > 0.0f ? fminf((float)xr, __fdividef(4294967296.0f * (float)(yr + 1), nearest) + 1.0f) : (float)xr;
    return 0.31f * q * q * (float)(B - A) * (1.0f / 4294967296.0f);
}

// Slopes a leaf is expected to list: its pairs, or its fractions where those are tried.
__device__ __forceinline__ float leaf_slopes(const DNode &lf, float gain, int xr, int yr)
{
    const float f = fractions(lf.a, lf.b, xr, yr), e = fmaxf(lf.est * gain, 1.0f);
    return f < FRACTIONS ? fminf(f + 1.0f, 4.0f * e + LEAF_FRACTIONS) : e;
}

// How many of the count leaves together are expected to list at most limit
// slopes (one at least), and how many slopes those are: every warp for itself,
// a leaf a lane.
template <int T, bool F>
__device__ __forceinline__ int leaves_within(const DNode *leaf, int count, float limit, float gain, int xr, int yr,
                                             float &slopes)
{
    constexpr int L = T >= 32 ? 32 : 1;
    const int lane = threadIdx.x % L;
    slopes = 0.0f;
    for (int l0 = 0; l0 < count; l0 += L) {
        const int l = l0 + lane;
        float v = 0.0f;
        if (l < count) v = F ? fmaxf(leaf[l].est * gain, 1.0f) : leaf_slopes(leaf[l], gain, xr, yr);
        if constexpr (L == 32) {
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const float o = __shfl_up_sync(FULL, v, d);
                if (lane >= d) v += o;
            }
        }
        const unsigned beyond = __ballot_sync(FULL, l > 0 && l < count && slopes + v > limit);
        if (beyond) {
            const int first = __clz((int)(beyond & (0u - beyond))) ^ 31;
            if (first > 0) slopes += __shfl_sync(FULL, v, (first - 1) % L);
            return l0 + first;
        }
        slopes += __shfl_sync(FULL, v, L - 1);
    }
    return count;
}

// The first cell start at or after position p of the held points in ord, which
// lie cell by cell (end[q]: where cell q ends).  CTAs that share a leaf take
// blocks of positions by turns (dense cells lie side by side), and the blocks
// start and end there: every CTA sorts the points into cells for itself, the
// order inside a cell differs between them, and a cell cut between two of them
// would lose pairs.
template <class CELL>
__device__ __forceinline__ int block_start(int p, int held, const unsigned *end, const unsigned short *ord, CELL cell_of)
{
    return p <= 0 ? 0 : p >= held ? held : (int)end[cell_of(ord[p - 1])];
}

// Shared bytes of list_pairs for NC cells and n points.
__host__ __device__ constexpr size_t pairs_bytes(int NC, int n)
{
    return 12 * (size_t)TABLE + 16 + 4 * (size_t)NC + 2 * (size_t)n;
}

// A superset of the distinct slopes of the pairs with key in [A, B), appended
// to the team's list by one CTA, which takes share `part` of `parts` of the
// pairs or fractions (CTAs sharing a leaf may list a slope twice, which only
// tests it twice).  wk: pairs_bytes(NC, n).  Narrow leaves hold
// few reduced fractions p / q with q <= X at all (about 0.31 X^2 times the
// width), far fewer than pairs when many pairs share a slope: up to
// FRACTIONS of them the CTA tries every q.  p / q lies in the leaf when
// g = -A q mod 2^32 is below (B - A) q: two 32-bit products a q, whatever the
// number of points (n = 65536, 10 leaves: 4.6 ms by pairs).  Otherwise the
// pairs are found by cells (see the head of the file); so are they when the
// leaf holds far more fractions than the pairs expected (most fractions are
// then no pair's slope, and each would be tested and scored).  Cells that hold many points hold
// quadratically many candidates with few distinct slopes.  Above the limit
// nothing is searched: points that repeat another one are left out (dup, once
// they are marked: 2048 points, 70% of them at one place, cost 35 ms of
// candidates), and for points on one line the leaf is tried by fractions, or
// false is returned and it is cut until it can be.
template <int T>
__device__ __noinline__ bool list_pairs(const int *pts, int n, const unsigned *dup, const DNode &lf, const Box &bx,
                                        int NC, unsigned char *wk, int *s_warp, const TeamMem &m,
                                        int *nlist, int *over, int HC,
                                        int part, int parts)
{
    const long long A = lf.a, B = lf.b;
    const int xr = bx.xhi - bx.xlo, yr = bx.yhi - bx.ylo;
    auto by_q = [&]() {
        const long long d = B - A;
        const int qmax = fraction_q(A, B, xr, yr);
        for (int q = 1 + part * T + (int)threadIdx.x; q <= qmax; q += T * parts) {
            const long long end = d * q;
            for (long long g = (unsigned)(0u - (unsigned)A * (unsigned)q); g < end; g += 1LL << 32) {
                const int y = (int)((A * q + g) >> 32);
                const unsigned ay = (unsigned)(y < 0 ? -y : y);
                if (ay > (unsigned)yr || gcd32(ay, (unsigned)q) != 1) continue;
                const int at = atomicAdd(nlist, 1);
                if (at < HC) {
                    m.lkey[at] = slope_key(y, q);
                    m.lden[at] = (unsigned)q;
                } else if (at == HC) {
                    atomicMax(over, 1);
                }
            }
        }
    };
    const float fr = fractions(A, B, xr, yr);
    if (fr < FRACTIONS && fr <= 4.0f * fmaxf(lf.est, 1.0f) + LEAF_FRACTIONS) {
        by_q();
        return true;
    }
    auto out = [&](int k) { return dup && (__ldcg(&dup[k >> 5]) >> (k & 31) & 1); };
    const SlopeTable tab = table_clear<T>(wk);
    unsigned *cnt = tab.den + TABLE + 4;
    unsigned short *ord = reinterpret_cast<unsigned short *>(cnt + NC);
    for (int q = threadIdx.x; q < NC; q += T) cnt[q] = 0u;
    __syncthreads();
    // beyond D_GUARD in units of 2^-26, the cells a little wider for the rounding
    const bool steep = A <= -D_GUARD || B >= D_GUARD;
    const int ys = steep ? 32 - STEEP : 32;
    const long long za = steep ? A >> STEEP : A, dk = steep ? ((B - A) >> STEEP) + 2 : B - A;
    {
        const long long width = (long long)xr * dk;
        int sh = 0;
        while ((1ull << sh) < (unsigned long long)width) ++sh;   // width < 2^63
        long long zlo, zhi;
        box_range(bx, za, ys, zlo, zhi);
        auto cell = [&](int p) { return (int)((unsigned long long)(z_at(p, za, ys) - zlo) >> sh) & (NC - 1); };
        for (int k = threadIdx.x; k < n; k += T)
            if (!out(k)) atomicAdd(&cnt[cell(pts[k])], 1u);
        __syncthreads();
        const int per = NC / T;
        unsigned sum = 0;
        float cand = 0.0f;   // candidates: the rest of a cell, and the next cell
        for (int r = 0; r < per; ++r) {
            const unsigned c = cnt[threadIdx.x * per + r], c2 = cnt[(threadIdx.x * per + r + 1) & (NC - 1)];
            sum += c;
            cand += (float)c * (0.5f * (float)c + (float)c2);
        }
        if (candidates_above<T>(cand, DENSE + DENSE_PER_POINT * (float)n, s_warp)) {
            // (every CTA that shares the leaf finds the same)
            if (dup && fr < FRACTIONS) by_q();
            __syncthreads();
            return dup && fr < FRACTIONS;
        }
        int held;
        unsigned run = (unsigned)cta_scan_ex<T>((int)sum, s_warp, held);
        for (int r = 0; r < per; ++r) {
            const unsigned c = cnt[threadIdx.x * per + r];
            cnt[threadIdx.x * per + r] = run;
            run += c;
        }
        __syncthreads();
        for (int k = threadIdx.x; k < n; k += T)
            if (!out(k)) ord[atomicAdd(&cnt[cell(pts[k])], 1u)] = (unsigned short)k;
        __syncthreads();
        // cnt[q] is now the end of cell q, cnt[q - 1] its start.  A warp takes
        // 32 points at a time, lays their candidates (the rest of the cell,
        // then the next cell) end to end and tests 32 of them at once.
        constexpr int L = T >= 32 ? 32 : 1;
        const int lane = threadIdx.x % L;
        auto cell_of = [&](int k) { return cell(pts[k]); };
        constexpr int BLOCK = T >= 32 ? T : 16;
        for (int blk = part * BLOCK; blk < held; blk += parts * BLOCK) {
            const int first = block_start(blk, held, cnt, ord, cell_of);
            const int last = block_start(blk + BLOCK, held, cnt, ord, cell_of);
            for (int e0 = first + threadIdx.x - lane; e0 < last; e0 += T) {
                const int e = e0 + lane;
                int pa = 0, n1 = 0, nn = 0, beg2 = 0;
                if (e < last) {
                    pa = pts[ord[e]];
                    const int q = cell(pa), q2 = (q + 1) & (NC - 1);
                    beg2 = q2 ? (int)cnt[q2 - 1] : 0;
                    n1 = (int)cnt[q] - e - 1;
                    nn = n1 + (int)cnt[q2] - beg2;
                }
                int pre = nn;   // inclusive prefix over the warp
                if constexpr (L == 32) {
#pragma unroll
                    for (int d = 1; d < 32; d <<= 1) {
                        const int o = __shfl_up_sync(FULL, pre, d);
                        if (lane >= d) pre += o;
                    }
                }
                const int total = L == 32 ? __shfl_sync(FULL, pre, 31) : pre;
                LMS_DIRECT_COUNT(M_DONE, total);
                for (int c0 = 0; c0 < total; c0 += L) {
                    const int c = c0 + lane;
                    int src = 0;   // the lane whose candidates hold c
                    if constexpr (L == 32) {
#pragma unroll
                        for (int d = 16; d >= 1; d >>= 1) {
                            const int v = __shfl_sync(FULL, pre, src + d - 1);
                            if (v <= c) src += d;
                        }
                        src = min(src, 31);
                    }
                    const int u = c - (__shfl_sync(FULL, pre, src) - __shfl_sync(FULL, nn, src));
                    const int k1 = __shfl_sync(FULL, n1, src), k2 = __shfl_sync(FULL, beg2, src);
                    const int p = __shfl_sync(FULL, pa, src);
                    if (c >= total) continue;
                    const int b = ord[u < k1 ? e0 + src + 1 + u : k2 + u - k1];
                    int dy, dx;
                    if (!pair_slope(p, pts[b], dy, dx)) continue;
                    const long long t = (long long)dy << 32;
                    if (!steep && (A * dx > t || B * dx <= t)) continue;
                    const long long k = slope_key(dy, dx);
                    if (k >= A && k < B) table_put(tab, k, dx);
                }
            }
        }
    }
    __syncthreads();
    table_append<T>(tab, m, nlist, over, HC, s_warp);
    return true;
}

// ------------------------------------------------------------------ float points
struct FloatSet {
    const float *x, *y;
    double xc, yc, sx, sy;   // grid = rint((v - c) * s), s a power of two
    double ratio;            // scaled slope = slope * ratio
    double rx, ry;           // rounding of a width in double: rx |K| + ry units of 2^-F_YS steps
};

__device__ __forceinline__ long long order_of(double v)
{
    const long long b = v == 0.0 ? 0LL : __double_as_longlong(v);
    return b < 0 ? (b ^ 0x7fffffffffffffffLL) : b;
}
__device__ __forceinline__ double of_order(long long k)
{
    return __longlong_as_double(k < 0 ? (k ^ 0x7fffffffffffffffLL) : k);
}
__device__ __forceinline__ bool slope_f32(const FloatSet &f, int i, int j, double &s)
{
    double dx = (double)f.x[j] - (double)f.x[i], dy = (double)f.y[j] - (double)f.y[i];
    if (dx == 0.0) return false;
    if (dx < 0.0) { dx = -dx; dy = -dy; }
    s = __ddiv_rn(dy, dx);
    return true;
}
__device__ __forceinline__ double z_f32(const FloatSet &f, int k, double s)
{
    return __dsub_rn((double)f.y[k], __dmul_rn(s, (double)f.x[k]));
}

// The distinct slopes of the pairs in the leaf [A, B) of scaled slope keys
// (their order_of words), listed by one CTA's share; with `want` instead the
// smallest index pair of that slope, lowered into *pair.  Cells of z(A) as in
// list_pairs; both points of a pair may lie half a step off the grid in x and
// y, which widens the cells by (1 + |s|) steps.  *over = 2 (nothing listed)
// when the cells hold too many candidates.
template <int T>
__device__ __noinline__ void list_pairs_f32(const int2 *pts, int n, long long A, long long B, const Box &bx,
                                            const FloatSet &f, int NC, unsigned char *wk, int *s_warp,
                                            const TeamMem &m, int *nlist, int *over, int HC, int part, int parts,
                                            const long long *want = nullptr, unsigned *pair = nullptr)
{
    const SlopeTable tab = table_clear<T>(wk);
    unsigned *cnt = tab.den + TABLE + 4;
    unsigned short *ord = reinterpret_cast<unsigned short *>(cnt + NC);
    for (int q = threadIdx.x; q < NC; q += T) cnt[q] = 0u;
    __syncthreads();
    const long long ka = max(A < 0 ? -A : A, B < 0 ? -B : B);
    const unsigned long long width = (unsigned long long)(bx.xhi - bx.xlo) * (unsigned long long)(B - A) +
                                     (1ull << F_YS) + (unsigned long long)ka + 4;
    int sh = 0;
    while (sh < 63 && (1ull << sh) < width) ++sh;
    long long zlo, zhi;
    box_range(bx, A, F_YS, zlo, zhi);
    auto cell = [&](int2 p) { return (int)((unsigned long long)(z_at(p, A, F_YS) - zlo) >> sh) & (NC - 1); };
    for (int k = threadIdx.x; k < n; k += T) atomicAdd(&cnt[cell(pts[k])], 1u);
    __syncthreads();
    const int per = NC / T;
    unsigned sum = 0;
    constexpr int L = T >= 32 ? 8 : 1, BLOCK = T >= 32 ? T / L : 16, HEAVY = 4 * BLOCK;
    float cand = 0.0f;
    int heavy = 0;
    for (int r = 0; r < per; ++r) {
        const unsigned c = cnt[threadIdx.x * per + r], c2 = cnt[(threadIdx.x * per + r + 1) & (NC - 1)];
        sum += c;
        cand += (float)c * (0.5f * (float)c + (float)c2);
        heavy |= c > (unsigned)HEAVY;
    }
    if (candidates_above<T>(cand, F_DENSE, s_warp) && !want) {
        if (threadIdx.x == 0) atomicMax(over, 2);
        __syncthreads();
        return;
    }
    heavy = __syncthreads_or(heavy);
    int total;
    unsigned run = (unsigned)cta_scan_ex<T>((int)sum, s_warp, total);
    for (int r = 0; r < per; ++r) {
        const unsigned c = cnt[threadIdx.x * per + r];
        cnt[threadIdx.x * per + r] = run;
        run += c;
    }
    __syncthreads();
    for (int k = threadIdx.x; k < n; k += T) ord[atomicAdd(&cnt[cell(pts[k])], 1u)] = (unsigned short)k;
    __syncthreads();
    const long long err = (1LL << F_YS) + ka + 4;
    auto cell_of = [&](int k) { return cell(pts[k]); };
    auto full = [&]() { return *reinterpret_cast<volatile int *>(tab.count) > TABLE * 3 / 4; };   // the leaf is cut instead
    auto test = [&](int a, int2 pa, int b) {
        const int2 pb = pts[b];
        // on the grid first: 0 <= dz < dx (B - A), widened
        long long dx = (long long)pb.x - pa.x, dz = z_at(pb, A, F_YS) - z_at(pa, A, F_YS);
        if (dx < 0) { dx = -dx; dz = -dz; }
        if (dz < -err || (double)dz > (double)(dx + 1) * (double)(B - A) + (double)err) return;
        double s;
        if (!slope_f32(f, a, b, s)) return;
        const double k = s * f.ratio * (double)(1LL << F_YS);
        if (!(k >= (double)A && k < (double)B)) return;
        if (want) {
            const unsigned ij = (unsigned)min(a, b) << 16 | (unsigned)max(a, b);
            if (order_of(s) == *want && *reinterpret_cast<volatile unsigned *>(pair) > ij) atomicMin(pair, ij);
        } else {
            table_put(tab, order_of(s), 0);
        }
    };
    for (int blk = part * BLOCK; blk < n; blk += parts * BLOCK) {
        const int first = block_start(blk, n, cnt, ord, cell_of);
        const int last = block_start(blk + BLOCK, n, cnt, ord, cell_of);
        for (int e = first + (int)threadIdx.x / L; e < last; e += T / L) {
            const int a = ord[e];
            const int2 pa = pts[a];
            const int q = cell(pa), q2 = (q + 1) & (NC - 1);
            if ((int)cnt[q] - (q ? (int)cnt[q - 1] : 0) > HEAVY) continue;
            const int beg2 = q2 ? (int)cnt[q2 - 1] : 0;
            const int n1 = (int)cnt[q] - e - 1, nn = n1 + (int)cnt[q2] - beg2;
            LMS_DIRECT_COUNT(M_DONE, nn);
            if (full()) break;
            for (int u = threadIdx.x % L; u < nn; u += L) test(a, pa, ord[u < n1 ? e + 1 + u : beg2 + u - n1]);
        }
    }
    if (heavy) {
        // cells of many points (points on one line) are shared too, by the points'
        // indices, which every CTA agrees on: each meets the later ones of its cell
        for (int blk = part * BLOCK; blk < n; blk += parts * BLOCK) {
            for (int a = blk + (int)threadIdx.x / L; a < min(n, blk + BLOCK); a += T / L) {
                const int2 pa = pts[a];
                const int q = cell(pa), q2 = (q + 1) & (NC - 1);
                const int beg1 = q ? (int)cnt[q - 1] : 0, n1 = (int)cnt[q] - beg1;
                if (n1 <= HEAVY) continue;
                const int beg2 = q2 ? (int)cnt[q2 - 1] : 0, nn = n1 + (int)cnt[q2] - beg2;
                if (full()) break;
                for (int u = threadIdx.x % L; u < nn; u += L) {
                    const int b = ord[u < n1 ? beg1 + u : beg2 + u - n1];
                    if (u >= n1 || b > a) test(a, pa, b);
                }
            }
        }
    }
    __syncthreads();
    if (!want) table_append<T>(tab, m, nlist, over, HC, s_warp);
}

// The best of the CTA's candidates (buf: one a warp).
template <int T>
__device__ __forceinline__ Cand cta_best(Cand c, Cand *buf)
{
    if constexpr (T >= 32) {
        c = warp_best(c);
        if ((threadIdx.x & 31) == 0) buf[threadIdx.x >> 5] = c;
        __syncthreads();
        c = (threadIdx.x & 31) < T / 32 ? buf[threadIdx.x & 31] : cand_empty();
        c = warp_best(c);
        __syncthreads();
    }
    return c;
}

// The smallest width of the CTA's threads and the first window that has it.
template <int T, class W>
__device__ __forceinline__ void cta_first_min(W &bw, int &ba, long long *s_red)
{
    if constexpr (T >= 32) {
#pragma unroll
        for (int d = 16; d >= 1; d >>= 1) {
            const W ow = __shfl_xor_sync(FULL, bw, d);
            const int oa = __shfl_xor_sync(FULL, ba, d);
            if (ow < bw || (ow == bw && oa < ba)) { bw = ow; ba = oa; }
        }
        if ((threadIdx.x & 31) == 0) {
            s_red[2 * (threadIdx.x >> 5)] = (long long)bw;
            s_red[2 * (threadIdx.x >> 5) + 1] = ba;
        }
        __syncthreads();
        for (int w = 0; w < T / 32; ++w) {
            const W ow = (W)s_red[2 * w];
            const int oa = (int)s_red[2 * w + 1];
            if (ow < bw || (ow == bw && oa < ba)) { bw = ow; ba = oa; }
        }
        __syncthreads();
    }
}

// The narrowest window at the double slope s, as the float sweep computes it:
// z = y - s x in double, w = z_hi - z_lo; ties take the lowest window.
template <int T>
__device__ __noinline__ void score_f32(const FloatSet &f, int n, int h, double s, unsigned char *wk, int wk_bytes,
                                       unsigned char *gs, long long *s_red, double &w, double &t)
{
    int P = T;
    while (P < n) P <<= 1;
    auto key = [&](int k) { return k < n ? order_of(z_f32(f, k, s)) : D_MAX; };
    long long *v = reinterpret_cast<long long *>(wk);
    if (2 * P * 8 <= wk_bytes && P <= 16 * T) {
        cta_fill_merge_sort_any(v, v + P, P, key);
    } else {
        long long *g = reinterpret_cast<long long *>(gs);
        v = cta_sort_chunked<4 * T>(v, g, g + P, P, key);
    }
    long long bw = D_MAX;   // widths are >= 0: their bits order like them
    int ba = 0x7fffffff;
    for (int a = threadIdx.x; a + h - 1 < n; a += T) {
        const long long d = order_of(__dsub_rn(of_order(v[a + h - 1]), of_order(v[a])));
        if (d < bw) { bw = d; ba = a; }
    }
    cta_first_min<T>(bw, ba, s_red);
    const double zb = of_order(v[ba]), zt = of_order(v[ba + h - 1]);
    w = zt - zb;
    t = 0.5 * (zb + zt);
    __syncthreads();
}

__device__ __forceinline__ bool candd_better(const CandD &a, const CandD &b)
{
    if (!a.valid) return false;
    if (!b.valid) return true;
    if (a.w != b.w) return a.w < b.w;
    if (a.s != b.s) return a.s < b.s;
    if (a.t != b.t) return a.t < b.t;
    return a.pair < b.pair;
}

// Frame of a float set: centre and power-of-two scales that bring both axes
// into the grid.  False (in every thread) when the set has values that are
// not finite, no x range, or exponents so far apart that the scales would
// leave the doubles' normal range: those are left to the sweep.
template <int T>
__device__ bool float_box(const float *x, const float *y, int n, FloatSet &f, Box &bx, long long *s_red)
{
    float xl = INFINITY, xh = -INFINITY, yl = INFINITY, yh = -INFINITY;
    int bad = 0;
    for (int k = threadIdx.x; k < n; k += T) {
        const float u = x[k], v = y[k];
        bad |= !(isfinite(u) && isfinite(v));
        xl = fminf(xl, u); xh = fmaxf(xh, u);
        yl = fminf(yl, v); yh = fmaxf(yh, v);
    }
    float *r = reinterpret_cast<float *>(s_red);
    if constexpr (T >= 32) {
#pragma unroll
        for (int d = 16; d >= 1; d >>= 1) {
            xl = fminf(xl, __shfl_xor_sync(FULL, xl, d)); xh = fmaxf(xh, __shfl_xor_sync(FULL, xh, d));
            yl = fminf(yl, __shfl_xor_sync(FULL, yl, d)); yh = fmaxf(yh, __shfl_xor_sync(FULL, yh, d));
        }
        if ((threadIdx.x & 31) == 0) {
            r[4 * (threadIdx.x >> 5)] = xl; r[4 * (threadIdx.x >> 5) + 1] = xh;
            r[4 * (threadIdx.x >> 5) + 2] = yl; r[4 * (threadIdx.x >> 5) + 3] = yh;
        }
        bad = __syncthreads_or(bad);
        for (int w = 0; w < T / 32; ++w) {
            xl = fminf(xl, r[4 * w]); xh = fmaxf(xh, r[4 * w + 1]);
            yl = fminf(yl, r[4 * w + 2]); yh = fmaxf(yh, r[4 * w + 3]);
        }
        __syncthreads();
    }
    const double dx = (double)xh - (double)xl, dy = (double)yh - (double)yl;
    if (bad || !(dx > 1e-30) || !(dy > 1e-30) || dx > 1e30 || dy > 1e30) return false;
    f.x = x;
    f.y = y;
    f.xc = 0.5 * ((double)xl + (double)xh);
    f.yc = 0.5 * ((double)yl + (double)yh);
    // |v - c| <= d / 2 < 2^(e - 1): scaled below 2^F_BITS
    int ex, ey;
    frexp(dx, &ex);
    frexp(dy, &ey);
    f.sx = ldexp(1.0, F_BITS + 1 - ex);
    f.sy = ldexp(1.0, F_BITS + 1 - ey);
    f.ratio = ldexp(1.0, ex - ey);
    // A projection y - s x computed in double is off by at most 2^-53 (|s x| +
    // |y - s x|), a width of two of them by 2^-52 (2 |s x| + |y|) and its own
    // rounding, far below one unit; 2^-51 covers both.  Not small beside the
    // grid: points 2^22 of their spread away from the origin move by two steps.
    f.rx = ldexp(fmax(fabs((double)xl), fabs((double)xh)) * f.sx, -50);
    f.ry = ldexp(fmax(fabs((double)yl), fabs((double)yh)) * f.sy, F_YS - 51);
    if (threadIdx.x == 0) {
        bx.xc = bx.yc = bx.dh = 0;
        bx.xlo = __double2int_rn(((double)xl - f.xc) * f.sx);
        bx.xhi = __double2int_rn(((double)xh - f.xc) * f.sx);
        bx.ylo = __double2int_rn(((double)yl - f.yc) * f.sy);
        bx.yhi = __double2int_rn(((double)yh - f.yc) * f.sy);
    }
    return true;
}

// ------------------------------------------------------------------ exact score
// The narrowest window at slope dy/dx: all projections sorted as exact
// integers; ties take the lowest window.  wk: shared memory; gs: global
// scratch for sets that do not fit.
template <int T, class W>
__device__ void min_window(const W *s, int n, int h, W &bw, int &ba, long long *s_red)
{
    bw = ~(W)0;
    ba = 0x7fffffff;
    for (int a = threadIdx.x; a + h - 1 < n; a += T) {
        const W w = s[a + h - 1] - s[a];
        if (w < bw) { bw = w; ba = a; }
    }
    cta_first_min<T>(bw, ba, s_red);
}

template <int T>
__device__ __noinline__ Cand score(const int *pts, int n, int h, int dy, int dx, const Box &bx, unsigned char *wk, int wk_bytes,
                      unsigned char *gs, long long *s_red)
{
    const long long u = (long long)bx.xlo * dy, v = (long long)bx.xhi * dy;
    const long long lo = (long long)bx.ylo * dx - max(u, v), hi = (long long)bx.yhi * dx - min(u, v);
    int P = T;
    while (P < n) P <<= 1;
    Cand c = cand_empty();
    c.dy = dy;
    c.dx = dx;
    // centred projections are (projection) - (yc dx - xc dy)
    const long long back = 2 * ((long long)bx.yc * dx - (long long)bx.xc * dy);
    if (hi - lo < 0xffffffffLL) {
        auto key = [&](int k) { return k < n ? (unsigned)(proj(pts[k], dy, dx) - lo) : 0xffffffffu; };
        unsigned *s = reinterpret_cast<unsigned *>(wk);
        if (2 * P * 4 <= wk_bytes && P <= 16 * T) {
            cta_fill_merge_sort_any(s, s + P, P, key);
        } else {
            unsigned *g = reinterpret_cast<unsigned *>(gs);
            s = cta_sort_chunked<8 * T>(s, g, g + P, P, key);
        }
        unsigned bw;
        int ba;
        min_window<T, unsigned>(s, n, h, bw, ba, s_red);
        c.w = (long long)bw;
        c.t = (long long)s[ba] + (long long)s[ba + h - 1] + 2 * lo + back;
    } else {
        auto key = [&](int k) {
            return k < n ? (unsigned long long)(proj(pts[k], dy, dx) - lo) : 0xffffffffffffffffull;
        };
        unsigned long long *s = reinterpret_cast<unsigned long long *>(wk);
        if (2 * P * 8 <= wk_bytes && P <= 16 * T) {
            cta_fill_merge_sort_any(s, s + P, P, key);
        } else {
            unsigned long long *g = reinterpret_cast<unsigned long long *>(gs);
            s = cta_sort_chunked<4 * T>(s, g, g + P, P, key);
        }
        unsigned long long bw;
        int ba;
        min_window<T, unsigned long long>(s, n, h, bw, ba, s_red);
        c.w = (long long)bw;
        c.t = (long long)s[ba] + (long long)s[ba + h - 1] + 2 * lo + back;
    }
    __syncthreads();
    return c;
}

// The same from histograms: bins of the exact integers y dx - x dy, first of
// [t0, t1 + U] (where a window no wider than U must lie, units of 2^-32),
// then of the regions where the narrowest ones start and end, down to single
// values.  Two or three passes instead of a sort.  False when the regions
// stay too wide (many windows near the narrowest): the caller sorts.  c.dx =
// 0: no window within U.
template <int T, int NB>
__device__ __noinline__ bool score_bins(const Group<T> &g, const int *pts, int n, int h, int dy, int dx, long long U,
                                        long long t0, long long t1, const Box &bx, int *hist, Cand &c)
{
    const long long u = (long long)bx.xlo * dy, v = (long long)bx.xhi * dy;
    const long long zlo = (long long)bx.ylo * dx - max(u, v), zhi = (long long)bx.yhi * dx - min(u, v);
    long long lim = D_MAX, lo1 = zlo, hi1 = zhi + 1, lo2 = zlo, hi2 = zhi + 1, sl = zhi + 1;
    if (U < (1LL << 60)) lim = (long long)(((__int128)U * dx) >> 32);
    if (t0 <= t1) {
        lo1 = lo2 = max(zlo, (long long)(((__int128)t0 * dx) >> 32));
        sl = min(sl, (long long)(((__int128)t1 * dx) >> 32) + 2);
        hi1 = hi2 = lim < zhi - sl ? sl + lim + 1 : zhi + 1;
    }
    bool two = false;
    int sh = 62, b0, b1, e0, bm;
    c = cand_empty();
    for (int pass = 0; pass < 4; ++pass) {
        int s2;
        if (two) {
            s2 = shift_below(max(hi1 - lo1, hi2 - lo2) - 1, NB / 2 - 1);
        } else {
            hi2 = max(hi1, hi2);
            lo1 = min(lo1, lo2);
            s2 = shift_below(hi2 - lo1 - 1, NB);
        }
        if (s2 >= sh) return false;
        sh = s2;
        g.sync();
        hist_zero<T, NB>(g, hist);
        int mid = 0;
#pragma unroll 2
        for (int k = g.lane; k < n; k += T) {
            const long long z = proj(pts[k], dy, dx);
            if (z < lo1 || z >= hi2) continue;
            if (!two || z < hi1) atomicAdd(&hist[slot_of<NB / T>((int)((z - lo1) >> sh))], 1);
            else if (z < lo2) ++mid;
            else atomicAdd(&hist[slot_of<NB / T>(NB / 2 + (int)((z - lo2) >> sh))], 1);
        }
        if (two && mid) atomicAdd(&hist[slot_of<NB / T>(NB / 2 - 1)], mid);
        hist_cumulate<T, NB>(g, hist);
        const int half = two ? NB / 2 : 0;
        const int nst = (int)min((long long)(two ? NB / 2 - 1 : NB), ((sl - 1 - lo1) >> sh) + 1);
        const long long w = window_search<T, NB>(g, hist, nst, h, lim, lo1, lo2, half, sh, b0, b1, e0, bm);
        if (w == D_MAX) return true;
        const long long o1 = lo1, o2 = lo2;
        auto left = [&](int b) {
            return half == 0 || b < half ? o1 + ((long long)b << sh) : o2 + ((long long)(b - half) << sh);
        };
        if (sh == 0) {
            c.dy = dy;
            c.dx = dx;
            c.w = w;
            c.t = 2 * left(bm) + w + 2 * ((long long)bx.yc * dx - (long long)bx.xc * dy);
            g.sync();
            return true;
        }
        lo1 = left(b0);
        hi1 = min(sl, left(b1) + (1LL << sh));
        lo2 = left(e0);
        hi2 = min(hi2, hi1 + w + 1);   // later points of a start bin end later than its first
        sl = hi1;
        two = lo2 > hi1;
    }
    return false;
}

// The order of the points along slope dy/dx: words (projection, index),
// ascending, in shared memory where they fit, else in gs (32 bytes a point).
template <int T>
__device__ __noinline__ unsigned long long *sort_points(const int *pts, int n, int dy, int dx, const Box &bx,
                                                        unsigned char *wk, int wk_bytes, unsigned char *gs)
{
    const long long u = (long long)bx.xlo * dy, v = (long long)bx.xhi * dy;
    const long long lo = (long long)bx.ylo * dx - max(u, v);
    int P = T;
    while (P < n) P <<= 1;
    auto key = [&](int k) {   // projections span less than 2^34
        return k < n ? (unsigned long long)(proj(pts[k], dy, dx) - lo) << 16 | (unsigned)k : 0xffffffffffffffffull;
    };
    unsigned long long *s = reinterpret_cast<unsigned long long *>(wk);
    if (2 * P * 8 <= wk_bytes && P <= 16 * T) {
        cta_fill_merge_sort_any(s, s + P, P, key);
        return s;
    }
    unsigned long long *g = reinterpret_cast<unsigned long long *>(gs);
    return cta_sort_chunked<4 * T>(s, g, g + P, P, key);
}

// The narrowest windows at count slopes in ascending order (their indices in
// idx), one CTA: the points stay sorted from one slope to the next.  Where
// the slopes that survive are dense (widths that many slopes share: points in
// a few columns, near-vertical lines), few points change places between two
// of them, so the order is repaired by odd-even exchanges (two or three
// passes over the points) and every width is read off it, instead of two or
// three histogram passes with their scans for each slope.
template <int T>
__device__ __noinline__ void score_run(const int *pts, int n, int h, const long long *ev, const unsigned *evd,
                                       const int *idx, int count, const Box &bx, unsigned char *wk, int wk_bytes,
                                       unsigned char *gs, long long *s_red, Cand *out)
{
    unsigned long long *s = nullptr;
    for (int k = 0; k < count; ++k) {
        const int dx = (int)__ldcg(&evd[idx[k]]), dy = dy_of(__ldcg(&ev[idx[k]]), dx);
        bool sorted = false;
        for (int it = 0; s != nullptr && it < EXCHANGES; ++it) {
            int moved = 0;
            for (int odd = 0; odd < 2; ++odd) {
                for (int p = 2 * (int)threadIdx.x + odd; p + 1 < n; p += 2 * T) {
                    const unsigned long long a = s[p], b = s[p + 1];
                    const int pa = pts[a & 0xffffu], pb = pts[b & 0xffffu];
                    if (proj(pb, dy, dx) < proj(pa, dy, dx)) {
                        s[p] = b;
                        s[p + 1] = a;
                        moved = 1;
                    }
                }
                __syncthreads();
            }
            if (!__syncthreads_or(moved)) {
                sorted = true;
                break;
            }
        }
        if (!sorted) s = sort_points<T>(pts, n, dy, dx, bx, wk, wk_bytes, gs);
        __syncthreads();
        long long bw = D_MAX;
        int ba = 0x7fffffff;
        for (int a = threadIdx.x; a + h - 1 < n; a += T) {
            const long long w = proj(pts[s[a + h - 1] & 0xffffu], dy, dx) - proj(pts[s[a] & 0xffffu], dy, dx);
            if (w < bw) { bw = w; ba = a; }
        }
        cta_first_min<T>(bw, ba, s_red);
        if (threadIdx.x == 0) {
            Cand c = cand_empty();
            c.dy = dy;
            c.dx = dx;
            c.w = bw;
            // centred projections are (projection) - (yc dx - xc dy)
            c.t = 2 * proj(pts[s[ba] & 0xffffu], dy, dx) + bw + 2 * ((long long)bx.yc * dx - (long long)bx.xc * dy);
            out[k] = c;
        }
        __syncthreads();
    }
}

// The smallest index pair (i < j) with slope dy/dx, lowered into *out (a
// pair is i << 16 | j).  Points on one line of that slope share y dx - x dy; a
// table in shared memory keeps the smallest index of every line, then each
// point with another x than its line's first point makes a pair with it.
// Lines are dealt into `rounds` shares by a hash; this CTA does the shares
// part, part + parts, ..  table: `slots` words (a power of two), at least
// twice a share's points.
template <int T>
__device__ __noinline__ void line_pair(const int *pts, int n, int dy, int dx, unsigned *tab, int slots, int rounds,
                                       int part, int parts, unsigned *out, int *bad)
{
    for (int r = part; r < rounds; r += parts) {
        __syncthreads();
        for (int k = threadIdx.x; k < slots; k += T) tab[k] = ~0u;
        __syncthreads();
        for (int step = 0; step < 2; ++step) {
            for (int k = threadIdx.x; k < n; k += T) {
                const int p = pts[k];
                const long long z = proj(p, dy, dx);
                const unsigned hs = mix32((unsigned)z ^ (unsigned)(z >> 32) * 0x9e3779b9u);
                if ((int)(hs & (unsigned)(rounds - 1)) != r) continue;
                unsigned s = (hs >> 8) & (unsigned)(slots - 1);
                int probe = 0;
                for (; probe < slots; ++probe, s = (s + 1) & (unsigned)(slots - 1)) {
                    unsigned cur = *reinterpret_cast<volatile unsigned *>(&tab[s]);
                    if (cur == ~0u) {
                        cur = atomicCAS(&tab[s], ~0u, (unsigned)k);
                        if (cur == ~0u) break;
                    }
                    const int f = pts[cur];
                    if (proj(f, dy, dx) != z) continue;
                    if (step == 0) {
                        if (cur > (unsigned)k) atomicMin(&tab[s], (unsigned)k);
                    } else if (px(f) != px(p)) {
                        const unsigned pair = cur << 16 | (unsigned)k;
                        if (*reinterpret_cast<volatile unsigned *>(out) > pair) atomicMin(out, pair);
                    }
                    break;
                }
                if (probe == slots) *bad = 1;   // the share did not fit: reported, never silent
            }
            __syncthreads();
        }
    }
}

// Sets the bit of every point that repeats one of a smaller index (the words
// of dup are 0 before).  Table, rounds and shares as in line_pair.
template <int T>
__device__ __noinline__ void mark_duplicates(const int *pts, int n, unsigned *tab, int slots, int rounds, int part,
                                             int parts, unsigned *dup, int *bad)
{
    for (int r = part; r < rounds; r += parts) {
        __syncthreads();
        for (int k = threadIdx.x; k < slots; k += T) tab[k] = ~0u;
        __syncthreads();
        for (int step = 0; step < 2; ++step) {
            for (int k = threadIdx.x; k < n; k += T) {
                const int p = pts[k];
                const unsigned hs = mix32((unsigned)p);
                if ((int)(hs & (unsigned)(rounds - 1)) != r) continue;
                unsigned s = (hs >> 8) & (unsigned)(slots - 1);
                int probe = 0;
                for (; probe < slots; ++probe, s = (s + 1) & (unsigned)(slots - 1)) {
                    unsigned cur = *reinterpret_cast<volatile unsigned *>(&tab[s]);
                    if (cur == ~0u) {
                        cur = atomicCAS(&tab[s], ~0u, (unsigned)k);
                        if (cur == ~0u) break;
                    }
                    if (pts[cur] != p) continue;
                    if (step == 0) {
                        if (cur > (unsigned)k) atomicMin(&tab[s], (unsigned)k);
                    } else if (cur != (unsigned)k) {
                        atomicOr(&dup[k >> 5], 1u << (k & 31));
                    }
                    break;
                }
                if (probe == slots) *bad = 1;
            }
            __syncthreads();
        }
    }
}

// ------------------------------------------------------------------ kernel
struct DirectArgs {
    const short *x, *y;           // points of every set
    const float *xf, *yf;         // points of a float set
    int *done;                    // set to 1 once a float set's record is written
    const long long *off;         // set offsets (null: one set of n points)
    const int *hvec;              // order statistics per set (null: h)
    const int *sets;              // set indices in the order they are fitted (null: one set)
    const float *pred;            // predicted slope of the one set (or null)
    lms_result *out;
    unsigned char *mem;           // teams' memory
    int *next;                    // next set (several sets)
    int *set_done;                // per set (or null): 0 when a set of at most small_max points is left to another kernel
    int small_max;
    int n, h, nsets;
    int algo, plain_max, bnb_min;   // reported path: PLAIN up to plain_max points, BNB from bnb_min on, else algo
    TeamShape shape;
};

__device__ __forceinline__ long long gcd64(long long a, long long b)
{
    while (b) { long long r = a % b; a = b; b = r; }
    return a;
}

__device__ inline void write_result(lms_result *out, const Cand &b, int algo, int err)
{
    lms_result r;
    r.algorithm = algo;
    if (b.dx <= 0 || err) {
        r.w_num = r.w_den = r.s_num = r.s_den = r.t_num = r.t_den = 0;
        r.theta1 = r.theta2 = r.med_sq = 0.0;
        r.i = r.j = -1;
        r.status = LMS_ERR_INTERNAL;
        *out = r;
        return;
    }
    const long long dx = b.dx, dy = b.dy;
    long long g = gcd64(dy < 0 ? -dy : dy, dx);
    if (g <= 0) g = 1;
    r.s_num = dy / g;
    r.s_den = dx / g;
    r.w_num = b.w / g;
    r.w_den = r.s_den;
    r.t_num = b.t / g;
    r.t_den = 2 * r.s_den;
    r.theta1 = __ddiv_rn((double)r.s_num, (double)r.s_den);
    r.theta2 = __ddiv_rn((double)r.t_num, (double)r.t_den);
    const double half = __ddiv_rn((double)r.w_num, (double)(2 * r.w_den));
    r.med_sq = __dmul_rn(half, half);
    r.i = b.i;
    r.j = b.j;
    r.status = b.i < 0 ? LMS_ERR_VERTICAL : LMS_OK;
    *out = r;
}

// Shared memory ahead of the points and the work area.  Every CTA of a team
// plans the phases for itself from the same inputs, so the plan needs no
// messages: only answers, listed slopes and scores pass through global memory.
template <int NS, int PM, int LC>
struct DShared {
    long long red[128];          // group reductions (4 words a warp) and CTA reductions
    long long smp[NS];           // sorted sampled slope keys
    DNode work[2][PM];           // this phase's intervals or runs, ascending; the next ones
    DNode leaf[LC];
    int keep[PM];                // indices of the surviving work items
    int xl[PM];                  // slopes to score
    int warp_a[32], warp_b[32];
    Box bx;
    int nsmp, set;
    long long t0, t1;
    // what listing has learned; kept here, not in registers, since every call of the
    // loop below saves what is live (read before a barrier, written by thread 0 after it)
    float gain;                  // slopes to expect for each pair expected
    int lcap, regrown, cuts;     // leaves listed at a time; times that leaves or lists were cut
    int marked;                  // duplicates are marked
};

// Children of a tree node: cut keys into c[1 .. count - 1] (c[0] = a, c[count] = b).
__device__ inline int cut_node(const DNode &nd, const long long *smp, int m, long long *c)
{
    const long long a = nd.a, b = nd.b;
    int k = 1;
    c[0] = a;
    auto add = [&](long long v) { if (v > c[k - 1] && v < b && k < NODE_F) c[k++] = v; };
    const long long one = 1LL << 32;
    if (a <= -D_GUARD && b >= D_GUARD) {
        add(-one);
        add(0);
        add(one);
    } else if (b >= D_GUARD && a < D_GUARD - 1) {
        const long long t = a < 0 ? 0 : 4 * a + one;
        add(t);
        add(4 * t + one < D_GUARD ? 4 * t + one : D_GUARD - 1);
        add(D_GUARD - 1);
    } else if (a <= -D_GUARD && b > -(D_GUARD - 1)) {
        const long long t = b > 0 ? 0 : 4 * b - one;
        add(-(D_GUARD - 1));
        add(4 * t - one > -D_GUARD ? 4 * t - one : -(D_GUARD - 1));
        add(t);
    } else {
        auto rank = [&](long long v) {   // samples < v
            int lo = 0, hi = m;
            while (lo < hi) {
                const int q = (lo + hi) >> 1;
                if (smp[q] < v) lo = q + 1; else hi = q;
            }
            return lo;
        };
        const int r0 = rank(a + 1), cnt = rank(b) - r0;
        if (cnt >= NODE_F - 1) {
            for (int f = 1; f < NODE_F; ++f) add(smp[r0 + (int)((long long)cnt * f / NODE_F)]);
        }
        if (k == 1) {
            const long long d = b - a, big = max(a < 0 ? -a : a, b < 0 ? -b : b);
            if (d > big / 2 && d > one / 4) {
                // a tail of the slopes: most of its pairs lie near the flat end
                const bool up = big == b;
                add(up ? a + d / 64 : b - d / 4);
                add(up ? a + d / 16 : b - d / 16);
                add(up ? a + d / 4 : b - d / 64);
            } else
            for (int f = 1; f < NODE_F; ++f) add(a + d / NODE_F * f + d % NODE_F * f / NODE_F);
        }
    }
    c[k] = b;
    return k;
}

template <int T, int G, int NB, int NBW, int PM, int LRUN, bool SP, bool F>
__global__ void __launch_bounds__(T) k_direct(const DirectArgs A)
{
    extern __shared__ __align__(16) unsigned char dsm[];
    using P_t = std::conditional_t<F, int2, int>;
    constexpr int GROUPS = T / G;
    constexpr int NS = T < 512 ? 512 : T;   // sampled slopes
    constexpr int LC = LRUN + PM;
    using Shared = DShared<NS, PM, LC>;
    Shared &S = *reinterpret_cast<Shared *>(dsm);
    const TeamShape &sh = A.shape;
    const unsigned C = cluster_ctas(), rank = cluster_rank();
    const int team = blockIdx.x / C;
    const TeamMem m = team_carve(A.mem + (long long)team * team_bytes(sh), sh);
    TeamState *st = m.st;
    unsigned char *gsort = m.sort + d_up(sh.sortw) * rank;
    auto team_sync = [&]() {
        if (C == 1) __syncthreads();
        else cluster_meet();
    };
    Group<G> g;
    g.id = threadIdx.x / G;
    g.lane = threadIdx.x % G;
    g.red = S.red + 4 * (G < 32 ? 0 : (threadIdx.x / G) * (G / 32));
    const int NG = GROUPS * (int)C, gi = g.id * (int)C + (int)rank;
    Group<T> gw;
    gw.id = 0;
    gw.lane = threadIdx.x;
    gw.red = S.red;

    for (int turn = 0;; ++turn) {
        // ---------------------------------------------------------- the next set
        int set = 0, n = A.n, h = A.h;
        long long base = 0;
        if (A.sets) {
            if (threadIdx.x == 0) S.set = atomicAdd(A.next, 1);
            __syncthreads();
            const int at = S.set;
            __syncthreads();
            if (at >= A.nsets) return;
            set = A.sets[at];
            base = A.off[set];
            n = (int)(A.off[set + 1] - base);
            h = A.hvec[set];
        } else if (turn) {
            return;
        }
        [[maybe_unused]] const short *x = A.x + base, *y = A.y + base;
        P_t *pts = SP ? reinterpret_cast<P_t *>(dsm + sizeof(Shared)) : reinterpret_cast<P_t *>(m.pts);
        unsigned char *wk = dsm + sizeof(Shared) + (SP ? (((int)sizeof(P_t) * n + 15) & ~15) : 0);
        const int wk_bytes = (int)smem_size() - (int)(wk - dsm);
        int *hist = reinterpret_cast<int *>(wk) + g.id * NB, *histw = reinterpret_cast<int *>(wk);

        // ---------------------------------------------------------- box, centred points
        FloatSet fs{};
        if constexpr (F) {
            if (!float_box<T>(A.xf, A.yf, n, fs, S.bx, S.red)) return;   // left to the sweep
            for (int k = (SP ? 0 : (int)rank * T) + (int)threadIdx.x; k < n; k += SP ? T : T * (int)C)
                pts[k] = make_int2(__double2int_rn(((double)A.xf[k] - fs.xc) * fs.sx),
                                   __double2int_rn(((double)A.yf[k] - fs.yc) * fs.sy));
        } else {
            int xl = 0x7fffffff, xh = -0x7fffffff, yl = 0x7fffffff, yh = -0x7fffffff;
            for (int k = threadIdx.x; k < n; k += T) {
                const int xv = x[k], yv = y[k];
                xl = min(xl, xv); xh = max(xh, xv);
                yl = min(yl, yv); yh = max(yh, yv);
                if (SP) pts[k] = pack_xy(xv, yv);
            }
            cta_min_max_i<T>(xl, xh, S.warp_a, S.warp_b);
            cta_min_max_i<T>(yl, yh, S.warp_a, S.warp_b);
            // the upper midrange: centred coordinates stay within int16
            const int xc = (xl + xh + 1) >> 1, yc = (yl + yh + 1) >> 1;
            if (SP) {
                for (int k = threadIdx.x; k < n; k += T) pts[k] = pack_xy(px(pts[k]) - xc, py(pts[k]) - yc);
            } else {
                for (int k = rank * T + threadIdx.x; k < n; k += T * C) pts[k] = pack_xy(x[k] - xc, y[k] - yc);
            }
            if (threadIdx.x == 0) {
                S.bx.xc = xc; S.bx.yc = yc;
                S.bx.xlo = xl - xc; S.bx.xhi = xh - xc;
                S.bx.ylo = yl - yc; S.bx.yhi = yh - yc;
                S.bx.dh = 0;
            }
        }
        if (rank == 0 && threadIdx.x == 0) {
            st->ub = D_MAX;
            st->bad = 0;
            st->pair[0] = st->pair[1] = 0xffffffffu;
            st->nlist[0] = st->nlist[1] = st->over[0] = st->over[1] = 0;
        }
        team_sync();
        auto brief = [&]() { return !F && A.set_done && n <= A.small_max; };
        auto phases = [&]() { return F ? F_PHASES : brief() ? SMALL_PHASES : PHASES_MAX; };
        const int algo = n <= A.plain_max ? LMS_ALGO_PLAIN : n >= A.bnb_min ? LMS_ALGO_BNB : A.algo;
        if constexpr (!F) {
        if (S.bx.xlo == S.bx.xhi) {
            // every x equal: the window at slope 0
            if (rank == 0) {
                Cand c = score<T>(pts, n, h, 0, 1, S.bx, wk, wk_bytes, gsort, S.red);
                c.i = c.j = -1;
                if (threadIdx.x == 0) {
                    write_result(A.out + set, c, algo, 0);
                    if (brief()) A.set_done[set] = 1;
                }
            }
            team_sync();
            continue;
        }
        }
        // a lower bound of the x-span of any h points: narrowest window of h
        // over the histogram of x, less its two end bins
        {
            const int xr = S.bx.xhi - S.bx.xlo, s = shift_below(xr, NBW - 1);
            hist_zero<T, NBW>(gw, histw);
            for (int k = threadIdx.x; k < n; k += T) atomicAdd(&histw[slot_of<NBW / T>((px(pts[k]) - S.bx.xlo) >> s)], 1);
            hist_cumulate<T, NBW>(gw, histw);
            int b0, b1, e0, bm;
            const long long w = window_search<T, NBW>(gw, histw, NBW, h, D_MAX, 0, 0, 0, s, b0, b1, e0, bm);
            if (threadIdx.x == 0) S.bx.dh = w == D_MAX ? 0 : (int)max(0LL, w + 2 - (2LL << s));
        }
        __syncthreads();
        const Box bx = S.bx;
        const int yr = bx.yhi - bx.ylo, xr = bx.xhi - bx.xlo;
        // above every pair's slope; float sets leave steeper ones to the bound below
        const long long kmax = F ? F_KMAX : ((long long)yr + 1) << 32;

        // Float sets: w at a slope differs by at most (1 + |s|) steps and the rounding
        // of its doubles from w of the grid points.  An upper bound is raised by that much, and an interval is
        // tested against the upper bound raised once more.
        auto grid_key = [&](double s) { return (long long)floor(s * fs.ratio * (double)(1LL << F_YS)); };
        auto grid_err = [&](long long K) {
            if (!F) return 0LL;
            const long long k = K < 0 ? -K : K;
            return (1LL << F_YS) + k + 4 + (long long)(fs.rx * (double)k + fs.ry);
        };

        // ---------------------------------------------------------- sampled slopes (the same in every CTA)
        {
            auto sample = [&](int k) -> long long {
                const unsigned u = mix32(2u * k + 0x51ed270bu), v = mix32(2u * k + 0x2545f491u);
                const int i = (int)__umulhi(u, (unsigned)n);
                int j = (int)__umulhi(v, (unsigned)(n - 1));
                j += j >= i;
                if constexpr (F) {
                    double v;
                    if (!slope_f32(fs, i, j, v)) return D_MAX;
                    v *= fs.ratio * (double)(1LL << F_YS);
                    return fabs(v) < (double)(F_KMAX - 1) ? (long long)floor(v) : D_MAX;
                } else {
                    int dy, dx;
                    if (!pair_slope(pts[i], pts[j], dy, dx)) return D_MAX;
                    return slope_key(dy, dx);
                }
            };
            long long *s = reinterpret_cast<long long *>(wk);
            cta_fill_merge_sort_any(s, s + NS, NS, sample);
            int mm = 0;
            for (int k = threadIdx.x; k < NS; k += T) {
                S.smp[k] = s[k];
                mm = max(mm, s[k] < D_MAX ? k + 1 : 0);
            }
            int dummy = 0;
            cta_min_max_i<T>(dummy, mm, S.warp_a, S.warp_b);
            if (threadIdx.x == 0) S.nsmp = mm;
            __syncthreads();
        }
        const int ms = S.nsmp;
        // root cuts: quantiles of the sample; each of them is an upper bound
        const int Q = ms ? sh.Q : 0;
        auto cut = [&](int q) { return S.smp[(int)((2LL * q + 1) * ms / (2 * Q))]; };
        auto seed = [&](int q, long long &K) {
            if (q < Q) {
                K = cut(q);
                if (q > 0 && cut(q - 1) == K) return false;
            } else {
                if (!A.pred) return false;
                const float v = *A.pred;
                if (!(fabsf(v) < 16000.0f)) return false;
                K = (long long)((double)v * 4294967296.0);   // float sets have no prediction
            }
            return K > -kmax && K < kmax;
        };
        // one coarse pass for each, then to the end for the narrowest (and those of the
        // same coarse width)
        for (int q = gi; q < Q + 1; q += NG) {
            long long K, lower = D_MAX;
            if (seed(q, K)) {
                lower = ub_at<G, NB>(g, pts, n, h, K, D_MAX, bx, hist, 1, 0, true);
                if (lower < D_MAX) lower += grid_err(K);
                if (g.lane == 0 && lower < D_MAX) atomicMin(&st->ub, lower);
            }
            if (g.lane == 0) m.ans[q].t0 = lower;   // the coarse width
        }
        team_sync();
        {
            const int per = (Q + T) / T;
            const int q0 = min(Q + 1, (int)threadIdx.x * per), q1 = min(Q + 1, q0 + per);
            const long long ub = __ldcg(&st->ub);   // stable: nobody lowers it before the next barrier
            int c = 0, ns;
            for (int q = q0; q < q1; ++q) c += __ldcg(&m.ans[q].t0) <= ub;
            int at = cta_scan_ex<T>(c, S.warp_a, ns);
            for (int q = q0; q < q1; ++q)
                if (__ldcg(&m.ans[q].t0) <= ub) S.keep[at++] = q;
            team_sync();   // everyone has read the coarse bound
            ns = min(ns, C > 1 ? (int)C : NG);   // one round: the tree looks further anyway
            auto refine = [&](auto &gr, auto nb, int *hs, int i) {
                constexpr int GG = std::remove_reference_t<decltype(gr)>::SIZE;
                long long K;
                if (!seed(S.keep[i], K)) return;
                const long long u = gr.first(__ldcg(&st->ub));   // others lower it meanwhile: one value for the group
                const long long w = ub_at<GG, decltype(nb)::value>(gr, pts, n, h, K, u, bx, hs, 1, 0);
                if (gr.lane == 0 && w < D_MAX / 2 && w + grid_err(K) < u) atomicMin(&st->ub, w + grid_err(K));
            };
            if (C > 1 && ns <= (int)C * WIDE_ITEMS) {
                for (int i = rank; i < ns; i += C) refine(gw, std::integral_constant<int, NBW>(), histw, i);
            } else {
                for (int i = gi; i < ns; i += NG) refine(g, std::integral_constant<int, NB>(), hist, i);
            }
        }
        if constexpr (F) {
            // steep slopes that stay in reach even at half the bound make the attempt useless
            team_sync();
            const long long U = __ldcg(&st->ub) / 2;
            if (!steep_above_at(F_KMAX, bx.dh, yr, U < D_MAX / 4 ? U + grid_err(F_KMAX) : D_MAX)) return;
        }
        for (int q = threadIdx.x; q <= Q; q += T) {
            DNode nd;
            nd.a = q == 0 ? -kmax : cut(q - 1);
            nd.b = q == Q ? kmax : cut(q);
            nd.t0 = 1;
            nd.t1 = 0;
            nd.force = 0;
            nd.est = nd.a < nd.b ? 0.5f * (float)n * (float)(n - 1) / (float)(Q + 1) : -1.0f;
            S.work[0][q] = nd;
        }
        // hash tables of line_pair and mark_duplicates
        auto table_slots = [&]() {
            int slots = 1024;
            while (slots * 8 <= wk_bytes && slots < 2 * n) slots <<= 1;
            return slots;
        };
        auto table_rounds = [&](int slots) {
            int rounds = 1;
            while (rounds < (int)C || (long long)rounds * slots < 2LL * n) rounds <<= 1;
            return rounds;
        };
        if (threadIdx.x == 0) {
            S.gain = 1.0f;
            S.lcap = LC;
            S.regrown = S.cuts = S.marked = 0;
        }
        // the plan: the same values in every thread of the team
        int mode = M_TREE, P = Q + 1, cur = 0, par = 0, lpar = 0, ppar = 0;
        int top = 0, etop = 0, nleaf = 0, lf0 = 0, lfn = 0, nx = 0, err = 0, scored = 0;
        bool flush = false;
        long long ux = D_MAX, uxl = D_MAX, bkey = D_MAX;
        Cand best = cand_empty();
        CandD bestd{};
        team_sync();
        for (int phase = 0; mode != M_DONE; ++phase) {
            DNode *work = S.work[cur], *next = S.work[cur ^ 1];
            LMS_DIRECT_COUNT(mode, mode == M_EXACT ? nx : mode == M_PAIRS ? lfn : P);
            if (mode == M_TREE || mode == M_EVENT) {
                const bool ev = mode == M_EVENT;
                // ------------------------------------------------ interval tests
                Answer *ans = m.ans + par * PM;
                auto test = [&](auto &gr, auto nb, int *hs, int k) {
                    constexpr int GG = std::remove_reference_t<decltype(gr)>::SIZE;
                    const DNode &nd = work[k];
                    long long ka = ev ? __ldcg(&m.ev[nd.a]) : nd.a;
                    long long kb = ev ? __ldcg(&m.ev[nd.b - 1]) + 1 : nd.b;
                    const bool right = F && !ev ? bestd.valid && ka > grid_key(bestd.s) + 1 : ka > bkey;
                    long long U = min(gr.first(__ldcg(&st->ub)), right ? uxl : ux);
                    if constexpr (F) {
                        if (ev) {
                            ka = grid_key(of_order(ka)) - 1;
                            kb = grid_key(of_order(kb - 1)) + 2;
                        }
                        if (U >= 0 && U < D_MAX / 2) U += max(grid_err(ka), grid_err(kb)) + 4;
                    }
                    long long t0 = nd.t0, t1 = nd.t1;
                    bool keep;
                    if ((!ev && nd.est < 0.0f) || (!F && steep_above(ka, kb, bx.dh, yr, U))) keep = false;
                    else
                        keep = may_hold<GG, decltype(nb)::value>(gr, pts, n, h, ka, kb, U, ev ? U >> 18 : U >> 12, bx,
                                                                 hs, t0, t1);
                    if (gr.lane == 0) {
                        ans[k].t0 = t0;
                        ans[k].t1 = t1;
                        ans[k].keep = keep;
                    }
                };
                if (C > 1 && P <= (int)C * WIDE_ITEMS) {
                    for (int k = rank; k < P; k += C) test(gw, std::integral_constant<int, NBW>(), histw, k);
                } else {
                    for (int k = gi; k < P; k += NG) test(g, std::integral_constant<int, NB>(), hist, k);
                }
                team_sync();
                // ------------------------------------------------ survivors, and an upper bound at the middle of each
                const int per = (P + T - 1) / T;
                const int k0 = min(P, (int)threadIdx.x * per), k1 = min(P, k0 + per);
                int c = 0, ns;
                for (int k = k0; k < k1; ++k) c += __ldcg(&ans[k].keep) != 0;
                int at = cta_scan_ex<T>(c, S.warp_a, ns);
                for (int k = k0; k < k1; ++k)
                    if (__ldcg(&ans[k].keep)) {
                        S.keep[at++] = k;
                        work[k].t0 = __ldcg(&ans[k].t0);
                        work[k].t1 = __ldcg(&ans[k].t1);
                    }
                __syncthreads();
                par ^= 1;
                auto bound = [&](auto &gr, auto nb, int *hs, int i) {
                    constexpr int GG = std::remove_reference_t<decltype(gr)>::SIZE;
                    const DNode &nd = work[S.keep[i]];
                    if (ev && nd.b - nd.a == 1) return;
                    long long K = ev ? __ldcg(&m.ev[(nd.a + nd.b) >> 1]) : nd.a + ((nd.b - nd.a) >> 1);
                    if (F && ev) K = grid_key(of_order(K));
                    const long long ub = gr.first(__ldcg(&st->ub));
                    const long long w = ub_at<GG, decltype(nb)::value>(gr, pts, n, h, K, ub, bx, hs, nd.t0, nd.t1);
                    if (gr.lane == 0 && w < D_MAX / 2 && w + grid_err(K) < ub) atomicMin(&st->ub, w + grid_err(K));
                };
                if (ns > 0) {
                    if (C > 1 && ns <= (int)C * WIDE_ITEMS) {
                        for (int i = rank; i < ns; i += C) bound(gw, std::integral_constant<int, NBW>(), histw, i);
                    } else {
                        for (int i = gi; i < ns; i += NG) bound(g, std::integral_constant<int, NB>(), hist, i);
                    }
                    team_sync();
                }
                // ------------------------------------------------ children and leaves, or runs and slopes to score
                // (intervals across D_GUARD are cut whatever their expected pairs)
                auto is_leaf = [&](const DNode &nd) {
                    if (nd.a < D_GUARD - 1 && nd.b >= D_GUARD) return false;
                    if (nd.b > -(D_GUARD - 1) && nd.a <= -D_GUARD) return false;
                    if (nd.b - nd.a == 1) return true;
                    if (nd.force > 0) return false;
                    const float f = F ? 0.0f : fractions(nd.a, nd.b, xr, yr);
                    return nd.est * S.gain <= sh.leaf || (!F && f <= LEAF_FRACTIONS);
                };
                const int pers = (ns + T - 1) / T;
                const int i0 = min(ns, (int)threadIdx.x * pers), i1 = min(ns, i0 + pers);
                long long cuts[NODE_F + 1];
                int kids = 0, ends = 0, tk;
                for (int i = i0; i < i1; ++i) {
                    const DNode &nd = work[S.keep[i]];
                    if (ev ? nd.b - nd.a == 1 : is_leaf(nd)) ++ends;
                    else kids += ev ? (int)min(nd.b - nd.a, (long long)EV_F) : cut_node(nd, S.smp, ms, cuts);
                }
                int ak = cta_scan_ex<T>(kids | ends << 16, S.warp_a, tk);
                int ae = ak >> 16;
                const int te = tk >> 16;
                ak &= 0xffff;
                tk &= 0xffff;
                int &tp = ev ? etop : top;
                DNode *stack = ev ? m.estack : m.stack;
                // the leftmost PM children are the next work; the rest waits on the stack
                const int spill = max(0, tk - PM);
                if (tp + spill > (ev ? estack_cap(sh) : stack_cap(sh)) || (!ev && nleaf + te > LC)) err = 1;
                if (!err) {
                    for (int i = i0; i < i1; ++i) {
                        const DNode nd = work[S.keep[i]];
                        if (ev ? nd.b - nd.a == 1 : is_leaf(nd)) {
                            if (ev) S.xl[ae++] = (int)nd.a;
                            else S.leaf[nleaf + ae++] = nd;
                            continue;
                        }
                        const int len = ev ? (int)(nd.b - nd.a) : 0;
                        const int f = ev ? min(len, EV_F) : pers == 1 ? kids : cut_node(nd, S.smp, ms, cuts);
                        for (int q = 0; q < f; ++q, ++ak) {
                            DNode ch = nd;
                            if (ev) {
                                ch.a = nd.a + (long long)len * q / f;
                                ch.b = nd.a + (long long)len * (q + 1) / f;
                            } else {
                                ch.a = cuts[q];
                                ch.b = cuts[q + 1];
                                ch.est = nd.est / NODE_F;
                                ch.force = max(0, nd.force - 1);
                            }
                            if (ak < PM) next[ak] = ch;
                            else if (rank == 0) stack[tp + tk - 1 - ak] = ch;
                        }
                    }
                }
                P = min(tk, PM);
                tp += spill;
                if (ev) nx = te;
                else nleaf += te;
                if (tk < PM && tp > 0) {
                    // entries on the stack are at least one barrier old here
                    const int more = min(tp, PM - tk);
                    for (int j = threadIdx.x; j < more; j += T) next[tk + j] = ld_node(&stack[tp - 1 - j]);
                    tp -= more;
                    P += more;
                }
                cur ^= 1;
                __syncthreads();
                if (ev && nx > 0) {
                    // scored before the next runs are tested: those wait on the stack
                    if (rank == 0)
                        for (int j = threadIdx.x; j < P; j += T) stack[tp + P - 1 - j] = S.work[cur][j];
                    tp += P;
                    P = 0;
                }
            } else if (mode == M_PAIRS) {
                // ------------------------------------------------ distinct slopes of the leaves
                int NC = T;
                while (NC < n && NC < CELLS_MAX) NC <<= 1;
                const int parts = max(1, (int)C / lfn);
                // (read here; thread 0 writes them behind the barrier)
                float gain = S.gain;
                int lcap = S.lcap, regrown = S.regrown, cuts_made = S.cuts;
                [[maybe_unused]] int marked = S.marked;
                for (int l = rank; l < lfn * parts; l += C) {
                    const DNode &lf = S.leaf[lf0 + l / parts];
                    if constexpr (F)
                        list_pairs_f32<T>(pts, n, lf.a, lf.b, bx, fs, NC, wk, S.warp_a, m, &st->nlist[lpar],
                                          &st->over[lpar], sh.HC, l % parts, parts);
                    else {
                        const bool listed = list_pairs<T>(pts, n, marked ? m.dup : nullptr, lf, bx, NC, wk, S.warp_a,
                                                          m, &st->nlist[lpar], &st->over[lpar], sh.HC,
                                                          l % parts, parts);
                        if (threadIdx.x == 0 && l % parts == 0) {
                            m.ans[l / parts].dense = !listed;   // (no test runs here; LC <= 2 PM answers)
                            if (!listed && !marked) atomicMax(&st->over[lpar], 2);
                        }
                    }
                }
                team_sync();
                const int over = __ldcg(&st->over[lpar]);
                const int nn = __ldcg(&st->nlist[lpar]);
                // slopes to expect for each pair expected: few where many pairs share a slope
                {
                    float held;
                    leaves_within<T, F>(S.leaf + lf0, lfn, 1e30f, gain, xr, yr, held);
                    if (F && (over == 2 || (over && (++cuts_made > F_CUTS || (lfn == 1 && S.leaf[lf0].b - S.leaf[lf0].a == 1)))))
                        err = 1;   // more slopes or candidates than the sweep is worth
                    if (over == 1 && lfn == 1) gain = fminf(64.0f, 4.0f * gain);
                    else if (8.0f * (float)nn < held) gain = fmaxf(1.0f / 4096, 0.25f * gain);
                }
                if constexpr (!F) {
                    if (over == 2) {
                        // the first leaf with too many candidates: duplicates are marked, the leaves listed again
                        for (int k = rank * T + threadIdx.x; k < (n + 31) / 32; k += T * C) m.dup[k] = 0u;
                        team_sync();
                        mark_duplicates<T>(pts, n, reinterpret_cast<unsigned *>(wk), table_slots(), table_rounds(table_slots()),
                                           (int)rank, (int)C, m.dup, &st->bad);
                        marked = 1;
                    }
                }
                if (rank == 0 && !over) {
                    long long *s = reinterpret_cast<long long *>(wk);
                    if (nn <= 512) {
                        // few slopes: each finds its rank
                        for (int k = threadIdx.x; k < nn; k += T) s[k] = __ldcg(&m.lkey[k]);
                        __syncthreads();
                        for (int k = threadIdx.x; k < nn; k += T) {
                            const long long v = s[k];
                            int r = 0;
                            for (int j = 0; j < nn; ++j) r += s[j] < v || (s[j] == v && j < k);
                            m.ev[r] = v;
                            m.evd[r] = __ldcg(&m.lden[k]);
                        }
                    } else {
                        int P2 = T;
                        while (P2 < nn) P2 <<= 1;
                        auto key = [&](int k) { return k < nn ? __ldcg(&m.lkey[k]) : D_MAX; };
                        if (16 * P2 <= wk_bytes) {
                            cta_fill_merge_sort_any(s, s + P2, P2, key);
                        } else {
                            long long *gk = reinterpret_cast<long long *>(gsort);
                            s = cta_sort_chunked<4 * T>(s, gk, gk + P2, P2, key);
                        }
                        for (int k = threadIdx.x; k < nn; k += T) {
                            m.ev[k] = s[k];
                            const long long v = __ldcg(&m.lkey[k]);
                            int lo = 0, hi = nn - 1;
                            while (lo < hi) {
                                const int q = (lo + hi) >> 1;
                                if (s[q] < v) lo = q + 1; else hi = q;
                            }
                            const unsigned den = __ldcg(&m.lden[k]);
                            for (; lo < nn && s[lo] == v; ++lo) m.evd[lo] = den;
                        }
                    }
                }
                if (rank == 0 && threadIdx.x == 0) st->nlist[lpar ^ 1] = st->over[lpar ^ 1] = 0;
                lpar ^= 1;
                if (!over) {
                    // where their windows can start: over all leaves listed
                    if (threadIdx.x == 0) {
                        long long t0 = D_MAX, t1 = -D_MAX;
                        bool known = true;
                        for (int k = lf0; k < lf0 + lfn; ++k) {
                            known = known && S.leaf[k].t0 <= S.leaf[k].t1;
                            t0 = min(t0, S.leaf[k].t0);
                            t1 = max(t1, S.leaf[k].t1);
                        }
                        S.t0 = known ? t0 : 1;
                        S.t1 = known ? t1 : 0;
                    }
                    __syncthreads();
                    const int runs = min(nn, min(PM, max(8, NG)));
                    for (int q = threadIdx.x; q < runs; q += T) {
                        DNode nd;
                        nd.a = (long long)nn * q / runs;
                        nd.b = (long long)nn * (q + 1) / runs;
                        nd.t0 = S.t0;
                        nd.t1 = S.t1;
                        nd.est = 0.0f;
                        nd.force = 0;
                        S.work[cur][q] = nd;
                    }
                    P = runs;
                    lcap = min(2 * lcap, LC);
                    if constexpr (!F) {
                        // leaves with too many candidates are cut before they are listed again
                        int any = 0;
                        for (int l = threadIdx.x; l < lfn; l += T) any |= __ldcg(&m.ans[l].dense);
                        if (__syncthreads_or(any)) {
                            int dense = 0;
                            for (int l = 0; l < lfn; ++l) dense += __ldcg(&m.ans[l].dense);
                            if (top + dense > stack_cap(sh)) err = 1;
                            for (int l = lfn - 1, at = top; l >= 0 && !err && rank == 0 && threadIdx.x == 0; --l)
                                if (__ldcg(&m.ans[l].dense)) {
                                    DNode nd = S.leaf[lf0 + l];
                                    nd.force = 2;
                                    m.stack[at++] = nd;
                                }
                            top += dense;
                        }
                    }
                    lf0 += lfn;
                    if (lf0 == nleaf) {
                        lf0 = nleaf = 0;
                        flush = false;
                    }
                } else if (over == 2) {
                    P = 0;
                } else if (regrown < REGROW && nleaf - lf0 > 1 && nleaf - lf0 <= PM) {
                    // more slopes than hoped: the leaves are cut and tested once more
                    const int left = nleaf - lf0;
                    for (int j = threadIdx.x; j < left; j += T) {
                        DNode nd = S.leaf[lf0 + j];
                        nd.force = 1;
                        S.work[cur][j] = nd;
                    }
                    ++regrown;
                    P = -left;
                    lf0 = nleaf = 0;
                    flush = false;
                } else if (lfn > 1) {
                    // fewer of them: as many as would have fitted
                    lfn = lcap = max(1, min(lfn / 2, (int)(0.6f * (float)lfn * (float)sh.HC / (float)max(nn, 1))));
                    P = 0;
                } else {
                    // one leaf with too many slopes: more intervals of it, the other leaves wait on the stack
                    const int rest = nleaf - lf0 - 1;
                    if (top + rest > stack_cap(sh)) err = 1;
                    if (rank == 0 && !err)
                        for (int j = threadIdx.x; j < rest; j += T) m.stack[top + rest - 1 - j] = S.leaf[lf0 + 1 + j];
                    if (threadIdx.x == 0) {
                        DNode nd = S.leaf[lf0];
                        nd.force = 3;
                        S.work[cur][0] = nd;
                    }
                    top += rest;
                    lf0 = nleaf = 0;
                    flush = false;
                    P = -1;   // minus the intervals for the tree
                }
                if (threadIdx.x == 0) {
                    S.gain = gain;
                    S.lcap = lcap;
                    S.regrown = regrown;
                    S.cuts = cuts_made;
                    S.marked = marked;
                }
                team_sync();
                if (over && P == 0) {
                    if (phase > phases()) err = 1;
                    mode = err ? M_DONE : M_PAIRS;
                    continue;
                }
                if (P < 0) {
                    P = -P;
                    mode = err ? M_DONE : M_TREE;
                    continue;
                }
            } else {
                // ------------------------------------------------ exact scores
                if constexpr (F) {
                    scored += nx;
                    if (scored > F_SCORES) err = 1;
                    for (int k = rank; k < nx && !err; k += C) {
                        CandD c;
                        c.s = of_order(__ldcg(&m.ev[S.xl[k]]));
                        c.pair = 0;   // found for the best slope alone
                        c.valid = 1;
                        score_f32<T>(fs, n, h, c.s, wk, wk_bytes, gsort, S.red, c.w, c.t);
                        if (threadIdx.x == 0) reinterpret_cast<CandD *>(m.xres)[k] = c;
                    }
                    team_sync();
                    for (int k = 0; k < nx && !err; ++k) {
                        const CandD *q = reinterpret_cast<const CandD *>(m.xres) + k;
                        CandD c;
                        c.w = __ldcg(&q->w);
                        c.s = __ldcg(&q->s);
                        c.t = __ldcg(&q->t);
                        c.pair = 0;
                        c.valid = 1;
                        if (candd_better(c, bestd)) bestd = c;
                    }
                    // the true width, rounded up, bounds the rest; nothing right of a width of 0 is better
                    if (bestd.valid) {
                        const double u = bestd.w * fs.sy * (double)(1LL << F_YS);
                        ux = u < 4e18 ? (long long)u + 2 : D_MAX;
                        uxl = bestd.w == 0.0 ? -1 : ux;
                        bkey = order_of(bestd.s);
                    }
                } else {
                const int r0 = (int)((long long)nx * rank / C), r1 = (int)((long long)nx * (rank + 1) / C);
                if (nx >= RUN_MIN * (int)C)
                    score_run<T>(pts, n, h, m.ev, m.evd, S.xl + r0, r1 - r0, bx, wk, wk_bytes, gsort, S.red,
                                 m.xres + r0);
                else
                for (int k = rank; k < nx; k += C) {
                    const int dx = (int)__ldcg(&m.evd[S.xl[k]]), dy = dy_of(__ldcg(&m.ev[S.xl[k]]), dx);
                    Cand c;
                    const long long U = min(gw.first(__ldcg(&st->ub)), ux);
                    if (!score_bins<T, NBW>(gw, pts, n, h, dy, dx, U, S.t0, S.t1, bx, histw, c)) {
                        __syncthreads();
                        c = score<T>(pts, n, h, dy, dx, bx, wk, wk_bytes, gsort, S.red);
                    }
                    if (threadIdx.x == 0) m.xres[k] = c;
                }
                team_sync();
                // the best of them that is a pair's slope (fractions need not be)
                const int slots = table_slots(), rounds = table_rounds(slots);
                for (int tries = 0; tries < nx; ++tries) {
                    Cand c = cand_empty();
                    for (int k = threadIdx.x; k < nx; k += T) {
                        Cand o = ld_cand(&m.xres[k]);
                        o.i = k;
                        if (S.xl[k] >= 0 && cand_better(o, c)) c = o;
                    }
                    c = cta_best<T>(c, reinterpret_cast<Cand *>(S.red));
                    const int at = c.i;
                    c.i = c.j = 0x7fffffff;   // (an equal slope is not better)
                    if (!cand_better(c, best)) break;
                    line_pair<T>(pts, n, c.dy, c.dx, reinterpret_cast<unsigned *>(wk), slots, rounds, (int)rank, (int)C,
                                 &st->pair[ppar], &st->bad);
                    team_sync();
                    const unsigned pr = __ldcg(&st->pair[ppar]);
                    if (rank == 0 && threadIdx.x == 0) st->pair[ppar ^ 1] = 0xffffffffu;
                    ppar ^= 1;
                    if (threadIdx.x == 0) S.xl[at] = -1;
                    team_sync();
                    if (pr != 0xffffffffu) {
                        c.i = (int)(pr >> 16);
                        c.j = (int)(pr & 0xffffu);
                        best = c;
                        break;
                    }
                }
                if (best.dx > 0) {
                    // W = w / dx in units of 2^-32
                    const long long q = best.w / best.dx, r = (best.w % best.dx) << 32;
                    ux = (q << 32) + r / best.dx;
                    uxl = (r % best.dx) ? ux : ux - 1;
                    bkey = slope_key(best.dy, best.dx);
                }
                }
                nx = 0;
                P = 0;
                __syncthreads();
            }
            // ---------------------------------------------------- the next phase
            const bool was_tree = mode == M_TREE;
            if (!F && nx > 0) scored += nx;
            if (err || phase > phases() || (brief() && scored > SMALL_SCORES)) {
                err = 1;
                mode = M_DONE;
            } else if (nx > 0) {
                mode = M_EXACT;
            } else if (!was_tree && (P > 0 || etop > 0)) {
                mode = M_EVENT;
                if (P == 0) {
                    P = min(etop, PM);
                    for (int j = threadIdx.x; j < P; j += T) S.work[cur][j] = ld_node(&m.estack[etop - 1 - j]);
                    etop -= P;
                    __syncthreads();
                }
            } else if (nleaf > 0 && (flush || nleaf >= LRUN || (was_tree ? P : 0) + top == 0)) {
                mode = M_PAIRS;
                if (was_tree && P > 0) {
                    if (top + P > stack_cap(sh)) err = 1;
                    if (rank == 0 && !err)
                        for (int j = threadIdx.x; j < P; j += T) m.stack[top + P - 1 - j] = S.work[cur][j];
                    top += P;
                    P = 0;
                }
                // as many of the leaves as the list is expected to hold
                float held;
                lfn = leaves_within<T, F>(S.leaf + lf0, min(nleaf - lf0, S.lcap), LIST_HOPE * (float)sh.HC, S.gain,
                                          xr, yr, held);
                flush = true;
            } else if (was_tree && P > 0) {
                mode = M_TREE;
            } else if (top > 0) {
                mode = M_TREE;
                P = min(top, PM);
                for (int j = threadIdx.x; j < P; j += T) S.work[cur][j] = ld_node(&m.stack[top - 1 - j]);
                top -= P;
                __syncthreads();
            } else {
                mode = M_DONE;
            }
        }
        if constexpr (F) {
            // the smallest index pair with the best slope
            if (bestd.valid && !err) {
                int NC = T;
                while (NC < n && NC < CELLS_MAX) NC <<= 1;
                const long long K = grid_key(bestd.s), want = order_of(bestd.s);
                list_pairs_f32<T>(pts, n, K - 1, K + 2, bx, fs, NC, wk, S.warp_a, m, &st->nlist[lpar], &st->over[lpar],
                                  sh.HC, (int)rank, (int)C, &want, &st->pair[0]);
                team_sync();
                bestd.pair = __ldcg(&st->pair[0]);
                if (bestd.pair == 0xffffffffu) err = 1;
            }
            // slopes beyond the tree's range must be out of reach
            const long long U = min(__ldcg(&st->ub), ux);
            const bool tails = steep_above_at(F_KMAX, bx.dh, yr, U < D_MAX / 2 ? U + grid_err(F_KMAX) : D_MAX);
            if (rank == 0 && threadIdx.x == 0 && !err && tails && bestd.valid) {
                lms_result r;
                r.w_num = r.w_den = r.s_num = r.s_den = r.t_num = r.t_den = 0;
                r.theta1 = bestd.s;
                r.theta2 = bestd.t;
                const double half = 0.5 * bestd.w;
                r.med_sq = half * half;
                r.i = (int)(bestd.pair >> 16);
                r.j = (int)(bestd.pair & 0xffffu);
                r.status = LMS_OK;
                r.algorithm = algo;
                *A.out = r;
                *A.done = 1;
            }
        } else {
            if (rank == 0 && threadIdx.x == 0) {
                const int bad = err | __ldcg(&st->bad);
                if (brief()) A.set_done[set] = !bad;
                if (!(brief() && bad)) write_result(A.out + set, best, algo, bad);
            }
        }
        team_sync();
    }
}

// ------------------------------------------------------------------ host
// The kernel's shapes: for one fit in a cluster by its size, and for batches.
template <int T_, int G_, int NB_, int NBW_, int PM_, int LRUN_, bool SP_, bool F_ = false>
struct Shape {
    static constexpr int T = T_, PM = PM_, LC = LRUN_ + PM_, NS = T_ < 512 ? 512 : T_, PT = F_ ? 8 : 4;
    // (a function: only the file that launches a shape compiles its kernel)
    static auto kernel() { return k_direct<T_, G_, NB_, NBW_, PM_, LRUN_, SP_, F_>; }
    // shared memory of a CTA whose largest set has n points
    static size_t smem(int n, int HC)
    {
        size_t P = T, NC = T, P2 = T;
        while (P < (size_t)n) P <<= 1;
        while (NC < (size_t)n && NC < CELLS_MAX) NC <<= 1;
        while (P2 < (size_t)HC) P2 <<= 1;
        size_t wk = std::max<size_t>((size_t)(T / G_) * NB_ * 4, (size_t)NBW_ * 4);
        wk = std::max<size_t>(wk, 16 * (size_t)NS);
        wk = std::max(wk, pairs_bytes((int)NC, n));
        wk = std::max(wk, 16 * P2);
        wk = std::max(wk, std::min<size_t>(8 * P, 64 * (size_t)T));   // 32-bit exact sort, or its chunks
        return sizeof(DShared<NS, PM, LC>) + (SP_ ? ((PT * (size_t)n + 15) & ~(size_t)15) : 0) + wk;
    }
    static TeamShape team(int nmax, int C, int HC, float leaf)
    {
        TeamShape t{};
        size_t P = T;
        while (P < (size_t)nmax) P <<= 1;
        t.PM = PM;
        t.LC = LC;
        t.HC = HC;
        t.Q = std::min(PM, 128) - 1;
        t.leaf = leaf;
        t.ptsn = SP_ ? 0 : (long long)nmax * (PT / 4);
        t.dupw = F_ ? 0 : (nmax + 31) / 32;
        t.sortw = 16LL * std::max<long long>(P, HC);
        t.C = C;
        return t;
    }
};
using Small = Shape<512, 32, 1024, 4096, 256, 64, true>;
using Mid = Shape<1024, 128, 2048, 4096, 256, 64, true>;
using Large = Shape<1024, 256, 4096, 8192, 128, 64, false>;
using FloatSmall = Shape<512, 32, 1024, 4096, 256, 64, true, true>;
using FloatMid = Shape<1024, 128, 2048, 4096, 256, 64, true, true>;
using Batch = Shape<256, 32, 1024, 1024, 64, 32, true>;

// The launches, each shape's in a file of its own (the kernels compile side
// by side): for one fit in a cluster, an error (not launched) also where the
// device cannot hold the cluster; for a batch's teams.
template <class SH>
cudaError_t launch_cluster(const DirectArgs &a, size_t smem, cudaStream_t st);
bool cluster_fits(const void *kernel, const cudaLaunchConfig_t &cfg);
int batch_teams_per_sm(size_t smem);   // 0 on failure
cudaError_t launch_batch(const DirectArgs &a, int nteams, size_t smem, cudaStream_t st);

}  // namespace direct
}  // namespace lms
