// collide_common.cuh -- device functions shared by the collision kernels: the exact overlap tests (narrow
// phase), candidate selection within a warp, the pair of a collision tile, asynchronous copies.
#pragma once
#include <cstdint>

#include "mhc_internal.cuh"

namespace mhc {
namespace {

constexpr float kEps = 1e-5f;
constexpr float kEps0 = 1e-4f;
constexpr float kFar = 1.0e6f;   // padding poses far outside any scene

__device__ __forceinline__ bool rect_rect(float dx, float dy, float ca, float sa, float la, float wa,
                                          float cb, float sb, float lb, float wb) {
    const float c = fabsf(fmaf(ca, cb, sa * sb));
    const float s = fabsf(fmaf(sa, cb, -ca * sb));
    const float pau = fabsf(fmaf(dx, ca, dy * sa));
    const float pav = fabsf(fmaf(dy, ca, -dx * sa));
    const float pbu = fabsf(fmaf(dx, cb, dy * sb));
    const float pbv = fabsf(fmaf(dy, cb, -dx * sb));
    return pau <= la + fmaf(lb, c, wb * s) && pav <= wa + fmaf(lb, s, wb * c) &&
           pbu <= lb + fmaf(la, c, wa * s) && pbv <= wb + fmaf(la, s, wa * c);
}

// rectangle at the origin of d (axis (c, s), half extents l, w) against a disc of radius r at offset d
__device__ __forceinline__ bool rect_disc(float dx, float dy, float c, float s, float l, float w, float r) {
    const float ex = fmaxf(fabsf(fmaf(dx, c, dy * s)) - l, 0.0f);
    const float ey = fmaxf(fabsf(fmaf(dy, c, -dx * s)) - w, 0.0f);
    return fmaf(ex, ex, ey * ey) <= r * r;
}

// Convex outlines (Section IV-C.1 lets an outline be as detailed as needed); in a pair with an outline a
// plain rectangle comes as a 4-gon.  Two convex polygons are disjoint iff the supporting line of some edge
// of one has the whole other polygon strictly on its outer side (the edges of their Minkowski difference
// are the edges of the two), so each edge is one test: edge e of A (body-frame vertex v_e, outward unit
// normal n_e, support h_e = n_e . v_e) separates iff min over B's vertices w of
// (R_a n_e) . (d + R_b w) > h_e, d = p_b - p_a.  The normal is turned into B's frame once per edge and B's
// vertices are read as stored.  Only the kernels instantiated for batches with outlines contain it.
// Does edge v of A separate the two: d = p_b - p_a, (cr, sr) the cosine and sine of psi_a - psi_b.  An edge of B: the
// roles exchanged, d and sr negated.
__device__ __forceinline__ bool edge_separates(const float4 v, float dx, float dy, float ca, float sa, float cr, float sr,
                                              const PolyVertex *B, int nb) {
    const float h = fmaf(v.z, v.x, v.w * v.y);
    const float nwx = fmaf(ca, v.z, -sa * v.w), nwy = fmaf(sa, v.z, ca * v.w);
    const float o = fmaf(nwx, dx, nwy * dy);
    const float mx = fmaf(cr, v.z, -sr * v.w), my = fmaf(sr, v.z, cr * v.w);
    float lo = INFINITY;
#pragma unroll 4
    for (int q = 0; q < nb; ++q) {
        const float4 w = B[q];
        lo = fminf(lo, fmaf(mx, w.x, my * w.y));
    }
    return o + lo > h;
}

__device__ __forceinline__ bool outline_outline(float dx, float dy, float ca, float sa, float cb, float sb,
                                               const PolyVertex *A, int na, const PolyVertex *B, int nb) {
    const float cr = fmaf(ca, cb, sa * sb), sr = fmaf(sa, cb, -ca * sb);   // R_b^T R_a = R(psi_a - psi_b)
    for (int e = 0; e < na; ++e)
        if (edge_separates(A[e], dx, dy, ca, sa, cr, sr, B, nb)) return false;
    for (int e = 0; e < nb; ++e)
        if (edge_separates(B[e], -dx, -dy, cb, sb, cr, -sr, A, na)) return false;
    return true;
}

// The edge of A that faces the point (qx, qy) of A's frame most: the one whose line it is furthest outside of.
__device__ __forceinline__ int facing_edge(const PolyVertex *A, int n, float qx, float qy) {
    float best = -INFINITY;
    int at = 0;
#pragma unroll 4
    for (int e = 0; e < n; ++e) {
        const float4 v = A[e];
        const float s = fmaf(v.z, qx - v.x, v.w * (qy - v.y));
        if (s > best) { best = s; at = e; }
    }
    return at;
}

// Sixteen sectors of directions around a rectangle of half extents l, w: signs, the longer side, near the diagonal or not.
__device__ __forceinline__ int sector_of(float qx, float qy, float l, float w) {
    const float x = qx * w, y = qy * l, ax = fabsf(x), ay = fabsf(y);
    return (x < 0.0f ? 1 : 0) | (y < 0.0f ? 2 : 0) | (ax > ay ? 4 : 0) | (2.4f * fminf(ax, ay) > fmaxf(ax, ay) ? 8 : 0);
}

// A point of the sector.
__device__ __forceinline__ float2 point_of(int sector, float l, float w) {
    const float shorter = sector & 8 ? 1.1f : 0.4f, x = sector & 4 ? 1.6f : shorter, y = sector & 4 ? shorter : 1.6f;
    return make_float2((sector & 1 ? -x : x) * l, (sector & 2 ? -y : y) * w);
}

// Does the edge of A that faces B most, or B's that faces A, separate the two?  Nine in ten pairs that are apart pass
// here, for two edges instead of all of them.  faces: the facing edges by sector, A's and B's (or null: searched).
__device__ __forceinline__ bool outlines_apart(float dx, float dy, float ca, float sa, float cb, float sb, float la, float wa,
                                              float lb, float wb, const PolyVertex *A, int na, const PolyVertex *B, int nb,
                                              const unsigned char *faces) {
    const float cr = fmaf(ca, cb, sa * sb), sr = fmaf(sa, cb, -ca * sb);
    const float ax = fmaf(dx, ca, dy * sa), ay = fmaf(dy, ca, -dx * sa);
    const float bx = -fmaf(dx, cb, dy * sb), by = -fmaf(dy, cb, -dx * sb);
    const int ea = faces ? faces[sector_of(ax, ay, la, wa)] : facing_edge(A, na, ax, ay);
    if (edge_separates(A[ea], dx, dy, ca, sa, cr, sr, B, nb)) return true;
    const int eb = faces ? faces[16 + sector_of(bx, by, lb, wb)] : facing_edge(B, nb, bx, by);
    return edge_separates(B[eb], -dx, -dy, cb, sb, cr, -sr, A, na);
}

// Squared distance of the point (qx, qy) from the edge v w.
__device__ __forceinline__ float edge_distance2(const float4 v, const float4 w, float qx, float qy) {
    const float ex = w.x - v.x, ey = w.y - v.y, px = qx - v.x, py = qy - v.y;
    const float t = fminf(fmaxf(fmaf(px, ex, py * ey) / fmaf(ex, ex, ey * ey), 0.0f), 1.0f);
    const float rx = fmaf(-t, ex, px), ry = fmaf(-t, ey, py);
    return fmaf(rx, rx, ry * ry);
}

// How far the point (qx, qy) of A's frame lies outside the edge's line that it is furthest outside of.
__device__ __forceinline__ float outside_by(const PolyVertex *A, int n, float qx, float qy) {
    float smax = -INFINITY;
#pragma unroll 4
    for (int e = 0; e < n; ++e) {
        const float4 v = A[e];
        smax = fmaxf(smax, fmaf(v.z, qx - v.x, v.w * (qy - v.y)));
    }
    return smax;
}

// Outline A at the origin of d (axis (c, s)) against a disc of radius r at offset d: the disc's centre in
// A's frame lies inside A, or within r of one of its edges (segment distance).
__device__ __forceinline__ bool outline_disc(float dx, float dy, float c, float s, const PolyVertex *A, int n,
                                            float r) {
    const float qx = fmaf(dx, c, dy * s), qy = fmaf(dy, c, -dx * s);
    const float smax = outside_by(A, n, qx, qy);
    if (smax > r) return false;   // beyond some edge's line by more than r
    if (smax <= 0.0f) return true; // centre inside
    float d2 = INFINITY;
    for (int e = 0; e < n; ++e) d2 = fminf(d2, edge_distance2(A[e], A[e + 1 == n ? 0 : e + 1], qx, qy));
    return d2 <= r * r;
}

// The exact test of one broad-phase candidate: d = p_b - p_a, (ca, sa) / (cb, sb) the body axes, la / wa
// and lb / wb the half extents of rectangles, ra / rb the radii of discs.  OUTL: the batch has outlines
// (combos 4..6); the kernels without them keep the short rectangle and disc tests alone.
// The shape combination of a pair and its outlines, copied out of the descriptor once per block: a field read
// through the descriptor in a loop with atomics would be read again after every atomic.
struct PairShape {
    int combo, poly_a, nv_a, poly_b, nv_b;
};

__device__ __forceinline__ PairShape shape_of(const PairDesc &P) { return {P.combo, P.poly_a, P.nv_a, P.poly_b, P.nv_b}; }

template <bool OUTL>
__device__ __forceinline__ bool narrow_hit(const PairShape P, const PolyVertex *polys, float dx, float dy,
                                           float2 qa, float2 qb, float la, float wa, float lb, float wb,
                                           float ra, float rb) {
    if (!OUTL) {
        switch (P.combo) {
            case 0: return rect_rect(dx, dy, qa.x, qa.y, la, wa, qb.x, qb.y, lb, wb);
            case 1: return rect_disc(dx, dy, qa.x, qa.y, la, wa, rb);
            case 2: return rect_disc(-dx, -dy, qb.x, qb.y, lb, wb, ra);
            default: return fmaf(dx, dx, dy * dy) <= (ra + rb) * (ra + rb);
        }
    }
    switch (P.combo) {
        case 0: return rect_rect(dx, dy, qa.x, qa.y, la, wa, qb.x, qb.y, lb, wb);
        case 1: return rect_disc(dx, dy, qa.x, qa.y, la, wa, rb);
        case 2: return rect_disc(-dx, -dy, qb.x, qb.y, lb, wb, ra);
        case 3: return fmaf(dx, dx, dy * dy) <= (ra + rb) * (ra + rb);
        case 4: return outline_outline(dx, dy, qa.x, qa.y, qb.x, qb.y, polys + P.poly_a, P.nv_a, polys + P.poly_b, P.nv_b);
        case 5: return outline_disc(dx, dy, qa.x, qa.y, polys + P.poly_a, P.nv_a, rb);
        default: return outline_disc(-dx, -dy, qb.x, qb.y, polys + P.poly_b, P.nv_b, ra);
    }
}

// A pair with an outline at a first look; undecided: narrow_hit says.  kApart comes from a part of the exact test itself.
// kOverlap: the centre of a disc inside the outline (the exact test's next line), or, of two outlines, the overlap of
// rectangles (half extents la, wa and lb, wb) that lie a millimetre inside them, far beyond the rounding of either test.
enum Verdict { kUndecided, kApart, kOverlap };

__device__ __forceinline__ Verdict outline_verdict(const PairShape P, const PolyVertex *polys, float dx, float dy,
                                                  float2 qa, float2 qb, float la, float wa, float lb, float wb, float ra,
                                                  float rb, const unsigned char *faces) {
    if (P.combo == 4) {
        if (rect_rect(dx, dy, qa.x, qa.y, la, wa, qb.x, qb.y, lb, wb)) return kOverlap;
        return outlines_apart(dx, dy, qa.x, qa.y, qb.x, qb.y, la, wa, lb, wb, polys + P.poly_a, P.nv_a, polys + P.poly_b, P.nv_b,
                              faces) ? kApart : kUndecided;
    }
    const float out = P.combo == 5 ? outside_by(polys + P.poly_a, P.nv_a, fmaf(dx, qa.x, dy * qa.y), fmaf(dy, qa.x, -dx * qa.y))
                                   : outside_by(polys + P.poly_b, P.nv_b, fmaf(-dx, qb.x, -dy * qb.y), fmaf(-dy, qb.x, dx * qb.y));
    return out > (P.combo == 5 ? rb : ra) ? kApart : (out <= 0.0f ? kOverlap : kUndecided);
}

// What edge g says of a pair that outline_verdict left undecided: of two outlines (A's edges, then B's) that it separates
// them, of an outline and a disc that the disc reaches it.
__device__ __forceinline__ bool outline_edge(const PairShape P, const PolyVertex *polys, float dx, float dy, float2 qa,
                                             float2 qb, float ra, float rb, int g) {
    const PolyVertex *A = polys + P.poly_a, *B = polys + P.poly_b;
    if (P.combo == 4) {
        const bool of_b = g >= P.nv_a;
        const float cr = fmaf(qa.x, qb.x, qa.y * qb.y), sr = fmaf(qa.y, qb.x, -qa.x * qb.y);
        return edge_separates(of_b ? B[g - P.nv_a] : A[g], of_b ? -dx : dx, of_b ? -dy : dy, of_b ? qb.x : qa.x,
                              of_b ? qb.y : qa.y, cr, of_b ? -sr : sr, of_b ? A : B, of_b ? P.nv_a : P.nv_b);
    }
    const bool of_a = P.combo == 5;
    const PolyVertex *V = of_a ? A : B;
    const int n = of_a ? P.nv_a : P.nv_b;
    const float c = of_a ? qa.x : qb.x, s = of_a ? qa.y : qb.y, x = of_a ? dx : -dx, y = of_a ? dy : -dy, r = of_a ? rb : ra;
    return edge_distance2(V[g], V[g + 1 == n ? 0 : g + 1], fmaf(x, c, y * s), fmaf(y, c, -x * s)) <= r * r;
}

// Narrow-phase work counters by shape class (CollideArgs::counters [2 + class]): 0 rectangle-rectangle,
// 1 rectangle-disc, 2 disc-disc, 3 outline-outline, 4 outline-disc (the PairDesc combos 0, 1|2, 3, 4, 5|6).
__device__ __forceinline__ int narrow_class(int combo) {
    return combo == 0 ? 0 : (combo <= 2 ? 1 : (combo <= 4 ? combo - 1 : 4));
}

__device__ __forceinline__ void count_narrow(const CollideArgs &a, int combo, unsigned long long n) {
    atomicAdd(a.counters + 1, n);
    atomicAdd(a.counters + 2 + narrow_class(combo), n);
}

// Queue slots of one compaction round: each lane brings cnt (0..8) candidates; off = the candidates of the
// lanes below it, total = all of them (one ballot per bit of cnt instead of a shuffle scan: four
// independent instructions, not a chain of five).  Returns false when no lane has any (uniform).
__device__ __forceinline__ bool queue_offsets(int cnt, int lane, int &off, int &total) {
    const unsigned b0 = __ballot_sync(0xffffffffu, cnt & 1), b1 = __ballot_sync(0xffffffffu, cnt & 2);
    const unsigned b2 = __ballot_sync(0xffffffffu, cnt & 4), b3 = __ballot_sync(0xffffffffu, cnt & 8);
    if (!(b0 | b1 | b2 | b3)) return false;
    const unsigned lt = (1u << lane) - 1u;
    off = __popc(b0 & lt) + 2 * __popc(b1 & lt) + 4 * __popc(b2 & lt) + 8 * __popc(b3 & lt);
    total = __popc(b0) + 2 * __popc(b1) + 4 * __popc(b2) + 8 * __popc(b3);
    return true;
}

// Position of the r-th set bit (r counted from 0, below popc(m)) of m, by halving popcounts.
__device__ __forceinline__ int nth_set_bit(unsigned m, int r) {
    int pos = 0, c = __popc(m & 0xffffu);
    if (r >= c) { r -= c; m >>= 16; pos += 16; }
    c = __popc(m & 0xffu);
    if (r >= c) { r -= c; m >>= 8; pos += 8; }
    c = __popc(m & 0xfu);
    if (r >= c) { r -= c; m >>= 4; pos += 4; }
    c = __popc(m & 0x3u);
    if (r >= c) { r -= c; m >>= 2; pos += 2; }
    return pos + (r >= (int)(m & 1u) ? 1 : 0);
}

// Candidate selection without a queue: lane L holds a mask `cand` of its candidates; slot s of the warp's
// candidates in (lane, bit) order belongs to the last lane whose exclusive count is <= s (a 5-step
// shuffle search), and is that lane's (s - its count)-th bit.  Every lane takes one slot per round, so the
// exact tests run with all lanes busy.  Calls fn(owner lane, bit) for each slot (warp-uniform call).
template <typename Fn>
__device__ __forceinline__ void for_each_candidate(unsigned cand, int lane, Fn &&fn) {
    const unsigned cnt = __popc(cand);
    unsigned incl = cnt;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const unsigned v = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += v;
    }
    const unsigned excl = incl - cnt;
    const unsigned total = __shfl_sync(0xffffffffu, incl, 31);
    for (unsigned s0 = 0; s0 < total; s0 += 32) {
        const unsigned s = s0 + lane;
        int owner = 0;
#pragma unroll
        for (int step = 16; step > 0; step >>= 1) {
            const unsigned e = __shfl_sync(0xffffffffu, excl, owner + step);
            if (e <= s) owner += step;
        }
        const unsigned m = __shfl_sync(0xffffffffu, cand, owner);
        const unsigned e = __shfl_sync(0xffffffffu, excl, owner);
        if (s < total) fn(owner, nth_set_bit(m, (int)(s - e)));
    }
}

// The last i in [0, n) with le(i), which holds for 0 and up to some entry of an ascending array.  A 64-way search by the
// whole warp (every lane must call it for the same array and value): each round the lanes probe 64 evenly spaced entries
// at once (two each) and keep the span between the last probe that holds and the next, so up to 64 entries take one
// round of loads and 4,096 two (a binary search is a chain of log2 n dependent loads).
template <typename Le>
__device__ __forceinline__ int last_where(int n, Le &&le) {
    const int lane = threadIdx.x & 31;
    int lo = 0, hi = n - 1;
    while (lo < hi) {
        const long long span = hi - lo + 1;
        const bool le0 = le(lo + (int)(span * (2 * lane) / 64));
        const bool le1 = le(lo + (int)(span * (2 * lane + 1) / 64));
        // probe q = 2 lane + (0 | 1); probe 0 always holds
        const unsigned even = __ballot_sync(0xffffffffu, le0), odd = __ballot_sync(0xffffffffu, le1);
        const int last0 = 31 - __clz(even), last1 = odd ? 31 - __clz(odd) : -1;   // last true even / odd probe
        const int L = 2 * last1 + 1 > 2 * last0 ? 2 * last1 + 1 : 2 * last0;      // the true probes form a prefix
        const int nlo = lo + (int)(span * L / 64);
        hi = L == 63 ? hi : lo + (int)(span * (L + 1) / 64) - 1;
        lo = nlo;
    }
    return lo;
}

// The pair of tile g: the last pair (in the order of a.pairs) whose first tile is <= g (every lane with the same g).
template <typename Args>
__device__ __forceinline__ int pair_of_tile(const Args &a, long long g) {
    return last_where(a.n_pairs, [&](int p) { return a.pairs[p].tile_start <= g; });
}

// Asynchronous 4- and 8-byte copies global -> shared (both addresses aligned to the size); cp_async_wait()
// returns once the calling thread's copies have landed (a barrier then shows them to the CTA).
__device__ __forceinline__ void cp_async4(void *dst, const void *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void cp_async8(void *dst, const void *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

}  // namespace
}  // namespace mhc
