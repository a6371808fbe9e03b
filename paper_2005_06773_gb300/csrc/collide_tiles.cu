// collide_tiles.cu -- collision layouts 4 and 7: a warp (4) or a CTA (7) per active 32 x 32 block of hypothesis pairs,
// in the objects' tile order.
//
// The bounds kernel has written each object's poses tile by tile (CollideArgs::tile_poses: 32 poses of one step side
// by side, in the compact order of hypothesis_at) together with the boxes around them, so that a block's active
// steps are few and a step's poses are one 16-byte load per lane and side.  Without that array (culling off, or an
// arena sized to the least) layout 4's kernel takes ascending tiles and reads the pose planes (large scenes without
// outlines: the kernel of whole tiles in collide.cu).
//
// A step of a block, by one warp: the 32 + 32 poses go to a shared slot, the broad phase runs on a 4 x 8 micro-block
// per lane (rows lr + 8 m, columns lc + 4 n), and the candidates are queued and tested one per lane.  Compact tiles
// put 30 to 70 candidates into an active step, on few lanes (the lane with the most has four to eight): a loop over
// each lane's own candidates would run the exact test with a quarter of the lanes busy, and one over the rows that
// have any (a lane per column) with a fifth (3.7 ms against 2.7 ms on 32 cars).
#include <algorithm>
#include <cstdint>

#include "collide_common.cuh"
#include "hit_terms.cuh"

namespace mhc {
namespace {

constexpr int MI = 4, MJ = 8;          // micro-block of a lane

// One step's poses in shared memory.
struct StepSlot {
    float4 pa[32], pb[32];             // x, y, h of the broad phase
    float4 qa[32], qb[32];             // x, y, c, s
};

// This lane's row of a and column of b at one step.
struct StepPoses {
    float4 a, b;
};

// One side's pose `idx` of the tile-ordered array, or of the planes; past the object's end: far from everything.
template <bool TILED>
__device__ __forceinline__ float4 load_pose(const CollideArgs &a, long long idx, bool ok, float far) {
    if (TILED) return __ldg(a.tile_poses + idx);     // x = NaN past the end: no test passes
    return ok ? make_float4(__ldg(a.x + idx), __ldg(a.y + idx), __ldg(a.c + idx), __ldg(a.s + idx))
              : make_float4(far, 0.0f, 1.0f, 0.0f);
}

// The shapes of a pair: the half extents of rectangles, the radii of discs.
struct Extents {
    float la, wa, ra, lb, wb, rb;
};

// Stages a step's poses in a slot and returns the lane's broad-phase candidates (bit MJ m + n).
__device__ __forceinline__ unsigned stage_and_sweep(StepSlot &S, const StepPoses &p, float rc2, int lane) {
    const int lr = lane >> 2, lc = lane & 3;
    const float ka = 0.5f * (1.0f - kEps);
    S.pa[lane] = make_float4(p.a.x, p.a.y, ka * fmaf(p.a.x, p.a.x, p.a.y * p.a.y), 0.0f);
    S.pb[lane] = make_float4(p.b.x, p.b.y, 0.5f * fmaf(1.0f - kEps, fmaf(p.b.x, p.b.x, p.b.y * p.b.y), -rc2), 0.0f);
    S.qa[lane] = p.a;
    S.qb[lane] = p.b;
    __syncwarp();
    float ax[MI], ay[MI], ah[MI];
#pragma unroll
    for (int m = 0; m < MI; ++m) {
        const float4 q = S.pa[lr + 8 * m];
        ax[m] = q.x; ay[m] = q.y; ah[m] = q.z;
    }
    unsigned cand = 0u;
#pragma unroll
    for (int n = 0; n < MJ; ++n) {
        const float4 q = S.pb[lc + 4 * n];
#pragma unroll
        for (int m = 0; m < MI; ++m)
            if (fmaf(ax[m], q.x, fmaf(ay[m], q.y, -q.z)) >= ah[m]) cand |= 1u << (MJ * m + n);
    }
    return cand;
}

// A queued candidate: lane << 5 | bit of its micro-block, and the row and column that means.
__device__ __forceinline__ int queued_row(int e) { return (e >> 7 & 7) + (e & 24); }
__device__ __forceinline__ int queued_col(int e) { return (e >> 5 & 3) + 4 * (e & 7); }

template <bool OUTL>
__device__ __forceinline__ bool overlap(const StepSlot &S, const PairShape &shape, const PolyVertex *polys,
                                        const Extents &x, int e) {
    const float4 qa = S.qa[queued_row(e)], qb = S.qb[queued_col(e)];
    return narrow_hit<OUTL>(shape, polys, qb.x - qa.x, qb.y - qa.y, make_float2(qa.z, qa.w), make_float2(qb.z, qb.w),
                            x.la, x.wa, x.lb, x.wb, x.ra, x.rb);
}

__device__ __forceinline__ Verdict first_look(const StepSlot &S, const PairShape &shape, const PolyVertex *polys,
                                              const Extents &x, int e, const unsigned char *faces) {
    const float4 qa = S.qa[queued_row(e)], qb = S.qb[queued_col(e)];
    return outline_verdict(shape, polys, qb.x - qa.x, qb.y - qa.y, make_float2(qa.z, qa.w), make_float2(qb.z, qb.w), x.la,
                           x.wa, x.lb, x.wb, x.ra, x.rb, faces);
}

__device__ __forceinline__ bool edge_decides(const StepSlot &S, const PairShape &shape, const PolyVertex *polys,
                                             const Extents &x, int e, int g, int edges) {
    const float4 qa = S.qa[queued_row(e)], qb = S.qb[queued_col(e)];
    return g < edges && outline_edge(shape, polys, qb.x - qa.x, qb.y - qa.y, make_float2(qa.z, qa.w),
                                     make_float2(qb.z, qb.w), x.ra, x.rb, g);
}

// A pair's outlines in shared memory, the vertices of two outlines padded to a multiple of four by copies of the first
// (another vertex, or edge, that is there already: no test changes).
constexpr int kOutlineSlots = 16;      // MHC_MAX_VERTICES
__device__ __forceinline__ void load_outline(PolyVertex *slot, const PolyVertex *polys, const PairDesc &P, int side, int lane) {
    const int first = side ? P.poly_b : P.poly_a, n = side ? P.nv_b : P.nv_a;
    if (lane < kOutlineSlots && n > 0) slot[lane] = polys[first + (lane < n ? lane : 0)];
}

__device__ __forceinline__ PairShape staged_shape(const PairDesc &P) {
    const int pad = P.combo == 4 ? 3 : 0;
    return {P.combo, 0, (P.nv_a + pad) & ~pad, kOutlineSlots, (P.nv_b + pad) & ~pad};
}

// The extents the tests of a pair use: of two outlines, the rectangles inside them.
__device__ __forceinline__ Extents extents_of(const CollideArgs &a, const PairDesc &P, bool outlines) {
    if (outlines && P.combo == 4) {
        const ObjDesc &A = a.objs[P.a], &B = a.objs[P.b];
        return {A.core_l, A.core_w, 0.0f, B.core_l, B.core_w, 0.0f};
    }
    return {P.hl_a, P.hw_a, P.rad_a, P.hl_b, P.hw_b, P.rad_b};
}

// The exact tests of outline pairs, by a warp: `rounds` of 32 candidates (take(round) gives the lane's, or -1).  A first
// look decides nine in ten; the others get the whole test one after another, a lane per edge (the edges of both: 16 lanes
// a candidate, 32 beyond 16 edges).  A lane per candidate would take the warp through every edge of both outlines, 860
// instructions, as soon as one candidate needs it.  Whole call, 11 objects with outlines: every candidate's whole test
// 133 us, the edges found by search first 120, outlines in shared memory 113, heavy blocks in halves 87, pairs found
// earlier in the batch dropped 80, overlaps and facing edges by rectangle and sector, a lane per edge 75.
template <typename Take, typename Look, typename Lanes, typename Hit>
__device__ __forceinline__ void test_outlines(int rounds, const PairShape &shape, Take &&take, Look &&look, Lanes &&lanes,
                                              Hit &&hit) {
    const int lane = threadIdx.x & 31;
    const int edges = shape.combo == 4 ? shape.nv_a + shape.nv_b : (shape.combo == 5 ? shape.nv_a : shape.nv_b);
    const int group = edges <= 16 ? 16 : 32, g = lane & (group - 1);
    const unsigned mine = group == 32 ? 0xffffffffu : 0xffffu << (lane & 16);
    for (int r = 0; r < rounds; ++r) {
        const int e = take(r);
        const Verdict v = e >= 0 ? look(e) : kApart;
        if (v == kOverlap) hit(e);
        const unsigned open = __ballot_sync(0xffffffffu, v == kUndecided);
        const int n = __popc(open);
        for (int c = lane / group; c - lane / group < n; c += 32 / group) {
            const int ec = __shfl_sync(0xffffffffu, e, nth_set_bit(open, min(c, n - 1)));
            const bool found = lanes(ec, g, edges);
            const bool any = __ballot_sync(0xffffffffu, found) & mine;
            if (g == 0 && c < n && any != (shape.combo == 4)) hit(ec);
        }
    }
}

__device__ __forceinline__ bool boxes_meet(const float4 &a, const float4 &b, float r) {
    return (a.x - r <= b.z) && (b.x - r <= a.z) && (a.y - r <= b.w) && (b.y - r <= a.w);
}

// ---- the list of active blocks ------------------------------------------------------------------------------
//
// The walk runs over the blocks that come close only (a fifth to a quarter of them), those with many active steps
// first: a warp that starts last then has little to do.  A warp lists `per_warp` consecutive 64 x 64
// tiles: lane 4 u + q keeps block q (rows 32 (q >> 1), columns 32 (q & 1)) of tile u.  Large scenes take 8 tiles per
// warp, one search for eight tiles and one pair of atomics per CTA; small ones 1, to use every SM.
constexpr int kListWarps = 8;
// Active steps from which a block is listed from the front.  Layout 4 runs for long enough that only its longest blocks
// need a head start (12 cars 0.70 -> 0.68 ms, 256 scenarios 6.39 -> 6.33 ms against 12 steps); of layout 7's, with outlines,
// the front is also what two CTAs share (from 12 steps 71 us, from 24 91 us).
constexpr int kHeavySteps = 12, kHeavyStepsWalk = 24;

__global__ void __launch_bounds__(32 * kListWarps) block_list_kernel(const CollideArgs a, int per_warp) {
    pdl_trigger();
    __shared__ int s_heavy[kListWarps], s_light[kListWarps];
    __shared__ unsigned long long s_at[2];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const long long g0 = ((long long)blockIdx.x * kListWarps + w) * per_warp;
    BlockRef ref{};
    int n = 0;                                      // active steps of this lane's block
    int pair = 0;
    if (g0 < a.n_tiles) pair = pair_of_tile(a, g0);   // uploaded data: before the wait
    pdl_wait();
    const int mine = lane >> 2, q = lane & 3;
    for (int u0 = 0; u0 < per_warp && g0 + u0 < a.n_tiles;) {
        while (pair + 1 < a.n_pairs && a.pairs[pair + 1].tile_start <= g0 + u0) ++pair;
        const PairDesc &P = a.pairs[pair];
        const int t = (int)(g0 + u0 - P.tile_start);   // < tiles_a x tiles_b <= n_tiles < 2^31
        const int ta = t / P.tiles_b, tb = t - ta * P.tiles_b, N = P.n_steps, hb = P.h_b;
        const int run = min(per_warp - u0, P.tiles_b - tb);   // tiles of the same rows: their boxes are loaded once
        const long long box_a = P.bounds_a + (long long)(2 * ta) * N, box_b = P.bounds_b + (long long)(2 * tb) * N;
        const bool two_a = ta * kTile + 32 < P.h_a;
        const float r = P.r_cull;
        if (mine - u0 >= 0 && mine - u0 < run) {
            ref.pair = pair;
            ref.tile_a = 2 * ta + (q >> 1);
            ref.tile_b = 2 * (tb + mine - u0) + (q & 1);
            ref.box_a = (int)(box_a + (q >> 1) * N);
            ref.box_b = (int)(box_b + (2 * (mine - u0) + (q & 1)) * N);
        }
        for (int k0 = 0; k0 < N; k0 += 32) {
            const int k = k0 + lane;
            const bool in = k < N;
            const float4 far = make_float4(INFINITY, INFINITY, -INFINITY, -INFINITY);   // meets no finite box
            const float4 a0 = in ? a.bounds[box_a + k] : far, a1 = in && two_a ? a.bounds[box_a + N + k] : far;
            for (int v = 0; v < run; ++v) {
                const long long bb = box_b + (long long)(2 * v) * N;
                const bool two_b = (tb + v) * kTile + 32 < hb;
                const float4 b0 = in ? a.bounds[bb + k] : far, b1 = in && two_b ? a.bounds[bb + N + k] : far;
                const unsigned m0 = __ballot_sync(0xffffffffu, boxes_meet(a0, b0, r));
                const unsigned m1 = __ballot_sync(0xffffffffu, boxes_meet(a0, b1, r));
                const unsigned m2 = __ballot_sync(0xffffffffu, boxes_meet(a1, b0, r));
                const unsigned m3 = __ballot_sync(0xffffffffu, boxes_meet(a1, b1, r));
                // (a tile past the object's end is never listed: `far` does meet the box of poses that have
                // overflowed to both infinities)
                if (mine == u0 + v && (two_a || q < 2) && (two_b || !(q & 1))) {
                    const unsigned m = q < 2 ? (q ? m1 : m0) : (q == 2 ? m2 : m3);
                    if (n == 0) { ref.k0 = k0; ref.mask = m; }
                    n += __popc(m);
                }
            }
        }
        u0 += run;
    }
    const unsigned active = __ballot_sync(0xffffffffu, n > 0), heavy = __ballot_sync(0xffffffffu, n >= (a.variant == 4 ? kHeavyStepsWalk : kHeavySteps));
    const unsigned light = active & ~heavy, lt = (1u << lane) - 1u;
    if (lane == 0) { s_heavy[w] = __popc(heavy); s_light[w] = __popc(light); }
    __syncthreads();
    int h0 = 0, l0 = 0, hn = 0, ln = 0;
#pragma unroll
    for (int v = 0; v < kListWarps; ++v) {
        if (v == w) { h0 = hn; l0 = ln; }
        hn += s_heavy[v];
        ln += s_light[v];
    }
    if (threadIdx.x == 0 && hn) s_at[0] = atomicAdd(a.list_counts, (unsigned long long)hn);
    if (threadIdx.x == 32 && ln) s_at[1] = atomicAdd(a.list_counts + 1, (unsigned long long)ln);
    __syncthreads();
    if (n == 0) return;
    // at most 4 blocks per tile: the front and the back never meet
    if (heavy >> lane & 1u) a.list[s_at[0] + h0 + __popc(heavy & lt)] = ref;
    else a.list[4 * a.n_tiles - 1 - (long long)(s_at[1] + l0 + __popc(light & lt))] = ref;
}

// Entry `it` of the list (heavy blocks first); `front`, `listed`: its heavy blocks and all.
__device__ __forceinline__ BlockRef listed_block(const CollideArgs &a, long long it, long long front) {
    return a.list[it < front ? it : 4 * a.n_tiles - 1 - (it - front)];
}

// ---- layout 4: a warp per block, its steps in ascending order -------------------------------------------------
//
// A block's steps come in order, so the first overlap of a pair is its first collision step: it is stored at once,
// and the pair's bit in `found` drops its later candidates.  The warps take the listed blocks one after another from
// a counter, until their CTA has walked kWalkSteps.
// Without the list (UNLISTED: culling off, or no room for the tile-ordered poses; kWholeTiles in collide.cu) they take
// every block of ascending tiles, strided, and read the pose planes.
//
// Bound by instruction issue while the list lasts (12 cars of 2,048 hypotheses, ncu: 74 % of the issue slots, 560 warp
// instructions per (block, step) item with its hits, set-up and listing order) and by the last blocks (SMs active 79 %
// of the launch); a shorter sweep alone did not shorten it.  Measured (collision stage, listing included): 32 cars 1.90
// ms, 256 uneven scenarios 6.00 ms; a warp per 64 x 64 tile of consecutive hypotheses took 4.77 and 11.8 ms (five and
// two times the executed tests), compact tiles without the list 2.67 and 8.9 ms (a third of the launch was its last
// warps), with it but with warps that stay until the list is empty 1.73 ms for the 32 cars (requests of higher priority
// then wait for the whole launch).
constexpr int kWalkWarps = 4;
constexpr int kWalkCtas = 7;            // per SM: bounds the registers to 72 (256 scenarios, collision stage: 6.00 ms; 5, 6, 8: 6.80, 6.33, 6.17)
constexpr int kWalkBlocks = 16;         // blocks per warp that the grid is sized for (its last CTAs take what is left)
// Steps after which a CTA makes room for a stream of higher priority (unless it is one of the last).  By steps and for the
// CTA as a whole: its warps end together.  A small request behind 32 cars in the serving loop is done 0.4 ms after its
// submission so, 0.9 to 1.2 ms with 16 blocks a warp or 1,024 steps; the whole call on 32 cars takes 2.66 ms, with 96
// steps 2.68, with 1,024 2.59; 256 scenarios (collision stage, at six CTAs per SM) 6.32, 6.40 and 6.18 ms, 6.33 with 16
// blocks a warp.
constexpr int kWalkSteps = 192;

struct WalkSlot {
    StepSlot step;
    unsigned short queue[8 * 32];      // the candidates of one round: at most 8 of each lane
    unsigned found[32];                // [lane] micro-block pairs that have hit
    int order[2][32];                  // hypotheses of the rows and columns
    float prob[2][32];                 // their probabilities (fused)
};

template <bool FUSED, bool OUTL, bool UNLISTED>
__device__ __forceinline__ int walk_block(const CollideArgs &a, const BlockRef &B, int lane, WalkSlot &S) {
    const PairDesc &P = a.pairs[B.pair];               // fields read where used (fewer live registers)
    const int ha = P.h_a, hb = P.h_b, N = P.n_steps;
    const int ia = 32 * B.tile_a + lane, jb = 32 * B.tile_b + lane;   // this lane's positions
    const long long box_a = UNLISTED ? P.bounds_a + (long long)B.tile_a * N : B.box_a;
    const long long box_b = UNLISTED ? P.bounds_b + (long long)B.tile_b * N : B.box_b;
    const float r_cull = P.r_cull;
    auto chunk = [&](int k0) -> unsigned {             // active steps among k0 .. k0 + 31
        const int k = k0 + lane;
        bool act = k < N;
        if (act && (!UNLISTED || a.cull)) act = boxes_meet(a.bounds[box_a + k], a.bounds[box_b + k], r_cull);
        return __ballot_sync(0xffffffffu, act);
    };
    int k0 = UNLISTED ? 0 : B.k0;
    unsigned mask = UNLISTED ? chunk(0) : B.mask;
    auto next = [&]() -> int {
        while (!mask) {
            k0 += 32;
            if (k0 >= N) return -1;
            mask = chunk(k0);
        }
        const int b = __ffs(mask) - 1;
        mask &= mask - 1u;
        return k0 + b;
    };
    int k = next();
    if (k < 0) return 0;
    StepPoses cur;
    auto load = [&](int kk) {
        if (UNLISTED) {
            cur.a = load_pose<false>(a, P.pose_a + (long long)kk * ha + ia, ia < ha, kFar);
            cur.b = load_pose<false>(a, P.pose_b + (long long)kk * hb + jb, jb < hb, -kFar);
        } else {
            cur.a = load_pose<true>(a, 32 * (box_a + kk) + lane, true, 0.0f);
            cur.b = load_pose<true>(a, 32 * (box_b + kk) + lane, true, 0.0f);
        }
    };
    load(k);
    {
        const int hi = UNLISTED ? ia : a.tile_order[32LL * (P.tile_a + B.tile_a) + lane];
        const int hj = UNLISTED ? jb : a.tile_order[32LL * (P.tile_b + B.tile_b) + lane];
        S.order[0][lane] = hi;
        S.order[1][lane] = hj;
        S.found[lane] = 0u;
        if (FUSED) {
            S.prob[0][lane] = ia < ha ? a.probf[P.traj_a + hi] : 0.0f;
            S.prob[1][lane] = jb < hb ? a.probf[P.traj_b + hj] : 0.0f;
        }
    }
    const PairShape shape = shape_of(P);
    const Extents ext = extents_of(a, P, OUTL);
    const float rc2 = P.rc2 + kEps0;
    const int ego_side = P.ego_side;
    unsigned narrow = 0;
    unsigned long long hit_cnt = 0, hit_mass = 0;
    int steps = 0;
    while (k >= 0) {
        __syncwarp();                   // the previous step's slot is no longer read
        unsigned cand = stage_and_sweep(S.step, cur, rc2, lane) & ~S.found[lane];
        const int kn = next();
        if (kn >= 0) load(kn);          // in flight while this step's candidates are tested
        ++steps;
        unsigned cnt = 0;
        unsigned long long mass = 0;
        for (;;) {                      // rounds of at most 8 candidates of each lane
            const int n = min(__popc(cand), 8);
            int off, total;
            if (!queue_offsets(n, lane, off, total)) break;
            for (int u = 0; u < n; ++u, cand &= cand - 1u) S.queue[off + u] = (unsigned short)(lane << 5 | (__ffs(cand) - 1));
            __syncwarp();
            narrow += total;
            auto hit_at = [&](int e) {
                atomicOr(&S.found[e >> 5], 1u << (e & 31));
                const int i = queued_row(e), j = queued_col(e), hi = S.order[0][i], hj = S.order[1][j];
                a.table[P.off + (long long)hi * hb + hj] = (int16_t)k;
                ++cnt;
                if (!FUSED) return;
                mass += to_fixed(S.prob[0][i] * S.prob[1][j], kFixProb);
                if (ego_side >= 0) {
                    const int eg = ego_side == 0 ? hi : hj;                              // the EGO hypothesis
                    const long long co = ego_side == 0 ? P.traj_b + hj : P.traj_a + hi;  // the CO hypothesis
                    atomicAdd(a.acc.mass + P.mass_base + (long long)eg * P.n_obj_s + P.co_local, a.pfix[co]);
                    atomicAdd(a.acc.hits + P.hits_base + eg, 1ull);
                    atomicAdd(a.acc.lsum + P.lsum_base + ((long long)eg * N + k) * P.n_obj_s + P.co_local, a.lfix[co]);
                }
            };
            if (OUTL && shape.combo >= 4) {
                test_outlines((total + 31) / 32, shape,
                    [&](int r) { return 32 * r + lane < total ? (int)S.queue[32 * r + lane] : -1; },
                    [&](int e) { return first_look(S.step, shape, a.polys, ext, e, nullptr); },
                    [&](int e, int g, int edges) { return edge_decides(S.step, shape, a.polys, ext, e, g, edges); }, hit_at);
            } else {
                for (int u = lane; u < total; u += 32) {
                    const int e = S.queue[u];
                    if (overlap<false>(S.step, shape, a.polys, ext, e)) hit_at(e);
                }
            }
            __syncwarp();
        }
        if (FUSED && __any_sync(0xffffffffu, cnt != 0u)) {   // the step's terms summed over the warp
            const unsigned c = __reduce_add_sync(0xffffffffu, cnt);
            mass = reduce_terms(mass);
            if (lane == 0) {
                atomicAdd(a.acc.count_k + P.kofs + k, (unsigned long long)c);
                atomicAdd(a.acc.H + P.kofs + k, mass);
            }
            hit_cnt += c;
            hit_mass += mass;
        }
        k = kn;
    }
    if (lane != 0) return steps;
    if (a.counters) {
        if (narrow) count_narrow(a, P.combo, narrow);
        atomicAdd(a.counters, (unsigned long long)steps * 32 * 32);
    }
    if (FUSED && hit_cnt) {
        atomicAdd(a.acc.count + P.index, hit_cnt);
        atomicAdd(a.acc.P + P.index, hit_mass);
    }
    return steps;
}

template <bool FUSED, bool OUTL, bool UNLISTED>
__global__ void __launch_bounds__(32 * kWalkWarps, kWalkCtas) walk_kernel(const CollideArgs a) {
    pdl_start();
    __shared__ WalkSlot slots[kWalkWarps];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    WalkSlot &S = slots[warp];
    if (UNLISTED) {                                 // every 32 x 32 block of every tile (four per tile)
        const long long stride = (long long)gridDim.x * kWalkWarps;
        for (long long gw = (long long)blockIdx.x * kWalkWarps + warp; gw < 4 * a.n_tiles; gw += stride) {
            BlockRef B;
            B.pair = pair_of_tile(a, gw >> 2);
            const PairDesc &P = a.pairs[B.pair];
            const int t = (int)((gw >> 2) - P.tile_start), ta = t / P.tiles_b, q = (int)(gw & 3);
            B.tile_a = 2 * ta + (q >> 1);
            B.tile_b = 2 * (t - ta * P.tiles_b) + (q & 1);
            if (32 * B.tile_a < P.h_a && 32 * B.tile_b < P.h_b) walk_block<FUSED, OUTL, true>(a, B, lane, S);
            __syncwarp();
        }
        return;
    }
    __shared__ int s_steps;                         // steps the CTA has walked
    if (threadIdx.x == 0) s_steps = 0;
    __syncthreads();
    const bool leaves = blockIdx.x + kWalkCtas * 152 < gridDim.x;   // not one of the last: others come after it
    const long long front = (long long)a.list_counts[0], listed = front + (long long)a.list_counts[1];
    unsigned long long taken = 0;
    if (lane == 0) taken = atomicAdd(a.list_counts + 2, 1ull);
    for (;;) {
        const long long it = (long long)__shfl_sync(0xffffffffu, taken, 0);
        if (it >= listed) return;
        int total = 0;
        if (lane == 0) {
            total = *(volatile int *)&s_steps;
            if (!leaves || total < kWalkSteps) taken = atomicAdd(a.list_counts + 2, 1ull);   // in flight meanwhile
        }
        const int steps = walk_block<FUSED, OUTL, false>(a, listed_block(a, it, front), lane, S);
        total = __shfl_sync(0xffffffffu, total, 0);
        if (leaves && total >= kWalkSteps) return;
        if (lane == 0) atomicAdd(&s_steps, steps);
        __syncwarp();
    }
}

// ---- layout 7: a CTA per active 32 x 32 block, its active steps spread over its warps ------------------------
//
// A scene of few tiles waits for its heaviest blocks, so a block gets a whole CTA.  It takes the block's active steps
// W at a time, one per warp: every warp stages its step's poses, sweeps the 32 x 32 pairs and puts its candidates
// into the CTA's queue; after a barrier all warps test the queue, 32 candidates a round.  A pair that overlapped in
// an earlier batch is dropped at the sweep (`found`: the batches ascend in time), two hits of one batch keep the
// earlier step (atomicMin).  At the end the CTA stores the first hits and adds their fused risk terms.
//
// Bound by latency: a batch of W steps is a chain of 2,300 cycles, the heaviest block has four, and a block's set-up
// and epilogue take as long as two more.  Measured (whole call replayed as one graph; before: a CTA of four warps per
// 32 consecutive hypotheses a side, listed or not, a queue per warp): EGO-only scene 154 -> 101 us, 11 objects with
// outlines 153 -> 133 (test_outlines: 75), with lane paths 150 -> 137, 11 objects 46.5 -> 46.8.  Four warps a CTA: 11 objects 53.6, outlines
// 178; sixteen: 51.3 and 135; four CTAs per SM: 49.5 and 158; the light blocks by a warp each: 50.7 and 140; in
// arbitrary order: 52.5 and 140.
constexpr int kBlockWarps = 8;
constexpr int kBlockCtas = 3;           // per SM: bounds the registers to 80
constexpr int kBlockSlots = 152 * kBlockCtas;   // CTAs on the chip at once

// With outlines a heavy block of a small scene is shared by two CTAs, 16 rows each: its exact tests, ten times as long,
// make the heaviest one three times the kernel's average load per CTA (11 objects: 114 us whole, 89 in halves, 92 in
// quarters; four such scenes at once, bound by the tests in all: 321, 349 and 394).
constexpr long long kHalvesBelow = 152 * 16;   // tiles

// queue_offsets for counts up to 32.
__device__ __forceinline__ bool queue_offsets6(int cnt, int lane, int &off, int &total) {
    if (!__any_sync(0xffffffffu, cnt > 15)) return queue_offsets(cnt, lane, off, total);
    const unsigned lt = (1u << lane) - 1u;
    off = total = 0;
#pragma unroll
    for (int b = 0; b < 6; ++b) {
        const unsigned m = __ballot_sync(0xffffffffu, cnt >> b & 1);
        off += __popc(m & lt) << b;
        total += __popc(m) << b;
    }
    return true;
}

constexpr int kFirstRow = 33;           // (odd: columns read without bank conflicts)

struct BlockSlot {
    StepSlot step[kBlockWarps];
    PolyVertex outline[2][kOutlineSlots];
    unsigned char faces[2][16];         // of two outlines: the edge that faces each sector
    unsigned short queue[kBlockWarps * 32 * 32];   // step slot << 10 | candidate: room for every pair of every slot
    int at[kBlockWarps];                // the slots' steps
    int queued[2];                      // candidates in the queue (of alternate batches)
    int first[32 * kFirstRow];          // first overlapping step of pair (i, j) at kFirstRow i + j
    unsigned found[32];                 // [lane] micro-block pairs that overlapped in an earlier batch
    int order[2][32];                   // hypotheses of the rows and columns
    float prob[2][32];                  // fused: their probabilities
    unsigned long long lfix[32], pfix[32];   // fused EGO pair: the CO side's fixed-point terms
};

// (mask 0: the block's active steps are not known yet, from step 0 on)
template <bool FUSED, bool OUTL>
__device__ __forceinline__ void block_work(const CollideArgs &a, const BlockRef &B, unsigned rows, BlockSlot &S) {
    constexpr int W = kBlockWarps, ROWS = 32 / W;
    constexpr int kNone = 0x7fffffff;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, tid = threadIdx.x;
    const PairDesc &P = a.pairs[B.pair];
    const long long box_a = B.box_a, box_b = B.box_b;
    StepPoses cur{};
    auto load = [&](int k) {
        cur.a = load_pose<true>(a, 32 * (box_a + k) + lane, true, 0.0f);
        cur.b = load_pose<true>(a, 32 * (box_b + k) + lane, true, 0.0f);
    };
    // the warp's step of the next batch: of the active steps in `mask` (bit b: step k0 + b), rank base + w
    int k0 = B.k0, base = 0;
    unsigned mask = B.mask;
    auto next_chunk = [&](int from) {               // the next 32 steps with an active one (mask 0: none)
        base = 0;
        for (k0 = from; k0 < P.n_steps; k0 += 32) {
            const int k = k0 + lane;
            mask = __ballot_sync(0xffffffffu, k < P.n_steps && boxes_meet(a.bounds[box_a + k], a.bounds[box_b + k], P.r_cull));
            if (mask) return;
        }
    };
    if (!mask) next_chunk(k0);
    if (!mask) return;                              // (uniform over the CTA)
    auto mine = [&]() -> int { return base + w < __popc(mask) ? k0 + nth_set_bit(mask, base + w) : -1; };
    int k = mine();
    if (k >= 0) load(k);
    for (int q = tid; q < 32 * kFirstRow; q += 32 * W) S.first[q] = kNone;
    if (w < 2) {                                    // warp 0: the rows, warp 1: the columns
        const int tile = w ? B.tile_b : B.tile_a;
        const bool ok = 32 * tile + lane < (w ? P.h_b : P.h_a);
        const int h = a.tile_order[32LL * ((w ? P.tile_b : P.tile_a) + tile) + lane];
        S.order[w][lane] = h;
        if (FUSED) {                                // asynchronous: the latency hides under the tests
            const long long traj = (w ? P.traj_b : P.traj_a) + h;
            if (ok) cp_async4(&S.prob[w][lane], a.probf + traj); else S.prob[w][lane] = 0.0f;
            if (ok && P.ego_side == 1 - w) {        // the CO's side
                cp_async8(S.lfix + lane, a.lfix + traj);
                cp_async8(S.pfix + lane, a.pfix + traj);
            }
        }
    }
    if (OUTL && P.combo >= 4 && w < 2) {
        load_outline(S.outline[w], a.polys, P, w, lane);
        if (P.combo == 4 && lane < 16) {
            const ObjDesc &o = a.objs[w ? P.b : P.a];
            const float2 q = point_of(lane, o.core_l, o.core_w);
            __syncwarp(0xffffu);
            S.faces[w][lane] = (unsigned char)facing_edge(S.outline[w], o.n_poly, q.x, q.y);
        }
    }
    if (w == W - 1) S.found[lane] = ~rows;          // (the other rows' pairs count as found)
    if (w == W - 2 && lane < 2) S.queued[lane] = 0;
    const PairShape shape = OUTL ? staged_shape(P) : shape_of(P);
    const Extents ext = extents_of(a, P, OUTL);
    const float rc2 = P.rc2 + kEps0;
    __syncthreads();                                // S.first, S.found, S.queued initialised
    unsigned narrow = 0;                            // this lane's exact tests
    int steps = 0, parity = 0;
    while (mask) {                                  // (uniform over the CTA)
        unsigned cand = 0u;
        if (k >= 0) cand = stage_and_sweep(S.step[w], cur, rc2, lane) & ~S.found[lane];
        if (lane == 0) S.at[w] = k;
        steps += k >= 0;
        base += W;
        if (base >= __popc(mask)) {
            mask = 0u;
            next_chunk(k0 + 32);
        }
        k = mine();
        if (k >= 0) load(k);                        // in flight while the candidates are tested
        int off, total, at = 0;
        if (queue_offsets6(__popc(cand), lane, off, total)) {
            if (lane == 0) at = atomicAdd(&S.queued[parity], total);
            off += __shfl_sync(0xffffffffu, at, 0);
            for (; cand; cand &= cand - 1u, ++off)
                S.queue[off] = (unsigned short)(w << 10 | lane << 5 | (__ffs(cand) - 1));
        }
        __syncthreads();
        const int queued = S.queued[parity];
        if (tid == 0) S.queued[parity ^ 1] = 0;
        auto hit_at = [&](int e) {
            atomicOr(&S.found[e >> 5 & 31], 1u << (e & 31));
            atomicMin(&S.first[kFirstRow * queued_row(e) + queued_col(e)], S.at[e >> 10]);
        };
        // (half the candidates with outlines overlap, most of them pairs that do so in several steps of the batch)
        auto beaten = [&](int e) { return S.first[kFirstRow * queued_row(e) + queued_col(e)] < S.at[e >> 10]; };
        if (OUTL && shape.combo >= 4) {
            test_outlines((queued + 32 * W - 1 - 32 * w) / (32 * W), shape,
                [&](int r) {
                    const int u = 32 * W * r + tid;
                    narrow += u < queued;
                    const int e = u < queued ? S.queue[u] : -1;
                    return u < queued && !beaten(e) ? e : -1;
                },
                [&](int e) { return first_look(S.step[e >> 10], shape, S.outline[0], ext, e, S.faces[0]); },
                [&](int e, int g, int edges) { return edge_decides(S.step[e >> 10], shape, S.outline[0], ext, e, g, edges); },
                hit_at);
        } else {
            for (int u = tid; u < queued; u += 64 * W) {   // two candidates of a lane in flight
                const int u2 = u + 32 * W, e = S.queue[u], e2 = S.queue[u2 < queued ? u2 : u];
                const bool h = overlap<false>(S.step[e >> 10], shape, S.outline[0], ext, e);
                const bool h2 = (u2 - lane < queued) && overlap<false>(S.step[e2 >> 10], shape, S.outline[0], ext, e2);
                narrow += u2 < queued ? 2 : 1;
                if (h) hit_at(e);
                if (h2 && u2 < queued) hit_at(e2);
            }
        }
        parity ^= 1;
        __syncthreads();
    }
    if (a.counters) {
        narrow = __reduce_add_sync(0xffffffffu, narrow);
        if (lane == 0) {
            if (narrow) count_narrow(a, P.combo, narrow);
            if (steps) atomicAdd(a.counters, (unsigned long long)steps * 32 * __popc(rows));
        }
    }
    if (FUSED) {
        cp_async_wait();
        __syncthreads();                            // the copies of the first warps
    }

    // ---- the first hits of the warp's ROWS lines (rows, or columns where b is the EGO object, so that a line is one
    // EGO hypothesis): the table entries and (fused) the risk terms
    const int ego_side = P.ego_side, l0 = w * ROWS, line = ego_side == 1 ? 1 : kFirstRow;
    const int across = ego_side == 1 ? kFirstRow : 1;
    int at[ROWS];                                   // first steps of this lane's pair in each line
    unsigned hits = 0u;                             // bit u: the pair in line u hit
#pragma unroll
    for (int u = 0; u < ROWS; ++u) {
        at[u] = S.first[line * (l0 + u) + across * lane];
        if (at[u] != kNone) hits |= 1u << u;
    }
    const int total = (int)__reduce_add_sync(0xffffffffu, (unsigned)__popc(hits));
    if (!total) return;
    const int hb = P.h_b;
    int16_t *tab = a.table + P.off;
    const int *line_h = S.order[ego_side == 1], hl = S.order[ego_side != 1][lane];   // the lines' hypotheses, the lane's
    unsigned long long wt[ROWS] = {};
#pragma unroll
    for (int u = 0; u < ROWS; ++u) {
        if (!(hits >> u & 1u)) continue;
        const int h = line_h[l0 + u];
        tab[ego_side == 1 ? (long long)hl * hb + h : (long long)h * hb + hl] = (int16_t)at[u];
        if (FUSED) wt[u] = to_fixed(S.prob[ego_side == 1][l0 + u] * S.prob[ego_side != 1][lane], kFixProb);
    }
    if constexpr (FUSED) {
        const bool ego = ego_side >= 0;
        add_hit_terms<ROWS>(a.acc, P, ego, at, hits, total, wt, [&](int u) { return line_h[l0 + u]; },
                            ego ? S.lfix[lane] : 0ull, ego ? S.pfix[lane] : 0ull);
    }
}

// LISTED: CTAs take the listed blocks in order, the heavy ones first.  Otherwise CTA g has block g of the ascending
// tiles: where all blocks fit on the chip at once the listing would only delay them (3 us of a 19 us call with two
// objects of 16 hypotheses; with 5,780 blocks, most of them empty, it saves 9 of 56 us).

template <bool FUSED, bool OUTL, bool LISTED>
__global__ void __launch_bounds__(32 * kBlockWarps, kBlockCtas) block_kernel(const CollideArgs a) {
    pdl_trigger();
    __shared__ BlockSlot S;
    if (!LISTED) {
        const long long g = blockIdx.x;
        BlockRef B{};
        B.pair = pair_of_tile(a, g >> 2);           // uploaded data: before the wait
        const PairDesc &P = a.pairs[B.pair];
        const int t = (int)((g >> 2) - P.tile_start), ta = t / P.tiles_b, q = (int)(g & 3);
        B.tile_a = 2 * ta + (q >> 1);
        B.tile_b = 2 * (t - ta * P.tiles_b) + (q & 1);
        B.box_a = (int)(P.bounds_a + (long long)B.tile_a * P.n_steps);
        B.box_b = (int)(P.bounds_b + (long long)B.tile_b * P.n_steps);
        const bool in = 32 * B.tile_a < P.h_a && 32 * B.tile_b < P.h_b;
        pdl_wait();
        if (in) block_work<FUSED, OUTL>(a, B, 0xffffffffu, S);
        return;
    }
    pdl_wait();
    const bool halves = OUTL && a.n_tiles < kHalvesBelow;
    const long long front = (long long)a.list_counts[0], listed = front + (long long)a.list_counts[1];
    const long long parts = halves ? 2 * front : 0, tasks = listed + parts / 2;
    for (long long it = blockIdx.x; it < tasks; it += gridDim.x) {
        // (a half: its rows' bits of every micro-block, MJ m + n at rows lr + 8 m)
        if (it < parts) block_work<FUSED, OUTL>(a, a.list[it >> 1], it & 1 ? 0xffff0000u : 0xffffu, S);
        else block_work<FUSED, OUTL>(a, listed_block(a, it - parts / 2, front), 0xffffffffu, S);
        if (it + gridDim.x < tasks) __syncthreads();   // the slots are no longer read
    }
}

template <bool OUTL, bool LISTED>
cudaError_t launch_blocks(const CollideArgs &a, long long ctas, cudaStream_t st, bool pdl) {
    if (ctas > 0x7fffffffLL) return cudaErrorInvalidValue;
    const dim3 grid((unsigned)ctas), block(32 * kBlockWarps);
    return a.probf ? launch_kernel(block_kernel<true, OUTL, LISTED>, grid, block, 0, st, pdl, a)
                   : launch_kernel(block_kernel<false, OUTL, LISTED>, grid, block, 0, st, pdl, a);
}

template <bool OUTL>
cudaError_t launch_listed(const CollideArgs &a, cudaStream_t st, bool pdl) {
    const long long blocks = 4 * a.n_tiles;
    if (a.variant == 7 && blocks <= kBlockSlots) return launch_blocks<OUTL, false>(a, blocks, st, pdl);
    // 8 tiles per warp once that still gives every SM a few warps
    const int per_warp = a.n_tiles >= 152LL * 8 * 32 ? 8 : 1;
    const long long tiles = (long long)kListWarps * per_warp;
    cudaError_t e = launch_kernel(block_list_kernel, dim3((unsigned)((a.n_tiles + tiles - 1) / tiles)), dim3(32 * kListWarps),
                                  0, st, pdl, a, per_warp);
    if (e != cudaSuccess) return e;
    if (a.variant == 7)                             // up to four waves of CTAs, further blocks in turn
        return launch_blocks<OUTL, true>(a, std::min(blocks, 4LL * kBlockSlots), st, true);
    // CTAs for every block of every tile (the warps of those past the last listed block leave at once)
    const long long ctas = (4 * a.n_tiles + kWalkWarps * kWalkBlocks - 1) / (kWalkWarps * kWalkBlocks);
    const dim3 grid((unsigned)ctas), walk(32 * kWalkWarps);
    return a.probf ? launch_kernel(walk_kernel<true, OUTL, false>, grid, walk, 0, st, true, a)
                   : launch_kernel(walk_kernel<false, OUTL, false>, grid, walk, 0, st, true, a);
}

template <bool OUTL>
cudaError_t launch_unlisted(const CollideArgs &a, cudaStream_t st, bool pdl) {
    long long ctas = a.n_tiles;                     // a warp per block
    if (a.max_ctas > 0 && ctas > a.max_ctas) ctas = a.max_ctas;
    const dim3 grid((unsigned)ctas), block(32 * kWalkWarps);
    return a.probf ? launch_kernel(walk_kernel<true, OUTL, true>, grid, block, 0, st, pdl, a)
                   : launch_kernel(walk_kernel<false, OUTL, true>, grid, block, 0, st, pdl, a);
}

}  // namespace

int tiles_launches(const CollideArgs &a) {
    return a.tile_poses && !(a.variant == 7 && 4 * a.n_tiles <= kBlockSlots) ? 2 : 1;
}

cudaError_t launch_tiles(const CollideArgs &a, cudaStream_t st, bool pdl) {
    if (a.tile_poses) {     // the table's -1s and the list's counts are written beforehand
        if (!a.tile_order || !a.list || !a.list_counts) return cudaErrorInvalidValue;
        return a.polys ? launch_listed<true>(a, st, pdl) : launch_listed<false>(a, st, pdl);
    }
    return a.polys ? launch_unlisted<true>(a, st, pdl) : launch_unlisted<false>(a, st, pdl);
}

}  // namespace mhc
