// hit_terms.cuh -- the risk terms of first hits, summed over a warp before they go out: shared by the fused collision
// kernel (layout 7) and the risk scan of a finished table.
#pragma once
#include "mhc_internal.cuh"

namespace mhc {
namespace {

// Sum of v over the warp (modulo 2^64): three 32-bit reductions.
__device__ __forceinline__ unsigned long long reduce_terms(unsigned long long v) {
    const unsigned m0 = __reduce_add_sync(0xffffffffu, (unsigned)v & 0xffffffu);
    const unsigned m1 = __reduce_add_sync(0xffffffffu, (unsigned)(v >> 24) & 0xffffffu);
    const unsigned m2 = __reduce_add_sync(0xffffffffu, (unsigned)(v >> 48));
    return m0 + ((unsigned long long)m1 << 24) + ((unsigned long long)m2 << 48);
}

constexpr int kHitsPerStep = 16;        // hits per step of a warp's lines from which its terms are summed step by step

// A warp's hits of one object pair P: `ROWS` lines of 32 pairs, lane l of line u with first step at[u] where bit u of
// `hits` is set (`total`: the hits of all lanes) and the pair's probability wt[u].  `ego`: line u is EGO hypothesis
// line_h(u), and the lane's CO hypothesis has the fixed-point terms lf (log-survival) and pf (probability).
//
// Many hits a step: a loop over the steps (one reduction per hit and sum, on few addresses, took up to 34 us for a block
// of 1,024 hits; EGO-only call 136 -> 101 us).  Else one reduction per hit: a turn of the loop is 150 instructions
// (always looping, the 11-object call takes 51.4 us instead of 48.1; from 8 hits a step 49.1).
template <int ROWS, typename LineH>
__device__ __forceinline__ void add_hit_terms(const RiskScratch &acc, const PairDesc &P, bool ego, const int (&at)[ROWS],
                                              unsigned hits, int total, const unsigned long long (&wt)[ROWS],
                                              LineH &&line_h, unsigned long long lf, unsigned long long pf) {
    constexpr int kNone = 0x7fffffff;
    const int lane = threadIdx.x & 31, N = P.n_steps, n_obj_s = P.n_obj_s, co_local = P.co_local;
    const long long kofs = P.kofs, lsum_base = P.lsum_base, mass_base = P.mass_base, hits_base = P.hits_base;
    unsigned count = 0;
    unsigned long long mass = 0;
    int lo = kNone, hi = 0;
#pragma unroll
    for (int u = 0; u < ROWS; ++u)
        if (hits >> u & 1u) { lo = min(lo, at[u]); hi = max(hi, at[u]); }
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    const bool dense = total >= kHitsPerStep * (hi - lo + 1);
    if (!dense) {
#pragma unroll
        for (int u = 0; u < ROWS; ++u) {
            if (!(hits >> u & 1u)) continue;
            atomicAdd(acc.count_k + kofs + at[u], 1ull);
            atomicAdd(acc.H + kofs + at[u], wt[u]);
            ++count;
            mass += wt[u];
            if (ego) atomicAdd(acc.lsum + lsum_base + ((long long)line_h(u) * N + at[u]) * n_obj_s + co_local, lf);
        }
        count = __reduce_add_sync(0xffffffffu, count);
        mass = reduce_terms(mass);
    }
    for (unsigned left = dense ? hits : 0u;;) {
        const unsigned lanes = __ballot_sync(0xffffffffu, left != 0u);
        if (!lanes) break;
        int k = kNone;                          // the lane's earliest step
#pragma unroll
        for (int u = 0; u < ROWS; ++u)
            if (left >> u & 1u) k = min(k, at[u]);
        k = __reduce_min_sync(0xffffffffu, k);
        unsigned c = 0;
        unsigned long long v = 0;
#pragma unroll
        for (int u = 0; u < ROWS; ++u) {
            const bool now = (left >> u & 1u) && at[u] == k;
            const unsigned m = __ballot_sync(0xffffffffu, now);
            if (!m) continue;
            if (now) {
                v += wt[u];
                left &= ~(1u << u);
            }
            c += __popc(m);
            if (!ego) continue;
            const unsigned long long sum = reduce_terms(now ? lf : 0ull);
            if (lane == 0)
                atomicAdd(acc.lsum + lsum_base + ((long long)line_h(u) * N + k) * n_obj_s + co_local, sum);
        }
        v = reduce_terms(v);
        if (lane == 0) {
            atomicAdd(acc.count_k + kofs + k, (unsigned long long)c);
            atomicAdd(acc.H + kofs + k, v);
        }
        count += c;
        mass += v;
    }
    if (ego) {
#pragma unroll
        for (int u = 0; u < ROWS; ++u) {
            const unsigned m = __ballot_sync(0xffffffffu, hits >> u & 1u);
            if (!m) continue;
            const unsigned long long sum = reduce_terms(hits >> u & 1u ? pf : 0ull);
            if (lane == 0) {
                const long long e = line_h(u);
                atomicAdd(acc.mass + mass_base + e * n_obj_s + co_local, sum);
                atomicAdd(acc.hits + hits_base + e, (unsigned long long)__popc(m));
            }
        }
    }
    if (lane == 0) {
        atomicAdd(acc.count + P.index, (unsigned long long)count);
        atomicAdd(acc.P + P.index, mass);
    }
}

}  // namespace
}  // namespace mhc
