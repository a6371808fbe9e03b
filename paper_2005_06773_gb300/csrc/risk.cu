// risk.cu -- risk assessment (Section IV-D) from the first-collision table.
//
//   prepare  zero the accumulators; L1-normalise each object's weights into probabilities (Section IV-D.1)
//   scan     a warp per 8 x 32 (large tables: 32 x 32) entries of the table: counts, first-step histograms and
//            probability masses per object pair (Eq. totalCrashProb per pair); for pairs containing the
//            EGO object also per-EGO-hypothesis hit counts, per-(hypothesis, CO object) masses and, per
//            (hypothesis, step, CO object) cell, the sum of -log(1 - p) over the cell's entries
//   ego      one warp per EGO hypothesis walks the cells in ascending (step, object) order: a cell with
//            survival factor 1 - q = exp(-sum) contributes S q and leaves S (1 - q), S being the survival
//            product of the earlier cells -- exactly the entry-by-entry scaling of Eq. p21 summed over
//            the cell (telescoping); plus the per-object independence measure and the scalar totals
//            and the escape-route ranks (Section VI-A); its last CTA converts the totals
//
// Collisions are rare and scattered inside a warp, so the per-hit work uses only FP32 and integer
// instructions: each term (p_a p_b, p, -log(1 - p)) is formed in FP32 and added exactly as unsigned
// 64-bit fixed point by integer atomics (exact, order-independent, bitwise reproducible).  FP64 -- a
// narrow pipe on this GPU -- runs only in dense per-warp steps.
#include "collide_common.cuh"
#include "hit_terms.cuh"
#include "mhc_internal.cuh"
#include "prepare.cuh"

namespace mhc {
namespace {

// value of a fixed-point sum with `frac` fractional bits (the scale is an exact power of two)
__device__ __forceinline__ double from_fixed(unsigned long long v, int frac) {
    return __ull2double_rn(v) * (1.0 / (double)(1ull << frac));
}

// blocks [0, n_obj) normalise one object each; every block zeroes a slice of the accumulators
__global__ void __launch_bounds__(256) prepare_kernel(const PrepArgs a) {
    pdl_start();
    prepare_block(a, blockIdx.x, gridDim.x);
}

// The terms of a finished table's first hits.  A warp takes 32 columns of some rows of one pair (a lane per column: the
// rows' loads coalesced and all in flight at once).  Where b is the EGO object the lanes are EGO hypotheses, and their
// masses and hits are sums over the lane's own rows.
//
// Small tables: 8 rows a warp, add_hit_terms sums what four rows' hits have in common.  Large ones (HIST): 32 rows a
// warp, with the counts and masses per step in a histogram of the warp's own in shared memory, since with many warps the
// reductions on a pair's few per-step sums would be the bound.  The whole call (preparation, scan, walk) on an 11-object
// table of 5.7 M entries 33.8 us (a CTA of 64 threads per 64 x 64 tile with the cells in shared memory: 57.6; HIST 40),
// EGO-only 63 us (392), 20 cars of 2,048 hypotheses, 1.6 GB, 1.51 ms (2.71; without the histograms 4.42).
constexpr int kScanLines = 4;              // rows whose terms are summed together
constexpr int kScanWarps = 4;
constexpr long long kScanHistTiles = 4864; // 32 tiles per SM: large
constexpr int kScanHistSteps = 1024;       // histograms (16 bytes a step and warp) up to this horizon
template <bool HIST> constexpr int kScanRows = HIST ? 32 : 8;
template <bool HIST> constexpr int kScanUnits = (kTile / 32) * (kTile / kScanRows<HIST>);   // warp tasks per 64 x 64 tile

template <bool HIST>
__global__ void __launch_bounds__(32 * kScanWarps) scan_kernel(const RiskArgs a) {
    constexpr int R = kScanRows<HIST>, UNITS = kScanUnits<HIST>;
    pdl_trigger();
    extern __shared__ unsigned s_hist[];   // HIST: [warp][step] count | [warp][3][step] 21-bit parts of the mass
    const long long gw = (long long)blockIdx.x * kScanWarps + (threadIdx.x >> 5);
    const long long g = gw / UNITS;
    const int lane = threadIdx.x & 31;
    if (g >= a.n_tiles) {
        pdl_wait();
        return;
    }
    const PairDesc &P = a.pairs[pair_of_tile(a, g)];   // uploaded data: before the wait
    const int t = (int)(g - P.tile_start), q = (int)(gw - g * UNITS);
    const int ta = t / P.tiles_b, tb = t - ta * P.tiles_b;
    const int i0 = ta * kTile + (q >> 1) * R, j = tb * kTile + (q & 1) * 32 + lane;
    const int rows = min(R, P.h_a - i0), N = P.n_steps, ego_side = P.ego_side, hb = P.h_b;
    const long long traj_a = P.traj_a + i0, traj_b = P.traj_b + j;
    const int16_t *row = a.table + P.off + (long long)i0 * hb + j;
    pdl_wait();
    if (rows <= 0) return;
    const bool col = j < hb;
    short first[R];
#pragma unroll
    for (int u = 0; u < R; ++u) first[u] = col && u < rows ? __ldg(row + (long long)u * hb) : (short)-1;
    unsigned any = 0u;
#pragma unroll
    for (int u = 0; u < R; ++u) {
        const bool hit = first[u] >= 0 && first[u] < N;   // -1: no collision; >= N cannot come from the collision kernel
        any |= (hit ? 1u : 0u) << u;
    }
    if (!__any_sync(0xffffffffu, any != 0u)) return;
    const float pb = col ? a.probf[traj_b] : 0.0f;
    const unsigned long long lf = ego_side == 0 && col ? a.lfix[traj_b] : 0ull, pf = ego_side == 0 && col ? a.pfix[traj_b] : 0ull;
    unsigned long long lane_mass = 0;
    if (ego_side == 1) {
#pragma unroll 4
        for (unsigned m = any; m; m &= m - 1u) lane_mass += a.pfix[traj_a + __ffs(m) - 1];
        if (any) {
            atomicAdd(a.acc.mass + P.mass_base + (long long)j * P.n_obj_s + P.co_local, lane_mass);
            atomicAdd(a.acc.hits + P.hits_base + j, (unsigned long long)__popc(any));
        }
    }
    if constexpr (HIST) {
        unsigned *cnt = s_hist + (size_t)(threadIdx.x >> 5) * 4 * N, *part = cnt + N;
        for (int k = lane; k < 4 * N; k += 32) cnt[k] = 0u;
        __syncwarp();
        unsigned long long mass = 0;
#pragma unroll
        for (int u = 0; u < R; ++u) {
            const bool hit = any >> u & 1u;
            const unsigned m = __ballot_sync(0xffffffffu, hit);
            if (!m) continue;
            const int k = first[u];
            if (hit) {
                const unsigned long long wt = to_fixed(a.probf[traj_a + u] * pb, kFixProb);
                mass += wt;
                atomicAdd(cnt + k, 1u);
                atomicAdd(part + k, (unsigned)wt & 0x1fffffu);              // 1,024 terms of 21 bits at most
                atomicAdd(part + N + k, (unsigned)(wt >> 21) & 0x1fffffu);
                atomicAdd(part + 2 * N + k, (unsigned)(wt >> 42));
                if (ego_side >= 0) {
                    const long long e = ego_side == 0 ? i0 + u : j;
                    atomicAdd(a.acc.lsum + P.lsum_base + (e * N + k) * P.n_obj_s + P.co_local,
                              ego_side == 0 ? lf : a.lfix[traj_a + u]);
                }
            }
            if (ego_side == 0) {
                const unsigned long long sum = reduce_terms(hit ? pf : 0ull);
                if (lane == 0) {
                    const long long e = i0 + u;
                    atomicAdd(a.acc.mass + P.mass_base + e * P.n_obj_s + P.co_local, sum);
                    atomicAdd(a.acc.hits + P.hits_base + e, (unsigned long long)__popc(m));
                }
            }
        }
        __syncwarp();
        for (int k = lane; k < N; k += 32)
            if (cnt[k]) {
                atomicAdd(a.acc.count_k + P.kofs + k, (unsigned long long)cnt[k]);
                atomicAdd(a.acc.H + P.kofs + k, part[k] + ((unsigned long long)part[N + k] << 21) +
                                                    ((unsigned long long)part[2 * N + k] << 42));
            }
        const unsigned total = __reduce_add_sync(0xffffffffu, (unsigned)__popc(any));
        mass = reduce_terms(mass);
        if (lane == 0) {
            atomicAdd(a.acc.count + P.index, (unsigned long long)total);
            atomicAdd(a.acc.P + P.index, mass);
        }
    } else {
#pragma unroll
        for (int u0 = 0; u0 < R; u0 += kScanLines) {
            const unsigned hits = any >> u0 & ((1u << kScanLines) - 1u);
            const int total = (int)__reduce_add_sync(0xffffffffu, (unsigned)__popc(hits));
            if (!total) continue;
            int at[kScanLines];
            unsigned long long wt[kScanLines];
#pragma unroll
            for (int u = 0; u < kScanLines; ++u) {
                at[u] = first[u0 + u];
                wt[u] = 0ull;
                if (!(hits >> u & 1u)) continue;
                wt[u] = to_fixed(a.probf[traj_a + u0 + u] * pb, kFixProb);
                if (ego_side == 1)
                    atomicAdd(a.acc.lsum + P.lsum_base + ((long long)j * N + at[u]) * P.n_obj_s + P.co_local,
                              a.lfix[traj_a + u0 + u]);
            }
            add_hit_terms<kScanLines>(a.acc, P, ego_side == 0, at, hits, total, wt, [&](int u) { return i0 + u0 + u; }, lf, pf);
        }
    }
}

template <bool HIST>
cudaError_t launch_scan(const RiskArgs &a, cudaStream_t st, bool pdl) {
    const long long ctas = (a.n_tiles * kScanUnits<HIST> + kScanWarps - 1) / kScanWarps;
    if (ctas > 0x7fffffffLL) return cudaErrorInvalidValue;
    const size_t per_step = HIST ? sizeof(unsigned) * 4 * kScanWarps : 0, smem = per_step * (size_t)a.max_steps;
    if (smem > 48 * 1024) {
        const cudaError_t e = allow_shared(scan_kernel<HIST>, per_step * kScanHistSteps);
        if (e != cudaSuccess) return e;
    }
    return launch_kernel(scan_kernel<HIST>, dim3((unsigned)ctas), dim3(32 * kScanWarps), smem, st, pdl, a);
}

// The caller's outputs from the accumulators (fixed point -> double), in two parts: the pair totals
// (count, P, count_k, H), final once the collision / scan launch has finished, and the totals the EGO walk
// itself accumulates (attr_obj, attr_step, scalars, n_escape).  Threads t of nt; each pass loads four
// elements before storing any, so the loads overlap.
__device__ void convert_pair_totals(const RiskArgs &a, long long t, long long nt) {
    const long long n = a.n_kofs + a.n_pairs;
    for (long long q0 = t; q0 < n; q0 += 4 * nt) {
        unsigned long long c[4], h[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const long long q = q0 + u * nt;
            c[u] = h[u] = 0ull;
            if (q < a.n_kofs) { c[u] = a.acc.count_k[q]; h[u] = a.acc.H[q]; }
            else if (q < n) { c[u] = a.acc.count[q - a.n_kofs]; h[u] = a.acc.P[q - a.n_kofs]; }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const long long q = q0 + u * nt;
            if (q < a.n_kofs) {
                if (a.count_k) a.count_k[q] = (long long)c[u];
                if (a.H) a.H[q] = from_fixed(h[u], kFixProb);
            } else if (q < n) {
                if (a.count) a.count[q - a.n_kofs] = (long long)c[u];
                if (a.P) a.P[q - a.n_kofs] = from_fixed(h[u], kFixProb);
            }
        }
    }
}

// One element per thread and pass, the four kinds in one index space: their loads overlap.
__device__ void convert_walk_totals(const RiskArgs &a, long long t, long long nt) {
    const long long b1 = a.n_obj, b2 = b1 + a.n_steps_total, b3 = b2 + 4LL * a.n_scen, n = b3 + a.n_scen;
    for (long long q = t; q < n; q += nt) {
        if (q < b2) {
            const unsigned long long v = q < b1 ? a.acc.attr_obj[q] : a.acc.attr_step[q - b1];
            double *out = q < b1 ? a.attr_obj : a.attr_step;
            if (out) out[q < b1 ? q : q - b1] = from_fixed(v, kFixProb);
        } else if (q < b3) {
            if (a.scalars) a.scalars[q - b2] = ((q - b2) & 3) < 3 ? a.acc.scalars[q - b2] : 0.0;
        } else {
            if (a.n_escape) a.n_escape[q - b3] = (int)a.acc.n_escape[q - b3];
        }
    }
}

// One warp per EGO hypothesis of the batch (its scenario found by binary search).
//  * collision-free hypothesis: its escape-route rank (Section VI-A) = the number of collision-free
//    hypotheses of its scenario more probable than it, ties by index, counted 32 at a time with ballots on
//    integer keys (probabilities are non-negative, so their bit patterns order like the values);
//  * otherwise the chronological walk: the (step, object) cells are copied to shared memory 416 at a time and the
//    non-empty ones moved together in ascending order, each with the prefix sum of the earlier cells' fixed-point
//    log-survival sums L (exact 64-bit integers), which gives it the survival S = exp(-sum of the
//    earlier cells' L), and the cell contributes S q with q = 1 - exp(-L) (Eq. p21 over the cell's collisions:
//    the product of their survival factors is exp(-L)).  Every term is formed in FP32 (relative error
//    below 5e-7) and the terms are summed in FP64.
// The attribution per object and step goes out with atomics, or (IN_PLACE, scenes of many cells) each term replaces
// its cell's sum, for attribution_kernel to add up: 2,048 hypotheses with 1,600 cells each spent 180 us of 215 in
// atomics on 82 addresses.
// The CTAs past the walk's convert the pair totals (within the walk's CTAs it held up the first of them by 1 us); the
// last CTA to finish converts the walk's own totals (or a later kernel does, for large batches).
// Bound by latency: a chain of loads (hits, masses and cells), the walk, a fence and the last CTA's conversion.  The
// loops stay rolled: each warp runs them about once, and fetching the unrolled code was most of a short walk (40 cells:
// 3.5 us).
constexpr float kLogScale = 1.0f / 1099511627776.0f;   // 2^-40: the fixed point of the log-survival sums

// exp(-x 2^-40) for a fixed-point log-survival sum x: x = hi + lo with hi the nearest FP32 value (exact
// as an integer) and lo the small remainder, so the FP32 rounding of x does not reach the exponent.
__device__ __forceinline__ float survival(unsigned long long x) {
    const float hi = __ull2float_rn(x);
    const long long lo = (long long)(x - __float2ull_rz(hi));
    return expf(-hi * kLogScale) * (1.0f - (float)lo * kLogScale);
}

constexpr int kEgoWarps = 2;
constexpr int kEscapeBatch = 8;    // escape ranking: 256 EGO hypotheses' keys in flight per round
constexpr int kWalkCells = 416;    // chronological walk: cells copied at once

// The last CTA of the launch to come here converts the totals, once every CTA's atomics are visible.  Every thread of
// every CTA calls it.
__device__ __forceinline__ void finish_totals(const RiskArgs &a) {
    __shared__ bool s_last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(a.acc.done, 1ull) == (unsigned long long)gridDim.x - 1;
    __syncthreads();
    if (s_last) {
        __threadfence();
        convert_walk_totals(a, threadIdx.x, blockDim.x);
    }
}

// The scenario of EGO hypothesis g of the batch.
__device__ __forceinline__ int scenario_of(const RiskArgs &a, long long g) {
    int lo = 0, hi = a.n_scen - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (a.scens[mid].e_base <= g) lo = mid; else hi = mid - 1;
    }
    return lo;
}

template <bool IN_PLACE>
__global__ void __launch_bounds__(32 * kEgoWarps) ego_kernel(const RiskArgs a) {
    pdl_trigger();
    __shared__ unsigned long long s_cells[kEgoWarps][kWalkCells], s_before[kEgoWarps][kWalkCells];
    __shared__ unsigned short s_index[kEgoWarps][kWalkCells];
    const int lane = threadIdx.x & 31;
    const long long g = (long long)blockIdx.x * kEgoWarps + (threadIdx.x >> 5);
    // the scenario of EGO hypothesis g and its descriptor: uploaded data, read before the wait
    const int lo = g < a.h_e ? scenario_of(a, g) : 0;
    const ScenDesc sd = g < a.h_e ? a.scens[lo] : ScenDesc{};
    pdl_wait();
    if (blockIdx.x >= a.walk_ctas)
        convert_pair_totals(a, (long long)(blockIdx.x - a.walk_ctas) * blockDim.x + threadIdx.x,
                            (long long)(gridDim.x - a.walk_ctas) * blockDim.x);
    const long long i = g - sd.e_base;
    if (g < a.h_e) {
        const unsigned long long hits = a.acc.hits[g];
        const double pe = a.prob[sd.e_traj + i];
        const float pef = a.probf[sd.e_traj + i];
        const int N = sd.n_steps, n_obj = sd.n_obj;
        double naive = 0.0, cond = 0.0, indep = 0.0;
        if (!hits) {
            if (a.escape) {
                const long long key = __double_as_longlong(pe);
                int rank = 0;
                for (int q0 = 0; q0 < sd.h_e; q0 += 32 * kEscapeBatch) {   // every load of a batch issued first
                    unsigned long long hq[kEscapeBatch];
                    long long kq[kEscapeBatch];
#pragma unroll
                    for (int u = 0; u < kEscapeBatch; ++u) {
                        const int q = q0 + 32 * u + lane;
                        hq[u] = q < sd.h_e ? a.acc.hits[sd.e_base + q] : 1ull;
                        kq[u] = q < sd.h_e ? __double_as_longlong(a.prob[sd.e_traj + q]) : 0ll;
                    }
#pragma unroll
                    for (int u = 0; u < kEscapeBatch; ++u) {
                        const int q = q0 + 32 * u + lane;
                        const bool above = hq[u] == 0ull && (kq[u] > key || (kq[u] == key && q < i));
                        rank += __popc(__ballot_sync(0xffffffffu, above));
                    }
                }
                if (lane == 0) a.escape[sd.e_base + rank] = (int)i;
            }
            if (lane == 0) atomicAdd(a.acc.n_escape + lo, 1ull);
        } else {
            unsigned long long *cell = s_cells[threadIdx.x >> 5];
            unsigned long long *before = s_before[threadIdx.x >> 5];
            unsigned short *index = s_index[threadIdx.x >> 5];
            unsigned long long *lc = a.acc.lsum + sd.lsum_base + i * N * n_obj;
            const long long cells = (long long)N * n_obj;
            // per-object masses: naive sum and independence product
            double surv = 1.0, mass_sum = 0.0, part = 0.0;
            const unsigned long long *ms = a.acc.mass + sd.mass_base + i * n_obj;
            unsigned long long carry = 0;     // L summed over every cell before the chunk
            for (long long g0 = 0; g0 < cells; g0 += kWalkCells) {
                const int n = (int)min((long long)kWalkCells, cells - g0);
                __syncwarp();
#pragma unroll 1
                for (int c = lane; c < n; c += 32) cp_async8(cell + c, lc + g0 + c);
                if (g0 == 0) {                // meanwhile
                    for (int b = lane; b < n_obj; b += 32) {
                        const double m = from_fixed(ms[b], kFixProb);
                        mass_sum += m;
                        surv *= 1.0 - m;
                    }
                }
                cp_async_wait();
                __syncwarp();
                // the lane's share of the window in ascending order (an odd number: no bank conflicts): its non-empty
                // cells and their sum, then both prefix sums, then the cells moved together with the sum before each
                const int per = ((n + 31) >> 5) | 1, c0 = min(lane * per, n), c1 = min(c0 + per, n);
                int count = 0;
                unsigned long long sum = 0;
                for (int c = c0; c < c1; ++c) {
                    const unsigned long long v = cell[c];
                    sum += v;
                    count += v != 0ull;
                }
                int at = count;
                unsigned long long incl = sum;
#pragma unroll
                for (int d = 1; d < 32; d <<= 1) {
                    const unsigned long long v = __shfl_up_sync(0xffffffffu, incl, d);
                    const int q = __shfl_up_sync(0xffffffffu, at, d);
                    if (lane >= d) { incl += v; at += q; }
                }
                const int filled = __shfl_sync(0xffffffffu, at, 31);
                unsigned long long earlier = carry + (incl - sum);
                carry += __shfl_sync(0xffffffffu, incl, 31);
                at -= count;
                for (int c = c0; c < c1; ++c) {
                    const unsigned long long v = cell[c];
                    if (!v) continue;
                    before[at] = earlier;
                    index[at++] = (unsigned short)c;
                    earlier += v;
                }
                __syncwarp();
                const int k0 = (int)(g0 / n_obj), b0 = (int)(g0 - (long long)k0 * n_obj);
#pragma unroll 1
                for (int q = lane; q < filled; q += 32) {
                    const int c = index[q];
                    const unsigned long long lf = cell[c];
                    const float eff = survival(before[q]) * -expm1f(-(float)lf * kLogScale);
                    part += (double)eff;
                    const unsigned long long w = to_fixed(pef * eff, kFixProb);
                    if (IN_PLACE) {
                        lc[g0 + c] = w;
                    } else {
                        const unsigned r = (unsigned)(b0 + c), k = r / (unsigned)n_obj;
                        atomicAdd(a.acc.attr_obj + sd.obj0 + (r - k * (unsigned)n_obj), w);
                        atomicAdd(a.acc.attr_step + sd.step_base + k0 + k, w);
                    }
                }
            }
#pragma unroll
            for (int d = 16; d > 0; d >>= 1) {
                surv *= __shfl_xor_sync(0xffffffffu, surv, d);
                mass_sum += __shfl_xor_sync(0xffffffffu, mass_sum, d);
                part += __shfl_xor_sync(0xffffffffu, part, d);
            }
            naive = mass_sum;
            indep = 1.0 - surv;
            cond = part;
        }
        if (lane < 3) {
            const double v = lane == 0 ? naive : (lane == 1 ? cond : indep);
            double *out = lane == 0 ? a.naive : (lane == 1 ? a.cond : a.indep);
            if (out) out[g] = v;
            if (v != 0.0) atomicAdd(a.acc.scalars + 4 * lo + lane, pe * v);
        }
        if (lane == 3 && a.hits) a.hits[g] = (int)hits;
    }
    if (a.convert_in_walk == 1) finish_totals(a);
}

// The attribution sums of scenes with many cells, from the terms the walk left in them: a CTA takes kAttrHyps EGO
// hypotheses of one scenario (its last CTA the rest), reads their cells coalesced (a thread per cell), adds the cells up
// per object and per step in shared memory and then into the totals: two atomics per object and step of a CTA instead of
// two per cell.  Cells the walk did not write are zero (a collision-free hypothesis's, or empty).  HBM-bound: it reads
// the cells once.  The CTAs' order takes the scenarios in turn, so that those that run together add to different totals
// (256 scenarios: risk stage 314 us, 351 in batch order).
constexpr int kAttrCells = 2048;

__global__ void __launch_bounds__(256) attribution_kernel(const RiskArgs a) {
    pdl_trigger();
    __shared__ unsigned long long s_sum[kAttrCells];
    // the CTAs as attr_rows rows of equal length (the last not full), taken column by column
    const unsigned rows = a.attr_rows, at = blockIdx.x % rows * (gridDim.x / rows) + blockIdx.x / rows;
    const int cta = (int)min((long long)at, a.attr_ctas - 1);
    const int s = last_where(a.n_scen, [&](int q) { return a.scens[q].attr_base <= cta; });   // uploaded data: before the wait
    const ScenDesc sd = a.scens[s];
    const long long i0 = (long long)(cta - sd.attr_base) * kAttrHyps;
    pdl_wait();
    const int hyps = at < a.attr_ctas ? (int)min((long long)kAttrHyps, sd.h_e - i0) : 0, n_obj = sd.n_obj;
    const long long cells = hyps ? (long long)sd.n_steps * n_obj : 0;
    const unsigned long long *term = a.acc.lsum + sd.lsum_base + i0 * cells;
    for (long long c0 = 0; c0 < cells; c0 += kAttrCells) {
        const int n = (int)min((long long)kAttrCells, cells - c0);
        for (int c = threadIdx.x; c < n; c += blockDim.x) {
            unsigned long long sum = 0;
#pragma unroll
            for (int u = 0; u < kAttrHyps; ++u)
                if (u < hyps) sum += term[u * cells + c0 + c];
            s_sum[c] = sum;
        }
        __syncthreads();
        const int k0 = (int)(c0 / n_obj), k1 = (int)((c0 + n - 1) / n_obj);   // the window's steps
        for (int q = threadIdx.x; q < n_obj + (k1 - k0 + 1); q += blockDim.x) {
            unsigned long long sum = 0;
            if (q < n_obj) {               // object q: every n_obj-th cell
                int c = (int)((q - c0 % n_obj + n_obj) % n_obj);
                for (; c < n; c += n_obj) sum += s_sum[c];
                if (sum) atomicAdd(a.acc.attr_obj + sd.obj0 + q, sum);
            } else {                       // step k: n_obj consecutive cells
                const long long k = k0 + (q - n_obj);
                const int c1 = (int)min((long long)n, (k + 1) * n_obj - c0);
                for (int c = (int)max(0LL, k * n_obj - c0); c < c1; ++c) sum += s_sum[c];
                if (sum) atomicAdd(a.acc.attr_step + sd.step_base + k, sum);
            }
        }
        __syncthreads();
    }
    if (a.convert_in_walk == 2) finish_totals(a);
}

// The walk's totals of a large batch, grid-wide after the walk (and the pair totals too when there is no
// EGO hypothesis to walk, which a valid scenario never has).
__global__ void __launch_bounds__(256) totals_kernel(const RiskArgs a) {
    pdl_start();
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x, nt = (long long)gridDim.x * blockDim.x;
    if (a.h_e == 0) convert_pair_totals(a, t, nt);
    convert_walk_totals(a, t, nt);
}

// Up to this many walk totals the walk's last CTA (64 threads) converts them, saving a launch; beyond it a
// grid-wide kernel does.
constexpr long long kConvertInWalk = 512;

long long convert_elements(const RiskArgs &a) {
    return a.n_obj + a.n_steps_total + 5LL * a.n_scen + (a.h_e == 0 ? 2 * (a.n_kofs + a.n_pairs) : 0);
}

}  // namespace

cudaError_t launch_risk_prepare(const RiskArgs &a, cudaStream_t st) {
    const int prep_blocks = a.n_obj > 304 ? a.n_obj : 304;
    prepare_kernel<<<prep_blocks, 256, 0, st>>>(prep_of(a));
    return cudaGetLastError();
}

// From this many cells (EGO hypotheses x steps x objects) the attribution is summed by its own kernel: the 11-object
// scene's 146 K cells take a launch less with atomics.
constexpr long long kAttrInPlace = 1LL << 19;

namespace {
bool attribution_alone(const RiskArgs &a) { return a.h_e > 0 && a.n_cells >= kAttrInPlace; }
}  // namespace

int risk_tail_launches(const RiskArgs &a) {
    const bool alone = attribution_alone(a);
    return (a.h_e > 0 ? 1 : 0) + (alone ? 1 : 0) + (a.h_e > 0 && convert_elements(a) <= kConvertInWalk ? 0 : 1);
}

cudaError_t launch_risk_tail(const RiskArgs &args, cudaStream_t st, bool pdl) {
    RiskArgs a = args;
    const long long conv = convert_elements(a);
    const bool alone = attribution_alone(a);
    a.convert_in_walk = a.h_e > 0 && conv <= kConvertInWalk ? (alone ? 2 : 1) : 0;
    if (a.h_e > 0) {
        a.walk_ctas = (a.h_e + kEgoWarps - 1) / kEgoWarps;
        const long long pair_ctas = std::min((a.n_kofs + a.n_pairs + 128 * kEgoWarps - 1) / (128 * kEgoWarps), 152LL * 8);
        const dim3 grid((unsigned)(a.walk_ctas + pair_ctas)), block(32 * kEgoWarps);
        cudaError_t e = alone ? launch_kernel(ego_kernel<true>, grid, block, 0, st, pdl, a)
                              : launch_kernel(ego_kernel<false>, grid, block, 0, st, pdl, a);
        if (e != cudaSuccess) return e;
        pdl = true;
        if (alone) {
            if (a.attr_ctas > 0x3fffffffLL) return cudaErrorInvalidValue;
            a.attr_rows = (int)std::min(a.attr_ctas, std::min((long long)a.n_scen, 1024LL));
            e = launch_kernel(attribution_kernel, dim3((unsigned)((a.attr_ctas + a.attr_rows - 1) / a.attr_rows * a.attr_rows)), dim3(256), 0, st, true, a);
            if (e != cudaSuccess) return e;
        }
    }
    if (!a.convert_in_walk) {
        long long blocks = (conv + 255) / 256;
        if (blocks > 152 * 8) blocks = 152 * 8;
        return launch_kernel(totals_kernel, dim3((unsigned)blocks), dim3(256), 0, st, pdl, a);
    }
    return cudaSuccess;
}

cudaError_t launch_risk(const RiskArgs &a, cudaStream_t st, bool with_prepare, bool pdl) {
    cudaError_t e = with_prepare ? launch_risk_prepare(a, st) : cudaSuccess;
    if (e != cudaSuccess) return e;
    pdl = pdl || with_prepare;
    if (a.n_tiles > 0) {
        if (a.n_tiles > 0x7fffffffLL) return cudaErrorInvalidValue;
        e = a.n_tiles >= kScanHistTiles && a.max_steps <= kScanHistSteps ? launch_scan<true>(a, st, pdl) : launch_scan<false>(a, st, pdl);
        if (e != cudaSuccess) return e;
        pdl = true;
    }
    return launch_risk_tail(a, st, pdl);
}

}  // namespace mhc
