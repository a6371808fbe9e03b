// gen.cu -- trajectory generation (Section IV-B): a warp per hypothesis with its sub-steps in parallel
// (scenarios with few hypotheses), or a thread per hypothesis with its sub-steps in order.
//
// Vehicles: one-track model (Eq. onetrack) with constant steering and acceleration, integrated by
// Eq. (EulerVelocity) with sub-step tau / K; the low-speed kinematic limit and the stop rule are applied
// on the sub-steps where the FP64 speed v_0 + n vdot tau_i crosses 2 m/s / zero (decided on the host in
// FP64, per object and acceleration value, and read from a table: no FP64 arithmetic runs here).  Arithmetic is FP32; x, y and psi are carried as
// compensated (hi, lo) sums so that 250+ sub-steps add no more than ~1e-6 m of rounding.
// Pedestrians: Eq. (pedestrianmotion) with a constant acceleration integrates exactly, so every output
// pose is evaluated in closed form (speed saturating at 0 or at the cap).
#include <algorithm>

#include "mhc_internal.cuh"
#include "prepare.cuh"
#include "quotient.h"

namespace mhc {
namespace {

// Kahan summation: (hi, c) carries the running sum hi - c; c is the compensation of the lost low part.
__device__ __forceinline__ void kahan_add(float &hi, float &c, float d) {
    const float y = __fsub_rn(d, c);
    const float t = __fadd_rn(hi, y);
    c = __fsub_rn(__fsub_rn(t, hi), y);
    hi = t;
}

// sincosf as one function body: inlined at every use it was most of the generation kernel's code, and a warp that runs
// its chain once fetches every instruction of it.
__device__ __noinline__ float2 sincos_any(float x) {
    float s, c;
    sincosf(x, &s, &c);
    return make_float2(s, c);
}

// sin / cos of the angle (a_hi + a_lo) to first order in the small part a_lo.
__device__ __forceinline__ void sincos2(float a_hi, float a_lo, float &sn, float &cs) {
    const float2 sc = sincos_any(a_hi);
    const float s0 = sc.x, c0 = sc.y;
    cs = fmaf(-s0, a_lo, c0);
    sn = fmaf(c0, a_lo, s0);
}

// sin / cos by the Taylor series to x^9 / x^10 (|x| <= 0.5: error < 2e-11).
__device__ __forceinline__ void sincos_half_series(float x, float &sn, float &cs) {
    const float x2 = x * x;
    float ps = fmaf(x2, 1.0f / 362880.0f, -1.0f / 5040.0f);
    ps = fmaf(x2, ps, 1.0f / 120.0f);
    ps = fmaf(x2, ps, -1.0f / 6.0f);
    sn = fmaf(x * x2, ps, x);
    float pc = fmaf(x2, -1.0f / 3628800.0f, 1.0f / 40320.0f);
    pc = fmaf(x2, pc, -1.0f / 720.0f);
    pc = fmaf(x2, pc, 1.0f / 24.0f);
    pc = fmaf(x2, pc, -0.5f);
    cs = fmaf(x2, pc, 1.0f);
}

// The series, sincosf beyond its range.
__device__ __forceinline__ void sincos_half(float x, float &sn, float &cs) {
    if (fabsf(x) > 0.5f) {
        const float2 sc = sincos_any(x);
        sn = sc.x;
        cs = sc.y;
        return;
    }
    sincos_half_series(x, sn, cs);
}

// sin / cos by the Taylor series to x^5 / x^6 (|x| <= 0.1: error < 3e-11).
__device__ __forceinline__ void sincos_tenth_series(float x, float &sn, float &cs) {
    const float x2 = x * x;
    sn = fmaf(x * x2, fmaf(x2, 1.0f / 120.0f, -1.0f / 6.0f), x);
    cs = fmaf(x2, fmaf(x2, fmaf(x2, -1.0f / 720.0f, 1.0f / 24.0f), -0.5f), 1.0f);
}

// The series, sincosf beyond its range.
__device__ __forceinline__ void sincos_tenth(float x, float &sn, float &cs) {
    if (fabsf(x) > 0.1f) {
        const float2 sc = sincos_any(x);
        sn = sc.x;
        cs = sc.y;
        return;
    }
    sincos_tenth_series(x, sn, cs);
}

__device__ void vehicle(const ObjDesc &o, float acc, float delta, const Regime &g, int N, int K, double tau_i_d,
                        long long base, int h, int i, float *X, float *Y, float *C, float *S) {
    const float dvf = (float)__dmul_rn((double)acc, tau_i_d);
    const int low_lo = g.low_lo, low_hi = g.low_hi, n_stop = g.n_stop;   // low regime on [low_lo, low_hi)

    const float ti = (float)tau_i_d;
    const float hti2 = 0.5f * ti * ti;
    const float dv = dvf;
    const float L = o.lf + o.lr;
    const float inv_m = 1.0f / o.m, inv_iz = 1.0f / o.Iz;
    const float k11 = -(o.caf + o.car) * inv_m;                 // a11 * v
    const float k12 = (o.car * o.lr - o.caf * o.lf) * inv_m;    // (a12 + 1) * v^2
    const float k21 = (o.car * o.lr - o.caf * o.lf) * inv_iz;   // a21
    const float k22 = -(o.caf * o.lf * o.lf + o.car * o.lr * o.lr) * inv_iz;  // a22 * v
    const float kb1 = o.caf * inv_m * delta;                    // b1 * v * delta
    const float kb2 = o.caf * o.lf * inv_iz * delta;            // b2 * delta
    const float tdel = tanf(delta);
    const float beta_kin = atanf(o.lr * tdel / L);
    const float kappa = cosf(beta_kin) * tdel / L;              // r = v * kappa in the kinematic limit
    const float stop_den = 0.5f / fabsf(acc == 0.0f ? 1.0f : acc);

    float xh = o.x0, xc = 0.0f, yh = o.y0, yc = 0.0f, ph = o.psi0, pc = 0.0f;   // Kahan sums
    float cps, sps;                      // cos / sin of the heading, carried between output steps
    sincos2(ph, -pc, sps, cps);
    float beta = 0.0f, r = 0.0f, ax = acc, ay = 0.0f;
    const int last = __reduce_max_sync(__activemask(), n_stop);   // every hypothesis of the warp has stopped after it
    bool stopped = false;
    int n = 0;
    for (int k = 0; k < N; ++k) {
        // (a warp whose hypotheses have all stopped only stores their poses)
        for (int q = 0; q < K && n <= last; ++q, ++n) {
            // every lane runs the same straight-line sub-step; regime and stop act through selects
            const bool low = n >= low_lo && n < low_hi;
            const bool stop_now = n == n_stop;
            const float v = fmaf((float)n, dv, o.v0);
            const float iv = __fdividef(1.0f, fmaxf(v, 1e-3f));
            const float bd_ot = fmaf(k11 * iv, beta, fmaf(fmaf(k12 * iv, iv, -1.0f), r, kb1 * iv));
            const float rd_ot = fmaf(k21, beta, fmaf(k22 * iv, r, kb2));
            const float b_use = low ? beta_kin : beta;
            const float r_use = low ? v * kappa : r;
            const float bd = low ? 0.0f : bd_ot;
            const float rd = low ? 0.0f : rd_ot;
            float sb, cb;
            sincos_half(b_use, sb, cb);
            const float cpb = fmaf(cps, cb, -sps * sb);          // course angle psi + beta
            const float spb = fmaf(sps, cb, cps * sb);
            const float d_stop = v * v * stop_den;
            const float dx = stop_now ? cpb * d_stop : fmaf(cpb * v, ti, fmaf(cps, ax, -sps * ay) * hti2);
            const float dy = stop_now ? spb * d_stop : fmaf(spb * v, ti, fmaf(sps, ax, cps * ay) * hti2);
            const float w = v * (bd + r_use);
            const float ax_n = fmaf(cb, acc, -sb * w);
            const float ay_n = fmaf(sb, acc, cb * w);
            const float dpsi = fmaf(r_use, ti, rd * hti2);
            const bool move = !stopped && !stop_now;             // a state update beyond the position
            kahan_add(xh, xc, stopped ? 0.0f : dx);
            kahan_add(yh, yc, stopped ? 0.0f : dy);
            kahan_add(ph, pc, move ? dpsi : 0.0f);
            if (move) {
                beta = fmaf(bd, ti, b_use);
                r = fmaf(rd, ti, r_use);
                ax = ax_n;
                ay = ay_n;
                float sd, cd;                                   // rotate (cos, sin) of the heading by dpsi
                sincos_tenth(dpsi, sd, cd);
                const float c2 = fmaf(cps, cd, -sps * sd);
                sps = fmaf(sps, cd, cps * sd);
                cps = c2;
            }
            stopped = stopped || stop_now;
        }
        sincos2(ph, -pc, sps, cps);                              // re-anchor on the exact heading
        const long long idx = base + (long long)k * h + i;
        X[idx] = xh - xc;
        Y[idx] = yh - yc;
        C[idx] = cps;
        S[idx] = sps;
    }
}

// Path hypotheses (Section IV-B.2b): before every sub-step the lateral controller of Eq. (controller) sets
// the front steering angle, in degrees, from the speed, the signed distance d_path from the centre of
// gravity predicted kCtrlTp ahead along the course to the active section's line (positive when the line
// lies to the left) and the yaw error e_psi = psi_section - psi; the angle is held within kDeltaMax and
// within kDeltaRate x tau_i of the previous sub-step's (0 before the first).  The one-track step is then
// the constant-steering one of `vehicle` with that angle.
constexpr float kCtrlTp = 0.5f;       // s: prediction time of the centre of gravity
constexpr float kDeltaMax = 0.5f;     // rad
constexpr float kDeltaRate = 0.5f;    // rad/s
constexpr float kPi = 3.14159265358979f;

struct PathConst {                     // of one hypothesis
    float acc, dv, v0, ti, hti2, lr, L, inv_L, k11, k12, k21, k22, kb1u, kb2u, stop_den, step_max;
};
struct PathSection {                   // point, direction, left normal
    float x, y, psi, nx, ny;
};
struct PathState {
    float xh, xc, yh, yc, ph, pc;      // Kahan sums
    float cps, sps;
    float beta, r, ax, ay, delta;
};

// One sub-step (n).  GENERAL: any state.  Otherwise for a sub-step outside the low-speed regime, without a branch;
// returns false if a slip angle or heading increment is out of the short series' range (the state is then not valid).
template <bool GENERAL>
__device__ __forceinline__ bool path_step(const PathConst &p, const PathSection &sec, PathState &s, int n, bool low,
                                          bool stop_now, bool stopped) {
    const float v = fmaf((float)n, p.dv, p.v0);
    float sb0, cb0;                                              // the course of the state before the step
    if (GENERAL) sincos_half(s.beta, sb0, cb0); else sincos_half_series(s.beta, sb0, cb0);
    bool ok = GENERAL || !(fabsf(s.beta) > 0.5f);
    {   // the controller, on the state before this sub-step
        const float px = (s.xh - s.xc) + kCtrlTp * v * fmaf(s.cps, cb0, -s.sps * sb0);
        const float py = (s.yh - s.yc) + kCtrlTp * v * fmaf(s.sps, cb0, s.cps * sb0);
        const float d_path = fmaf(sec.x - px, sec.nx, (sec.y - py) * sec.ny);
        float e_psi = sec.psi - (s.ph - s.pc);
        e_psi -= 2.0f * kPi * floorf((e_psi + kPi) * (0.5f / kPi));
        const float gd = fabsf(fmaf(-0.018f, v, 1.5f) * d_path);
        const float cmd = ((gd + 0.5f) * d_path + (9.5f - gd) * (3.8197f * e_psi)) * (kPi / 180.0f);
        const float delta = fminf(fmaxf(s.delta + fminf(fmaxf(cmd - s.delta, -p.step_max), p.step_max), -kDeltaMax), kDeltaMax);
        s.delta = stopped ? s.delta : delta;
    }
    const float kb1 = p.kb1u * s.delta, kb2 = p.kb2u * s.delta;
    float beta_kin = 0.0f, kappa = 0.0f;
    float sb = sb0, cb = cb0;                                    // the one-track step keeps the course
    if (GENERAL && low) {                                        // the kinematic limit at the new angle
        const float tdel = tanf(s.delta);
        beta_kin = atanf(quotient(p.lr * tdel, p.L, p.inv_L));
        kappa = quotient(cosf(beta_kin) * tdel, p.L, p.inv_L);
        sincos_half(beta_kin, sb, cb);
    }
    const float iv = __fdividef(1.0f, fmaxf(v, 1e-3f));
    const float bd_ot = fmaf(p.k11 * iv, s.beta, fmaf(fmaf(p.k12 * iv, iv, -1.0f), s.r, kb1 * iv));
    const float rd_ot = fmaf(p.k21, s.beta, fmaf(p.k22 * iv, s.r, kb2));
    const float b_use = low ? beta_kin : s.beta;
    const float r_use = low ? v * kappa : s.r;
    const float bd = low ? 0.0f : bd_ot;
    const float rd = low ? 0.0f : rd_ot;
    const float cpb = fmaf(s.cps, cb, -s.sps * sb);
    const float spb = fmaf(s.sps, cb, s.cps * sb);
    const float d_stop = v * v * p.stop_den;
    const float dx = stop_now ? cpb * d_stop : fmaf(cpb * v, p.ti, fmaf(s.cps, s.ax, -s.sps * s.ay) * p.hti2);
    const float dy = stop_now ? spb * d_stop : fmaf(spb * v, p.ti, fmaf(s.sps, s.ax, s.cps * s.ay) * p.hti2);
    const float w = v * (bd + r_use);
    const float ax_n = fmaf(cb, p.acc, -sb * w);
    const float ay_n = fmaf(sb, p.acc, cb * w);
    const float dpsi = fmaf(r_use, p.ti, rd * p.hti2);
    const bool move = !stopped && !stop_now;                     // a state update beyond the position
    kahan_add(s.xh, s.xc, stopped ? 0.0f : dx);
    kahan_add(s.yh, s.yc, stopped ? 0.0f : dy);
    kahan_add(s.ph, s.pc, move ? dpsi : 0.0f);
    float sd, cd;                                                // rotate (cos, sin) of the heading by dpsi
    if (GENERAL) sincos_tenth(move ? dpsi : 0.0f, sd, cd); else sincos_tenth_series(dpsi, sd, cd);
    ok = ok && (GENERAL || !move || !(fabsf(dpsi) > 0.1f));
    const float c2 = fmaf(s.cps, cd, -s.sps * sd);
    const float s2 = fmaf(s.sps, cd, s.cps * sd);
    const float b2 = fmaf(bd, p.ti, b_use), r2 = fmaf(rd, p.ti, r_use);
    s.beta = move ? b2 : s.beta;
    s.r = move ? r2 : s.r;
    s.ax = move ? ax_n : s.ax;
    s.ay = move ? ay_n : s.ay;
    s.sps = move ? s2 : s.sps;
    s.cps = move ? c2 : s.cps;
    return ok;
}

// One path hypothesis, in order: the controller feeds each sub-step's state back.  Latency-bound: a sub-step is a chain
// of some 170 instructions.  Outside the low-speed regime the warp runs the short body (no branch but the votes), inside
// it the general one (three times as long: tanf, atanf, cosf and the short series' other case); a hypothesis that has
// stopped is not in the regime, and a warp whose hypotheses have all stopped only stores their poses.  3,087 path
// hypotheses (11-object scene): generation 57 us (60 under ncu), 90 with the low regime run to the horizon's end, section values indexed
// in local memory and two divisions per low sub-step (a hypothesis braking at 9 m/s^2 spent three quarters of its time
// after its stop).
__device__ void vehicle_path(const ObjDesc &o, float acc, const float *path, const Regime &g, int N, int K,
                             double tau_i_d, long long base, int h, int i, float *X, float *Y, float *C, float *S) {
    const unsigned lanes = __activemask();
    const int low_lo = g.low_lo, low_hi = g.low_hi, n_stop = g.n_stop, n1 = o.path_n1, n2 = o.path_n2;
    PathConst p;
    p.acc = acc;
    p.dv = (float)__dmul_rn((double)acc, tau_i_d);
    p.v0 = o.v0;
    p.ti = (float)tau_i_d;
    p.hti2 = 0.5f * p.ti * p.ti;
    p.lr = o.lr;
    p.L = o.lf + o.lr;
    p.inv_L = 1.0f / p.L;
    const float inv_m = 1.0f / o.m, inv_iz = 1.0f / o.Iz;
    p.k11 = -(o.caf + o.car) * inv_m;
    p.k12 = (o.car * o.lr - o.caf * o.lf) * inv_m;
    p.k21 = (o.car * o.lr - o.caf * o.lf) * inv_iz;
    p.k22 = -(o.caf * o.lf * o.lf + o.car * o.lr * o.lr) * inv_iz;
    p.kb1u = o.caf * inv_m;                                     // b1 * v per rad of steering
    p.kb2u = o.caf * o.lf * inv_iz;                             // b2 per rad of steering
    p.stop_den = 0.5f / fabsf(acc == 0.0f ? 1.0f : acc);
    p.step_max = kDeltaRate * p.ti;
    PathState s{o.x0, 0.0f, o.y0, 0.0f, o.psi0, 0.0f};
    sincos2(s.ph, -s.pc, s.sps, s.cps);
    s.beta = s.r = s.ay = s.delta = 0.0f;
    s.ax = acc;
    // over the warp: the sub-step after which every hypothesis has stopped, and the sub-steps with a low-speed one
    const int last = __reduce_max_sync(lanes, n_stop), low_end = min(low_hi, n_stop + 1);
    const int any_lo = __reduce_min_sync(lanes, low_lo < low_end ? low_lo : 0x7fffffff);
    const int any_hi = __reduce_max_sync(lanes, low_lo < low_end ? low_end : 0);
    PathSection sec{};
    int n = 0;
    for (int k = 0; k < N; ++k) {
        // (a warp whose hypotheses have all stopped only stores their poses)
        for (int q = 0; q < K && n <= last; ++q, ++n) {
            if (n == 0 || n == n1 || n == n2) {                  // the section of the sub-steps from here on
                const float *pt = path + (n < n1 ? 0 : (n < n2 ? 3 : 6));
                sec.x = pt[0];
                sec.y = pt[1];
                sec.psi = pt[2];
                const float2 sc = sincos_any(sec.psi);
                sec.nx = -sc.x;
                sec.ny = sc.y;
            }
            const bool stop_now = n == n_stop, stopped = n > n_stop;
            const bool low = n >= low_lo && n < low_hi && !stopped;   // (a stopped hypothesis's values are not used)
            if (n < any_lo || n >= any_hi) {
                PathState next = s;
                const bool ok = path_step<false>(p, sec, next, n, false, stop_now, stopped);
                if (!__any_sync(lanes, !ok)) {
                    s = next;
                    continue;
                }
            }
            path_step<true>(p, sec, s, n, low, stop_now, stopped);
        }
        sincos2(s.ph, -s.pc, s.sps, s.cps);
        const long long idx = base + (long long)k * h + i;
        X[idx] = s.xh - s.xc;
        Y[idx] = s.yh - s.yc;
        C[idx] = s.cps;
        S[idx] = s.sps;
    }
}

// output steps k0, k0 + dk, ... of one pedestrian hypothesis (closed form)
__device__ void pedestrian(const ObjDesc &o, float ga, float gb, int N, float tau, long long base, int h, int i,
                           float *X, float *Y, float *C, float *S, int k0 = 0, int dk = 1) {
    const bool accel = (o.flags & kPedAccelGrid) != 0;
    const float v0 = accel ? o.v0 : ga;
    const float a = accel ? ga : 0.0f;
    const float th = o.psi0 + gb;
    float st, ct;
    sincosf(th, &st, &ct);
    // saturation time of the speed (cap when accelerating, zero when braking)
    float ts = INFINITY, s_sat = 0.0f, v_sat = v0;
    if (a > 0.0f && o.v_max > 0.0f) {
        if (v0 >= o.v_max) { ts = 0.0f; s_sat = 0.0f; v_sat = v0; }
        else { ts = (o.v_max - v0) / a; s_sat = v0 * ts + 0.5f * a * ts * ts; v_sat = o.v_max; }
    } else if (a < 0.0f) {
        ts = v0 / -a; s_sat = v0 * v0 / (-2.0f * a); v_sat = 0.0f;
    }
    for (int k = k0; k < N; k += dk) {
        const float t = (float)(k + 1) * tau;
        const float s = t < ts ? fmaf(0.5f * a * t, t, v0 * t) : fmaf(v_sat, t - ts, s_sat);
        const long long idx = base + (long long)k * h + i;
        X[idx] = fmaf(ct, s, o.x0);
        Y[idx] = fmaf(st, s, o.y0);
        C[idx] = ct;
        S[idx] = st;
    }
}

// ---- parallel-in-time generation: one warp per hypothesis ----------------------------------------------
//
// Every sub-step maps the lateral state s = (beta, r) affinely: s' = M_n s + c_n, with M_n, c_n functions of
// the speed v_n alone (one-track model: M = I + tau_i A(v_n), c = tau_i b(v_n); kinematic limit: M = 0,
// c = (beta_kin, v_n kappa); stopped: M = I, c = 0).  The warp's lanes take 8 consecutive sub-steps each,
// compose their maps, and one warp scan of the compositions gives every lane its start state; each lane
// then runs its sub-steps in order.  Heading and position are sums of per-sub-step increments, so they
// are prefix sums (double-float: an FP32 (hi, lo) pair per value, exact two-sum additions) over the lanes.

// (hi, lo) + (bh, bl), renormalised
__device__ __forceinline__ void df_add(float &hi, float &lo, float bh, float bl) {
    const float s = __fadd_rn(hi, bh);
    const float bb = __fsub_rn(s, hi);
    float e = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bb)), __fsub_rn(bh, bb));
    e = __fadd_rn(e, __fadd_rn(lo, bl));
    hi = __fadd_rn(s, e);
    lo = __fsub_rn(e, __fsub_rn(hi, s));
}

// inclusive warp scan of double-float values (lane order = time order)
__device__ __forceinline__ void df_scan(float &hi, float &lo, int lane) {
#pragma unroll 1
    for (int d = 1; d < 32; d <<= 1) {
        const float h2 = __shfl_up_sync(0xffffffffu, hi, d), l2 = __shfl_up_sync(0xffffffffu, lo, d);
        if (lane >= d) {
            float th = h2, tl = l2;
            df_add(th, tl, hi, lo);
            hi = th;
            lo = tl;
        }
    }
}

// df_scan of two values at once
__device__ __forceinline__ void df_scan2(float &ah, float &al, float &bh, float &bl, int lane) {
#pragma unroll 1
    for (int d = 1; d < 32; d <<= 1) {
        float a2 = __shfl_up_sync(0xffffffffu, ah, d), a3 = __shfl_up_sync(0xffffffffu, al, d);
        float b2 = __shfl_up_sync(0xffffffffu, bh, d), b3 = __shfl_up_sync(0xffffffffu, bl, d);
        if (lane >= d) {
            df_add(a2, a3, ah, al);
            df_add(b2, b3, bh, bl);
            ah = a2; al = a3;
            bh = b2; bl = b3;
        }
    }
}

// Affine map of the lateral state: s' = [m00 m01; m10 m11] s + (c0, c1).
struct Aff {
    float m00, m01, m10, m11, c0, c1;
};

// second after first: the map that applies `first`, then `second`
__device__ __forceinline__ Aff aff_then(const Aff &first, const Aff &second) {
    Aff r;
    r.m00 = fmaf(second.m00, first.m00, second.m01 * first.m10);
    r.m01 = fmaf(second.m00, first.m01, second.m01 * first.m11);
    r.m10 = fmaf(second.m10, first.m00, second.m11 * first.m10);
    r.m11 = fmaf(second.m10, first.m01, second.m11 * first.m11);
    r.c0 = fmaf(second.m00, first.c0, fmaf(second.m01, first.c1, second.c0));
    r.c1 = fmaf(second.m10, first.c0, fmaf(second.m11, first.c1, second.c1));
    return r;
}

// What a lane keeps of its sub-steps between the phases of a round: one slot per sub-step in shared memory (the loops
// over them stay rolled, a fifth of the unrolled code: the warp runs this chain once, and fetching straight-line code
// was most of its time).  Latency-bound where a scene has few hypotheses: 32 of them end 6.0 us after the descriptor
// copy, 11.4 us with the loops unrolled and sincosf inlined at its 17 uses; the 11-object scene's 3,571, six warps per
// scheduler and by then bound by issue, 11.0 us against 12.8.
constexpr int kScanSteps = 5;          // sub-steps per lane and round: a 150-sub-step horizon takes one round
struct ScanSlot {                      // [slip sine, cosine, heading increment, next accelerations, dx, dy][sub-step][lane]
    float v[7][kScanSteps][32];
    __device__ __forceinline__ float &at(int q, int c, int lane) { return v[q][c][lane]; }
};

// One vehicle hypothesis by the whole warp (every lane calls it).  Rounds of 32 x 5 sub-steps; lane L
// takes sub-steps L*5 .. L*5+4 of the round.  Per round: compose and scan the lanes'
// state maps, run the lanes' sub-steps from their start states (the same per-sub-step arithmetic as the
// sequential integration), scan the heading increments, form the position increments (heading trig
// exact at the lane's first sub-step, then rotated by each increment as the sequential integration
// rotates it), scan them, and store the poses of the output steps that end in each lane's sub-steps
// (exact heading trig).
__device__ void vehicle_scan(const ObjDesc &o, float acc, float delta, const Regime &g, int N, int K, int lane,
                             long long base, int h, int i, float *X, float *Y, float *C, float *S, ScanSlot &slot) {
    constexpr int CS = kScanSteps;
    enum { kSb, kCb, kDps, kAx, kAy, kDx, kDy };
    const int NK = N * K;
    const int low_lo = g.low_lo, low_hi = g.low_hi, n_stop = g.n_stop;
    const float ti = (float)o.tau_i_d;
    const float hti2 = 0.5f * ti * ti;
    const float dv = (float)__dmul_rn((double)acc, o.tau_i_d);
    const float v0 = o.v0;
    const float L = o.lf + o.lr;
    const float inv_m = 1.0f / o.m, inv_iz = 1.0f / o.Iz;
    const float k11 = -(o.caf + o.car) * inv_m;
    const float k12 = (o.car * o.lr - o.caf * o.lf) * inv_m;
    const float k21 = (o.car * o.lr - o.caf * o.lf) * inv_iz;
    const float k22 = -(o.caf * o.lf * o.lf + o.car * o.lr * o.lr) * inv_iz;
    const float kb1 = o.caf * inv_m * delta;
    const float kb2 = o.caf * o.lf * inv_iz * delta;
    float beta_kin = 0.0f, kappa = 0.0f;
    if (low_lo < min(low_hi, NK)) {                   // (uniform over the warp) the hypothesis enters the low regime
        const float tdel = tanf(delta);
        beta_kin = atanf(o.lr * tdel / L);
        kappa = cosf(beta_kin) * tdel / L;
    }
    const float stop_den = 0.5f / fabsf(acc == 0.0f ? 1.0f : acc);

    float beta = 0.0f, r = 0.0f;                      // lateral state at the round's first sub-step
    float ax = acc, ay = 0.0f;                        // acceleration used by the round's first sub-step
    float ph = o.psi0, pl = 0.0f, xh = o.x0, xl = 0.0f, yh = o.y0, yl = 0.0f;
    for (int nr = 0; nr < NK; nr += 32 * CS) {
        // sub-steps per lane this round: CS for full rounds, fewer for the last (100 sub-steps: 4 per lane)
        const int csa = min(CS, (min(NK - nr, 32 * CS) + 31) / 32);
        const int n0 = nr + lane * csa;
        // 1. the lane's state map, composed over its sub-steps, and the warp scan of the maps
        Aff F{1.0f, 0.0f, 0.0f, 1.0f, 0.0f, 0.0f};
#pragma unroll 1
        for (int c = 0; c < csa; ++c) {
            const int n = n0 + c;
            if (n >= NK || n >= n_stop) continue;     // past the end / frozen state: identity
            const float v = fmaf((float)n, dv, v0);
            Aff m;
            if (n >= low_lo && n < low_hi) {
                m = Aff{0.0f, 0.0f, 0.0f, 0.0f, beta_kin, v * kappa};
            } else {
                const float iv = __fdividef(1.0f, fmaxf(v, 1e-3f));
                m = Aff{fmaf(ti, k11 * iv, 1.0f), ti * fmaf(k12 * iv, iv, -1.0f), ti * k21, fmaf(ti, k22 * iv, 1.0f),
                        ti * (kb1 * iv), ti * kb2};
            }
            F = aff_then(F, m);
        }
        Aff P = F;
#pragma unroll 1
        for (int d = 1; d < 32; d <<= 1) {
            Aff q;
            q.m00 = __shfl_up_sync(0xffffffffu, P.m00, d); q.m01 = __shfl_up_sync(0xffffffffu, P.m01, d);
            q.m10 = __shfl_up_sync(0xffffffffu, P.m10, d); q.m11 = __shfl_up_sync(0xffffffffu, P.m11, d);
            q.c0 = __shfl_up_sync(0xffffffffu, P.c0, d);   q.c1 = __shfl_up_sync(0xffffffffu, P.c1, d);
            if (lane >= d) P = aff_then(q, P);
        }
        Aff E;   // the maps of the earlier lanes (identity for lane 0)
        E.m00 = __shfl_up_sync(0xffffffffu, P.m00, 1); E.m01 = __shfl_up_sync(0xffffffffu, P.m01, 1);
        E.m10 = __shfl_up_sync(0xffffffffu, P.m10, 1); E.m11 = __shfl_up_sync(0xffffffffu, P.m11, 1);
        E.c0 = __shfl_up_sync(0xffffffffu, P.c0, 1);   E.c1 = __shfl_up_sync(0xffffffffu, P.c1, 1);
        if (lane == 0) E = Aff{1.0f, 0.0f, 0.0f, 1.0f, 0.0f, 0.0f};
        float bs = fmaf(E.m00, beta, fmaf(E.m01, r, E.c0));
        float rs = fmaf(E.m10, beta, fmaf(E.m11, r, E.c1));

        // 2. the lane's sub-steps in order: slip trig, heading increments and their sum, next accelerations
        float ax_last = 0.0f, ay_last = 0.0f;             // the acceleration after the lane's last sub-step
        float dh = 0.0f, dl = 0.0f;
#pragma unroll 1
        for (int c = 0; c < csa; ++c) {
            const int n = n0 + c;
            const bool move = n < NK && n < n_stop;
            const bool low = n >= low_lo && n < low_hi;
            const float v = fmaf((float)n, dv, v0);
            const float iv = __fdividef(1.0f, fmaxf(v, 1e-3f));
            const float bd_ot = fmaf(k11 * iv, bs, fmaf(fmaf(k12 * iv, iv, -1.0f), rs, kb1 * iv));
            const float rd_ot = fmaf(k21, bs, fmaf(k22 * iv, rs, kb2));
            const float b_use = low ? beta_kin : bs;
            const float r_use = low ? v * kappa : rs;
            const float bd = low ? 0.0f : bd_ot;
            const float rd = low ? 0.0f : rd_ot;
            float sb, cb;
            sincos_half(b_use, sb, cb);
            const float w = v * (bd + r_use);
            const float dp = move ? fmaf(r_use, ti, rd * hti2) : 0.0f;
            ax_last = fmaf(cb, acc, -sb * w);
            ay_last = fmaf(sb, acc, cb * w);
            slot.at(kSb, c, lane) = sb;
            slot.at(kCb, c, lane) = cb;
            slot.at(kDps, c, lane) = dp;
            slot.at(kAx, c, lane) = ax_last;
            slot.at(kAy, c, lane) = ay_last;
            df_add(dh, dl, dp, 0.0f);
            if (move) {
                bs = fmaf(bd, ti, b_use);
                rs = fmaf(rd, ti, r_use);
            }
        }
        // the next round starts from the state after every lane's maps
        {
            const float m00 = __shfl_sync(0xffffffffu, P.m00, 31), m01 = __shfl_sync(0xffffffffu, P.m01, 31);
            const float m10 = __shfl_sync(0xffffffffu, P.m10, 31), m11 = __shfl_sync(0xffffffffu, P.m11, 31);
            const float c0 = __shfl_sync(0xffffffffu, P.c0, 31), c1 = __shfl_sync(0xffffffffu, P.c1, 31);
            const float b2 = fmaf(m00, beta, fmaf(m01, r, c0));
            r = fmaf(m10, beta, fmaf(m11, r, c1));
            beta = b2;
        }

        // 3. heading at every sub-step start: lane sums, scanned
        float ih = dh, il = dl;
        df_scan(ih, il, lane);
        float hh = ph, hl = pl;                                       // heading at the lane's first sub-step
        {
            const float eh = __shfl_up_sync(0xffffffffu, ih, 1), el = __shfl_up_sync(0xffffffffu, il, 1);
            if (lane > 0) df_add(hh, hl, eh, el);
        }
        const float th = __shfl_sync(0xffffffffu, ih, 31), tl = __shfl_sync(0xffffffffu, il, 31);

        // 4. position increments
        float axu = __shfl_up_sync(0xffffffffu, ax_last, 1), ayu = __shfl_up_sync(0xffffffffu, ay_last, 1);
        if (lane == 0) { axu = ax; ayu = ay; }
        float sxh = 0.0f, sxl = 0.0f, syh = 0.0f, syl = 0.0f;
        float sp, cp;                                  // heading trig: exact at the lane start, then rotated
        sincos2(hh, hl, sp, cp);
#pragma unroll 1
        for (int c = 0; c < csa; ++c) {
            const int n = n0 + c;
            const float sb = slot.at(kSb, c, lane), cb = slot.at(kCb, c, lane), dp = slot.at(kDps, c, lane);
            const float cpb = fmaf(cp, cb, -sp * sb);
            const float spb = fmaf(sp, cb, cp * sb);
            const float v = fmaf((float)n, dv, v0);
            const bool stop_now = n == n_stop;
            const float d_stop = v * v * stop_den;
            float dx = stop_now ? cpb * d_stop : fmaf(cpb * v, ti, fmaf(cp, axu, -sp * ayu) * hti2);
            float dy = stop_now ? spb * d_stop : fmaf(spb * v, ti, fmaf(sp, axu, cp * ayu) * hti2);
            if (n >= NK || n > n_stop) dx = dy = 0.0f;
            slot.at(kDx, c, lane) = dx;
            slot.at(kDy, c, lane) = dy;
            df_add(sxh, sxl, dx, 0.0f);
            df_add(syh, syl, dy, 0.0f);
            axu = slot.at(kAx, c, lane);
            ayu = slot.at(kAy, c, lane);
            if (dp != 0.0f) {                          // rotate (cos, sin) of the heading by the increment
                float sd, cd;
                sincos_tenth(dp, sd, cd);
                const float c2 = fmaf(cp, cd, -sp * sd);
                sp = fmaf(sp, cd, cp * sd);
                cp = c2;
            }
        }
        float ixh = sxh, ixl = sxl, iyh = syh, iyl = syl;
        df_scan2(ixh, ixl, iyh, iyl, lane);

        // 5. poses of the output steps ending in this lane's sub-steps
        float px = xh, pxl = xl, py = yh, pyl = yl;
        {
            const float eh = __shfl_up_sync(0xffffffffu, ixh, 1), el = __shfl_up_sync(0xffffffffu, ixl, 1);
            const float fh = __shfl_up_sync(0xffffffffu, iyh, 1), fl = __shfl_up_sync(0xffffffffu, iyl, 1);
            if (lane > 0) {
                df_add(px, pxl, eh, el);
                df_add(py, pyl, fh, fl);
            }
        }
        int k = n0 / K, left = K - (n0 - k * K);       // the output step in progress, its sub-steps still to do
#pragma unroll 1
        for (int c = 0; c < csa; ++c) {
            df_add(px, pxl, slot.at(kDx, c, lane), 0.0f);
            df_add(py, pyl, slot.at(kDy, c, lane), 0.0f);
            df_add(hh, hl, slot.at(kDps, c, lane), 0.0f);
            if (--left == 0) {                               // the pose stores the exact heading trig
                if (n0 + c < NK) {
                    float so, co;
                    sincos2(hh, hl, so, co);
                    const long long idx = base + (long long)k * h + i;
                    X[idx] = __fadd_rn(px, pxl);
                    Y[idx] = __fadd_rn(py, pyl);
                    C[idx] = co;
                    S[idx] = so;
                }
                left = K;
                ++k;
            }
        }

        // 6. carried into the next round
        df_add(ph, pl, th, tl);
        df_add(xh, xl, __shfl_sync(0xffffffffu, ixh, 31), __shfl_sync(0xffffffffu, ixl, 31));
        df_add(yh, yl, __shfl_sync(0xffffffffu, iyh, 31), __shfl_sync(0xffffffffu, iyl, 31));
        ax = __shfl_sync(0xffffffffu, ax_last, 31);       // used only after a full round (csa = 5)
        ay = __shfl_sync(0xffffffffu, ay_last, 31);
    }
}

// LAYOUTS: 1 every task is a warp per hypothesis, 2 every task is a thread per hypothesis, 3 both (a kernel
// holding one layout only has a smaller instruction footprint).  Bounded to 80 registers (six CTAs per SM), where the
// integration has no spills.
// table[0, n) = -1 by CTA b of nb (16-byte stores on the aligned body).
__device__ __forceinline__ void fill_part(int16_t *table, long long n, long long b, long long nb) {
    const long long tid = b * blockDim.x + threadIdx.x, stride = nb * blockDim.x;
    const long long head = min(n, (long long)((16 - ((uintptr_t)table & 15)) & 15) / 2);
    if (tid < head) table[tid] = (int16_t)-1;
    const long long body = (n - head) / 8;
    int4 *v = reinterpret_cast<int4 *>(table + head);
    const int4 ones = make_int4(-1, -1, -1, -1);
    for (long long q = tid; q < body; q += stride) v[q] = ones;
    for (long long q = head + body * 8 + tid; q < n; q += stride) table[q] = (int16_t)-1;
}

// CTAs [0, fill_blocks) write the table's -1s (HBM-bound, beside the latency-bound integration: the table is
// read by nothing before the collision kernel), then come the generation CTAs, then the risk preparation.
// The last k in [0, n) with v[k] <= x (v ascending, v[0] <= x), by the whole warp: each round the lanes
// probe 64 evenly spaced entries (two each) and keep the span between the last probe <= x and the next, so
// up to 64 entries take one round of loads.
__device__ __forceinline__ int last_le(const int *v, int n, int x, int lane) {
    int lo = 0, hi = n - 1;
    while (lo < hi) {
        const long long span = hi - lo + 1;
        const bool le0 = v[lo + (int)(span * (2 * lane) / 64)] <= x;
        const bool le1 = v[lo + (int)(span * (2 * lane + 1) / 64)] <= x;
        const unsigned even = __ballot_sync(0xffffffffu, le0), odd = __ballot_sync(0xffffffffu, le1);
        const int le = 31 - __clz(even), lo2 = odd ? 31 - __clz(odd) : -1;   // last true even / odd probe
        const int L = 2 * lo2 + 1 > 2 * le ? 2 * lo2 + 1 : 2 * le;           // the true probes form a prefix
        const int nlo = lo + (int)(span * L / 64);
        hi = L == 63 ? hi : lo + (int)(span * (L + 1) / 64) - 1;
        lo = nlo;
    }
    return lo;
}

template <int LAYOUTS>
__global__ void __launch_bounds__(128, 6) gen_kernel(const GenArgs a) {
    // wait first: launched as a dependent of the descriptor copy kernel, this kernel lets its own dependents
    // (which read descriptors before their wait) start only once the copy is complete
    pdl_wait();
    pdl_trigger();
    if ((int)blockIdx.x < a.fill_blocks) {
        fill_part(a.fill, a.n_fill, blockIdx.x, a.fill_blocks);
        return;
    }
    const int bid = (int)blockIdx.x - a.fill_blocks;
    if (bid >= a.gen_blocks) {                           // the risk preparation, independent of generation
        prepare_block(a.prep, bid - a.gen_blocks, a.prep_blocks);
        return;
    }
    int w = bid * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (w >= a.n_warps) return;                          // whole warps leave
    if (LAYOUTS == 3) w = a.n_warps - 1 - w;             // the long sequential chains start first (24 uneven scenarios:
                                                         // 0.18 ms, 0.22 when they ended the launch)
    if ((LAYOUTS & 1) && (LAYOUTS == 1 || w < a.n_scan)) {   // one hypothesis by the whole warp
        __shared__ ScanSlot slots[4];
        const int lane = threadIdx.x & 31;
        int first, obj;
        if (a.n_scan_objs <= 32) {                       // one round of loads: entry `lane` and its object
            const bool in = lane < a.n_scan_objs;
            first = in ? a.warp_first[lane] : 0x7fffffff;
            obj = in ? a.warp_obj[lane] : 0;
            const int k = 31 - __clz(__ballot_sync(0xffffffffu, first <= w));
            first = __shfl_sync(0xffffffffu, first, k);
            obj = __shfl_sync(0xffffffffu, obj, k);
        } else {
            const int k = last_le(a.warp_first, a.n_scan_objs, w, lane);
            first = a.warp_first[k];
            obj = a.warp_obj[k];
        }
        const ObjDesc &o = a.objs[obj];
        const int i = w - first;
        const int ia = i / o.n_b, ib = i - ia * o.n_b;
        const float ga = a.grids[o.grid_off + ia];
        const float gb = a.grids[o.grid_off + o.n_a + ib];
        if (o.kind == kVehicle)
            vehicle_scan(o, ga, gb, a.regimes[o.regime_off + ia], o.n_steps, o.substeps, lane, o.pose_base, o.h, i,
                         a.x, a.y, a.c, a.s, slots[threadIdx.x >> 5]);
        else
            pedestrian(o, ga, gb, o.n_steps, o.tau, o.pose_base, o.h, i, a.x, a.y, a.c, a.s, lane, 32);
        return;
    }
    if (!(LAYOUTS & 2)) return;
    if ((threadIdx.x & 31) >= a.lanes) return;
    const int e = a.n_scan_objs + (w - a.n_scan);
    const ObjDesc &o = a.objs[a.warp_obj[e]];
    const int i = a.warp_first[e] + (threadIdx.x & 31);
    if (i >= o.h) return;
    const int ia = i / o.n_b, ib = i - ia * o.n_b;
    const float ga = a.grids[o.grid_off + ia];
    const float gb = a.grids[o.grid_off + o.n_a + ib];
    if (o.kind == kVehicle && o.path_off >= 0)
        vehicle_path(o, ga, a.paths + 9LL * (o.path_off + ib), a.regimes[o.regime_off + ia], o.n_steps, o.substeps,
                     o.tau_i_d, o.pose_base, o.h, i, a.x, a.y, a.c, a.s);
    else if (o.kind == kVehicle)
        vehicle(o, ga, gb, a.regimes[o.regime_off + ia], o.n_steps, o.substeps, o.tau_i_d, o.pose_base, o.h, i,
                a.x, a.y, a.c, a.s);
    else
        pedestrian(o, ga, gb, o.n_steps, o.tau, o.pose_base, o.h, i, a.x, a.y, a.c, a.s);
}

// Bounding box of the 32 pose centres of each bound tile at each step: one warp per (32-hypothesis group,
// chunk of 8 steps).  Lane i loads hypothesis i's x and y at the chunk's 8 steps (16 loads in flight),
// then a butterfly reduce-scatter over the 32 values (step s, quantity q = x min, y min, x max, y max;
// value 4 s + q) halves the values at each of its five levels, so that lane L ends with the finished value
// L and the 8 boxes go out as one 128-byte store.  The descriptors are read before the wait for the
// generation kernel, the poses after it.  With `fill` set, the CTAs past the bounds write the table's -1s
// (16-byte stores on the aligned body) before the wait: nothing earlier in the launch sequence reads the
// table, so the HBM-rate fill overlaps the generation kernel's tail, and the collision kernel stores first
// hits only.  TILED: the tiles are taken in the objects' tile order (hypothesis_at) and the poses go out once more,
// 512 bytes per tile and step, so that the walk reads a step of a tile with one 16-byte load per lane: 35 us
// instead of 15 on the 32-vehicle scene, 0.28 ms instead of 0.11 on the 256-scenario batch (HBM: 52 and 340 MB of
// poses read and written), for collision kernels 2.9 and 5.4 ms shorter.
constexpr int kFillCtas = 152 * 4;
// Fill CTAs of the generation launch (the rest of each SM integrates).  Two per SM spread the fill's stores
// over every SM, which a table much larger than the generation work needs to reach the HBM rate (32-vehicle
// scene: 0.74 ms at two per SM, 0.94 ms at one); when the generation work is comparable, one per SM leaves it more room
// and both finish sooner (256-scenario batch: 1.69 ms, 1.78 with half as many, 1.83 with twice).
constexpr int kGenFillCtas = 152 * 2;
constexpr int kGenFillCtasShared = 152;
constexpr long long kFillPerHypothesis = 8192;   // table entries per hypothesis above which the fill dominates
constexpr int kBoundSteps = 8;          // steps per warp task

__device__ __forceinline__ float box_op(bool is_max, float u, float v) { return is_max ? fmaxf(u, v) : fminf(u, v); }

template <bool TILED>
__global__ void __launch_bounds__(256) bounds_kernel(const BoundsArgs a) {
    pdl_trigger();
    const int chunks = (a.max_steps + kBoundSteps - 1) / kBoundSteps;
    const long long total = (long long)a.n_warps * chunks;
    const int warps = blockDim.x >> 5;
    const long long bound_ctas = (total + warps - 1) / warps;
    if ((long long)blockIdx.x >= bound_ctas) {   // a fill CTA
        fill_part(a.fill, a.n_fill, (long long)blockIdx.x - bound_ctas, (long long)gridDim.x - bound_ctas);
        pdl_wait();
        return;
    }
    const long long g = (long long)blockIdx.x * warps + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    bool live = g < total;
    int k0 = 0, first = 0, h = 0, n_steps = 0, i = 0, tile = 0;
    long long pose_base = 0, bounds_base = 0;
    if (live) {
        const int w = (int)(g / chunks);
        k0 = (int)(g - (long long)w * chunks) * kBoundSteps;
        const ObjDesc &o = a.objs[a.warp_obj[w]];
        first = a.warp_first[w];
        h = o.h;
        n_steps = o.n_steps;
        pose_base = o.pose_base;
        bounds_base = o.bounds_base + (long long)(first / kBoundTile) * n_steps;
        i = first + lane;                           // past the object's end: not loaded
        tile = w;
        if (TILED && i < h) i = hypothesis_at(o, i);
    }
    pdl_wait();
    if (a.zero_counts && g == 0 && lane == 0) {
        a.zero_counts[0] = 0ull;
        a.zero_counts[1] = 0ull;
        a.zero_counts[2] = 0ull;
    }
    if (!live || k0 >= n_steps) return;             // uniform over the warp
    if (TILED && k0 == 0) a.tile_order[32LL * tile + lane] = i;
    float v[4 * kBoundSteps];                       // value 4 s + q of step k0 + s
    float cv[kBoundSteps], sv[kBoundSteps];         // the headings, for the poses in tile order
#pragma unroll
    for (int s = 0; s < kBoundSteps; ++s) {
        const bool ok = i < h && k0 + s < n_steps;
        const long long idx = pose_base + (long long)(k0 + s) * h + i;
        const float x = ok ? a.x[idx] : INFINITY, y = ok ? a.y[idx] : INFINITY;
        cv[s] = TILED && ok ? a.c[idx] : 1.0f;
        sv[s] = TILED && ok ? a.s[idx] : 0.0f;
        v[4 * s] = x;
        v[4 * s + 1] = y;
        v[4 * s + 2] = ok ? x : -INFINITY;
        v[4 * s + 3] = ok ? y : -INFINITY;
    }
    if (TILED) {
        float4 *tp = a.tile_poses + 32 * (bounds_base + k0) + lane;
#pragma unroll
        for (int s = 0; s < kBoundSteps; ++s)
            if (k0 + s < n_steps) tp[32 * s] = make_float4(i < h ? v[4 * s] : NAN, v[4 * s + 1], cv[s], sv[s]);
    }
    // levels 16, 8, 4: the kept values keep their quantity (q = index mod 4)
#pragma unroll
    for (int d = 16, n = 16; d >= 4; d >>= 1, n >>= 1) {
        const bool upper = lane & d;
#pragma unroll
        for (int j = 0; j < n; ++j) {
            const float send = upper ? v[j] : v[j + n], keep = upper ? v[j + n] : v[j];
            v[j] = box_op((j & 3) >= 2, keep, __shfl_xor_sync(0xffffffffu, send, d));
        }
    }
    {   // level 2: values q = 0, 1 (minima) or 2, 3 (maxima) kept
        const bool upper = lane & 2;
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const float send = upper ? v[j] : v[j + 2], keep = upper ? v[j + 2] : v[j];
            v[j] = box_op(upper, keep, __shfl_xor_sync(0xffffffffu, send, 2));
        }
    }
    {   // level 1
        const bool upper = lane & 1;
        const float send = upper ? v[0] : v[1], keep = upper ? v[1] : v[0];
        v[0] = box_op(lane & 2, keep, __shfl_xor_sync(0xffffffffu, send, 1));
    }
    const int s = lane >> 2;                        // lane L holds value L: step k0 + L / 4, quantity L % 4
    if (k0 + s < n_steps) {
        float *out = reinterpret_cast<float *>(a.bounds + bounds_base + k0);
        out[lane] = v[0];
    }
}

}  // namespace

cudaError_t launch_generate(const GenArgs &args, cudaStream_t st, bool pdl) {
    GenArgs a = args;
    if (a.n_warps <= 0 && a.prep_blocks <= 0) return cudaSuccess;
    // few warps: one warp per block so that the latency-bound integration spreads over all SMs; the
    // preparation CTAs (if any) then have 128 threads as well
    const int warps_per_block = a.n_warps < 4 * 152 ? 1 : 4;
    a.gen_blocks = (a.n_warps + warps_per_block - 1) / warps_per_block;
    const long long hyps = (long long)a.n_scan + (long long)(a.n_warps - a.n_scan) * a.lanes;
    const long long cap = a.n_fill > kFillPerHypothesis * std::max(1LL, hyps) ? kGenFillCtas : kGenFillCtasShared;
    a.fill_blocks = a.fill && a.n_fill > 0 ? (int)std::min(cap, (a.n_fill / 8 + 127) / 128 + 1) : 0;
    const long long blocks = (long long)a.fill_blocks + a.gen_blocks + (a.prep_blocks > 0 ? a.prep_blocks : 0);
    if (blocks > 0x7fffffffLL) return cudaErrorInvalidValue;
    auto kernel = a.n_scan >= a.n_warps ? gen_kernel<1> : (a.n_scan <= 0 ? gen_kernel<2> : gen_kernel<3>);
    return launch_kernel(kernel, dim3((unsigned)blocks), dim3(32 * warps_per_block), 0, st, pdl, a);
}

cudaError_t launch_bounds(const BoundsArgs &a, cudaStream_t st, bool pdl) {
    const long long total = (long long)a.n_warps * ((a.max_steps + kBoundSteps - 1) / kBoundSteps);
    if (total <= 0) return cudaSuccess;
    const int warps = total < 152 * 8 ? 2 : 8;       // few tasks: spread over the SMs (11 objects: 1 us less than 8)
    long long blocks = (total + warps - 1) / warps;
    if (a.fill && a.n_fill > 0) blocks += std::min((long long)kFillCtas * 8 / warps, (a.n_fill / 8 + 32 * warps - 1) / (32 * warps) + 1);
    if (blocks > 0x7fffffffLL) return cudaErrorInvalidValue;
    return a.tile_poses ? launch_kernel(bounds_kernel<true>, dim3((unsigned)blocks), dim3(32 * warps), 0, st, pdl, a)
                        : launch_kernel(bounds_kernel<false>, dim3((unsigned)blocks), dim3(32 * warps), 0, st, pdl, a);
}

}  // namespace mhc
