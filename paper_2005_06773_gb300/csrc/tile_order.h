// tile_order.h -- the order of an object's hypotheses in its collision tiles (host only, plain C++).
#pragma once
#include <algorithm>
#include <cmath>

#include "mhc.h"

namespace mhc {
namespace host {

// How an object's hypotheses lie in space t seconds ahead: the distance of neighbours along grid_a and along grid_b.
// Vehicles: da t^2 / 2 and, for steering angles, v^2 db t^2 / (2 L); path hypotheses: the paths' mean distance at
// their last section.  Pedestrians: da t for speeds (da t^2 / 2 for accelerations) and speed x heading step x t.
inline void neighbour_distance(const mhc_object &o, double t, double &along_a, double &along_b) {
    float a_lo = o.grid_a[0], a_hi = a_lo, b_lo = o.grid_b[0], b_hi = b_lo;
    for (int q = 1; q < o.n_a; ++q) { a_lo = std::min(a_lo, o.grid_a[q]); a_hi = std::max(a_hi, o.grid_a[q]); }
    for (int q = 1; q < o.n_b; ++q) { b_lo = std::min(b_lo, o.grid_b[q]); b_hi = std::max(b_hi, o.grid_b[q]); }
    const double da = o.n_a > 1 ? ((double)a_hi - a_lo) / (o.n_a - 1) : 0.0;
    const double db = o.n_b > 1 ? ((double)b_hi - b_lo) / (o.n_b - 1) : 0.0;
    const double far = std::max(std::fabs((double)a_lo), std::fabs((double)a_hi));
    if (o.kind == MHC_VEHICLE && o.paths) {
        const float *p = o.paths + 6, *q = o.paths + 9LL * (o.n_b - 1) + 6;
        along_b = o.n_b > 1 ? std::hypot((double)q[0] - p[0], (double)q[1] - p[1]) / (o.n_b - 1) : 0.0;
    } else if (o.kind == MHC_VEHICLE) {
        along_b = (double)o.v0 * o.v0 * db * t * t / (2.0 * 2.7);
    } else {
        along_b = (o.flags & MHC_PED_ACCEL_GRID ? 0.5 * far * t : far) * db * t;
    }
    along_a = o.kind == MHC_PEDESTRIAN && !(o.flags & MHC_PED_ACCEL_GRID) ? da * t : 0.5 * da * t * t;
}

// The order of an object's hypotheses in its collision tiles (hypothesis_at): strips of w grid_b values, such that
// a tile of w x 32 / w hypotheses is about as long as it is wide: w^2 = 32 along_a / along_b, doubled because braking
// hypotheses fan out less than along_b says (11 objects: w = 5, where 4 to 6 leave the fewest active steps; 12 cars
// of 64 x 32: 3, best at 3 and 4).  Where even 32 grid_b values are narrow (the paper's EGO, 343 of them), strips of
// few grid_a values run along grid_b instead.  Path hypotheses keep their order (a few paths per acceleration:
// already compact).
inline int tile_order(const mhc_object &o) {
    if (o.paths || o.n_a < 2 || o.n_b < 2) return 0;
    double along_a, along_b;
    neighbour_distance(o, 1.0, along_a, along_b);
    if (!(along_a > 0.0) || !(along_b > 0.0)) return 0;
    const double w = std::sqrt(64.0 * along_a / along_b);
    if (w >= 22.0 && o.n_b > 16) return 2 * 1 + 1;         // one grid_a value per strip
    if (w >= 12.0 && o.n_b > 16) return 2 * 2 + 1;
    return 2 * std::max(1, (int)std::min((double)o.n_b, w + 0.5));   // (w passes 2^31 for a car that all but stands)
}

}  // namespace host
}  // namespace mhc
