// cull_constants.h -- the per-(instance, view) constants of the conservative cull.
#pragma once
#include <cmath>

#include "device.cuh"

namespace curast {

__host__ __device__ inline double larger(double a, double b) { return a < b ? b : a; }
__host__ __device__ inline double smaller(double a, double b) { return b < a ? b : a; }

// Constants of the conservative tiny-triangle cull of one (instance, view).
// The estimate X'_f = (fn_x . p) / (fn_w . p) uses FMA rows and an
// approximate reciprocal; the exact path is the FP32 sequence of the
// projection (Eq. 2) and the snap.  Forward error analysis of both, with
// S_r = sum_j |m_rj a_j| + |m_r3| (a_j the largest |coordinate| of the mesh
// bounds), bounds their distance by max(1/w) (ka + kb |X'|) + kc |X'| + kd
// pixels (the terms are listed below).  wsafe keeps the exact depth of every
// vertex above the near plane.
// Runs on the host for the context's frames and on the device for the call
// that has no bounds until its own kernels find them; both give the same bits
// (double arithmetic without contraction).
__host__ __device__ inline void cull_constants(PairDev &p, bool bounded, const double (&lo)[3], const double (&hi)[3],
                                               const ViewDev &v) {
    for (int j = 0; j < 12; ++j) p.fn[j] = 0.0f;
    for (int j = 0; j < 4; ++j) p.fk[j] = 0.0f;
    for (int j = 0; j < 3; ++j) p.fs[j] = 0.0f;
    p.nlo = -INFINITY;
    p.wsafe = INFINITY;
    p.win = 0.0f;
    if (!bounded) return;
    // u: FP32 unit roundoff; rho: relative error assumed for rcp.approx.ftz.f32
    // (8x the documented one ulp)
    const double u = 0x1p-24, rho = 0x1p-20;
    double amax[3], S[3];
    for (int j = 0; j < 3; ++j) amax[j] = larger(fabs(lo[j]), fabs(hi[j]));
    for (int r = 0; r < 3; ++r) {
        S[r] = fabs((double)p.mv[4 * r + 3]);
        for (int j = 0; j < 3; ++j) S[r] += fabs((double)p.mv[4 * r + j]) * amax[j];
    }
    const double hw = v.hw, hh = v.hh, fx = v.fx, fy = v.fy;
    const double ax = hw * fx, bx = hw - 0.5, ay = hh * fy, by = hh - 0.5;
    for (int j = 0; j < 4; ++j) {
        const double wr = -(double)p.mv[8 + j];
        p.fn[j] = (float)(ax * (double)p.mv[j] + bx * wr);
        p.fn[4 + j] = (float)(ay * (double)p.mv[4 + j] + by * wr);
        p.fn[8 + j] = (float)wr;
    }
    // Near plane: the w row holds the exact path's own coefficients, negated,
    // so the FMA estimate and the exact path's w (three products and sums
    // without FMA) are each within 3.01 u S_z of the true value; a vertex
    // whose estimate lies below near - 8 u S_z is beyond the near plane in
    // the exact path, and a triangle with all three there is dropped by it.
    {
        const double nl = (double)v.nearv - 8 * u * S[2];
        float f = (float)nl;
        if ((double)f > nl) f = nextafterf(f, -INFINITY);
        p.nlo = f;
    }
    // Error budget per coordinate (pixels), exact path plus estimate:
    //   (9.002u a S_axis + 4.001u b S_z + 4.001u h S_z + 7.002u (|X'| + 1) S_z) / w
    //   + (|X'| + 1)(rho + 7.01u) + 5.01u (h + 1) + 1/512 (the snap),
    // with 1/w <= max(1/w~) (1 + 4u S_z / wsafe) / (1 - rho) for the estimated w~.
    double ws = v.nearv * (1 + 1e-3) + 8 * u * S[2];
    const double F = 1.01 * (1 + 4 * u * S[2] / ws) / (1 - rho);
    const double kax = 9.002 * ax * S[0] + 4.001 * bx * S[2] + 4.001 * hw * S[2] + 7.002 * S[2];
    const double kay = 9.002 * ay * S[1] + 4.001 * by * S[2] + 4.001 * hh * S[2] + 7.002 * S[2];
    const double ka = F * u * larger(kax, kay);
    const double kb = F * u * 7.002 * S[2];
    const double kc = 1.01 * (rho + 7.01 * u);
    const double kd = 1.01 * (5.01 * u * (larger(hw, hh) + 1) + rho + 7.01 * u) + 1.0 / 512;
    // The test applies where w > wsafe and |X'|, |Y'| < win = 100 min(W/2,
    // H/2).  wsafe is raised until the margin stays below 20 min(W/2, H/2)
    // there (the reciprocal may read 1 + rho high), so every exact vertex of a
    // tested triangle has |X'|, |Y'| < 120 min(W/2, H/2): well inside the
    // guard band (|X - W/2| <= 128 W/2, likewise for Y), where the exact path
    // snaps it and never clips.  The bound is linear in |X'| and holds at any
    // size of the margin; a margin of many pixels only culls less.
    const double hm = smaller(hw, hh);
    const double win = 100.0 * hm;
    const double room = 20.0 * hm - kc * win - kd;
    if (!(room > 0.0)) return;
    ws = larger(ws, 1.01 * (1 + rho) * (ka + kb * win) / room);
    if (!(ka < INFINITY) || !(ws < INFINITY) || ka > 1e30 || ws > 1e30) return;
    // round the constants up (the window down) so the float copies stay conservative
    p.fk[0] = (float)(ka * (1 + 1e-6));
    p.fk[1] = (float)(kb * (1 + 1e-6));
    p.fk[2] = (float)(kc * (1 + 1e-6));
    p.fk[3] = (float)(kd * (1 + 1e-6));
    // the rows' magnitude over the mesh bounds is at most ax S_0 + bx S_2,
    // ay S_1 + by S_2 and S_2; 2^-19 of it covers the rounding of the group
    // test's box arithmetic (centre, half extent, row sums: a few u each)
    p.fs[0] = (float)((0x1p-19 * (ax * S[0] + bx * S[2])) * (1 + 1e-6));
    p.fs[1] = (float)((0x1p-19 * (ay * S[1] + by * S[2])) * (1 + 1e-6));
    p.fs[2] = (float)((0x1p-19 * (S[2])) * (1 + 1e-6));
    p.wsafe = (float)(ws * (1 + 1e-6));
    p.win = (float)win;
}

}  // namespace curast
