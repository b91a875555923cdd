// pd_device.cuh -- device code shared by the multi-kernel and the persistent
// step paths: per-node phase functions (displacement update, forces) and the
// contact / wall / precision helpers they use.
#pragma once

#include <type_traits>

#include "pd_internal.h"
#include "peridem.h"

namespace pd {

// Loads of state that other blocks write in an earlier phase of the same
// persistent launch.  The persistent kernel's grid barrier orders them: every
// block fences its writes before it arrives and fences again once it has seen
// the new generation (the pattern of a cooperative grid synchronisation), so
// ordinary loads after the barrier, L1 included, see the other blocks' writes
// (the persistent-vs-graph tests compare FP64 trajectories bit for bit).
// PERSIST is kept to mark those loads.
template <bool PERSIST, class T>
__device__ __forceinline__ T ldm(const T *p) {
    return *p;
}

// ---------------------------------------------------------------------------
// contact search grid

// Square cells of side >= R_c + skin.  Each aggregate has a grid of gw x gh
// cells in row order behind its base; a cell coordinate outside the grid wraps
// around (the grid covers the wall box unless that has more than four cells per
// node).  Every pair closer than R_c + skin lies in the 3 x 3 cell block around
// either node; wrapped cells only add candidates, which the distance test
// rejects.  The three cells of a row of the block are neighbours in memory, and
// so are those of nearby nodes (a hash of the cell instead scattered every
// node's nine buckets over the whole table).
// Grid cell of a coordinate (inv_cell = 1 / cell side).  Only the
// binning kernel calls this; the force kernels read the stored cells.
__device__ __forceinline__ int cell_coord_f(float x, float inv_cell) {
    float f = floorf(x * inv_cell);
    if (!(f > -1048576.0f)) return -1048576;  // also catches NaN
    if (f > 1048576.0f) return 1048576;
    return (int)f;
}

__device__ __forceinline__ int cell_coord(double x, double origin, double inv_cell) {
    double f = floor((x - origin) * inv_cell);
    if (!(f > -1048576.0)) return -1048576;  // also catches NaN
    if (f > 1048576.0) return 1048576;
    return (int)f;
}

__device__ __forceinline__ int wrap_cell(int c, int n) {
    if ((unsigned)c < (unsigned)n) return c;
    const int r = c % n;
    return r < 0 ? r + n : r;
}
__device__ __forceinline__ int grid_cell(const AggParams &A, int cx, int cy) {
    return A.gbase + wrap_cell(cy, A.gh) * A.gw + wrap_cell(cx, A.gw);
}

// ---------------------------------------------------------------------------
// materials (Sec. 4.1): contact between bulk moduli k1, k2 uses the harmonic
// mean 2 k1 k2 / (k1 + k2) in K_n = 18 k / (pi eps_c^5); damping the harmonic
// mean of the two densities; equal values give the value itself
__device__ __forceinline__ double harmonic64(double a, double b) { return a == b ? a : 2.0 * a * b / (a + b); }
// (float: the contact stiffnesses reach 1e25, so a * b would overflow; a * (b / (a + b)) does not)
__device__ __forceinline__ float harmonic32(float a, float b) { return a == b ? a : 2.0f * a * (b / (a + b)); }

// ---------------------------------------------------------------------------
// FP64 laws

// Normal damping (Sec. 4.3, Kelvin-Voigt: -beta_d V_x V_y (v(x,y).e) e with
// beta_d = 2 r_d sqrt(K_n rho_d / V_y)) and regularised Coulomb friction
// (Sec. 4.2: slip -mu |F_r| v_perp/|v_perp| when |v_perp| > v_thr =
// mu |F_r| dt / (rho V_x), else the sticking force -(rho V_x / dt) v_perp).
// e points from x to y, (vrx, vry) = v(x) - v(y), Fr = |F_r|, Vy the partner
// volume (|S_l| for a wall); rho_d the pair's density (the harmonic mean of
// the two grains' densities), rho the density of x.  Adds to (fx, fy).
__device__ __forceinline__ void damping_friction64(const KParams &k, double Kn, double rho_d, double rho,
                                                   double ex, double ey, double vrx, double vry, double Fr, double Vx,
                                                   double Vy, double &fx, double &fy) {
    double beta = 2.0 * k.rd * sqrt(Kn * rho_d / Vy);
    double vn = vrx * ex + vry * ey;
    double cd = beta * Vx * Vy * vn;
    double Fdx = -cd * ex, Fdy = -cd * ey;
    double vtx = vrx - vn * ex, vty = vry - vn * ey;
    double vt = sqrt(vtx * vtx + vty * vty);
    double vthr = k.mu * Fr * k.dt / (rho * Vx);
    double c = (vt > vthr) ? (k.mu * Fr / vt) : (rho * Vx / k.dt);
    double Ffx = -c * vtx, Ffy = -c * vty;
    fx += Fdx + Ffx;
    fy += Fdy + Ffy;
}

// Taylor coefficients, about theta = 0, of the shape functions of the wall
// contact regions (Sec. 4.5), evaluated by the C++ front end at compile time:
//   h1(theta) / theta^3 = sum_{k>=1} H_k theta^(2k-2),
//       H_1 = 2/3, H_{k+1} = -4 H_k / ((2k+2)(2k+3))  (theta - sin theta cos theta);
//   g(theta) / theta^5 = sum_{k>=2} G_k theta^(2k-4),  G_k = a_k - b_k - e_k, the
//       terms of 3^(2k+1)/6, 4^k and 1/2 over (2k+1)! with alternating signs
//       (h1 - 2/3 sin^3 theta);
//   f(x) / x^3 = sum_{k>=1} F_k x^(2k-2),  F_1 = 1/6, F_{k+1} = -F_k / ((2k+2)(2k+3))
//       (x - sin x).
// Below theta = 0.3 (x = 0.5) nine, nine and eight terms leave a tail below
// 1e-18 of the sum.
__host__ __device__ constexpr double seg_h1_coef(int k) {
    double c = 4.0 / 6.0;
    for (int m = 1; m < k; ++m) c *= -4.0 / ((2.0 * m + 2.0) * (2.0 * m + 3.0));
    return c;
}
__host__ __device__ constexpr double seg_g_coef(int k) {
    double a = 243.0 / 6.0 / 120.0, b = 16.0 / 120.0, e = 0.5 / 120.0;
    for (int m = 2; m < k; ++m) {
        const double den = (2.0 * m + 2.0) * (2.0 * m + 3.0);
        a *= -9.0 / den;
        b *= -4.0 / den;
        e *= -1.0 / den;
    }
    return a - b - e;
}
__host__ __device__ constexpr double seg_f_coef(int k) {
    double c = 1.0 / 6.0;
    for (int m = 1; m < k; ++m) c *= -1.0 / ((2.0 * m + 2.0) * (2.0 * m + 3.0));
    return c;
}
constexpr int kSegH1Terms = 9, kSegGTerms = 9, kSegFTerms = 8;

// Horner evaluation of sum_{k=K..KMAX} C_k t2^(k-K0) with the coefficients above
// (WHICH: 0 = H, 1 = G, 2 = F), one FMA per term: a dependent chain of FMAs
// instead of the recurrence's chain of divisions, which at GB300's FP64 rate
// held a whole step back on the one node that touched a wall.
template <int WHICH, int K, int KMAX>
__device__ __forceinline__ double seg_horner(double t2) {
    constexpr double c = WHICH == 0 ? seg_h1_coef(K) : (WHICH == 1 ? seg_g_coef(K) : seg_f_coef(K));
    if constexpr (K == KMAX) return c;
    else return fma(seg_horner<WHICH, K + 1, KMAX>(t2), t2, c);
}

// Circular segment of B_R(p) beyond a line at distance d < R (Sec. 4.5).
// With theta = acos(d/R) = atan2(sqrt(R^2 - d^2), d) the paper's closed forms
// read |S| = R^2 (theta - sin theta cos theta) and
// R - |c - p| = R (h1 - 2/3 sin^3 theta) / h1; both are evaluated without
// cancellation (Taylor series in theta below 0.3), because the printed
// pi R^2/2 - R^2 asin(d/R) - d sqrt(R^2 - d^2) loses all digits as d -> R.
__device__ __forceinline__ void wall_segment_stable(double d, double R, double &area, double &gap) {
    const double y = sqrt((R - d) * (R + d));
    const double th = atan2(y, d);
    double h1, g;
    if (th < 0.3) {
        const double t2 = th * th;
        h1 = (th * t2) * seg_horner<0, 1, kSegH1Terms>(t2);
        g = (t2 * t2 * th) * seg_horner<1, 2, kSegGTerms + 1>(t2);
    } else {
        // sin and cos of the rounded angle itself: with sqrt(R^2 - d^2) / R and
        // d / R instead, the cancellation in g (about 30-fold at theta = 0.3)
        // doubles the rounding error of the gap
        double sn, cs;
        sincos(th, &sn, &cs);
        h1 = th - sn * cs;
        g = h1 - (2.0 / 3.0) * sn * sn * sn;
    }
    area = R * R * h1;
    gap = R * g / h1;
}

// Corner region S_li cap S_lj (Sec. 4.5) in the frame x -> wall i, y -> wall j:
// {x >= di, y >= dj, |.| <= R}, split into the triangle Q P1 P2 (Q = (di, dj),
// P1 = (b, dj), P2 = (di, c) on the circle) and the circular segment cut by
// the chord P1 P2, so the area and the centroid stay accurate as the corner
// point approaches the circle (the paper's polar integrals cancel there).
__device__ __forceinline__ void corner_region_stable(double di, double dj, double R, double &area, double &cx,
                                                     double &cy) {
    const double b = sqrt((R - dj) * (R + dj)), c = sqrt((R - di) * (R + di));
    const double w = (R - di) * (R + di) - dj * dj;
    const double bmi = w / (b + di), cmj = w / (c + dj);
    const double T = 0.5 * bmi * cmj;
    const double dth = atan2(b * cmj + dj * bmi, b * di + dj * c);
    double f;
    if (dth < 0.5) {
        const double t2 = dth * dth;
        f = (dth * t2) * seg_horner<2, 1, kSegFTerms>(t2);
    } else {
        f = dth - sin(dth);
    }
    const double Sg = 0.5 * R * R * f;
    const double mx = b + di, my = dj + c, ml = sqrt(mx * mx + my * my);
    const double s2 = sin(0.5 * dth);
    const double sd = (dth > 0.0) ? R * (4.0 * s2 * s2 * s2) / (3.0 * f) : R;
    const double A = Sg + T;
    area = A;
    cx = (Sg * (sd * mx / ml) + T * ((di + b + di) / 3.0)) / A;
    cy = (Sg * (sd * my / ml) + T * ((dj + dj + c) / 3.0)) / A;
}

// Wall contact (Sec. 4.5, eq:wall-repulsive, eq:wall-total) of a node at p
// with velocity v, volume Vx, contact stiffness Kn and density rho (its own
// material: a wall is rigid) against the four walls of its aggregate at
// time t (position w0 + v_w t, normal velocity v_w).  The repulsion of each
// wall uses the circular segment S_l of B_Rc(p) beyond it; corners subtract
// the S_li cap S_lj term (inclusion-exclusion); friction and damping follow by
// substituting e -> e^l, V_y -> |S_l|, p(y) -> c_l.  A node past a wall is
// treated as touching it and counted in status[PD_STATUS_PENETRATION].
//
// Distance of the node from wall l, not below 0 (the node past the wall: past).
__device__ __forceinline__ double wall_distance(const AggParams &A, int l, double t, double px, double py, bool &past) {
    const double w = A.w0[l] + A.wv[l] * t;
    const double x = l < 2 ? px : py;
    const double d = (l & 1) ? w - x : x - w;
    past = d < 0.0;
    return past ? 0.0 : d;
}
// The own-segment term of wall l at distance d.
__device__ __forceinline__ void wall_single64(const KParams &k, const AggParams &A, double Kn, double rho, int l, double d,
                                              double vx, double vy, double Vx, double &gx, double &gy) {
    gx = gy = 0.0;
    const double Rc = A.Rc;
    if (!(d < Rc)) return;
    double Ar, gap;
    wall_segment_stable(d, Rc, Ar, gap);
    if (!(Ar > 0.0) || !(gap > 0.0)) return;
    const double Fr = Kn * gap * Vx * Ar;
    const double ex = l == 0 ? -1.0 : (l == 1 ? 1.0 : 0.0), ey = l == 2 ? -1.0 : (l == 3 ? 1.0 : 0.0);
    const double wvx = (l < 2) ? A.wv[l] : 0.0, wvy = (l < 2) ? 0.0 : A.wv[l];
    gx = -Fr * ex, gy = -Fr * ey;
    damping_friction64(k, Kn, rho, rho, ex, ey, vx - wvx, vy - wvy, Fr, Vx, Ar, gx, gy);
}
// The term of corner c, (x_lo|x_hi) x (y_lo|y_hi), at distances di, dj from its walls.
__device__ __forceinline__ void wall_corner64(const KParams &k, const AggParams &A, double Kn, double rho, int c, double di,
                                              double dj, double vx, double vy, double Vx, double &gx, double &gy) {
    gx = gy = 0.0;
    const double Rc = A.Rc;
    const int i = c >> 1, j = 2 + (c & 1);
    if (!(di < Rc) || !(dj < Rc) || !(sqrt(di * di + dj * dj) < Rc)) return;
    double Ar, lx, ly;
    corner_region_stable(di, dj, Rc, Ar, lx, ly);
    if (!(Ar > 0.0)) return;
    const double cx = (i == 0 ? -1.0 : 1.0) * lx, cy = (j == 2 ? -1.0 : 1.0) * ly;
    const double cd = sqrt(cx * cx + cy * cy);
    if (!(cd < Rc) || !(cd > 0.0)) return;
    const double ux = cx / cd, uy = cy / cd;
    const double Fr = Kn * (Rc - cd) * Vx * Ar;
    gx = -Fr * ux, gy = -Fr * uy;
    damping_friction64(k, Kn, rho, rho, ux, uy, vx - A.wv[i], vy - A.wv[j], Fr, Vx, Ar, gx, gy);
}
__device__ __forceinline__ void wall_terms64(const KParams &k, const AggParams &A, double Kn, double rho, double t,
                                             double px, double py, double vx, double vy, double Vx,
                                             double (&single)[4][2], double (&corner)[4][2], int *status) {
    double d[4];
    bool near = false;
#pragma unroll
    for (int l = 0; l < 4; ++l) {
        single[l][0] = single[l][1] = corner[l][0] = corner[l][1] = 0.0;
        bool past;
        d[l] = wall_distance(A, l, t, px, py, past);
        if (past && status) atomicAdd(&status[PD_STATUS_PENETRATION], 1);
        near |= d[l] < A.Rc;
    }
    if (!near) return;
    for (int l = 0; l < 4; ++l) wall_single64(k, A, Kn, rho, l, d[l], vx, vy, Vx, single[l][0], single[l][1]);
    for (int c = 0; c < 4; ++c)
        wall_corner64(k, A, Kn, rho, c, d[c >> 1], d[2 + (c & 1)], vx, vy, Vx, corner[c][0], corner[c][1]);
}

// Wall force on a node at (px, py) with velocity (vx, vy) and volume Vx:
// eq:wall-total, the walls' own segments in order minus the corner terms.
__device__ __forceinline__ void wall_force64(const KParams &k, const AggParams &A, double Kn, double rho, double t,
                                             double px, double py, double vx, double vy, double Vx, double &Fx_out,
                                             double &Fy_out, int *status) {
    double single[4][2], corner[4][2];
    wall_terms64(k, A, Kn, rho, t, px, py, vx, vy, Vx, single, corner, status);
    double Fx = 0.0, Fy = 0.0;
#pragma unroll
    for (int l = 0; l < 4; ++l) {
        Fx += single[l][0];
        Fy += single[l][1];
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        Fx -= corner[c][0];
        Fy -= corner[c][1];
    }
    Fx_out = Fx;
    Fy_out = Fy;
}

// ---------------------------------------------------------------------------
// float-float helpers of the FP32-split path

__device__ __forceinline__ void two_prod(float a, float b, float &p, float &e) {
    p = __fmul_rn(a, b);
    e = fmaf(a, b, -p);
}

__device__ __forceinline__ void two_sum(float a, float b, float &s, float &e) {
    s = __fadd_rn(a, b);
    float bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

// |d|^2 of d = (dxh + dxl, dyh + dyl) as a float-float pair (hi, lo).  The low
// parts are not small against one ulp of the high parts (they carry the
// position bits below the float grid of the box coordinates), so the square
// keeps dxl^2 + dyl^2 as well as the cross terms.
__device__ __forceinline__ void len2_ff(float dxh, float dxl, float dyh, float dyl, float &hi, float &lo) {
    float px, ex, py, ey, s, es;
    two_prod(dxh, dxh, px, ex);
    two_prod(dyh, dyh, py, ey);
    two_sum(px, py, s, es);
    float r = es + (ex + ey) + (2.f * (dxh * dxl + dyh * dyl) + (dxl * dxl + dyl * dyl));
    hi = __fadd_rn(s, r);
    lo = __fsub_rn(r, __fsub_rn(hi, s));
}

// (ah + al) - (bh + bl) rounded to float; the high-part difference is exact
// when the two values are within a factor of two of each other.
__device__ __forceinline__ float ff_diff(float ah, float al, float bh, float bl) {
    return __fsub_rn(ah, bh) + (al - bl);
}

// Square root and reciprocal of the bond loop by the approximate special-function
// instructions (relative error about 2^-22) instead of the correctly rounded
// sequences: the FP32-split bond force carries a 1e-5 tolerance, and stretches
// within 1e-4 of the critical one are re-decided in FP64 after the loop, so
// the break decisions do not change.  The flush-to-zero forms are one
// instruction each; the others scale subnormal operands, which take lattices
// finer than 1e-12 m to occur.
__device__ __forceinline__ float sqrt_approx(float x) {
    float r;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float rcp_approx(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

__device__ __forceinline__ void damping_friction32(float rd, float Kn, float rho_d, float rho, float dt, float mu,
                                                   float ex, float ey, float vrx, float vry, float Fr, float Vx,
                                                   float Vy, float &fx, float &fy) {
    // sqrt(K_n) sqrt(rho_d / V_y): K_n of GPa-range materials (~1e28) times a
    // density over a node volume would overflow float
    float beta = 2.0f * rd * sqrtf(Kn) * sqrtf(rho_d / Vy);
    float vn = vrx * ex + vry * ey;
    float cd = beta * Vx * Vy * vn;
    float vtx = vrx - vn * ex, vty = vry - vn * ey;
    float vt = sqrtf(vtx * vtx + vty * vty);
    float vthr = mu * Fr * dt / (rho * Vx);
    float c = (vt > vthr) ? (mu * Fr / vt) : (rho * Vx / dt);
    fx += -cd * ex - c * vtx;
    fy += -cd * ey - c * vty;
}

// Float Horner evaluation of the wall-region series (coefficients as above).
template <int WHICH, int K, int KMAX>
__device__ __forceinline__ float seg_horner_f(float t2) {
    constexpr float c = (float)(WHICH == 0 ? seg_h1_coef(K) : (WHICH == 1 ? seg_g_coef(K) : seg_f_coef(K)));
    if constexpr (K == KMAX) return c;
    else return fmaf(seg_horner_f<WHICH, K + 1, KMAX>(t2), t2, c);
}

// Wall force of the FP32-split path (Sec. 4.5, eq:wall-total): the same terms
// as wall_force64, with the single-wall segments in float.  Each wall distance
// d is formed in FP64 and the segment is evaluated from R_c - d and R_c + d,
// each rounded once to float, so the small-angle quantities keep float's
// relative precision (the gap to about 1e-6 relative).  The small-angle series
// covers theta < 0.6 (six and eight terms leave a tail below 1e-8), where
// the closed form's cancellation in g stays below tenfold.  A node within R_c
// of a corner takes the FP64 terms.  Knf, rhof: the node's own contact
// stiffness and density as floats; Kn, rho, V: the same in FP64.
__device__ __forceinline__ void wall_force32(const KParams &k, const AggParams &A, float Knf, float rhof, double Kn,
                                             double rho, double t, double px, double py, double vx, double vy,
                                             double V, double &Fx_out, double &Fy_out, int *status) {
    const double Rc = A.Rc;
    double d[4];
    d[0] = px - (A.w0[0] + A.wv[0] * t);
    d[1] = (A.w0[1] + A.wv[1] * t) - px;
    d[2] = py - (A.w0[2] + A.wv[2] * t);
    d[3] = (A.w0[3] + A.wv[3] * t) - py;
    bool near = false, corner = false;
#pragma unroll
    for (int l = 0; l < 4; ++l) near |= d[l] < Rc;
    if (!near) {
        Fx_out = Fy_out = 0.0;
        return;
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const double di = fmax(d[c >> 1], 0.0), dj = fmax(d[2 + (c & 1)], 0.0);
        corner |= di * di + dj * dj < Rc * Rc;
    }
    if (corner) {
        wall_force64(k, A, Kn, rho, t, px, py, vx, vy, V, Fx_out, Fy_out, status);
        return;
    }
    const float Rf = (float)Rc, Vx = (float)V, rd = k.rdf, dt = k.dtf, mu = k.muf;
    float Fx = 0.f, Fy = 0.f;
#pragma unroll
    for (int l = 0; l < 4; ++l) {
        if (d[l] < 0.0) {
            if (status) atomicAdd(&status[PD_STATUS_PENETRATION], 1);
            d[l] = 0.0;
        }
        if (!(d[l] < Rc)) continue;
        const float e = (float)(Rc - d[l]), sp = (float)(Rc + d[l]), df = (float)d[l];
        const float y = sqrtf(e * sp);
        const float th = atan2f(y, df);
        float h1, g;
        if (th < 0.6f) {
            const float t2 = th * th;
            h1 = (th * t2) * seg_horner_f<0, 1, 6>(t2);
            g = (t2 * t2 * th) * seg_horner_f<1, 2, 9>(t2);
        } else {
            float sn, cs;
            sincosf(th, &sn, &cs);
            h1 = th - sn * cs;
            g = h1 - (2.0f / 3.0f) * sn * sn * sn;
        }
        const float Ar = Rf * Rf * h1, gap = Rf * g / h1;
        // (a region below 1e-30 R_c^2 carries no force float can represent)
        if (!(h1 > 1e-30f) || !(gap > 0.f)) continue;
        const float Fr = ((Knf * gap) * Vx) * Ar;
        const float ex = (l == 0) ? -1.f : (l == 1 ? 1.f : 0.f), ey = (l == 2) ? -1.f : (l == 3 ? 1.f : 0.f);
        const float vrx = (float)(vx - ((l < 2) ? A.wv[l] : 0.0)), vry = (float)(vy - ((l < 2) ? 0.0 : A.wv[l]));
        float gx = -Fr * ex, gy = -Fr * ey;
        damping_friction32(rd, Knf, rhof, rhof, dt, mu, ex, ey, vrx, vry, Fr, Vx, Ar, gx, gy);
        Fx += gx;
        Fy += gy;
    }
    Fx_out = (double)Fx;
    Fy_out = (double)Fy;
}

// ---------------------------------------------------------------------------
// plain FP64 path on GB300's narrow FP64 pipe
//
// GB300 issues FP64 at 2 lanes per SM cycle, against 64 for 32-bit integer and
// 128 for FP32 arithmetic.  The FP64 bond loop therefore keeps in FP64 only the
// operations whose rounding the stretch s = (L - |xi|) / |xi| depends on (the
// coordinate differences, |d|^2 and L - |xi|, which cancels), takes the correctly
// rounded L = sqrt(|d|^2) from integer and FP32 arithmetic, and forms the rest of
// the bond force in float-float arithmetic (about 2^-47 relative), far inside the
// 1e-12 per-step force tolerance of the path.

// Float-float (hi + lo) of a double from its bits: hi holds the top 24
// significand bits, lo the next 24 (the last five are dropped: 2^-48 relative).
// Integer operations and one conversion of a 24-bit integer, no FP64
// instruction.  Magnitudes below 2^-79 lose lo, below 2^-126 become 0; beyond
// the float range, inf and NaN are carried as inf or NaN.  Without branches, so
// that the chains of several bonds interleave (see bond_terms64).
__device__ __forceinline__ void dbl_to_ff(double x, float &hi, float &lo) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const unsigned sign = (unsigned)(b >> 32) & 0x80000000u;
    const int e = (int)((b >> 52) & 0x7FF);
    const unsigned long long m = b & 0xFFFFFFFFFFFFFull;
    // fraction bits 28..5 carry the weight 2^(e - 1023 - 47)
    const float scale = e > 943 ? __uint_as_float((unsigned)(e - 943) << 23) : 0.f;
    const float h = __uint_as_float(sign | ((unsigned)(e - 896) << 23) | (unsigned)(m >> 29));
    const float l = __uint_as_float(sign | __float_as_uint(__uint2float_rn((unsigned)(m >> 5) & 0xFFFFFFu) * scale));
    const float big = e == 2047 && m ? __int_as_float(0x7FC00000) : __uint_as_float(sign | 0x7F800000u);
    const float off = e < 897 ? 0.f : big;
    const bool in = (unsigned)(e - 897) <= 1150u - 897u;
    hi = in ? h : off;
    lo = in ? l : off;
}

// Correctly rounded (to nearest) square root of a positive normal double, in
// integer and FP32 arithmetic.  With x = M 2^(E - 52), M the 53-bit significand,
// let N = M 2^(52 + (E & 1)); then sqrt(x) = sqrt(N) 2^(floor(E / 2) - 52) with
// sqrt(N) in [2^52, 2^53), and the result's significand is Q = round(sqrt(N)).
//  1. y = sqrt(A), A = N 2^-104 in [1, 4): the FP32 reciprocal square root, one
//     FP32 Newton step, then one Newton step with the float-float residual
//     A - y^2 (relative error below 2^-44): Y = y 2^52 is within 2^9 of sqrt(N).
//  2. Newton's correction in integers: Q = Y + round((N - Y^2) / (2 Y)), with the
//     residual exact in 128 bits (|N - Y^2| < 2^63) and its top bits converted,
//     leaves |Q - sqrt(N)| < 1.
//  3. Exact decision from R = N - Q^2 (|R| < 2^55): Q - 1 if R < 0 (then
//     R += 2 Q - 1), and round up when R > Q, since (Q + 1/2)^2 = Q^2 + Q + 1/4
//     and sqrt(N) is never a half-integer.
// The result equals the IEEE square root (checked against the hardware's on
// random inputs by pd_check_sqrt).
__device__ __forceinline__ double sqrt_rn_int(double x) {
    const unsigned long long D = (unsigned long long)__double_as_longlong(x);
    const bool same = D == 0ull || (D >> 52) >= 0x7FFull;   // 0, inf, NaN (negative inputs do not occur)
    const int E = (int)(D >> 52) - 1023;
    const unsigned long long M = (D & 0xFFFFFFFFFFFFFull) | (1ull << 52);
    const int odd = E & 1;
    const int eL = (E - odd) / 2;
    // A = M 2^(odd - 52) as a float-float: the top 24 bits and the remaining 29
    const float a_hi = __uint_as_float(((unsigned)(127 + odd) << 23) | (unsigned)((M >> 29) & 0x7FFFFFu));
    const float a_lo = __uint2float_rn((unsigned)(M & 0x1FFFFFFFu)) * __uint_as_float((unsigned)(75 + odd) << 23);
    float r;
    asm("rsqrt.approx.f32 %0, %1;" : "=f"(r) : "f"(a_hi));
    r = r * fmaf(-0.5f * a_hi, r * r, 1.5f);
    const float y0 = a_hi * r;
    float p, pe;
    two_prod(y0, y0, p, pe);
    const float res = (__fsub_rn(a_hi, p) - pe) + a_lo;     // A - y0^2
    const unsigned yb = __float_as_uint(y0);
    const int ey = (int)(yb >> 23) - 127;                   // -1, 0 or 1
    long long Y = (long long)((yb & 0x7FFFFFu) | 0x800000u) << (29 + ey);
    Y += (long long)__float2int_rn(res * (0.5f * r) * 4503599627370496.0f);   // + (A - y0^2) / (2 y0) 2^52
    // R = N - Y^2 in 128 bits (hi:lo)
    const unsigned long long n_lo = M << (52 + odd), n_hi = M >> (12 - odd);
    const unsigned long long yy_lo = (unsigned long long)Y * (unsigned long long)Y;
    const unsigned long long yy_hi = __umul64hi((unsigned long long)Y, (unsigned long long)Y);
    const unsigned long long r_lo = n_lo - yy_lo;
    const unsigned long long r_hi = n_hi - yy_hi - (n_lo < yy_lo ? 1ull : 0ull);
    // R / 2^32 fits 32 bits (|R| < 2^63); its dropped low bits move R / (2 Y) by < 2^-21
    // (32-bit conversions only: GB300 converts 64-bit integers at the FP64 rate)
    const float rf = __int2float_rn((int)(long long)((r_hi << 32) | (r_lo >> 32))) * 4294967296.0f;
    long long Q = Y + __float2int_rn(rf * (r * 1.1102230246251565e-16f));   // R / (2 Y), 1 / (2 Y) = r 2^-53
    long long R = (long long)(n_lo - (unsigned long long)Q * (unsigned long long)Q);
    const long long Q1 = Q - 1;
    const bool below = R < 0;
    Q = below ? Q1 : Q;
    R += below ? 2 * Q1 + 1 : 0;
    Q += R > Q ? 1 : 0;
    const double root = __longlong_as_double(((long long)(eL + 1023) << 52) + (Q - (1ll << 52)));
    return same ? x : root;
}

// float-float arithmetic (Dekker / Knuth error-free transformations with FMA)
struct ff {
    float hi, lo;
};
__device__ __forceinline__ ff ff_mul(ff a, ff b) {
    float p, e;
    two_prod(a.hi, b.hi, p, e);
    e = fmaf(a.hi, b.lo, fmaf(a.lo, b.hi, e));
    const float s = __fadd_rn(p, e);
    return {s, __fsub_rn(e, __fsub_rn(s, p))};
}
__device__ __forceinline__ ff ff_add(ff a, ff b) {
    float s, e;
    two_sum(a.hi, b.hi, s, e);
    e += a.lo + b.lo;
    const float h = __fadd_rn(s, e);
    return {h, __fsub_rn(e, __fsub_rn(h, s))};
}
// 1 / a to about 2^-46 relative: the approximate reciprocal and two Newton
// steps x + x (1 - a x) with the residual formed in float-float.
__device__ __forceinline__ ff ff_rcp(ff a) {
    float x;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(x) : "f"(a.hi));
    float t = fmaf(-a.hi, x, 1.0f) - a.lo * x;
    x = fmaf(x, t, x);
    t = fmaf(-a.hi, x, 1.0f) - a.lo * x;
    const float c = x * t;
    const float h = __fadd_rn(x, c);
    return {h, __fsub_rn(c, __fsub_rn(h, x))};
}
__device__ __forceinline__ ff to_ff(double x) {
    ff r;
    dbl_to_ff(x, r.hi, r.lo);
    return r;
}

// Exact widening of a float to a double by bit operations: a conversion
// instruction occupies GB300's 2-lane FP64 pipe like an FP64 operation.
// Subnormal floats become zero; inf and NaN stay inf and NaN.
__device__ __forceinline__ double f2d_bits(float f) {
    const unsigned b = __float_as_uint(f);
    const unsigned e = (b >> 23) & 0xFFu;
    const unsigned long long sign = (unsigned long long)(b >> 31) << 63;
    if (e == 0u) return __longlong_as_double((long long)sign);
    const unsigned long long ed = e == 255u ? 2047ull : (unsigned long long)(e + 896u);
    return __longlong_as_double((long long)(sign | (ed << 52) | ((unsigned long long)(b & 0x7FFFFFu) << 29)));
}
// The float part of a double's float-float split (its top 24 significand bits).
__device__ __forceinline__ float d2f_hi_bits(double x) {
    float hi, lo;
    dbl_to_ff(x, hi, lo);
    return hi;
}

// ---------------------------------------------------------------------------
// per-node phases

// The persistent kernel's current displacement and positions: the buffers of
// its step's parity, set by thread 0 of every block at the start of the step
// (one kernel body serves both parities).
__shared__ double2 *s_cur_u;
__shared__ float4 *s_cur_pq;
// Likewise its time, its wall cells and the word its rebuild test raises.
__shared__ double s_cur_t;
__shared__ int4 *s_cur_wall;
__shared__ int *s_raise;

// Current displacement / positions of the kernel: the device pointers' own on
// the multi-kernel path (the host sets them per launch), the persistent
// kernel's per-step choice otherwise.
template <bool PERSIST>
__device__ __forceinline__ double2 *cur_u(const DevPtrs &d) {
    if constexpr (PERSIST) return s_cur_u;
    else return d.u;
}
template <bool PERSIST>
__device__ __forceinline__ float4 *cur_pq(const DevPtrs &d) {
    if constexpr (PERSIST) return s_cur_pq;
    else return d.pq;
}

// What a node's velocity and displacement update reads besides its forces.
struct Update32 {
    double2 v, u, xs;       // velocity, displacement, reference position + shift
    float4 sref;            // position at the last rebuild
    float2 a;               // previous acceleration
    int2 cell;
};

template <bool PERSIST>
__device__ __forceinline__ const int4 *cur_wall(const DevPtrs &d) {
    if constexpr (PERSIST) return s_cur_wall;
    else return d.wall_cell;
}
template <bool PERSIST>
__device__ __forceinline__ double cur_time(const DevPtrs &d) {
    if constexpr (PERSIST) return s_cur_t;
    else return *d.t_now;
}

// Shifted position xs + u of node i as a float-float pair into q_out[i], and
// the rebuild test: the displacement since the last rebuild from the float-float
// positions (error ~1e-7 of the displacement, far below the trigger's margin);
// xs, r: the node's reference position + shift and its position at the last rebuild.
__device__ __forceinline__ bool position32(const DevPtrs &d, const KParams &k, int i, double2 u, double2 xs, float4 r,
                                           float4 *q_out) {
    const double qx = xs.x + u.x, qy = xs.y + u.y;
    // float-float split by bit operations (no FP64-pipe conversions)
    float4 q;
    dbl_to_ff(qx, q.x, q.z);
    dbl_to_ff(qy, q.y, q.w);
    q_out[i] = q;
    const float ex = __fsub_rn(q.x, r.x) + (q.z - r.z), ey = __fsub_rn(q.y, r.y) + (q.w - r.w);
    return !(ex * ex + ey * ey <= k.dmax2);
}

// FP32-split displacement update of node i (Algorithm 1): u += dt v + dt^2/2 a
// with the FP32 acceleration widened exactly, written to u_out, and its shifted
// position as a float-float pair to q_out; true when the node has moved
// kSkinTrigger * skin since the last rebuild.  The persistent kernel's velocity
// update calls it for the next step with the same operands that the update
// phase would load, so both give the same bits.
__device__ __forceinline__ bool advance_node32(const DevPtrs &d, const KParams &k, int i, double2 u, double2 v,
                                               float ax, float ay, double2 xs, float4 r, double2 *u_out,
                                               float4 *q_out) {
    u.x = fma(k.dt, v.x, fma(k.half_dt2, f2d_bits(ax), u.x));
    u.y = fma(k.dt, v.y, fma(k.half_dt2, f2d_bits(ay), u.y));
    u_out[i] = u;
    return position32(d, k, i, u, xs, r, q_out);
}

// Algorithm 1: u <- u + dt v + dt^2/2 a (when advancing) and the positions.
// Returns true when the node has moved farther than kSkinTrigger * skin since
// the last rebuild of the candidate lists (or its position is not finite).
//  * FP64 path: p = X + u in FP64, every operation rounded as written (no FMA).
//  * FP32 split: u advances in FP64 with fused multiply-adds; the shifted
//    position q = (X + shift) + u is kept only as a float-float pair (the FP64
//    p is formed where it is needed: walls, near-threshold bonds, readout).
//    GB300 issues FP64 at 2 lanes per SM cycle, so the node update is written
//    with as few FP64 operations as the FP64 state allows.
// With advance, u^(n-1) is read from ub[vin] and u^n written to d.u
// (= ub[vin ^ 1]); without, only the positions of d.u.
template <bool PERSIST>
__device__ __forceinline__ bool predict_node(const DevPtrs &d, const KParams &k, int i, int vin, int advance) {
    double2 *const uc = cur_u<PERSIST>(d);
    double2 u = advance ? ldm<PERSIST>(&d.ub[vin][i]) : ldm<PERSIST>(&uc[i]);
    const float dmax2 = k.dmax2;
    if (d.pq) {
        const double2 xs = __ldg(&d.xs[i]);
        const float4 r = ldm<PERSIST>(&d.sref[i]);
        if (advance) {
            const double2 v = ldm<PERSIST>(&d.v[vin][i]);
            const float2 a = ldm<PERSIST>(&d.af[i]);       // FP32 acceleration, widened exactly
            return advance_node32(d, k, i, u, v, a.x, a.y, xs, r, uc, cur_pq<PERSIST>(d));
        }
        return position32(d, k, i, u, xs, r, cur_pq<PERSIST>(d));
    }
    if (advance) {
        // explicit round-to-nearest operations: never contracted into FMAs
        const double2 v = ldm<PERSIST>(&d.v[vin][i]), a = ldm<PERSIST>(&d.a[i]);
        u.x = __dadd_rn(__dadd_rn(u.x, __dmul_rn(k.dt, v.x)), __dmul_rn(k.half_dt2, a.x));
        u.y = __dadd_rn(__dadd_rn(u.y, __dmul_rn(k.dt, v.y)), __dmul_rn(k.half_dt2, a.y));
        uc[i] = u;
    }
    const double2 X = __ldg(&d.X[i]);
    d.p[i] = make_double2(__dadd_rn(X.x, u.x), __dadd_rn(X.y, u.y));
    // |u - u at the last rebuild| in float: its rounding (1e-7 |u|) is far below the margin
    // (1/2 - kSkinTrigger) skin of the trigger
    const float4 r = ldm<PERSIST>(&d.sref[i]);
    const float ex = d2f_hi_bits(u.x) - r.x, ey = d2f_hi_bits(u.y) - r.y;
    return !(ex * ex + ey * ey <= dmax2);
}

// FP64 position X + u of node i (the FP32-split path does not store p).
template <bool PERSIST>
__device__ __forceinline__ double2 position64(const DevPtrs &d, int i) {
    const double2 X = __ldg(&d.X[i]), u = ldm<PERSIST>(&cur_u<PERSIST>(d)[i]);
    return make_double2(__dadd_rn(X.x, u.x), __dadd_rn(X.y, u.y));
}

// Grid cell of node i at its current position.
template <bool PERSIST>
__device__ __forceinline__ int2 node_cell(const DevPtrs &d, const AggParams &A, int i) {
    if (d.pq) {
        // FP32-split: the cell from the shifted float position (error below 1e-3
        // cell; the cells of this path are 0.4 % wider to absorb it)
        const float4 q = ldm<PERSIST>(&cur_pq<PERSIST>(d)[i]);
        return make_int2(cell_coord_f((q.x - A.oxs) + q.z, A.inv_cell_f), cell_coord_f((q.y - A.oys) + q.w, A.inv_cell_f));
    }
    const double2 p = ldm<PERSIST>(&d.p[i]);
    return make_int2(cell_coord(p.x, A.ox, A.inv_cell), cell_coord(p.y, A.oy, A.inv_cell));
}

// Rebuild, step 1: cells of the nodes i, i + stride, ... (kBinBatch of them,
// those below N), each counted into its cell; its rank there is its place in
// the counting sort.  The batch's atomics are in flight together.
constexpr int kBinBatch = 4;
template <bool PERSIST>
__device__ __forceinline__ void bin_nodes(const DevPtrs &d, const KParams &k, int i, int stride) {
    int2 c[kBinBatch];
    int key[kBinBatch], rank[kBinBatch];
#pragma unroll
    for (int m = 0; m < kBinBatch; ++m) {
        const long long at = i + (long long)m * stride;
        key[m] = -1;
        if (at >= k.N) continue;
        const AggParams &A = d.agg[__ldg(&d.g_agg[__ldg(&d.grain[at])])];
        c[m] = node_cell<PERSIST>(d, A, (int)at);
        key[m] = grid_cell(A, c[m].x, c[m].y);
    }
#pragma unroll
    for (int m = 0; m < kBinBatch; ++m)
        if (key[m] >= 0) rank[m] = atomicAdd(&d.count[key[m]], 1);
#pragma unroll
    for (int m = 0; m < kBinBatch; ++m) {
        if (key[m] < 0) continue;
        const size_t at = i + (size_t)m * stride;
        d.cell[at] = c[m];
        d.key[at] = key[m];
        d.rank[at] = rank[m];
    }
}

// L2 prefetch of a byte range, one 128-byte line per index of a grid stride g
// that counts on from range to range (a hint: it never faults, and every
// address issued lies inside the range).
__device__ __forceinline__ void prefetch_range(const void *p, size_t bytes, long long &g, long long nt) {
    const long long lines = (long long)((bytes + 127) >> 7);
    for (; g < lines; g += nt) asm volatile("prefetch.global.L2 [%0];" ::"l"((const char *)p + (g << 7)));
    g -= lines;
}

// The read-only arrays of the force phase (CSR rows, grain ids, broken-bond
// words, candidate-list lengths and first rows, bond columns, per-grain and
// per-aggregate constants) and the lines of the step counter, rebuild flag,
// status words and grid barrier, prefetched into L2 by all threads of a grid
// before the displacement update: their DRAM latency then overlaps the update
// instead of lengthening the dependent load chains that follow.  Off
// (k.pf_bonds = 0) when the arrays do not fit comfortably in L2.
__device__ __forceinline__ void prefetch_force_inputs(const DevPtrs &d, const KParams &k, long long t, long long nt) {
    if (k.pf_bonds <= 0) return;
    const size_t N = (size_t)k.N, nb = (size_t)k.pf_bonds, G = (size_t)k.G;
    long long g = t;
    prefetch_range(d.step, sizeof(long long), g, nt);
    prefetch_range(d.rebuild, sizeof(int), g, nt);
    prefetch_range(d.status, sizeof(int) * PD_STATUS_COUNT, g, nt);
    prefetch_range(d.bar, 3 * sizeof(unsigned), g, nt);
    prefetch_range(d.g_agg, 4 * G, g, nt);
    prefetch_range(d.agg, sizeof(AggParams) * (size_t)k.n_agg, g, nt);
    if (d.pq) {
        prefetch_range(d.gq, 16 * G, g, nt);
        prefetch_range(d.gc, 16 * G, g, nt);
        prefetch_range(d.g_invm, 8 * G, g, nt);
        if (k.mat) prefetch_range(d.g_kf, 4 * G, g, nt);
    } else {
        prefetch_range(d.g_cw, 8 * G, g, nt);
        prefetch_range(d.g_s0, 8 * G, g, nt);
        prefetch_range(d.g_eps, 8 * G, g, nt);
        if (k.mat) {
            prefetch_range(d.g_rho, 8 * G, g, nt);
            prefetch_range(d.g_k, 8 * G, g, nt);
        }
    }
    // (bond tiles read the stencils instead of rows and columns.  FP32 split, L2
    // flushed before every step, 89136 nodes: 31.9 us with rows and columns, 29.8.)
    const bool tiles = k.lanes == 1 && k.pair;
    if (tiles) prefetch_range(d.stn, 16 * N, g, nt);
    else prefetch_range(d.row_ptr, 4 * (N + 1), g, nt);
    prefetch_range(d.grain, 4 * N, g, nt);
    prefetch_range(d.bits, 4 * N * (size_t)k.wpn, g, nt);
    prefetch_range(d.nbr_cnt, 4 * N, g, nt);
    prefetch_range(d.nbr, 4 * N * (size_t)kPrefetchListRows, g, nt);
    if (tiles) {
        if (!d.pq) prefetch_range(d.xif, 96 * N, g, nt);
    } else if (d.pq) {
        prefetch_range(d.colx, 4 * nb, g, nt);
    } else {
        prefetch_range(d.col, 4 * nb, g, nt);
        prefetch_range(d.xi, 8 * nb, g, nt);
    }
}

// Grid cells of the four walls of every aggregate at time t (written once
// per force evaluation by the threads of one block, one aggregate each): a node
// two or more cells away from all of them is farther than R_c from every wall
// and feels no wall force.
__device__ __forceinline__ void wall_cells(const DevPtrs &d, const KParams &k, double t, int4 *out) {
    for (int a = threadIdx.x; a < k.n_agg; a += blockDim.x) {
        const AggParams &A = d.agg[a];
        out[a] = make_int4(cell_coord(A.w0[0] + A.wv[0] * t, A.ox, A.inv_cell),
                                   cell_coord(A.w0[1] + A.wv[1] * t, A.ox, A.inv_cell),
                                   cell_coord(A.w0[2] + A.wv[2] * t, A.oy, A.inv_cell),
                                   cell_coord(A.w0[3] + A.wv[3] * t, A.oy, A.inv_cell));
    }
}

// The node cell is the one of the last rebuild: the node has moved less than
// kSkinTrigger * skin since, and cells are wider than R_c + skin, so two cells
// from a wall's cell still means farther than R_c from the wall.
template <bool PERSIST>
__device__ __forceinline__ bool far_from_walls(const DevPtrs &d, int i, int ag) {
    const int2 c = ldm<PERSIST>(&d.cell[i]);
    const int4 w = ldm<PERSIST>(&cur_wall<PERSIST>(d)[ag]);
    return c.x - w.x >= 2 && w.y - c.x >= 2 && c.y - w.z >= 2 && w.w - c.y >= 2;
}

// The same test on a cell and wall-cell record already loaded.
__device__ __forceinline__ bool cells_far_from_walls(int2 c, int4 w) {
    return c.x - w.x >= 2 && w.y - c.x >= 2 && c.y - w.z >= 2 && w.w - c.y >= 2;
}

// Counting-sort scatter of the nodes i, i + stride, ... (kBinBatch of them) into
// their cells, with their position records.
template <bool PERSIST>
__device__ __forceinline__ void scatter_nodes(const DevPtrs &d, const KParams &k, int i, int stride) {
    int pos[kBinBatch];
    uint4 rec[kBinBatch];
#pragma unroll
    for (int m = 0; m < kBinBatch; ++m) {
        const long long at = i + (long long)m * stride;
        pos[m] = -1;
        if (at >= k.N) continue;
        pos[m] = ldm<PERSIST>(&d.start[ldm<PERSIST>(&d.key[at])]) + ldm<PERSIST>(&d.rank[at]);
        if (k.fp32) {
            const float4 q = ldm<PERSIST>(&cur_pq<PERSIST>(d)[at]);
            rec[m] = make_uint4(__float_as_uint(q.x), __float_as_uint(q.y), __float_as_uint(q.z), __float_as_uint(q.w));
        } else {
            const double2 p = ldm<PERSIST>(&d.p[at]);
            rec[m] = make_uint4((unsigned)__double2loint(p.x), (unsigned)__double2hiint(p.x),
                                (unsigned)__double2loint(p.y), (unsigned)__double2hiint(p.y));
        }
    }
#pragma unroll
    for (int m = 0; m < kBinBatch; ++m) {
        if (pos[m] < 0) continue;
        d.sorted[pos[m]] = (int)(i + (long long)m * stride);
        d.srec[pos[m]] = rec[m];
    }
}

// sqrt(di^2 + dj^2) of the stencil offsets (compile-time for a fixed offset)
__host__ __device__ constexpr float stn_sqrt_n(int n) {
    return n == 1 ? 1.0f : (n == 2 ? 1.41421356f : (n == 4 ? 2.0f : (n == 5 ? 2.23606798f : 2.82842712f)));
}

// Offset o (0..23) of the bond stencil: the 5 x 5 lattice block without its
// centre, in (dj, di) order.
__host__ __device__ constexpr int stn_di(int o) { return (o + (o >= 12 ? 1 : 0)) % 5 - 2; }
__host__ __device__ constexpr int stn_dj(int o) { return (o + (o >= 12 ? 1 : 0)) / 5 - 2; }

// Offset of the neighbour row dj from a stencil record.
__device__ __forceinline__ int stn_row(const uint4 &st, int dj) {
    return dj == -2 ? (int)(short)(st.y & 0xFFFFu) : (dj == -1 ? (int)(short)(st.y >> 16)
           : (dj == 0 ? 0 : (dj == 1 ? (int)(short)(st.z & 0xFFFFu) : (int)(short)(st.z >> 16))));
}
// Where the bond at offset o of node ii (it has one there) leads, as a difference
// of node numbers; gap: the node's columns tell (see kStnGap).  (Left to the
// general bond loop, these nodes and the markers that their neighbours found
// held a tile's other warps up: a box of 233k nodes with seven in a thousand at
// the edge of a hole took 68 us a step in the FP32 split and 193 in FP64, now 30
// and 118; as many nodes without holes, 25 and 88.  The tile functions come
// twice, for warps with and without such a node: a test at each bond cost 4 %.)
__device__ __forceinline__ int stn_to(const DevPtrs &d, const uint4 &st, bool gap, int ii, int o) {
    int off = stn_di(o) + stn_row(st, stn_dj(o));
    if (gap) off = __ldg(&d.col[(int)st.w + __popc(st.x & ((1u << o) - 1u))]) - ii;
    return off;
}
// Bits of the stencil's intact bonds: the broken-bond bits w follow the order
// of the node's bonds (the rank of the offset among the stencil bits), so each
// set bit clears the stencil bit of that rank (a node seldom has a broken
// bond: the loop is skipped).
__device__ __forceinline__ uint32_t stn_alive(uint32_t mask, uint32_t w) {
    uint32_t alive = mask;
    for (; w; w &= w - 1u) {
        uint32_t m = mask;
        for (int t = __ffs(w) - 1; t > 0; --t) m &= m - 1u;
        alive &= ~(m & (0u - m));
    }
    return alive;
}
// Is the node whose number differs by `delta` the partner of one of the intact
// stencil bonds?
__device__ __forceinline__ bool stn_bonded(const uint4 &st, uint32_t alive, int delta) {
    bool hit = false;
#pragma unroll
    for (int dj = -2; dj <= 2; ++dj) {
        const int di = delta - stn_row(st, dj), oo = (dj + 2) * 5 + di + 2, o = oo < 12 ? oo : oo - 1;
        if (di >= -2 && di <= 2 && oo != 12) hit |= (alive >> o) & 1u;
    }
    return hit;
}

// Is the bond i -> j (rows r0..r1) intact?  (eight columns in flight at a time:
// a search would be a chain of loads, and so were eight loads each behind its
// own bounds test, 31.5 us a step of a settled box of 19681 nodes, FP64, 4
// threads per node, now 27.7; broken flags read past L1, since other lanes may
// have just set them.  From the middle of the row outwards: pairs near enough to
// ask for are mostly lattice neighbours, and columns ascend: horizon 4 h, 19681
// nodes, a step that rebuilds the lists, FP32 split 96 to 91 us, FP64 117 to 110.)
__device__ __forceinline__ bool bonded_intact(const DevPtrs &d, const KParams &k, int i, int r0, int r1, int j) {
    const int n = (r1 - r0 + 7) >> 3;
    for (int t = 0; t < n; ++t) {
        const int b0 = r0 + 8 * ((n >> 1) + ((t & 1) ? -((t + 1) >> 1) : t >> 1));
        int c[8], hit = -1;
#pragma unroll
        for (int m = 0; m < 8; ++m) c[m] = __ldg(&d.col[min(b0 + m, r1 - 1)]);
#pragma unroll
        for (int m = 0; m < 8; ++m)
            if (c[m] == j) hit = min(b0 + m, r1 - 1) - r0;
        if (hit >= 0) return !((__ldcg(&d.bits[(size_t)i * k.wpn + (hit >> 5)]) >> (hit & 31)) & 1u);
    }
    return false;
}

// The node's bonds broken since the last rebuild, whose partners its candidate
// list leaves out: their number (any: it may have broken bonds; words read past
// L1, since its lanes may have just set them), and the partner of the m-th.
__device__ __forceinline__ uint32_t fresh_word(const DevPtrs &d, const KParams &k, int i, int w) {
    const size_t at = (size_t)i * k.wpn + w;
    return __ldcg(&d.bits[at]) & ~__ldcg(&d.bref[at]);
}
__device__ __forceinline__ int fresh_bonds(const DevPtrs &d, const KParams &k, int i, bool any) {
    int n = 0;
    if (any)
        for (int w = 0; w < k.wpn; ++w) n += __popc(fresh_word(d, k, i, w));
    return n;
}
__device__ __forceinline__ int fresh_partner(const DevPtrs &d, const KParams &k, int i, int r0, int m) {
    for (int w = 0;; ++w) {
        uint32_t b = fresh_word(d, k, i, w);
        const int n = __popc(b);
        if (m < n || w + 1 == k.wpn) {
            for (; m > 0; --m) b &= b - 1u;
            return __ldg(&d.col[r0 + 32 * w + __ffs(b) - 1]);
        }
        m -= n;
    }
}

// Rebuild, last step: the candidate list of node i -- every node y != i of
// its aggregate with |p(y) - p(i)| < R_c + skin that it has no intact bond with
// (an intact bond excludes self-contact: without this rule the nodes of every
// grain whose spacing is within 4.5 % of the smallest list their four lattice
// neighbours; bonds that break later come from their bits, see fresh_bonds) --
// gathered from the 3 x 3 block of grid cells around its cell (cells are wider
// than R_c + skin) and kept in ascending node index, and the position and the
// broken bits it was built at.  The records hold the positions in cell order,
// so only nodes inside the radius are looked up, and the bonds of a stencil
// node are told from the difference of the node numbers.
template <bool PERSIST>
__device__ __forceinline__ void build_list_node(const DevPtrs &d, const KParams &k, int i) {
    const int gi = __ldg(&d.grain[i]);
    const int2 cc = ldm<PERSIST>(&d.cell[i]);
    const int rank = ldm<PERSIST>(&d.rank[i]), key = ldm<PERSIST>(&d.key[i]);
    const uint4 st = k.stencil ? __ldg(&d.stn[i]) : make_uint4(kStnIrregular, 0u, 0u, 0u);
    const uint32_t w0 = __ldcg(&d.bits[(size_t)i * k.wpn]);
    float4 qi = make_float4(0.f, 0.f, 0.f, 0.f);
    double2 pi = make_double2(0.0, 0.0), ui = pi;
    if (d.pq) {
        qi = ldm<PERSIST>(&cur_pq<PERSIST>(d)[i]);
    } else {
        pi = ldm<PERSIST>(&d.p[i]);
        ui = ldm<PERSIST>(&cur_u<PERSIST>(d)[i]);
    }
    const AggParams &A = d.agg[__ldg(&d.g_agg[gi])];
    const int s0 = __ldg(&d.g_start[gi]), s1 = __ldg(&d.g_start[gi + 1]);
    const int own = ldm<PERSIST>(&d.start[key]) + rank;          // the node's own record
    // the block's rows, each one range of records unless it wraps around
    const int wx = wrap_cell(cc.x, A.gw);
    const bool whole = wx > 0 && wx < A.gw - 1;
    int row[3], t0[3], m[3];
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        row[r] = A.gbase + wrap_cell(cc.y + r - 1, A.gh) * A.gw;
        t0[r] = ldm<PERSIST>(&d.start[row[r] + max(wx - 1, 0)]);
        m[r] = whole ? ldm<PERSIST>(&d.start[row[r] + wx + 2]) - t0[r] : 0;
    }
    int lst[kMaxList];
    int n = 0, over = 0;
    auto inside = [&](const uint4 &rec) {
        float dx, dy;
        if (d.pq) {
            dx = (__uint_as_float(rec.x) - qi.x) + (__uint_as_float(rec.z) - qi.z);
            dy = (__uint_as_float(rec.y) - qi.y) + (__uint_as_float(rec.w) - qi.w);
        } else {
            dx = (float)(__hiloint2double((int)rec.y, (int)rec.x) - pi.x);
            dy = (float)(__hiloint2double((int)rec.w, (int)rec.z) - pi.y);
        }
        return dx * dx + dy * dy < A.rs2;
    };
    auto take = [&](int j) {
        if (j >= s0 && j < s1) {
            if (st.x & kStnIrregular) {
                if (bonded_intact(d, k, i, __ldg(&d.row_ptr[i]), __ldg(&d.row_ptr[i + 1]), j)) return;
            } else if (stn_bonded(st, stn_alive(st.x, w0), j - i)) {
                return;
            }
        }
        if (n < kMaxList) {
            int w = n++;
            while (w > 0 && lst[w - 1] > j) {
                lst[w] = lst[w - 1];
                --w;
            }
            lst[w] = j;
        } else {
            over = 1;
        }
    };
    // kListBatch records in flight together, then the node numbers of those inside
    constexpr int kListBatch = 6;
    const int tot = m[0] + m[1] + m[2];
    for (int e0 = 0; e0 < tot; e0 += kListBatch) {
        int t[kListBatch];
        uint4 rec[kListBatch];
#pragma unroll
        for (int q = 0; q < kListBatch; ++q) {
            const int e = e0 + q;
            t[q] = e < m[0] ? t0[0] + e : (e < m[0] + m[1] ? t0[1] + (e - m[0]) : t0[2] + (e - m[0] - m[1]));
            if (e >= tot || t[q] == own) t[q] = -1;
            rec[q] = ldm<PERSIST>(&d.srec[max(t[q], 0)]);
        }
        int jb[kListBatch];
#pragma unroll
        for (int q = 0; q < kListBatch; ++q) jb[q] = t[q] >= 0 && inside(rec[q]) ? ldm<PERSIST>(&d.sorted[t[q]]) : -1;
#pragma unroll
        for (int q = 0; q < kListBatch; ++q)
            if (jb[q] >= 0) take(jb[q]);
    }
    if (!whole) {
        // (a grid has at least three cells each way: the nine are different)
        for (int c = 0; c < 9; ++c) {
            const int cell = row[c / 3] + wrap_cell(cc.x + c % 3 - 1, A.gw);
            for (int t = ldm<PERSIST>(&d.start[cell]), e = ldm<PERSIST>(&d.start[cell + 1]); t < e; ++t)
                if (t != own && inside(ldm<PERSIST>(&d.srec[t]))) take(ldm<PERSIST>(&d.sorted[t]));
        }
    }
    d.bref[(size_t)i * k.wpn] = w0;
    for (int w = 1; w < k.wpn; ++w) d.bref[(size_t)i * k.wpn + w] = __ldcg(&d.bits[(size_t)i * k.wpn + w]);
    const size_t N = (size_t)k.N;
    for (int q = 0; q < n; ++q) d.nbr[q * N + i] = lst[q];
    d.nbr_cnt[i] = n;
    if (d.pq) {
        d.sref[i] = qi;
    } else {
        d.sref[i] = make_float4((float)ui.x, (float)ui.y, 0.f, 0.f);
    }
    if (over) atomicAdd(&d.status[PD_STATUS_OVERFLOW], 1);
}

// Acceleration and velocity update of node i (Algorithm 1) plus the optional
// per-part force output; run by one lane per node.  m = rho V, or with RECIP
// inv_m = 1 / (rho V): a = F (1 / m) + g and the velocity update fused, about
// one ulp of a from the quotient (the forces themselves are unchanged), for
// the two FP64 divisions per node that GB300's FP64 pipe makes costly.
template <bool PERSIST, bool RECIP = false>
__device__ __forceinline__ void finish_node(const DevPtrs &d, const KParams &k, int i, int vin, int update_v,
                                            double2 vi, double m, double Fbx, double Fby, double Fsx, double Fsy,
                                            double Fnx, double Fny, double Fwx, double Fwy, double inv_m = 0.0) {
    const double Fx = __dadd_rn(__dadd_rn(__dadd_rn(Fbx, Fsx), Fnx), Fwx);
    const double Fy = __dadd_rn(__dadd_rn(__dadd_rn(Fby, Fsy), Fny), Fwy);
    double ax, ay;
    if constexpr (RECIP) {
        ax = fma(Fx, inv_m, k.gx);
        ay = fma(Fy, inv_m, k.gy);
    } else {
        ax = __dadd_rn(__ddiv_rn(Fx, m), k.gx);
        ay = __dadd_rn(__ddiv_rn(Fy, m), k.gy);
    }
    if (update_v) {
        const double2 ao = ldm<PERSIST>(&d.a[i]);
        double2 vn;
        if constexpr (RECIP) {
            vn.x = fma(k.half_dt, ao.x + ax, vi.x);
            vn.y = fma(k.half_dt, ao.y + ay, vi.y);
        } else {
            vn.x = __dadd_rn(vi.x, __dmul_rn(k.half_dt, __dadd_rn(ao.x, ax)));
            vn.y = __dadd_rn(vi.y, __dmul_rn(k.half_dt, __dadd_rn(ao.y, ay)));
        }
        d.v[vin ^ 1][i] = vn;
    }
    d.a[i] = make_double2(ax, ay);
    if ((((unsigned)__double2hiint(ax) | 0x800FFFFFu) == 0xFFFFFFFFu) || (((unsigned)__double2hiint(ay) | 0x800FFFFFu) == 0xFFFFFFFFu))   // inf or NaN
        atomicAdd(&d.status[PD_STATUS_NONFINITE], 1);
    if (k.store) {
        d.F[i] = make_double2(Fx, Fy);
        d.parts[i] = make_double2(Fbx, Fby);
        d.parts[k.N + i] = make_double2(Fsx, Fsy);
        d.parts[2 * (size_t)k.N + i] = make_double2(Fnx, Fny);
        d.parts[3 * (size_t)k.N + i] = make_double2(Fwx, Fwy);
    }
}

// FP32-split update: the lane-summed parts are added in FP32 (their rounding is
// far below the path's force error), the wall force in FP64 where there is one;
// a = F (1 / m) + g is formed and stored in FP32 (the force carries FP32
// precision already), the velocity-Verlet increment dt/2 (a_old + a) is
// formed in FP32 and added to the FP64 velocity: two FP64 additions per node
// on GB300's narrow FP64 pipe.  (ao: the previous acceleration, loaded by the
// caller with the node's other independent loads.)
//
// The persistent kernel (PERSIST) also takes the next step's displacement
// update here, from the velocity and acceleration just formed and the node's
// current displacement ui: u and pq of the next step go to ub[vin] / pqb[vin]
// (free: this step reads ub[vin ^ 1] / pqb[vin ^ 1]), and a node past the
// rebuild trigger raises the next step's flag.  The next step then skips its
// update phase, which would have read u, v and a back from memory.
template <bool PERSIST>
__device__ __forceinline__ void finish_node32_total(const DevPtrs &d, const KParams &k, int i, int vin, int update_v,
                                                    const Update32 &n, float fx, float fy, bool walls, double Fwx,
                                                    double Fwy, float inv_m) {
    float ax, ay;
    if (walls) {
        ax = fmaf(__double2float_rn(f2d_bits(fx) + Fwx), inv_m, k.gxf);
        ay = fmaf(__double2float_rn(f2d_bits(fy) + Fwy), inv_m, k.gyf);
    } else {
        ax = fmaf(fx, inv_m, k.gxf);
        ay = fmaf(fy, inv_m, k.gyf);
    }
    if (update_v) {
        const float hdt = 0.5f * k.dtf;
        const double2 vn = make_double2(n.v.x + f2d_bits(hdt * (n.a.x + ax)), n.v.y + f2d_bits(hdt * (n.a.y + ay)));
        d.v[vin ^ 1][i] = vn;
        if constexpr (PERSIST) {
            if (advance_node32(d, k, i, n.u, vn, ax, ay, n.xs, n.sref, d.ub[vin], d.pqb[vin]))
                *(volatile int *)s_raise = 1;
        }
    }
    d.af[i] = make_float2(ax, ay);
    // finiteness from the exponent bits (no FP64 compare)
    if (((__float_as_uint(ax) | 0x807FFFFFu) == 0xFFFFFFFFu) || ((__float_as_uint(ay) | 0x807FFFFFu) == 0xFFFFFFFFu))
        atomicAdd(&d.status[PD_STATUS_NONFINITE], 1);
}

// FP64 update from the total of the lane-summed parts, T = (F_b + F_s) + F_n
// (as finish_node forms it), and the wall force: the same roundings as
// finish_node with the reciprocal mass, without the per-part output.
template <bool PERSIST>
__device__ __forceinline__ void finish_node64_total(const DevPtrs &d, const KParams &k, int i, int vin, int update_v,
                                                    double2 vi, double2 ao, double Tx, double Ty, bool walls,
                                                    double Fwx, double Fwy, double inv_m) {
    const double Fx = walls ? __dadd_rn(Tx, Fwx) : Tx, Fy = walls ? __dadd_rn(Ty, Fwy) : Ty;
    const double ax = fma(Fx, inv_m, k.gx), ay = fma(Fy, inv_m, k.gy);
    if (update_v)
        d.v[vin ^ 1][i] = make_double2(fma(k.half_dt, ao.x + ax, vi.x), fma(k.half_dt, ao.y + ay, vi.y));
    d.a[i] = make_double2(ax, ay);
    if ((((unsigned)__double2hiint(ax) | 0x800FFFFFu) == 0xFFFFFFFFu) || (((unsigned)__double2hiint(ay) | 0x800FFFFFu) == 0xFFFFFFFFu))   // inf or NaN
        atomicAdd(&d.status[PD_STATUS_NONFINITE], 1);
}

template <int LANES, class T>
__device__ __forceinline__ T lane_sum(T v) {
#pragma unroll
    for (int off = 1; off < LANES; off <<= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    return v;
}

// Bond tile: the bonds of a run of consecutive nodes, each evaluated once.
//
// The bond loop is bound by instruction issue (FP32 split) or by the FP64 pipe
// (FP64 path), and a bond's force on its two nodes differs in sign only: both
// paths' arithmetic is odd in d, so the second evaluation gives the same bits.
// With one thread per node a block therefore takes its run of nodes in tiles of
// BLOCK consecutive ones: every thread evaluates the forward half of its node's
// stencil (offsets 12..23, towards higher node indices) into shared memory,
// and after a block barrier sums its backward half from the slots of the nodes
// that evaluated it.  Nodes of a grain are numbered row by row, so those lie
// at most two lattice rows back; what a tile needs of the one before it is
// carried over (the last kCarry nodes' slots; KParams::pair says that no row
// is longer), and the first tile of a run is preceded by a pass that forms the
// slots of the kCarry nodes before the run.  Each node still adds its bonds in
// the order of the stencil, so a sum does not depend on where tiles begin and
// the results of every path and block size agree.
//
// A slot whose force was not formed holds a marker (a NaN no operation makes):
// kPairNone (no such bond in the evaluating node's list, its bonds are not
// stencil bonds, or it is broken there), kPairBroken (breaks at this
// evaluation), kPairGuard (FP32 split: in the guard band, each node decides it
// in FP64).  Any NaN sends the reader to its general loop.
constexpr unsigned kPairNone = 0x7FC0D000u, kPairBroken = 0x7FC0D001u, kPairGuard = 0x7FC0D002u;
constexpr int kPairHalf = 12;     // forward offsets of the stencil
// What a node's bond pass leaves to do: bonds in the guard band to decide, and
// that one of its bonds broke at this evaluation.
// (kNoteSeen: one of its broken-bond words has a bit; see fresh_bonds)
constexpr unsigned kNoteGuard = 1u, kNoteBroke = 2u, kNoteSeen = 4u;
template <class Slot, int BLOCK>
struct PairTile {
    static constexpr int kStride = kCarry + BLOCK;      // carried slots, then the tile's
    static constexpr int kBytes = kPairHalf * kStride * (int)sizeof(Slot);
    static_assert(kCarry <= BLOCK, "the carried slots must not overlap their source");
    static __device__ __forceinline__ void carry(Slot *slot) {
        for (int e = threadIdx.x; e < kPairHalf * kCarry; e += BLOCK) {
            const int o = e / kCarry, q = e % kCarry;
            slot[o * kStride + q] = slot[o * kStride + BLOCK + q];
        }
    }
};

// Asynchronous copies of 4, 8 or 16 bytes into the calling thread's own places
// in shared memory; commit closes a group, wait<n> returns when all but the
// last n groups of the thread have arrived.
template <class T>
__device__ __forceinline__ void copy_async(T *dst, const T *src) {
    const unsigned a = (unsigned)__cvta_generic_to_shared(dst);
    if constexpr (sizeof(T) == 16) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(a), "l"(src) : "memory");
    else asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(a), "l"(src), "n"(sizeof(T)) : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void copy_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// The broken-bond bit of offset o.
__device__ __forceinline__ uint32_t stn_bit(uint32_t mask, int o) { return 1u << __popc(mask & ((1u << o) - 1u)); }

// Whether some thread of the node's LANES says so.
template <int LANES>
__device__ __forceinline__ bool any_lane(bool v) {
    if constexpr (LANES == 1) return v;
    const unsigned all = __ballot_sync(0xffffffffu, v);
    return (all >> ((threadIdx.x & 31) / LANES * LANES)) & ((1u << LANES) - 1u);
}

// FP64 forces of node i (eq:full, Algorithm 1), LANES threads per node: lane l
// takes bonds l, l + LANES, ... and grid cells l, l + LANES, ...; partial sums
// meet in a fixed xor-butterfly (deterministic).  With LANES = 1 every sum is
// in the textbook order (bonds in CSR order, contacts in ascending index).
// Every thread of the warp must call this (shuffles); inactive lanes pass
// active = false.
// Lane-summed per-node force parts (bond, self-contact, contact), handed from
// the lanes of a node to the node's epilogue thread.
struct Sums64 {
    double bx, by, sx, sy, nx, ny;
};
struct Sums32 {
    float bx, by, sx, sy, nx, ny;
};

// One FP64 bond (eq:peri, eq:pmb, Sec. 3.1) of a node at pi towards pj with
// reference length xi: false when it breaks at this evaluation, else its force
// (fx, fy) on the node.  The stretch's cancelling difference L - |xi| is formed
// exactly as the FP64 definition rounds it: dx, dy and |d|^2 in FP64, L =
// sqrt(|d|^2) correctly rounded (integer square root), L - |xi| in FP64.  The
// quotient by |xi|, the break decision away from the threshold and the bond
// force c_w w s V_x V_y (d / L) are float-float (relative error ~1e-14; a bond
// whose stretch lies within 1e-6 of s0 is decided by the FP64 quotient).
// c = c_w w V^2 (one grain: V_y = V_x; w = 1, or 1 - |xi| / eps for the conic
// micromodulus).
//
// A bond is a chain of some 200 dependent 32-bit operations.  bond_terms64 has
// no branch, so a thread's bonds of a batch run interleaved; the rare decisions
// (near the threshold, broken) follow the batch.  (Bond tiles of 1.03M nodes
// with a branch at each special case and at each bond, the 12 bonds unrolled:
// 37% of the issue slots, a sixth of the stalls for instructions to arrive.)
__device__ __forceinline__ ff bond_conic64(ff cwVV, double xi, ff inv_eps) {
    const ff x = to_ff(xi);
    return ff_mul(cwVV, ff_add({1.0f, 0.f}, ff_mul({-x.hi, -x.lo}, inv_eps)));
}
__device__ __forceinline__ double bond_diff64(double2 pi, double2 pj, double xi, double &dx, double &dy, double &L) {
    dx = __dsub_rn(pj.x, pi.x);
    dy = __dsub_rn(pj.y, pi.y);
    L = sqrt_rn_int(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)));
    return __dsub_rn(L, xi);                                    // |xi| s, exact as in FP64
}
// The bond's force, as if it held, and the float decision: broken, and whether
// it is near the threshold and takes bond_breaks64's.
__device__ __forceinline__ void bond_terms64(double2 pi, double2 pj, double xi, ff c, float s0f, ff &fx, ff &fy,
                                             bool &broken, bool &near) {
    double dx, dy, L;
    const ff dff = to_ff(bond_diff64(pi, pj, xi, dx, dy, L)), xff = to_ff(xi);
    const float lhs = fabsf(dff.hi), rhs = s0f * xff.hi;        // |diff| > s0 |xi|
    broken = lhs > rhs;
    near = fabsf(lhs - rhs) <= 1e-6f * rhs;
    const ff t = ff_mul(ff_mul(c, dff), ff_rcp(ff_mul(xff, to_ff(L))));     // c (diff / |xi|) / L
    fx = ff_mul(t, to_ff(dx));
    fy = ff_mul(t, to_ff(dy));
}
__device__ __forceinline__ bool bond_breaks64(double2 pi, double2 pj, double xi, double s0) {
    double dx, dy, L;
    return fabs(__ddiv_rn(bond_diff64(pi, pj, xi, dx, dy, L), xi)) > s0;
}
// One bond: false when it breaks at this evaluation.
__device__ __forceinline__ bool bond_force64(double2 pi, double2 pj, double xi, ff cwVV, ff inv_eps, float s0f,
                                             double s0, int micro, ff &fx, ff &fy) {
    bool broken, near;
    bond_terms64(pi, pj, xi, micro ? bond_conic64(cwVV, xi, inv_eps) : cwVV, s0f, fx, fy, broken, near);
    if (near) broken = bond_breaks64(pi, pj, xi, s0);
    return !broken;
}

// The forward half of node ii's stencil bonds (alive: the intact ones), FP64
// path, into the thread's slots; returns the offsets whose force is there.
// own: the block owns the node and records its broken bonds.
template <bool PERSIST, int BLOCK, bool GAP>
__device__ __forceinline__ uint32_t tile_forward64(const DevPtrs &d, const KParams &k, int ii, uint32_t alive,
                                                   const uint4 &st, bool gap, double2 pi, ff cwVV, ff inv_eps,
                                                   float s0f, double s0, float4 *slot, unsigned &note, bool own) {
    constexpr int S = PairTile<float4, BLOCK>::kStride;
    const int at = kCarry + (int)threadIdx.x;
    uint32_t formed = 0u;
    constexpr int kBatch = 4;
#pragma unroll 1
    for (int m0 = 0; m0 < kPairHalf; m0 += kBatch) {
        const uint32_t live = alive >> (kPairHalf + m0);
        const auto to = [&](int m) { return ii + stn_to(d, st, GAP && gap, ii, kPairHalf + m0 + m); };
        double2 pb[kBatch];
        double xb[kBatch];
#pragma unroll
        for (int m = 0; m < kBatch; ++m) {
            pb[m] = ldm<PERSIST>(&d.p[(live >> m) & 1u ? to(m) : ii]);
            xb[m] = (live >> m) & 1u ? __ldg(&d.xif[(size_t)(m0 + m) * k.N + ii]) : 1.0;
        }
        ff c[kBatch], fx[kBatch], fy[kBatch];
        uint32_t broken = 0u, near = 0u;
#pragma unroll
        for (int m = 0; m < kBatch; ++m) c[m] = cwVV;
        if (k.micro) {
#pragma unroll
            for (int m = 0; m < kBatch; ++m) c[m] = bond_conic64(cwVV, xb[m], inv_eps);
        }
#pragma unroll
        for (int m = 0; m < kBatch; ++m) {
            bool b, n;
            bond_terms64(pi, pb[m], xb[m], c[m], s0f, fx[m], fy[m], b, n);
            broken |= (b && ((live >> m) & 1u)) ? 1u << m : 0u;
            near |= (n && ((live >> m) & 1u)) ? 1u << m : 0u;
        }
        for (; near; near &= near - 1u) {
            const int m = __ffs(near) - 1;
            const bool b = bond_breaks64(pi, ldm<PERSIST>(&d.p[to(m)]), __ldg(&d.xif[(size_t)(m0 + m) * k.N + ii]), s0);
            broken = b ? broken | (1u << m) : broken & ~(1u << m);
        }
        if (broken) {
            note |= kNoteBroke;
            for (uint32_t b = broken; own && b; b &= b - 1u)
                atomicOr(&d.bits[(size_t)ii * k.wpn], stn_bit(st.x, kPairHalf + m0 + __ffs(b) - 1));
        }
#pragma unroll
        for (int m = 0; m < kBatch; ++m) {
            const unsigned mark = !((live >> m) & 1u) ? kPairNone : ((broken >> m) & 1u) ? kPairBroken : 0u;
            slot[(m0 + m) * S + at] = make_float4(mark ? __uint_as_float(mark) : fx[m].hi, fx[m].lo, fy[m].hi, fy[m].lo);
        }
        formed |= (live & ((1u << kBatch) - 1u) & ~broken) << (kPairHalf + m0);
    }
    return formed;
}

// The bond sum of node ii, FP64 path: the backward half from the slots of the
// nodes that formed it, then the node's own forward slots.
template <bool PERSIST, int BLOCK, bool GAP>
__device__ __forceinline__ void tile_sum64(const DevPtrs &d, const KParams &k, int ii, uint32_t alive, uint32_t formed,
                                           const uint4 &st, bool gap, double2 pi, ff cwVV, ff inv_eps, float s0f,
                                           double s0, const float4 *slot, ff &Fx, ff &Fy, unsigned &note) {
    constexpr int S = PairTile<float4, BLOCK>::kStride;
    const int at = kCarry + (int)threadIdx.x;
    const uint32_t back = alive & ((1u << kPairHalf) - 1u);
    uint32_t got = 0u;
#pragma unroll
    for (int o = 0; o < kPairHalf; ++o) {
        const bool in = (back >> o) & 1u;
        const float4 v = slot[(kPairHalf - 1 - o) * S + at + (in ? stn_to(d, st, GAP && gap, ii, o) : 0)];
        const bool ok = in && v.x == v.x;
        if (ok) got |= 1u << o;
        Fx = ff_add(Fx, ok ? ff{-v.x, -v.y} : ff{0.f, 0.f});
        Fy = ff_add(Fy, ok ? ff{-v.z, -v.w} : ff{0.f, 0.f});
    }
    if (back != got) {
        // some slot holds a marker: the half again, in order
        Fx = Fy = {0.f, 0.f};
        for (uint32_t m = back; m; m &= m - 1u) {
            const int o = __ffs(m) - 1;
            const int off = stn_to(d, st, GAP && gap, ii, o);
            const float4 v = slot[(kPairHalf - 1 - o) * S + at + off];
            unsigned mark = __float_as_uint(v.x);
            if (mark == kPairNone) {
                ff fx, fy;
                const int b = (int)st.w + __popc(st.x & ((1u << o) - 1u));
                if (bond_force64(pi, ldm<PERSIST>(&d.p[ii + off]), __ldg(&d.xi[b]), cwVV, inv_eps, s0f, s0, k.micro,
                                 fx, fy)) {
                    Fx = ff_add(Fx, fx);
                    Fy = ff_add(Fy, fy);
                    continue;
                }
                mark = kPairBroken;
            }
            if (mark == kPairBroken) {
                atomicOr(&d.bits[(size_t)ii * k.wpn], stn_bit(st.x, o));
                note |= kNoteBroke;
                continue;
            }
            Fx = ff_add(Fx, ff{-v.x, -v.y});
            Fy = ff_add(Fy, ff{-v.z, -v.w});
        }
    }
#pragma unroll
    for (int o = kPairHalf; o < 2 * kPairHalf; ++o) {
        const float4 v = slot[(o - kPairHalf) * S + at];
        const bool ok = (formed >> o) & 1u;
        Fx = ff_add(Fx, ok ? ff{v.x, v.y} : ff{0.f, 0.f});
        Fy = ff_add(Fy, ok ? ff{v.z, v.w} : ff{0.f, 0.f});
    }
}

// Contact force of candidate j on node ii, FP64 path: self-contact (Sec. 4.4)
// into fs, inter-grain contact (Secs. 4.1-4.3) into fn, zero beyond R_c.
template <bool PERSIST>
__device__ __forceinline__ void contact_pair64(const DevPtrs &d, const KParams &k, const AggParams &A, int ii, int j,
                                               int vin, int gi, int r0, int r1, double2 pi, double2 pj, double2 vi,
                                               double &fsx, double &fsy, double &fnx, double &fny) {
    fsx = fsy = fnx = fny = 0.0;
    const double Rc = A.Rc;
    // |d|^2 above R_c^2 (1 + 1e-12) means sqrt(|d|^2) rounds to R_c or more:
    // candidates that far are dropped before the square root
    const double rc2_out = Rc * Rc * (1.0 + 1e-12);
    double dx = pj.x - pi.x, dy = pj.y - pi.y;
    const double dd2 = dx * dx + dy * dy;
    if (!(dd2 <= rc2_out)) return;
    double dd = dd2 > 0.0 ? sqrt_rn_int(dd2) : 0.0;
    if (!(dd < Rc)) return;
    if (dd == 0.0) {
        atomicAdd(&d.status[PD_STATUS_COINCIDENT], 1);
        return;
    }
    const double Vi = __ldg(&d.V[ii]), cw = __ldg(&d.g_cw[gi]);
    const double2 Xi = __ldg(&d.X[ii]);
    const double rho_i = k.mat ? __ldg(&d.g_rho[gi]) : k.rho;
    double ex = dx / dd, ey = dy / dd;
    const double Vj = __ldg(&d.V[j]);
    const double2 vj = ldm<PERSIST>(&d.v[vin][j]);
    double vrx = vi.x - vj.x, vry = vi.y - vj.y;
    const int gj = __ldg(&d.grain[j]);
    if (gj == gi) {
        if (bonded_intact(d, k, ii, r0, r1, j)) return;
        const double2 Xj = __ldg(&d.X[j]);
        double xix = Xj.x - Xi.x, xiy = Xj.y - Xi.y;
        double xi = sqrt(xix * xix + xiy * xiy);
        double m;
        if (xi < Rc)
            m = (dd < xi) ? cw * (dd - xi) / xi : 0.0;
        else
            m = cw * (dd - Rc) / Rc;
        if (m == 0.0) return;
        double f = m * Vi * Vj;
        double gx = f * ex, gy = f * ey;
        const double Kn = k.mat ? 18.0 * __ldg(&d.g_k[gi]) / A.pe5 : A.Kn;
        damping_friction64(k, Kn, rho_i, rho_i, ex, ey, vrx, vry, -f, Vi, Vj, gx, gy);
        fsx = gx;
        fsy = gy;
    } else {
        double Kn = A.Kn, rho_d = rho_i;
        if (k.mat) {
            Kn = 18.0 * harmonic64(__ldg(&d.g_k[gi]), __ldg(&d.g_k[gj])) / A.pe5;
            rho_d = harmonic64(rho_i, __ldg(&d.g_rho[gj]));
        }
        double Fr = Kn * (Rc - dd) * Vi * Vj;
        double gx = -Fr * ex, gy = -Fr * ey;
        damping_friction64(k, Kn, rho_d, rho_i, ex, ey, vrx, vry, Fr, Vi, Vj, gx, gy);
        fnx = gx;
        fny = gy;
    }
}

// Candidate q of node ii, in ascending node index: the nc of its list and the nb
// partners of the bonds broken since the rebuild, merged; together every pair
// closer than R_c without an intact bond.  (The order of a node's contact forces
// then does not depend on when the lists were last rebuilt: a run continued from
// a stored state, or batched with other aggregates, adds them as any other.)
template <bool PERSIST>
__device__ __forceinline__ int candidate(const DevPtrs &d, const KParams &k, int ii, int nc, int nb, int r0, int q) {
    const auto listed = [&](int at) { return ldm<PERSIST>(&d.nbr[(size_t)at * k.N + ii]); };
    int at = 0;                             // list entries taken
    for (int m = 0; m < nb; ++m) {
        // (few nodes have one; both sequences ascend)
        const int p = fresh_partner(d, k, ii, r0, m);
        while (at < nc && listed(at) < p) {
            if (at + m == q) return listed(at);
            ++at;
        }
        if (at + m == q) return p;
    }
    return listed(q - nb);
}

// Adds the v of a group of LANES threads, thread by thread (the first n of them),
// to the running sum `acc` of all its threads.
template <int LANES, class T>
__device__ __forceinline__ T add_in_order(T acc, T v, int n) {
#pragma unroll
    for (int l = 0; l < LANES; ++l) {
        const T w = __shfl_sync(0xffffffffu, v, l, LANES);
        if (l < n) acc += w;
    }
    return acc;
}

// Not a zero of either sign (no FP64 instruction).
__device__ __forceinline__ bool nonzero(double v) { return (unsigned long long)__double_as_longlong(v) << 1; }
__device__ __forceinline__ bool nonzero(float v) { return __float_as_uint(v) << 1; }

// The n candidates of a node by its LANES threads, a candidate each:
// pair(q, sx, sy, nx, ny) for candidate q; the forces are then added in the
// order of the candidates, so the sums are those of one thread working through
// them, in every thread of the node.  A contact is a chain of divisions and
// square roots (FP64: about 4 us on the 2-lane pipe).  Four or eight threads
// work through their own node's: see warp_contacts.  (FP64: additions of zeros
// only, as most candidates lie beyond R_c, are left out; 28.0 to 27.6 us a step.)
// Every thread of the warp calls it.
template <int LANES, class T, class Pair>
__device__ __forceinline__ void group_contacts(int lane, int n, T &Fsx, T &Fsy, T &Fnx, T &Fny, Pair pair) {
    for (int q0 = 0; __any_sync(0xffffffffu, q0 < n); q0 += LANES) {
        T a = 0, b = 0, c = 0, e = 0;
        if (q0 + lane < n) pair(q0 + lane, a, b, c, e);
        if (sizeof(T) == 4 || __any_sync(0xffffffffu, nonzero(a) || nonzero(b))) {
            Fsx = add_in_order<LANES>(Fsx, a, n - q0);
            Fsy = add_in_order<LANES>(Fsy, b, n - q0);
        }
        if (sizeof(T) == 4 || __any_sync(0xffffffffu, nonzero(c) || nonzero(e))) {
            Fnx = add_in_order<LANES>(Fnx, c, n - q0);
            Fny = add_in_order<LANES>(Fny, e, n - q0);
        }
    }
}

// What a contact takes from its own node, handed from the node's thread to the
// one that works on the contact.
struct ContactNode64 {
    double px, py, vx, vy;
    int ii, gi, ag, r0, r1, nc, nb, pad;
};
struct ContactNode32 {
    float4 q;
    double vx, vy;
    int ii, gi, ag, r0, r1, nc, nb, pad;
};
template <class Node>
__device__ __forceinline__ Node shfl_node(const Node &v, int src) {
    constexpr int kWords = sizeof(Node) / 4 - 1;          // (not the padding)
    Node r;
#pragma unroll
    for (int w = 0; w < kWords; ++w)
        reinterpret_cast<int *>(&r)[w] = __shfl_sync(0xffffffffu, reinterpret_cast<const int *>(&v)[w], src);
    return r;
}

// The candidates of the nodes of a warp (several threads per node: thread 0 of
// each gives its node and the number n of its candidates, the others n = 0), one
// per thread, 32 at a time: pair(node, q, sx, sy, nx, ny) for candidate q of a
// node.  Each node's forces are then added in the order of its candidates, into
// its thread 0.  A contact is a chain of divisions and square roots (FP64: about
// 4 us on the 2-lane pipe, which a warp occupies as long for one pair as for
// 32), and few nodes of a warp have any.
// Two threads per node share their contacts so: a node's own two take half as
// many chains as it has candidates, one after the other.  A step of a settled
// box of 19681 nodes, by the node's own threads and dealt to the warp, hot and
// with L2 flushed: FP64, 2 threads 31.7 and 28.1, 46.2 and 43.6 us; 4 threads 27.9
// and 28.7, 40.1 and 42.1; FP32 split, 2 threads 13.4 and 12.7, 4 threads 12.8 and
// 13.3.  (Without the node's data handed over, each contact began with a chain of
// loads for it: FP64, 2 threads 31.0, flushed 48.3.)
// Every thread of the warp calls it.
template <class T, class Node, class Pair>
__device__ __forceinline__ void warp_contacts(const Node &mine, int n, T &Fsx, T &Fsy, T &Fnx, T &Fny, Pair pair) {
    constexpr unsigned kAll = 0xffffffffu;
    if (!__any_sync(kAll, n > 0)) return;
    const int lane = threadIdx.x & 31;
    int start = n;                          // exclusive prefix of n
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const int y = __shfl_up_sync(kAll, start, off);
        if (lane >= off) start += y;
    }
    const int total = __shfl_sync(kAll, start, 31);
    start -= n;
    for (int p0 = 0; p0 < total; p0 += 32) {
        // pair p belongs to the last thread whose prefix is not beyond p
        const int p = p0 + lane;
        int own = 0;
#pragma unroll
        for (int off = 16; off > 0; off >>= 1)
            if (__shfl_sync(kAll, start, own + off) <= p) own += off;
        const int q = p - __shfl_sync(kAll, start, own);
        const Node node = shfl_node(mine, own);
        T a = 0, b = 0, c = 0, e = 0;
        if (p < total) pair(node, q, a, b, c, e);
        // (most candidates lie beyond R_c; adding their zeros changes no sum)
        const unsigned some = __ballot_sync(kAll, nonzero(a) || nonzero(b) || nonzero(c) || nonzero(e));
        const int lo = max(start - p0, 0), hi = min(start + n - p0, 32);
        unsigned left = hi > lo ? some & (kAll >> (32 - hi)) & (kAll << lo) : 0u;
        while (__any_sync(kAll, left != 0u)) {
            const int src = left ? __ffs(left) - 1 : lane;
            const T va = __shfl_sync(kAll, a, src), vb = __shfl_sync(kAll, b, src);
            const T vc = __shfl_sync(kAll, c, src), ve = __shfl_sync(kAll, e, src);
            if (left) {
                Fsx += va;
                Fsy += vb;
                Fnx += vc;
                Fny += ve;
            }
            left &= left - 1u;
        }
    }
}

// Contact forces of node ii, FP64 path, by one thread: its nc + nb candidates.
template <bool PERSIST>
__device__ __forceinline__ void contacts64(const DevPtrs &d, const KParams &k, int ii, int vin, int gi, int nc, int nb,
                                           int r0, int r1, double2 pi, double &Fsx, double &Fsy, double &Fnx,
                                           double &Fny) {
    const AggParams &A = d.agg[__ldg(&d.g_agg[gi])];
    const double2 vi = ldm<PERSIST>(&d.v[vin][ii]);
    for (int q = 0; q < nc + nb; ++q) {
        const int j = candidate<PERSIST>(d, k, ii, nc, nb, r0, q);
        double a, b, c, e;
        contact_pair64<PERSIST>(d, k, A, ii, j, vin, gi, r0, r1, pi, ldm<PERSIST>(&d.p[j]), vi, a, b, c, e);
        Fsx += a;
        Fsy += b;
        Fnx += c;
        Fny += e;
    }
}

// (slot: the bond tile of a block of BLOCK threads with one thread per node,
// and warm the pass before a run, which forms slots only and leaves `out`;
// without a tile BLOCK is 0.  contact: the node has contact candidates; without
// INLINE (one thread per node) its contact forces are left to a later pass.)
template <bool PERSIST, int LANES, int BLOCK, bool INLINE = true>
__device__ __forceinline__ void force_node64(const DevPtrs &d, const KParams &k, int i, int lane, bool active,
                                             int vin, Sums64 &out, float4 *slot, bool warm, bool &contact) {
    contact = false;
    const int ii = active ? i : 0;
    const double2 pi = ldm<PERSIST>(&d.p[ii]);
    const double Vi = __ldg(&d.V[ii]);
    const int gi = __ldg(&d.grain[ii]);
    const double cw = __ldg(&d.g_cw[gi]), s0 = __ldg(&d.g_s0[gi]), eps = __ldg(&d.g_eps[gi]);
    uint32_t *bw = d.bits + (size_t)ii * k.wpn;

    ff Fbx = {0.f, 0.f}, Fby = {0.f, 0.f};
    const uint32_t w0 = active ? __ldcg(bw) : 0u;      // the row's first 32 broken bits (own bonds only)
    const float s0f = (float)s0;
    const ff cwVV = to_ff(cw * Vi * Vi);                // one grain: V_y = V_x
    const ff inv_eps = ff_rcp(to_ff(eps));
    bool csr = true;           // bonds from the CSR columns
    unsigned note = 0u;
    int r0, r1;
    if constexpr (BLOCK > 0) {
        uint4 st = active ? __ldg(&d.stn[ii]) : make_uint4(kStnIrregular, 0u, 0u, 0u);
        const bool gap = st.x & kStnGap;
        csr = (st.x & kStnIrregular) && !gap;
        st.x &= kStnBits;
        r0 = (int)st.w;
        r1 = r0 + __popc(st.x);
        if (csr) {
            r0 = active ? __ldg(&d.row_ptr[ii]) : 0;
            r1 = active ? __ldg(&d.row_ptr[ii + 1]) : 0;
        }
        const uint32_t alive = csr ? 0u : stn_alive(st.x, w0);
        const bool gaps = __any_sync(0xffffffffu, gap);
        const uint32_t formed =
            gaps ? tile_forward64<PERSIST, BLOCK, true>(d, k, ii, alive, st, gap, pi, cwVV, inv_eps, s0f, s0, slot,
                                                        note, !warm)
                 : tile_forward64<PERSIST, BLOCK, false>(d, k, ii, alive, st, gap, pi, cwVV, inv_eps, s0f, s0, slot,
                                                         note, !warm);
        if (warm) return;
        __syncthreads();
        if (gaps) tile_sum64<PERSIST, BLOCK, true>(d, k, ii, alive, formed, st, gap, pi, cwVV, inv_eps, s0f, s0, slot,
                                                   Fbx, Fby, note);
        else tile_sum64<PERSIST, BLOCK, false>(d, k, ii, alive, formed, st, gap, pi, cwVV, inv_eps, s0f, s0, slot, Fbx,
                                               Fby, note);
    } else {
        r0 = active ? __ldg(&d.row_ptr[ii]) : 0;
        r1 = active ? __ldg(&d.row_ptr[ii + 1]) : 0;
    }
    // six bonds loaded, three evaluated at a time: a full row of 24 is 4, 2, 1
    // rounds of loads and 8, 4, 2, 1 of evaluations with 1, 2, 4, 8 threads.
    // (One copy of the evaluation for both halves of a round, which moves the
    // second half's operands down: a bond is some 200 instructions, and a step
    // that starts with cold caches waits for its code more than for data.  Two
    // copies, 4 threads per node: 49.7 us a step of a settled box of 19681 nodes
    // with L2 flushed before it, one: 45.0; 48 bonds a node, 87340 nodes: 104.7
    // and 98.2.  Two bonds a time, of four: 306907 nodes, 4 threads per node 182 us
    // for 172, 8 threads 260 for 227, but horizon 2 h, whose rows of eight leave
    // the third place empty, 2 threads 71 for 88.)
    constexpr int kLoad = 6, kEval = 3;
    static_assert(kLoad == 2 * kEval, "a round is two evaluations");
    for (int b0 = r0 + lane; b0 < r1 && csr; b0 += kLoad * LANES) {
        int jb[kLoad];
        uint32_t wb[kLoad];
        double xb[kLoad];
        double2 pb[kLoad];
#pragma unroll
        for (int m = 0; m < kLoad; ++m) {
            const int b = b0 + m * LANES;
            jb[m] = b < r1 ? __ldg(&d.col[b]) : -1;
            xb[m] = b < r1 ? __ldg(&d.xi[b]) : 1.0;
            wb[m] = b - r0 < 32 ? w0 : (b < r1 ? __ldcg(&bw[(b - r0) >> 5]) : 0u);
        }
        uint32_t live = 0u;
#pragma unroll
        for (int m = 0; m < kLoad; ++m) {
            pb[m] = ldm<PERSIST>(&d.p[jb[m] < 0 ? ii : jb[m]]);
            live |= (jb[m] >= 0 && !((wb[m] >> ((b0 + m * LANES - r0) & 31)) & 1u)) ? 1u << m : 0u;
            note |= wb[m] ? kNoteSeen : 0u;
        }
#pragma unroll 1
        for (int bm = b0; live; bm += kEval * LANES, live >>= kEval) {
            ff c[kEval], fx[kEval], fy[kEval];
            uint32_t broken = 0u, near = 0u;
#pragma unroll
            for (int m = 0; m < kEval; ++m) c[m] = cwVV;
            if (k.micro) {
#pragma unroll
                for (int m = 0; m < kEval; ++m) c[m] = bond_conic64(cwVV, xb[m], inv_eps);
            }
#pragma unroll
            for (int m = 0; m < kEval; ++m) {
                bool b, n;
                bond_terms64(pi, pb[m], xb[m], c[m], s0f, fx[m], fy[m], b, n);
                broken |= b ? 1u << m : 0u;
                near |= n ? 1u << m : 0u;
            }
            const uint32_t now = live & ((1u << kEval) - 1u);
            broken &= now;
            for (near &= now; near; near &= near - 1u) {
                const int m = __ffs(near) - 1, b = bm + m * LANES;
                const bool brk = bond_breaks64(pi, ldm<PERSIST>(&d.p[__ldg(&d.col[b])]), __ldg(&d.xi[b]), s0);
                broken = brk ? broken | (1u << m) : broken & ~(1u << m);
            }
            for (uint32_t m = broken; m; m &= m - 1u) {
                const int kk = bm + (__ffs(m) - 1) * LANES - r0;
                atomicOr(&bw[kk >> 5], 1u << (kk & 31));
                note |= kNoteBroke;
            }
#pragma unroll
            for (int m = 0; m < kEval; ++m) {
                const bool ok = ((now & ~broken) >> m) & 1u;
                Fbx = ff_add(Fbx, ok ? fx[m] : ff{0.f, 0.f});
                Fby = ff_add(Fby, ok ? fy[m] : ff{0.f, 0.f});
                pb[m] = pb[kEval + m];
                xb[m] = xb[kEval + m];
            }
        }
    }
    __syncwarp();

    const int nc = active ? ldm<PERSIST>(&d.nbr_cnt[ii]) : 0;
    const int nb = fresh_bonds(d, k, ii, any_lane<LANES>(w0 != 0u || note != 0u));
    double Fsx = 0.0, Fsy = 0.0, Fnx = 0.0, Fny = 0.0;
    contact = nc + nb > 0;
    if constexpr (LANES == 1) {
        if (INLINE && contact) contacts64<PERSIST>(d, k, ii, vin, gi, nc, nb, r0, r1, pi, Fsx, Fsy, Fnx, Fny);
    } else if constexpr (LANES == 2) {
        ContactNode64 mine = {};
        if (contact) {
            const double2 vi = ldm<PERSIST>(&d.v[vin][ii]);
            mine = {pi.x, pi.y, vi.x, vi.y, ii, gi, __ldg(&d.g_agg[gi]), r0, r1, nc, nb, 0};
        }
        warp_contacts(mine, lane == 0 ? nc + nb : 0, Fsx, Fsy, Fnx, Fny,
                      [&](const ContactNode64 &x, int q, double &sx, double &sy, double &nx, double &ny) {
                          const int j = candidate<PERSIST>(d, k, x.ii, x.nc, x.nb, x.r0, q);
                          contact_pair64<PERSIST>(d, k, d.agg[x.ag], x.ii, j, vin, x.gi, x.r0, x.r1,
                                                  make_double2(x.px, x.py), ldm<PERSIST>(&d.p[j]),
                                                  make_double2(x.vx, x.vy), sx, sy, nx, ny);
                      });
    } else {
        group_contacts<LANES>(lane, nc + nb, Fsx, Fsy, Fnx, Fny,
                              [&](int q, double &sx, double &sy, double &nx, double &ny) {
                                  const int j = candidate<PERSIST>(d, k, ii, nc, nb, r0, q);
                                  contact_pair64<PERSIST>(d, k, d.agg[__ldg(&d.g_agg[gi])], ii, j, vin, gi, r0, r1, pi,
                                                          ldm<PERSIST>(&d.p[j]), ldm<PERSIST>(&d.v[vin][ii]), sx, sy,
                                                          nx, ny);
                              });
    }
    __syncwarp();
    out.bx = lane_sum<LANES>(f2d_bits(Fbx.hi) + f2d_bits(Fbx.lo));
    out.by = lane_sum<LANES>(f2d_bits(Fby.hi) + f2d_bits(Fby.lo));
    out.sx = Fsx;
    out.sy = Fsy;
    out.nx = Fnx;
    out.ny = Fny;
}

// Wall forces and the update of node i from its lane sums, one thread per node
// (the FP64 work runs with converged warps).
template <bool PERSIST>
__device__ __forceinline__ void node_epilogue64(const DevPtrs &d, const KParams &k, int i, int vin, int update_v,
                                                const Sums64 &f, bool total = false) {
    // the node's independent loads first, all in flight together (the pass is
    // bound by memory latency): velocity, previous acceleration, grain, cell
    const double2 vi = ldm<PERSIST>(&d.v[vin][i]);
    const double2 ao = update_v ? ldm<PERSIST>(&d.a[i]) : make_double2(0.0, 0.0);
    const int gi = __ldg(&d.grain[i]);
    const int2 cell = ldm<PERSIST>(&d.cell[i]);
    const int ag = __ldg(&d.g_agg[gi]);
    const double inv_m = __ldg(&d.g_invm[gi]);
    const int4 wc = ldm<PERSIST>(&cur_wall<PERSIST>(d)[ag]);
    double Fwx = 0.0, Fwy = 0.0;
    const bool walls = !cells_far_from_walls(cell, wc);
    if (walls) {
        const double2 pi = ldm<PERSIST>(&d.p[i]);
        const AggParams &A = d.agg[ag];
        const double rho = k.mat ? __ldg(&d.g_rho[gi]) : k.rho;
        const double Kn = k.mat ? 18.0 * __ldg(&d.g_k[gi]) / A.pe5 : A.Kn;
        wall_force64(k, A, Kn, rho, cur_time<PERSIST>(d), pi.x, pi.y, vi.x, vi.y, __ldg(&d.V[i]), Fwx, Fwy,
                     d.status);
    }
    if (k.store) {
        finish_node<PERSIST, true>(d, k, i, vin, update_v, vi, 0.0, f.bx, f.by, f.sx, f.sy, f.nx, f.ny, Fwx, Fwy,
                                   inv_m);
    } else {
        // total: the parts were summed by the lane-sum pass, f.bx / f.by hold T
        const double Tx = total ? f.bx : __dadd_rn(__dadd_rn(f.bx, f.sx), f.nx);
        const double Ty = total ? f.by : __dadd_rn(__dadd_rn(f.by, f.sy), f.ny);
        finish_node64_total<PERSIST>(d, k, i, vin, update_v, vi, ao, Tx, Ty, walls, Fwx, Fwy, inv_m);
    }
}

// FP32-split geometry of one bond to a neighbour at qj (float-float shifted
// position), lattice offset code nn = di^2 + dj^2 and sqn = sqrt(nn):
// num = |d|^2 - |xi|^2 (|xi|^2 = n h^2 exact to float-float), den = |xi| (L + |xi|),
// so that s = num / den.  The square |d|^2 is (s, r): s the rounded sum of the
// squared high parts and r everything below it.  With a >= b the magnitudes of
// the high parts, p = RN(a^2) and s = RN(b^2 + p) satisfy s/2 <= p <= s (one
// last place aside), so p - s is exact and fma(b, b, p - s) is the rounding
// error of s: eight operations where two exact products and an exact sum take
// ten.  r keeps the low parts' own squares too (see len2_ff) and stays apart
// from s until |xi|^2 has been taken off: s - n h^2 is exact for moderate
// stretches, so nothing is renormalised first.  Every operation is even in d,
// so both nodes of a bond get the same num and den.
struct BondGeom32 {
    float dx, dy, L, num, den, xi;
};
// (pow2: n is a power of two, so n h^2 is exact in float-float without a
// product residual; callers that know n at compile time pass it as a constant)
__device__ __forceinline__ void bond_geom32(float4 qj, float2 phi, float2 pli, float nn, float sqn, float4 gq,
                                            BondGeom32 &g, bool pow2 = false) {
    const float dxh = __fsub_rn(qj.x, phi.x), dxl = __fsub_rn(qj.z, pli.x);
    const float dyh = __fsub_rn(qj.y, phi.y), dyl = __fsub_rn(qj.w, pli.y);
    const float a = fmaxf(fabsf(dxh), fabsf(dyh)), b = fminf(fabsf(dxh), fabsf(dyh));
    const float p = __fmul_rn(a, a), ep = fmaf(a, a, -p);
    const float s = fmaf(b, b, p), es = fmaf(b, b, __fsub_rn(p, s));
    // ep + es + dxl (2 dxh + dxl) + dyl (2 dyh + dyl)
    const float r = __fadd_rn(es, fmaf(dxl, fmaf(2.f, dxh, dxl), fmaf(dyl, fmaf(2.f, dyh, dyl), ep)));
    float q, eq;                                         // |xi|^2 = n h^2 as a float-float pair
    if (pow2) {
        q = __fmul_rn(nn, gq.y);
        eq = __fmul_rn(nn, gq.z);
    } else {
        two_prod(nn, gq.y, q, eq);
        eq = fmaf(nn, gq.z, eq);
    }
    g.num = __fadd_rn(__fsub_rn(s, q), __fsub_rn(r, eq));
    g.xi = __fmul_rn(gq.x, sqn);
    g.L = sqrt_approx(__fadd_rn(s, r));
    g.den = fmaf(g.xi, g.L, q);                          // |xi| L + |xi|^2
    g.dx = __fadd_rn(dxh, dxl);
    g.dy = __fadd_rn(dyh, dyl);
}
// Break decision of a bond: 0 = intact, 1 = broken at this evaluation (|s| >
// s0), 2 = |s| in the guard band around s0 (decided in FP64 after the loop).
// The tests compare |num| with s0 den: no division.  A NaN stretch counts as
// intact.
__device__ __forceinline__ float bond_excess32(const BondGeom32 &g, float s0_lo) {
    return fmaf(-s0_lo, g.den, fabsf(g.num));           // > 0: not clearly intact
}
__device__ __forceinline__ int bond_state32(const BondGeom32 &g, float s0_lo, float s0_hi) {
    if (!(bond_excess32(g, s0_lo) > 0.f)) return 0;
    return fabsf(g.num) < __fmul_rn(s0_hi, g.den) ? 2 : 1;
}
__device__ __forceinline__ int bond_classify32(float4 qj, float2 phi, float2 pli, float nn, float sqn, float4 gq,
                                               float s0_lo, float s0_hi, BondGeom32 &g, bool pow2 = false) {
    bond_geom32(qj, phi, pli, nn, sqn, gq, g, pow2);
    return bond_state32(g, s0_lo, s0_hi);
}

// Bond force c_w w V^2 s (d / L) of an intact bond (w = 1 - |xi| / eps for the
// conic micromodulus).  The products are rounded by themselves (no FMA into a
// running sum): a bond's force on its other node is then the exact negative,
// whichever of the two nodes evaluates it.
__device__ __forceinline__ float2 bond_force32(const BondGeom32 &g, float cw, float inv_eps, float VV, int micro) {
    const float c = micro ? cw * fmaf(-g.xi, inv_eps, 1.0f) : cw;
    const float qf = __fmul_rn(__fmul_rn(__fmul_rn(c, VV), g.num), rcp_approx(__fmul_rn(g.den, g.L)));
    return make_float2(__fmul_rn(qf, g.dx), __fmul_rn(qf, g.dy));
}
__device__ __forceinline__ void bond_add32(const BondGeom32 &g, float cw, float inv_eps, float VV, int micro,
                                           float &Fbx, float &Fby) {
    const float2 f = bond_force32(g, cw, inv_eps, VV, micro);
    Fbx = __fadd_rn(Fbx, f.x);
    Fby = __fadd_rn(Fby, f.y);
}

// FP32-split forces of node i: the same laws and lane layout, with the bond,
// self-contact and contact arithmetic on the FP32 pipe.  Positions are
// float-float pairs of the shifted position (every coordinate of a box lies in
// [L, 2L), so high-part differences of nearby nodes are exact), |d|^2 is a
// float-float pair built with exact FMA products, and the reference
// |xi|^2 = h^2 (di^2 + dj^2) comes from the integer lattice offset: the stretch
// s = (|d|^2 - |xi|^2) / (|xi| (|d| + |xi|)) (eq:pmb, rearranged) and the
// contact overlap R_c - |d| = (R_c^2 - |d|^2) / (R_c + |d|) keep ~1e-7 relative
// accuracy.  Bonds whose FP32 stretch lies within guard * s0 of s0 are
// re-decided with the FP64 stretch, so break decisions are the FP64 ones.
// The learned surrogate is used only while none of its bounded tensor-core
// waits has given up (status[PD_STATUS_TIMEOUT], the networks' error word): a
// step in which one gives up still runs on the surrogate in the kernels that
// started before it, every later step uses the full bond kernel.
__device__ __forceinline__ bool sur_healthy(const DevPtrs &d) {
    return __ldcg(&d.status[PD_STATUS_TIMEOUT]) == 0 && (d.mlp_err == nullptr || __ldcg(d.mlp_err) == 0);
}

// Shared memory of an FP32-split tile: the bond slots, the positions of the
// tile and of the one after it (by tile parity; the even tile's first ones again
// behind the odd tile, so that no index wraps), and the streams of the tile's
// nodes.  A step reads about 180 bytes a node in a chain of dependent loads,
// and with the bonds evaluated once the warps that fit no longer hide that
// chain: with every load on the spot the same loop took 347 us on 2.28M nodes
// (16 warps an SM, 60 % of their time waiting for memory).  So every thread
// copies its next node's streams asynchronously while it works on the present
// one, and the bond loop's gathers are shared-memory reads.  A step of that
// ensemble (kernel alone) went from 226 us, with the loop that evaluates each
// bond twice from L1-cached gathers, to about 140 us; 1,119 instead of 2,350
// thread instructions a node.
template <int BLOCK>
struct Tile32 {
    float2 slot[kPairHalf * PairTile<float2, BLOCK>::kStride];
    static constexpr int kAhead = kCarry + 8;           // farthest forward place read, absent bonds included
    float4 q[2 * BLOCK + kAhead];
    uint4 st[BLOCK];
    double2 v[BLOCK], u[BLOCK], xs[BLOCK];
    float4 sref[BLOCK];
    float2 a[BLOCK];
    int2 cell[BLOCK];
    int gi[BLOCK], nc[BLOCK];
    uint32_t bits[BLOCK];
};

// What the bond loop takes from a node's grain and list.
struct BondNode32 {
    float4 qi, gq, gc;      // position; (h, h^2 hi, h^2 lo, V); (c_w, s0, eps, rho)
    uint4 st;               // stencil record (its 24 bits)
    bool gap;               // of a node with kStnGap
};

// The forward half of a node's stencil bonds: their forces into the thread's
// slots and their sum in (Fx, Fy).  alive: the intact ones of st.x.  win: the
// node's place in the position window.  Straight-line code over all twelve
// offsets: a slot of an absent bond holds what the arithmetic makes of the
// wrong position (nobody reads it: bonds are in both nodes' lists), and one
// comparison over the largest excess of a stretch tells whether the general
// pass after it is needed.  own: the block owns the node (broken-bond word bw)
// and records its broken bonds.
template <int BLOCK, bool GAP>
__device__ __forceinline__ void tile_forward32(const DevPtrs &d, const KParams &k, int ii, uint32_t alive,
                                               const BondNode32 &nd, const float4 *win, float2 *mine, uint32_t *bw, float &Fx, float &Fy, unsigned &note, bool own,
                                               bool micro) {
    constexpr int S = PairTile<float2, BLOCK>::kStride;
    const float2 phi = make_float2(nd.qi.x, nd.qi.y), pli = make_float2(nd.qi.z, nd.qi.w);
    const float VV = nd.gq.w * nd.gq.w, inv_eps = micro ? 1.0f / nd.gc.z : 0.f;
    const float s0_lo = nd.gc.y * (1.0f - k.guard);
    const float4 *const row[3] = {win, win + stn_row(nd.st, 1), win + stn_row(nd.st, 2)};
    float excess = 0.f;
    Fx = Fy = 0.f;
    constexpr int kBatch = 4;
#pragma unroll
    for (int m0 = 0; m0 < kPairHalf; m0 += kBatch) {
        float4 qb[kBatch];
        if (!GAP || !nd.gap) {
#pragma unroll
            for (int m = 0; m < kBatch; ++m) {
                const int o = kPairHalf + m0 + m;
                qb[m] = row[stn_dj(o)][stn_di(o)];
            }
        } else {
#pragma unroll
            for (int m = 0; m < kBatch; ++m) {
                const int o = kPairHalf + m0 + m;
                qb[m] = win[(nd.st.x >> o) & 1u ? stn_to(d, nd.st, true, ii, o) : 0];
            }
        }
#pragma unroll
        for (int m = 0; m < kBatch; ++m) {
            const int o = kPairHalf + m0 + m, di = stn_di(o), dj = stn_dj(o), n = di * di + dj * dj;
            BondGeom32 g;
            bond_geom32(qb[m], phi, pli, (float)n, stn_sqrt_n(n), nd.gq, g, (n & (n - 1)) == 0);
            const float2 f = bond_force32(g, nd.gc.x, inv_eps, VV, micro);
            mine[(m0 + m) * S] = f;
            if ((alive >> o) & 1u) {
                excess = fmaxf(excess, bond_excess32(g, s0_lo));      // (a NaN stretch counts as intact)
                Fx = __fadd_rn(Fx, f.x);
                Fy = __fadd_rn(Fy, f.y);
            }
        }
    }
    // broken bonds (their other node has them broken too, unless the caller set
    // the bits of one direction only)
    for (uint32_t m = nd.st.x & ~alive & ~((1u << kPairHalf) - 1u); m; m &= m - 1u)
        mine[(__ffs(m) - 1 - kPairHalf) * S].x = __uint_as_float(kPairNone);
    if (excess > 0.f) {
        // a bond breaks or lies in the guard band: markers and the sum again
        Fx = Fy = 0.f;
        for (uint32_t m = alive & ~((1u << kPairHalf) - 1u); m; m &= m - 1u) {
            const int o = __ffs(m) - 1, di = stn_di(o), dj = stn_dj(o), n = di * di + dj * dj;
            float2 *const at = &mine[(o - kPairHalf) * S];
            BondGeom32 g;
            const int r = bond_classify32(win[stn_to(d, nd.st, GAP && nd.gap, ii, o)], phi, pli, (float)n, stn_sqrt_n(n), nd.gq, s0_lo,
                                          nd.gc.y * (1.0f + k.guard), g);
            if (r == 0) {
                Fx = __fadd_rn(Fx, at->x);
                Fy = __fadd_rn(Fy, at->y);
                continue;
            }
            at->x = __uint_as_float(r == 1 ? kPairBroken : kPairGuard);
            if (r == 2) {
                note |= kNoteGuard;
            } else if (own) {
                atomicOr(bw, stn_bit(nd.st.x, o));
                note |= kNoteBroke;
            }
        }
    }
}

// The backward half of node ii's bonds, from the slots of the nodes that formed
// them: its sum in (Fx, Fy).
template <bool PERSIST, int BLOCK, bool GAP>
__device__ __forceinline__ void tile_backward32(const DevPtrs &d, const KParams &k, int ii, uint32_t alive,
                                                const BondNode32 &nd, const float2 *mine, float &Fx, float &Fy,
                                                unsigned &note) {
    constexpr int S = PairTile<float2, BLOCK>::kStride;
    const float2 *const row[3] = {mine + stn_row(nd.st, -2), mine + stn_row(nd.st, -1), mine};
    Fx = Fy = 0.f;
    if (!GAP || !nd.gap) {
#pragma unroll
        for (int o = 0; o < kPairHalf; ++o) {
            // (a row without bonds has offset 0: some slot of the tile)
            const float2 v = row[stn_dj(o) + 2][(kPairHalf - 1 - o) * S + stn_di(o)];
            if ((alive >> o) & 1u) {
                Fx = __fsub_rn(Fx, v.x);
                Fy = __fsub_rn(Fy, v.y);
            }
        }
    } else {
        int off[kPairHalf];
#pragma unroll
        for (int o = 0; o < kPairHalf; ++o) off[o] = (alive >> o) & 1u ? stn_to(d, nd.st, true, ii, o) : 0;
#pragma unroll
        for (int o = 0; o < kPairHalf; ++o) {
            if (!((alive >> o) & 1u)) continue;
            const float2 v = mine[(kPairHalf - 1 - o) * S + off[o]];
            Fx = __fsub_rn(Fx, v.x);
            Fy = __fsub_rn(Fy, v.y);
        }
    }
    if (Fx != Fx) {
        // some slot holds a marker (or a force is not finite): the half again
        const float2 phi = make_float2(nd.qi.x, nd.qi.y), pli = make_float2(nd.qi.z, nd.qi.w);
        Fx = Fy = 0.f;
        for (uint32_t m = alive & ((1u << kPairHalf) - 1u); m; m &= m - 1u) {
            const int o = __ffs(m) - 1, di = stn_di(o), dj = stn_dj(o), off = stn_to(d, nd.st, GAP && nd.gap, ii, o);
            const float2 v = mine[(kPairHalf - 1 - o) * S + off];
            unsigned mark = __float_as_uint(v.x);
            if (mark == kPairNone) {
                const int n = di * di + dj * dj;
                BondGeom32 g;
                const int r = bond_classify32(ldm<PERSIST>(&cur_pq<PERSIST>(d)[ii + off]), phi, pli, (float)n,
                                              stn_sqrt_n(n), nd.gq, nd.gc.y * (1.0f - k.guard),
                                              nd.gc.y * (1.0f + k.guard), g);
                if (r == 0) {
                    bond_add32(g, nd.gc.x, 1.0f / nd.gc.z, nd.gq.w * nd.gq.w, k.micro, Fx, Fy);
                    continue;
                }
                mark = r == 1 ? kPairBroken : kPairGuard;
            }
            if (mark == kPairBroken) {
                atomicOr(&d.bits[(size_t)ii * k.wpn], stn_bit(nd.st.x, o));
                note |= kNoteBroke;
            } else if (mark == kPairGuard) {
                note |= kNoteGuard;
            } else {
                Fx = __fsub_rn(Fx, v.x);
                Fy = __fsub_rn(Fy, v.y);
            }
        }
    }
}

// The bonds of a node that lie in the guard band, in the order of its list
// (every step-th from lane): FP64 break decision, else the FP32 force.
template <bool PERSIST>
__device__ __forceinline__ void guard_bonds32(const DevPtrs &d, const KParams &k, int ii, int r0, int r1, int lane, int step,
                                           bool stencil, float2 phi, float2 pli, float4 gq, float4 gc, int gi,
                                           float s0_lo, float s0_hi, uint32_t *bw, float &Fbx, float &Fby,
                                              unsigned &note) {
    for (int b = r0 + lane; b < r1; b += step) {
        const int kk = b - r0;
        if ((__ldcg(&bw[kk >> 5]) >> (kk & 31)) & 1u) continue;
        const uint32_t c = __ldg(&d.colx[b]);
        const int j = (int)(c & kColMask);
        const float4 qj = ldm<PERSIST>(&cur_pq<PERSIST>(d)[j]);
        const float nn = (float)(c >> kColBits);
        // the same classification as the loop (stencil: sqrt(n) from the table)
        const float sqn = stencil ? stn_sqrt_n((int)nn) : sqrt_approx(nn);
        BondGeom32 bg;
        if (bond_classify32(qj, phi, pli, nn, sqn, gq, s0_lo, s0_hi, bg) != 2) continue;
        const double2 pi = position64<PERSIST>(d, ii), pj = position64<PERSIST>(d, j);
        const double ddx = __dsub_rn(pj.x, pi.x), ddy = __dsub_rn(pj.y, pi.y);
        const double L64 = __dsqrt_rn(__dadd_rn(__dmul_rn(ddx, ddx), __dmul_rn(ddy, ddy)));
        const double xi64 = __ldg(&d.xi[b]);
        if (fabs(__ddiv_rn(__dsub_rn(L64, xi64), xi64)) > __ldg(&d.g_s0[gi])) {
            atomicOr(&bw[kk >> 5], 1u << (kk & 31));
            note |= kNoteBroke;
            continue;
        }
        bond_add32(bg, gc.x, 1.0f / gc.z, gq.w * gq.w, k.micro, Fbx, Fby);
    }
}

// Contact force of candidate j on node ii, FP32 split: self-contact into fs,
// inter-grain contact into fn, zero beyond R_c (exact in float-float).
template <bool PERSIST>
__device__ __forceinline__ void contact_pair32(const DevPtrs &d, const KParams &k, const AggParams &A, int ii, int j,
                                               int vin, int gi, int r0, int r1, float2 phi, float2 pli, float4 gq,
                                               float4 gc, float4 qj, double2 vi64, float &fsx, float &fsy, float &fnx,
                                               float &fny) {
    fsx = fsy = fnx = fny = 0.f;
    const float Rc = A.rcf, Kn = A.knf, Vi = gq.w, cw = gc.x;
    const float rd = k.rdf, rho = gc.w, dt = k.dtf, mu = k.muf;     // rho: this grain's density
    const float dxh = __fsub_rn(qj.x, phi.x), dxl = qj.z - pli.x;
    const float dyh = __fsub_rn(qj.y, phi.y), dyl = qj.w - pli.y;
    float L2h, L2l;
    len2_ff(dxh, dxl, dyh, dyl, L2h, L2l);
    if (!(ff_diff(A.rc2_hi, A.rc2_lo, L2h, L2l) > 0.f)) return;
    const float dd = sqrtf(L2h);
    if (dd == 0.f) {
        atomicAdd(&d.status[PD_STATUS_COINCIDENT], 1);
        return;
    }
    const float ex = (dxh + dxl) / dd, ey = (dyh + dyl) / dd;
    const float overlap = ff_diff(A.rc2_hi, A.rc2_lo, L2h, L2l) / (Rc + dd);   // R_c - |d|
    const int gj = __ldg(&d.grain[j]);
    const float Vj = __ldg(&d.gq[gj]).w;
    // v(x) - v(y) in FP64, rounded once to float (nearby nodes move alike:
    // a float difference of float velocities would cancel)
    const double2 vj64 = ldm<PERSIST>(&d.v[vin][j]);
    const float vrx = (float)__dsub_rn(vi64.x, vj64.x), vry = (float)__dsub_rn(vi64.y, vj64.y);
    if (gj == gi) {
        if (bonded_intact(d, k, ii, r0, r1, j)) return;
        const int2 li = __ldg(&d.lat[ii]), lj = __ldg(&d.lat[j]);
        const int di = lj.x - li.x, dj = lj.y - li.y;
        const float nn = (float)(di * di + dj * dj);
        const float xi = gq.x * sqrtf(nn);
        float m;
        if (xi < Rc) {
            float q2, eq2;
            two_prod(nn, gq.y, q2, eq2);
            const float dl = ff_diff(L2h, L2l, q2, eq2 + nn * gq.z) / (dd + xi);   // |d| - |xi|
            m = (dl < 0.f) ? cw * dl / xi : 0.f;
        } else {
            m = -cw * overlap / Rc;
        }
        if (m == 0.f) return;
        const float f = m * Vi * Vj;
        float gx = f * ex, gy = f * ey;
        const float Kns = k.mat ? __ldg(&d.g_kf[gi]) : Kn;
        damping_friction32(rd, Kns, rho, rho, dt, mu, ex, ey, vrx, vry, -f, Vi, Vj, gx, gy);
        fsx = gx;
        fsy = gy;
    } else {
        // the harmonic mean of the grains' own K_n is K_n of the harmonic-mean modulus
        const float Knp = k.mat ? harmonic32(__ldg(&d.g_kf[gi]), __ldg(&d.g_kf[gj])) : Kn;
        const float Fr = Knp * overlap * Vi * Vj;
        float gx = -Fr * ex, gy = -Fr * ey;
        damping_friction32(rd, Knp, harmonic32(rho, __ldg(&d.gc[gj]).w), rho, dt, mu, ex, ey, vrx, vry, Fr, Vi,
                           Vj, gx, gy);
        fnx = gx;
        fny = gy;
    }
}

// Contact forces of node ii, FP32 split, by one thread: its nc + nb candidates.
template <bool PERSIST>
__device__ __forceinline__ void contacts32(const DevPtrs &d, const KParams &k, int ii, int vin, int gi, int nc, int nb,
                                           int r0, int r1, float2 phi, float2 pli, float4 gq, float4 gc, float &Fsx,
                                           float &Fsy, float &Fnx, float &Fny) {
    const AggParams &A = d.agg[__ldg(&d.g_agg[gi])];
    const double2 vi64 = ldm<PERSIST>(&d.v[vin][ii]);      // start-of-step velocity
    for (int q = 0; q < nc + nb; ++q) {
        const int j = candidate<PERSIST>(d, k, ii, nc, nb, r0, q);
        float a, b, c, e;
        contact_pair32<PERSIST>(d, k, A, ii, j, vin, gi, r0, r1, phi, pli, gq, gc, ldm<PERSIST>(&cur_pq<PERSIST>(d)[j]),
                                vi64, a, b, c, e);
        Fsx += a;
        Fsy += b;
        Fnx += c;
        Fny += e;
    }
}

// The bonds of node ii from its CSR columns (a row with a gap, a horizon
// without the stencil): every LANES-th from lane.
template <bool PERSIST, int LANES>
__device__ __forceinline__ void csr_bonds32(const DevPtrs &d, const KParams &k, int ii, int lane, int r0, int r1,
                                            float2 phi, float2 pli, float4 gq, float4 gc, float s0_lo, float s0_hi,
                                            uint32_t w0, float &Fbx, float &Fby, unsigned &note) {
    constexpr int kBondBatch = 4;
    uint32_t *bw = d.bits + (size_t)ii * k.wpn;
    const float cw = gc.x, VV = gq.w * gq.w, inv_eps = 1.0f / gc.z;
    for (int b0 = r0 + lane; b0 < r1; b0 += kBondBatch * LANES) {
        uint32_t cb[kBondBatch], wb[kBondBatch];
#pragma unroll
        for (int m = 0; m < kBondBatch; ++m) {
            const int b = b0 + m * LANES;
            cb[m] = b < r1 ? __ldg(&d.colx[b]) : 0xFFFFFFFFu;
            // the node's first broken-bond word is loaded once (rows of up to 32 bonds)
            wb[m] = b - r0 < 32 ? w0 : (b < r1 ? __ldcg(&bw[(b - r0) >> 5]) : 0u);
        }
        float4 qb[kBondBatch];
#pragma unroll
        for (int m = 0; m < kBondBatch; ++m) {
            const int j = cb[m] == 0xFFFFFFFFu ? ii : (int)(cb[m] & kColMask);
            qb[m] = ldm<PERSIST>(&cur_pq<PERSIST>(d)[j]);
        }
#pragma unroll
        for (int m = 0; m < kBondBatch; ++m) {
            const int b = b0 + m * LANES;
            const int kk = b - r0;
            note |= wb[m] ? kNoteSeen : 0u;
            if (cb[m] == 0xFFFFFFFFu || ((wb[m] >> (kk & 31)) & 1u)) continue;
            const float nn = (float)(cb[m] >> kColBits);         // lattice offset di^2 + dj^2
            BondGeom32 bg;
            const int r = bond_classify32(qb[m], phi, pli, nn, sqrt_approx(nn), gq, s0_lo, s0_hi, bg);
            if (r == 0) {
                bond_add32(bg, cw, inv_eps, VV, k.micro, Fbx, Fby);
            } else if (r == 2) {
                note |= kNoteGuard;
            } else {
                atomicOr(&bw[kk >> 5], 1u << (kk & 31));
                note |= kNoteBroke;
            }
        }
    }
}

template <bool PERSIST, int LANES>
__device__ __forceinline__ void force_node32(const DevPtrs &d, const KParams &k, int i, int lane, bool active,
                                             int vin, Sums32 &out) {
    const int ii = active ? i : 0;
    const float4 qi = ldm<PERSIST>(&cur_pq<PERSIST>(d)[ii]);
    const float2 phi = make_float2(qi.x, qi.y), pli = make_float2(qi.z, qi.w);
    const int gi = __ldg(&d.grain[ii]);
    const int ag = __ldg(&d.g_agg[gi]);
    const float4 gq = __ldg(&d.gq[gi]);                   // (h, h^2 hi, h^2 lo, V)
    const float4 gc = __ldg(&d.gc[gi]);                   // (c_w, s0, eps) as floats
    const float cw = gc.x, s0 = gc.y, inv_eps = 1.0f / gc.z;
    const float s0_lo = s0 * (1.0f - k.guard), s0_hi = s0 * (1.0f + k.guard);
    // lattice stencil of the node's bonds (regular nodes: the neighbour at
    // offset o is node ii + di + D[dj], no column load), else the CSR columns
    const uint4 st = (k.stencil && active) ? __ldg(&d.stn[ii]) : make_uint4(kStnIrregular, 0u, 0u, 0u);
    const bool stencil = !(st.x & kStnIrregular);
    int r0 = 0, r1 = 0;
    if (stencil) {
        r0 = (int)st.w;
        r1 = r0 + __popc(st.x);
    } else if (active) {
        r0 = __ldg(&d.row_ptr[ii]);
        r1 = __ldg(&d.row_ptr[ii + 1]);
    }
    uint32_t *bw = d.bits + (size_t)ii * k.wpn;
    float Fbx = 0.f, Fby = 0.f;
    const float VV = gq.w * gq.w;
    // learned modal surrogate: between judge steps an active grain skips the
    // bond loop; the epilogue adds its surrogate bond force instead
    bool sur = false, judge = false;
    if constexpr (!PERSIST) {
        if (k.sur && active) {
            sur = d.sur_active[gi] != 0 && sur_healthy(d);
            judge = (*d.step) % k.judge_every == 0;
        }
    }
    const bool bonds = !(sur && !judge);
    // broken-bond bits of the node's first 32 bonds: only the node's own threads
    // set them, each for its own bonds, so one load at the start serves the loop
    const uint32_t w0 = active ? __ldcg(bw) : 0u;
    unsigned note = 0u;
    // bonds in batches of kBondBatch per lane: the column indices, broken words and
    // neighbour positions of a batch are all in flight before any is used (the
    // per-lane summation order is unchanged: bonds lane, lane + LANES, ...)
    constexpr int kBondBatch = 4;
    if (stencil && bonds) {
        const uint32_t mask = st.x, alive = stn_alive(mask, w0);
        constexpr int kPerLane = (24 + LANES - 1) / LANES;
        // fully unrolled (a loop over the batches was 30 % slower on the compaction)
#pragma unroll
        for (int m0 = 0; m0 < kPerLane; m0 += kBondBatch) {
            float4 qb[kBondBatch];
            bool live[kBondBatch];
#pragma unroll
            for (int m = 0; m < kBondBatch; ++m) {
                const int o = (m0 + m) * LANES + lane;
                live[m] = (m0 + m) < kPerLane && o < 24 && ((alive >> o) & 1u);
                qb[m] = ldm<PERSIST>(&cur_pq<PERSIST>(d)[live[m] ? ii + stn_di(o) + stn_row(st, stn_dj(o)) : ii]);
            }
#pragma unroll
            for (int m = 0; m < kBondBatch; ++m) {
                if (!live[m]) continue;
                const int o = (m0 + m) * LANES + lane;
                const int dj = stn_dj(o), di = stn_di(o);
                const int n = di * di + dj * dj;
                BondGeom32 bg;
                const int r = bond_classify32(qb[m], phi, pli, (float)n, stn_sqrt_n(n), gq, s0_lo, s0_hi, bg);
                if (r == 0) {
                    bond_add32(bg, cw, inv_eps, VV, k.micro, Fbx, Fby);
                } else if (r == 2) {
                    note |= kNoteGuard;
                } else {
                    atomicOr(bw, stn_bit(mask, o));
                    note |= kNoteBroke;
                }
            }
        }
    }
    if (!stencil && bonds)
        csr_bonds32<PERSIST, LANES>(d, k, ii, lane, r0, r1, phi, pli, gq, gc, s0_lo, s0_hi, w0, Fbx, Fby, note);
    // (all threads of the node: they share its offsets out in the loop above, its
    // bonds in this pass, and a node without some offset has other ranks)
    if (any_lane<LANES>(note & kNoteGuard))
        guard_bonds32<PERSIST>(d, k, ii, r0, r1, lane, LANES, stencil, phi, pli, gq, gc, gi, s0_lo, s0_hi, bw, Fbx, Fby,
                                note);
    __syncwarp();
    float Fsx = 0.f, Fsy = 0.f, Fnx = 0.f, Fny = 0.f;
    const int nc = active ? ldm<PERSIST>(&d.nbr_cnt[ii]) : 0;
    const int nb = fresh_bonds(d, k, ii, any_lane<LANES>(w0 != 0u || (note & ~kNoteGuard) ||
                                                         (active && !bonds && k.wpn > 1)));
    if constexpr (LANES == 1) {
        if (nc + nb > 0)
            contacts32<PERSIST>(d, k, ii, vin, gi, nc, nb, r0, r1, phi, pli, gq, gc, Fsx, Fsy, Fnx, Fny);
    } else if constexpr (LANES == 2) {
        ContactNode32 mine = {};
        if (nc + nb > 0) {
            const double2 vi = ldm<PERSIST>(&d.v[vin][ii]);
            mine = {qi, vi.x, vi.y, ii, gi, ag, r0, r1, nc, nb, 0};
        }
        warp_contacts(mine, lane == 0 ? nc + nb : 0, Fsx, Fsy, Fnx, Fny,
                      [&](const ContactNode32 &x, int q, float &sx, float &sy, float &nx, float &ny) {
                          const int j = candidate<PERSIST>(d, k, x.ii, x.nc, x.nb, x.r0, q);
                          contact_pair32<PERSIST>(d, k, d.agg[x.ag], x.ii, j, vin, x.gi, x.r0, x.r1,
                                                  make_float2(x.q.x, x.q.y), make_float2(x.q.z, x.q.w),
                                                  __ldg(&d.gq[x.gi]), __ldg(&d.gc[x.gi]),
                                                  ldm<PERSIST>(&cur_pq<PERSIST>(d)[j]), make_double2(x.vx, x.vy), sx, sy,
                                                  nx, ny);
                      });
    } else {
        group_contacts<LANES>(lane, nc + nb, Fsx, Fsy, Fnx, Fny,
                              [&](int q, float &sx, float &sy, float &nx, float &ny) {
                                  const int j = candidate<PERSIST>(d, k, ii, nc, nb, r0, q);
                                  contact_pair32<PERSIST>(d, k, d.agg[ag], ii, j, vin, gi, r0, r1, phi, pli, gq, gc,
                                                          ldm<PERSIST>(&cur_pq<PERSIST>(d)[j]), ldm<PERSIST>(&d.v[vin][ii]),
                                                          sx, sy, nx, ny);
                              });
    }
    out.bx = lane_sum<LANES>(Fbx);
    out.by = lane_sum<LANES>(Fby);
    out.sx = Fsx;
    out.sy = Fsy;
    out.nx = Fnx;
    out.ny = Fny;
    if (sur && judge && lane == 0) d.sur_fb[i] = make_float2(out.bx, out.by);   // full bond force for the judge
}

// FP32 split, one thread per node: forces of the nodes [lo, hi) by the calling
// block, in tiles (see PairTile, Tile32).  All threads call out(i, sums, place,
// active, contact) with each node's sums, its update streams in shared memory at
// `place` when `update`; without INLINE the contact forces are left to a later
// pass (contact: the node has candidates).
template <bool PERSIST, int BLOCK, bool INLINE, class Out>
__device__ __forceinline__ void tile_nodes32(const DevPtrs &d, const KParams &k, int lo, int hi, int vin, bool update,
                                             Tile32<BLOCK> &sm, Out out) {
    if (lo >= hi) return;
    const int tid = threadIdx.x;
    const float4 *const pq = cur_pq<PERSIST>(d);
    const double2 *const cu = cur_u<PERSIST>(d);
    // positions are read up to kCarry nodes past the run
    const int qend = min(hi + kCarry, k.N);
    auto copy_q = [&](int i, int half) {
        if (i >= qend) return;
        copy_async(&sm.q[half * BLOCK + tid], &pq[i]);
        if (half == 0 && tid < Tile32<BLOCK>::kAhead) copy_async(&sm.q[2 * BLOCK + tid], &pq[i]);
    };
    auto copy_list = [&](int i) {
        if (i >= hi) return;
        copy_async(&sm.st[tid], &d.stn[i]);
        copy_async(&sm.gi[tid], &d.grain[i]);
        copy_async(&sm.nc[tid], &d.nbr_cnt[i]);
        copy_async(&sm.bits[tid], &d.bits[(size_t)i * k.wpn]);
    };
    auto copy_update = [&](int i) {
        if (i >= hi || !update) return;
        copy_async(&sm.v[tid], &d.v[vin][i]);
        copy_async(&sm.a[tid], &d.af[i]);
        copy_async(&sm.cell[tid], &d.cell[i]);
        copy_async(&sm.u[tid], &cu[i]);
        copy_async(&sm.xs[tid], &d.xs[i]);
        copy_async(&sm.sref[tid], &d.sref[i]);
    };
    // the pass before the run takes the nodes [lo - BLOCK, lo), of which the last kCarry have slots
    const int first = lo > 0 ? lo - BLOCK : lo;
    const int skip = lo > 0 ? BLOCK - kCarry : 0;      // threads without a node in the first pass
    int half = 0;                                      // the tile's half of the position window
    if (tid >= skip && first + tid >= 0) {
        copy_q(first + tid, 0);
        copy_list(first + tid);
    }
    copy_q(first + BLOCK + tid, 1);
    copy_commit();
    if (first == lo) copy_update(lo + tid);
    copy_commit();
    copy_wait<1>();
    __syncthreads();
    for (int node0 = first; node0 < hi; node0 += BLOCK, half ^= 1) {
        const int i = node0 + tid;
        const bool warm = node0 < lo;
        const bool active = i < hi && !(warm && (tid < skip || i < 0));
        const float4 *const win = sm.q + half * BLOCK + tid;
        float2 *const mine = sm.slot + kCarry + tid;
        BondNode32 nd;
        nd.st = make_uint4(kStnIrregular, 0u, 0u, 0u);
        nd.qi = *win;
        int gi = 0, nc = 0;
        uint32_t w0 = 0u;
        if (active) {
            nd.st = sm.st[tid];
            gi = sm.gi[tid];
            nc = sm.nc[tid];
            w0 = sm.bits[tid];
        }
        nd.gq = __ldg(&d.gq[gi]);
        nd.gc = __ldg(&d.gc[gi]);
        nd.gap = nd.st.x & kStnGap;
        const bool gaps = __any_sync(0xffffffffu, nd.gap);
        const bool stencil = !(nd.st.x & kStnIrregular) || nd.gap;
        nd.st.x &= kStnBits;
        // learned modal surrogate: between judge steps an active grain skips the
        // bond loop; the epilogue adds its surrogate bond force instead
        bool sur = false, judge = false;
        if constexpr (!PERSIST) {
            if (k.sur && active) {
                sur = d.sur_active[gi] != 0 && sur_healthy(d);
                judge = (*d.step) % k.judge_every == 0;
            }
        }
        const bool bonds = active && !(sur && !judge);
        const uint32_t alive = bonds && stencil ? stn_alive(nd.st.x, w0) : 0u;
        unsigned note = 0u;
        uint32_t *bw = &d.bits[(size_t)(active ? i : 0) * k.wpn];
        float fx = 0.f, fy = 0.f;
        if (bonds && stencil) {
            if (gaps) tile_forward32<BLOCK, true>(d, k, i, alive, nd, win, mine, bw, fx, fy, note, !warm, k.micro != 0);
            else if (k.micro) tile_forward32<BLOCK, false>(d, k, i, alive, nd, win, mine, bw, fx, fy, note, !warm, true);
            else tile_forward32<BLOCK, false>(d, k, i, alive, nd, win, mine, bw, fx, fy, note, !warm, false);
        } else {
#pragma unroll
            for (int q = 0; q < kPairHalf; ++q)
                mine[q * PairTile<float2, BLOCK>::kStride].x = __uint_as_float(kPairNone);
        }
        __syncthreads();
        // the tile's positions and lists have been read: the next ones' take their places
        copy_q(i + 2 * BLOCK, half);
        copy_list(i + BLOCK);
        copy_commit();
        if (!warm) {
            Sums32 f{0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
            bool contact = false;
            if (active) {
                if (gaps) tile_backward32<PERSIST, BLOCK, true>(d, k, i, alive, nd, mine, f.bx, f.by, note);
                else tile_backward32<PERSIST, BLOCK, false>(d, k, i, alive, nd, mine, f.bx, f.by, note);
                f.bx = __fadd_rn(f.bx, fx);
                f.by = __fadd_rn(f.by, fy);
                const float2 phi = make_float2(nd.qi.x, nd.qi.y), pli = make_float2(nd.qi.z, nd.qi.w);
                int r0 = (int)nd.st.w, r1 = r0 + __popc(nd.st.x);
                if (!stencil || note) {
                    const float s0_lo = nd.gc.y * (1.0f - k.guard), s0_hi = nd.gc.y * (1.0f + k.guard);
                    if (!stencil) {
                        r0 = __ldg(&d.row_ptr[i]);
                        r1 = __ldg(&d.row_ptr[i + 1]);
                        if (bonds)
                            csr_bonds32<PERSIST, 1>(d, k, i, 0, r0, r1, phi, pli, nd.gq, nd.gc, s0_lo, s0_hi, w0, f.bx,
                                                    f.by, note);
                    }
                    if (note & kNoteGuard)
                        guard_bonds32<PERSIST>(d, k, i, r0, r1, 0, 1, stencil, phi, pli, nd.gq, nd.gc, gi, s0_lo, s0_hi,
                                               bw, f.bx, f.by, note);
                }
                const int nb = fresh_bonds(d, k, i, w0 != 0u || (note & kNoteBroke));
                contact = nc + nb > 0;
                if (INLINE && contact)
                    contacts32<PERSIST>(d, k, i, vin, gi, nc, nb, r0, r1, phi, pli, nd.gq, nd.gc, f.sx, f.sy, f.nx,
                                           f.ny);
                if (sur && judge) d.sur_fb[i] = make_float2(f.bx, f.by);   // full bond force for the judge
            }
            copy_wait<1>();              // the node's update streams
            out(i, f, tid, active, contact);
        }
        copy_update(i + BLOCK);
        copy_commit();
        copy_wait<1>();                  // the next tile's positions and lists
        __syncthreads();
        PairTile<float2, BLOCK>::carry(sm.slot);
        __syncthreads();
    }
    copy_wait<0>();
}

// The update streams of node i from memory, all in flight together.
template <bool PERSIST>
__device__ __forceinline__ Update32 load_update32(const DevPtrs &d, int i, int vin, int update_v) {
    Update32 n{};
    n.v = ldm<PERSIST>(&d.v[vin][i]);
    n.cell = ldm<PERSIST>(&d.cell[i]);
    if (update_v) {
        n.a = ldm<PERSIST>(&d.af[i]);
        if (PERSIST) {
            // for the next step's displacement update
            n.u = ldm<PERSIST>(&cur_u<PERSIST>(d)[i]);
            n.xs = __ldg(&d.xs[i]);
            n.sref = ldm<PERSIST>(&d.sref[i]);
        }
    }
    return n;
}

template <bool PERSIST>
__device__ __forceinline__ void node_epilogue32(const DevPtrs &d, const KParams &k, int i, int gi, int vin, int update_v,
                                                const Sums32 &fin, const Update32 &n, bool total = false) {
    const double2 vi = n.v;
    const int ag = __ldg(&d.g_agg[gi]);
    const float inv_m = __ldg(&d.g_invmf[gi]);
    const int4 wc = ldm<PERSIST>(&cur_wall<PERSIST>(d)[ag]);
    Sums32 f = fin;
    if constexpr (!PERSIST) {
        // learned modal surrogate: between judge steps an active grain's bond force
        // is R(theta + phi) Phi f E h (expanded on the tensor cores), in place of
        // the bond loop the sums skipped
        if (k.sur && d.sur_active[gi] && (*d.step) % k.judge_every != 0 && sur_healthy(d)) {
            const float2 sf = d.sur_f[i];                     // Phi f, lattice frame, units of E h
            const float2 rot = d.sur_rot[gi];
            const float Eh = k.E * __ldg(&d.gq[gi]).x;
            f.bx += (rot.x * sf.x - rot.y * sf.y) * Eh;
            f.by += (rot.y * sf.x + rot.x * sf.y) * Eh;
        }
    }
    double Fwx = 0.0, Fwy = 0.0;
    const bool walls = !cells_far_from_walls(n.cell, wc);
    if (walls) {
        const double2 pi = position64<PERSIST>(d, i);
        const AggParams &A = d.agg[ag];
        const double Kn = k.mat ? 18.0 * __ldg(&d.g_k[gi]) / A.pe5 : A.Kn;
        const double rho = k.mat ? __ldg(&d.g_rho[gi]) : k.rho;
        const float Knf = k.mat ? __ldg(&d.g_kf[gi]) : A.knf, rhof = __ldg(&d.gc[gi]).w;
        wall_force32(k, A, Knf, rhof, Kn, rho, cur_time<PERSIST>(d), pi.x, pi.y, vi.x, vi.y, __ldg(&d.V[i]), Fwx,
                     Fwy, d.status);
    }
    // the lane-sum pass may have summed the parts already (f.bx / f.by hold the total)
    const float fx = total ? f.bx : (f.bx + f.sx) + f.nx, fy = total ? f.by : (f.by + f.sy) + f.ny;
    if (k.store) {
        // per-part output in FP64 (the parts as the lanes summed them, the total as the update uses it)
        d.F[i] = make_double2(f2d_bits(fx) + Fwx, f2d_bits(fy) + Fwy);
        d.parts[i] = make_double2((double)f.bx, (double)f.by);
        d.parts[k.N + i] = make_double2((double)f.sx, (double)f.sy);
        d.parts[2 * (size_t)k.N + i] = make_double2((double)f.nx, (double)f.ny);
        d.parts[3 * (size_t)k.N + i] = make_double2(Fwx, Fwy);
    }
    finish_node32_total<PERSIST>(d, k, i, vin, update_v, n, fx, fy, walls, Fwx, Fwy, inv_m);
}

// ---------------------------------------------------------------------------
// special nodes of the persistent kernel with one thread per node: those with
// contact candidates or near a wall.  They are few, but each takes several
// times as long as a plain node, and a block's run of nodes can hold many: in
// place, the blocks whose grains touch set the time of the step.  So the tile
// pass puts such a node's bond sum aside and the node on a list (one atomic per
// warp), and after a grid barrier all threads share the list.

// Appends the calling warp's nodes i with `take` set to the list.
__device__ __forceinline__ void list_special(const DevPtrs &d, int which, int i, bool take) {
    const unsigned m = __ballot_sync(0xffffffffu, take);
    if (m == 0u) return;
    const int lane = threadIdx.x & 31, lead = __ffs(m) - 1;
    int at = 0;
    if (lane == lead) at = atomicAdd(&d.spec_n[which], __popc(m));
    at = __shfl_sync(0xffffffffu, at, lead);
    if (take) d.spec[at + __popc(m & ((1u << lane) - 1u))] = i;
}

// A group of kSpecialLanes threads takes one special node: each thread a
// candidate (and, FP64 path, a wall or a corner), whose forces are then added
// in the candidates' order, so the sums are those of one thread working through
// them.  A contact is a chain of divisions and square roots -- on the 2-lane
// FP64 pipe about 4 us -- and a node has up to a dozen.
constexpr int kSpecialLanes = 8;

// (node: the group has one; every thread of the warp calls it)
template <bool PERSIST>
__device__ __forceinline__ void special_node32(const DevPtrs &d, const KParams &k, int i, bool node, int vin) {
    const int lane = threadIdx.x & (kSpecialLanes - 1);
    const int ii = node ? i : 0;
    const float2 b = reinterpret_cast<const float2 *>(d.fsum)[ii];
    const float4 qi = ldm<PERSIST>(&cur_pq<PERSIST>(d)[ii]);
    const int gi = __ldg(&d.grain[ii]), nc = node ? ldm<PERSIST>(&d.nbr_cnt[ii]) : 0;
    const int r0 = __ldg(&d.row_ptr[ii]), r1 = __ldg(&d.row_ptr[ii + 1]);
    const Update32 n = load_update32<PERSIST>(d, ii, vin, 1);
    const int nb = node ? fresh_bonds(d, k, ii, true) : 0;
    const AggParams &A = d.agg[__ldg(&d.g_agg[gi])];
    const float4 gq = __ldg(&d.gq[gi]), gc = __ldg(&d.gc[gi]);
    Sums32 f{b.x, b.y, 0.f, 0.f, 0.f, 0.f};
    for (int q0 = 0; __any_sync(0xffffffffu, q0 < nc + nb); q0 += kSpecialLanes) {
        float sx = 0.f, sy = 0.f, nx = 0.f, ny = 0.f;
        if (q0 + lane < nc + nb) {
            const int j = candidate<PERSIST>(d, k, ii, nc, nb, r0, q0 + lane);
            contact_pair32<PERSIST>(d, k, A, ii, j, vin, gi, r0, r1, make_float2(qi.x, qi.y), make_float2(qi.z, qi.w), gq,
                                    gc, ldm<PERSIST>(&cur_pq<PERSIST>(d)[j]), n.v, sx, sy, nx, ny);
        }
        const int m = nc + nb - q0;
        f.sx = add_in_order<kSpecialLanes>(f.sx, sx, m);
        f.sy = add_in_order<kSpecialLanes>(f.sy, sy, m);
        f.nx = add_in_order<kSpecialLanes>(f.nx, nx, m);
        f.ny = add_in_order<kSpecialLanes>(f.ny, ny, m);
    }
    if (node && lane == 0) node_epilogue32<PERSIST>(d, k, ii, gi, vin, 1, f, n);
}

template <bool PERSIST>
__device__ __forceinline__ void special_node64(const DevPtrs &d, const KParams &k, int i, bool node, int vin) {
    const int lane = threadIdx.x & (kSpecialLanes - 1);
    const int ii = node ? i : 0;
    const double2 b = reinterpret_cast<const double2 *>(d.fsum)[ii];
    const double2 pi = ldm<PERSIST>(&d.p[ii]), vi = ldm<PERSIST>(&d.v[vin][ii]), ao = ldm<PERSIST>(&d.a[ii]);
    const int gi = __ldg(&d.grain[ii]), nc = node ? ldm<PERSIST>(&d.nbr_cnt[ii]) : 0;
    const int r0 = __ldg(&d.row_ptr[ii]), r1 = __ldg(&d.row_ptr[ii + 1]);
    const int2 cell = ldm<PERSIST>(&d.cell[ii]);
    const int nb = node ? fresh_bonds(d, k, ii, true) : 0;
    const int ag = __ldg(&d.g_agg[gi]);
    const AggParams &A = d.agg[ag];
    Sums64 f{b.x, b.y, 0.0, 0.0, 0.0, 0.0};
    for (int q0 = 0; __any_sync(0xffffffffu, q0 < nc + nb); q0 += kSpecialLanes) {
        double sx = 0.0, sy = 0.0, nx = 0.0, ny = 0.0;
        if (q0 + lane < nc + nb) {
            const int j = candidate<PERSIST>(d, k, ii, nc, nb, r0, q0 + lane);
            contact_pair64<PERSIST>(d, k, A, ii, j, vin, gi, r0, r1, pi, ldm<PERSIST>(&d.p[j]), vi, sx, sy, nx, ny);
        }
        const int m = nc + nb - q0;
        f.sx = add_in_order<kSpecialLanes>(f.sx, sx, m);
        f.sy = add_in_order<kSpecialLanes>(f.sy, sy, m);
        f.nx = add_in_order<kSpecialLanes>(f.nx, nx, m);
        f.ny = add_in_order<kSpecialLanes>(f.ny, ny, m);
    }
    // walls: thread l takes wall l, thread 4 + c corner c
    const bool walls = node && !cells_far_from_walls(cell, ldm<PERSIST>(&cur_wall<PERSIST>(d)[ag]));
    double Fwx = 0.0, Fwy = 0.0;
    if (__any_sync(0xffffffffu, walls)) {
        double gx = 0.0, gy = 0.0;
        if (walls) {
            const double rho = k.mat ? __ldg(&d.g_rho[gi]) : k.rho;
            const double Kn = k.mat ? 18.0 * __ldg(&d.g_k[gi]) / A.pe5 : A.Kn;
            const double t = cur_time<PERSIST>(d), V = __ldg(&d.V[ii]);
            bool past, past2;
            if (lane < 4) {
                const double dl = wall_distance(A, lane, t, pi.x, pi.y, past);
                if (past) atomicAdd(&d.status[PD_STATUS_PENETRATION], 1);
                wall_single64(k, A, Kn, rho, lane, dl, vi.x, vi.y, V, gx, gy);
            } else {
                const int c = lane - 4;
                wall_corner64(k, A, Kn, rho, c, wall_distance(A, c >> 1, t, pi.x, pi.y, past),
                              wall_distance(A, 2 + (c & 1), t, pi.x, pi.y, past2), vi.x, vi.y, V, gx, gy);
                gx = -gx;
                gy = -gy;
            }
        }
        Fwx = add_in_order<kSpecialLanes>(0.0, gx, kSpecialLanes);
        Fwy = add_in_order<kSpecialLanes>(0.0, gy, kSpecialLanes);
    }
    if (!node || lane != 0) return;
    const double inv_m = __ldg(&d.g_invm[gi]);
    if (k.store)
        finish_node<PERSIST, true>(d, k, ii, vin, 1, vi, 0.0, f.bx, f.by, f.sx, f.sy, f.nx, f.ny, Fwx, Fwy, inv_m);
    else
        finish_node64_total<PERSIST>(d, k, ii, vin, 1, vi, ao, __dadd_rn(__dadd_rn(f.bx, f.sx), f.nx),
                                     __dadd_rn(__dadd_rn(f.by, f.sy), f.ny), walls, Fwx, Fwy, inv_m);
}

}  // namespace pd
