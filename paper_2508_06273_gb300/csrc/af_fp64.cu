// af_fp64.cu -- the step in FP64 (AF_OPT_FP64): storage, reconstruction,
// EG2 with the correction term, Simpson fluxes and the average update all in
// double precision.  It exists for accuracy studies below the FP32 floor of
// the point values (Tables 1 and 2 of Sec. 2 at 512 and 1024 cells), not for
// speed: this GPU's FP64 rate is a small fraction of its FP32 rate.
//
// Scope: Alg. 1 with the linearisations of Sec. 2 and Sec. 3.1 (averaged,
// node value, Alg. 1's dt/4 step) and Corollary 1's correction; periodic,
// outflow and solid-wall boundaries.  The limiters and switches of Sec. 3
// (Alg. 2, Alg. 3, the Sec. 3.4 blend, the flux limiter) are not part of this
// path: the host refuses a step with any of them on.
//
// Layout: the padded planes of the FP32 path with 8-byte elements; the cell
// records (9 monomial coefficients of each variable's biquadratic about the
// cell centre, then Ubar) are built once per step by their own kernel into a
// global array, and the node kernel reads them through the L1 cache.
#include <cuda_runtime.h>

#include "af_common.cuh"
#include "af_kernels.h"

namespace af {

namespace {

// a cell record: 4 variables x 8 monomial coefficients (x, x^2, y, y^2, xy,
// x y^2, x^2 y, x^2 y^2), the four values at the centre, Ubar (4)
constexpr int REC64 = REC64_DOUBLES, M00_64 = 32, UBAR_64 = 36;
constexpr double PI_D = 3.14159265358979323846;

__host__ __device__ __forceinline__ long long cell_index(const Grid &g, int i, int j) {
#if defined(AF_CHECK_BOUNDS) && defined(__CUDA_ARCH__)
  if (!bounds_ok(i + OX >= 0 && i + OX < g.P && j + OY >= 0 && j + OY < g.H, BD_RECORD64)) return 0;
#endif
  return (long long)(j + OY) * g.P + (i + OX);
}

__device__ __forceinline__ void p2c_d(const double U[4], double gm1i, double Q[4]) {
  Q[0] = U[0];
  Q[1] = U[0] * U[1];
  Q[2] = U[0] * U[2];
  Q[3] = U[3] * gm1i + 0.5 * U[0] * (U[1] * U[1] + U[2] * U[2]);
}
__device__ __forceinline__ void c2p_d(const double Q[4], double gm1, double U[4]) {
  const double ir = 1.0 / Q[0];
  U[0] = Q[0];
  U[1] = Q[1] * ir;
  U[2] = Q[2] * ir;
  U[3] = gm1 * (Q[3] - 0.5 * (Q[1] * Q[1] + Q[2] * Q[2]) * ir);
}
__device__ __forceinline__ void ld4d(const Grid &g, const double *p, int i, int j, double U[4]) {
#pragma unroll
  for (int v = 0; v < NV; v++) U[v] = p[at(g, v, i, j)];
}
__device__ __forceinline__ void st4d(double *p, const Grid &g, int i, int j, const double U[4]) {
#pragma unroll
  for (int v = 0; v < NV; v++) p[at(g, v, i, j)] = U[v];
}

// ---- cell prep (Sec. 2) and the cell record
// nodal values f[k][l] at local (k/2, l/2) -> coefficients m[a][b] of x^a y^b
// (x, y in [-1/2, 1/2] about the cell centre)
__device__ __forceinline__ void to_monomial_d(const double f[3][3], double m[3][3]) {
  double r[3][3];
#pragma unroll
  for (int l = 0; l < 3; l++) {
    r[0][l] = f[1][l];
    r[1][l] = f[2][l] - f[0][l];
    r[2][l] = 2.0 * (f[0][l] + f[2][l]) - 4.0 * f[1][l];
  }
#pragma unroll
  for (int a = 0; a < 3; a++) {
    m[a][0] = r[a][1];
    m[a][1] = r[a][2] - r[a][0];
    m[a][2] = 2.0 * (r[a][0] + r[a][2]) - 4.0 * r[a][1];
  }
}

// record of cell (ci, cj): Q_c by Simpson's rule solved for the centre,
// U_c = C2P(Q_c), Ubar (Simpson over the primitive point values, or C2P of the
// average with ubar_c2p), and the biquadratic of each primitive variable
__device__ void build_record(const Grid &g, double gam, const double *avg, const double *vtx, const double *xe,
                             const double *ye, int ci, int cj, double *rec) {
  const double gm1 = gam - 1.0, gm1i = 1.0 / gm1;
  double N[8][4];  // corners (ll, lr, ul, ur), then edges (left, right, bottom, top)
  ld4d(g, vtx, ci, cj, N[0]);
  ld4d(g, vtx, ci + 1, cj, N[1]);
  ld4d(g, vtx, ci, cj + 1, N[2]);
  ld4d(g, vtx, ci + 1, cj + 1, N[3]);
  ld4d(g, xe, ci, cj, N[4]);
  ld4d(g, xe, ci + 1, cj, N[5]);
  ld4d(g, ye, ci, cj, N[6]);
  ld4d(g, ye, ci, cj + 1, N[7]);
  double Qs[4] = {0, 0, 0, 0}, Us[4] = {0, 0, 0, 0}, Qa[4], Qc[4], Uc[4], Ub[4];
  for (int n = 0; n < 8; n++) {
    double Q[4];
    p2c_d(N[n], gm1i, Q);
    const double w = n < 4 ? 1.0 : 4.0;
    for (int v = 0; v < NV; v++) {
      Qs[v] += w * Q[v];
      Us[v] += w * N[n][v];
    }
  }
  ld4d(g, avg, ci, cj, Qa);
  for (int v = 0; v < NV; v++) Qc[v] = (36.0 * Qa[v] - Qs[v]) / 16.0;
  c2p_d(Qc, gm1, Uc);
  if (g.ubar_c2p) {
    c2p_d(Qa, gm1, Ub);
  } else {
    for (int v = 0; v < NV; v++) Ub[v] = (Us[v] + 16.0 * Uc[v]) / 36.0;
  }
  for (int v = 0; v < NV; v++) {
    const double f[3][3] = {{N[0][v], N[4][v], N[2][v]}, {N[6][v], Uc[v], N[7][v]}, {N[1][v], N[5][v], N[3][v]}};
    double m[3][3];
    to_monomial_d(f, m);
    double2 *r2 = reinterpret_cast<double2 *>(rec + 8 * v);
    r2[0] = make_double2(m[1][0], m[2][0]);
    r2[1] = make_double2(m[0][1], m[0][2]);
    r2[2] = make_double2(m[1][1], m[1][2]);
    r2[3] = make_double2(m[2][1], m[2][2]);
    rec[M00_64 + v] = m[0][0];
    rec[UBAR_64 + v] = Ub[v];
  }
}

// ---- EG2 (eq. (EG2)) in FP64: the FP32 kernel's sums in truncated-power form
// (af_pointvalue.cuh, "EG2 arc sums in the truncated-power form"; the same
// symbols and recurrences), in double and reading the records through L1.
// The kernel is bound by the FP64 pipe (2 multiply-adds a clock and SM), so what
// counts is the number of FP64 operations: the tables come from recurrences on
// (a, sqrt(1 - a^2), acos a) without sin or cos calls, one division and one
// reciprocal square root serve the linearisation state.  The form before it
// built three full 5 x 5 tables with sines and cosines of the arcs' ends and
// contracted four cells' nine coefficients.  Now 2380 FP64 instructions a cell
// at 88 % of the pipe; node updates at 192^2 381 -> 180 us, a whole step 468 ->
// 241 us (512^2: 3.03 -> 1.67 ms).
__device__ __forceinline__ void taylor_d(double a0, double a1, double a2, double x0, double &t0, double &t1) {
  const double t = fma(a2, x0, a1);
  t0 = fma(t, x0, a0);
  t1 = fma(a2, x0, t);
}
__device__ __forceinline__ double horner_d(double a0, double a1, double a2, double x0) {
  return fma(fma(a2, x0, a1), x0, a0);
}
struct Coef64 {
  double m10, m20, m01, m02, m11, m12, m21, m22;
};
__device__ __forceinline__ Coef64 coef_d(const double *rec, int v) {
  const double2 *r = reinterpret_cast<const double2 *>(rec) + 4 * v;
  const double2 a = __ldg(r), b = __ldg(r + 1), c = __ldg(r + 2), d = __ldg(r + 3);
  return Coef64{a.x, a.y, b.x, b.y, c.x, c.y, d.x, d.y};
}
__device__ __forceinline__ double eval_at_d(const Coef64 &m, double m00, double x0, double y0) {
  return horner_d(horner_d(m00, m.m10, m.m20, x0), horner_d(m.m01, m.m11, m.m21, x0),
                  horner_d(m.m02, m.m12, m.m22, x0), y0);
}
struct Circle64 {
  double x0, y0, rx, ry, rx2, ry2;
};
// whole-circle sums of the reference cell's polynomial, divided by pi
template <int VAR>
__device__ __forceinline__ void circle_sums_d(const Coef64 &m, double m00, const Circle64 &c, double s[3],
                                              double &centre) {
  constexpr bool YF = VAR == 2;
  const double f0 = YF ? c.y0 : c.x0, s0 = YF ? c.x0 : c.y0;
  const double m20 = YF ? m.m02 : m.m20, m21 = YF ? m.m12 : m.m21;
  double r00, r10, r01, r11, r02, r12;
  taylor_d(m00, YF ? m.m01 : m.m10, m20, f0, r00, r10);
  taylor_d(YF ? m.m10 : m.m01, m.m11, m21, f0, r01, r11);
  taylor_d(YF ? m.m20 : m.m02, YF ? m.m21 : m.m12, m.m22, f0, r02, r12);
  double t00, t01, t10, t11;
  taylor_d(r00, r01, r02, s0, t00, t01);
  taylor_d(r10, r11, r12, s0, t10, t11);
  const double t20 = horner_d(m20, m21, m.m22, s0);
  const double rf = YF ? c.ry : c.rx, rs = YF ? c.rx : c.ry, rf2 = YF ? c.ry2 : c.rx2, rs2 = YF ? c.rx2 : c.ry2;
  centre = t00;
  if (VAR == 0) {
    const double t21 = fma(2.0 * s0, m.m22, m21);
    s[0] = fma(2.0, t00, fma(rf2, fma(0.25 * rs2, m.m22, t20), rs2 * r02));
    s[1] = rf * fma(0.25 * rs2, r12, t10);
    s[2] = rs * fma(0.25 * rf2, t21, t01);
  } else {
    s[0] = rf * fma(0.25 * rs2, r12, t10);
    s[1] = fma(rf2, fma(0.125 * rs2, m.m22, t20), t00);
    s[2] = (0.25 * rf) * (rs * t11);
  }
}

// moments over {cos > a} divided by pi, [times sin^2][X, X^2]
struct Half64 {
  double one[2][2], c[2][2], K[2][2], V[2][2];
};
__device__ __forceinline__ void half_table_d(double a, double s, double al, double r, double r2, Half64 &H) {
  const double q = s * s;
  const double L0 = (2.0 / PI_D) * al, L1 = (2.0 / PI_D) * fma(-a, al, s);
  const double L2 = 0.5 * fma(q, L0, -3.0 * (a * L1));
  const double N0 = fma(a, L1, L2);
  const double N1 = fma((2.0 / (3.0 * PI_D)) * q, s, -a * N0);
  const double N2 = 0.25 * fma(q, N0, -5.0 * (a * N1));
  const double N3 = fma(0.4 * q, N1, -1.4 * (a * N2));
  const double N4 = fma(0.5 * q, N2, -1.5 * (a * N3));
  const double CN1 = fma(a, N1, N2), CN2 = fma(a, N2, N3), CN3 = fma(a, N3, N4);
  H.one[0][0] = r * L1;
  H.one[0][1] = r2 * L2;
  H.one[1][0] = r * N1;
  H.one[1][1] = r2 * N2;
  H.c[0][0] = r * N0;
  H.c[0][1] = (2.0 * r2) * N1;
  H.c[1][0] = r * CN1;
  H.c[1][1] = r2 * CN2;
  const double W[2] = {(3.0 * r) * CN2, (2.0 * r2) * CN3};
#pragma unroll
  for (int k = 0; k < 2; k++) {
    H.K[0][k] = fma(1.5, H.one[0][k], -2.0 * H.one[1][k]);
    H.K[1][k] = fma(1.5, H.one[1][k], -W[k]);
    H.V[0][k] = H.one[0][k] - H.K[0][k];
    H.V[1][k] = fma(-0.5, H.one[1][k], W[k]);
  }
}

// jumps across a vertical (YL = false) or horizontal grid line: d[k][n], the
// coefficients of X^(k+1) and the tangential power n
template <bool YL>
__device__ __forceinline__ void jumps_d(const Coef64 &R, const Coef64 &O, double f, double d[2][3]) {
  const double r1[3] = {YL ? R.m01 : R.m10, R.m11, YL ? R.m21 : R.m12}, r2[3] = {YL ? R.m02 : R.m20, YL ? R.m12 : R.m21, R.m22};
  const double o1[3] = {YL ? O.m01 : O.m10, O.m11, YL ? O.m21 : O.m12}, o2[3] = {YL ? O.m02 : O.m20, YL ? O.m12 : O.m21, O.m22};
#pragma unroll
  for (int n = 0; n < 3; n++) {
    d[0][n] = fma(f, o1[n] - r1[n], -(o2[n] + r2[n]));
    d[1][n] = o2[n] - r2[n];
  }
}
// VAR 0: p; 1: the velocity normal to the line; 2: the tangential one
template <int VAR>
__device__ __forceinline__ void half_sums_d(const double d[2][3], double t0, double rt, double rt2, const Half64 &H,
                                            double &m0, double &m1, double &m2) {
#pragma unroll
  for (int k = 0; k < 2; k++) {
    double e0, e1;
    taylor_d(d[k][0], d[k][1], d[k][2], t0, e0, e1);
    e1 *= rt;
    const double e2 = d[k][2] * rt2;
    if (VAR == 0) {
      m0 = fma(e0, H.one[0][k], fma(e2, H.one[1][k], m0));
      m1 = fma(e0, H.c[0][k], fma(e2, H.c[1][k], m1));
      m2 = fma(e1, H.one[1][k], m2);
    } else if (VAR == 1) {
      m0 = fma(e0, H.c[0][k], fma(e2, H.c[1][k], m0));
      m1 = fma(e0, H.K[0][k], fma(e2, H.K[1][k], m1));
      m2 = fma(e1, H.c[1][k], m2);
    } else {
      m0 = fma(e1, H.one[1][k], m0);
      m1 = fma(e0, H.V[0][k], fma(e2, H.V[1][k], m1));
      m2 = fma(e1, H.c[1][k], m2);
    }
  }
}

// moments over the quarter (asin b, acos a), divided by pi: XY, X^2 Y, X Y^2, X^2 Y^2
struct Quarter64 {
  double one[4], c[4], s[4], K[4], V[4], Z[4];
};
__device__ __forceinline__ void quarter_moments_d(double a, double b, double sa, double sb, double phi, Quarter64 &T) {
  constexpr double IP = 1.0 / PI_D;
  const double kap = fma(-a, a, fma(-b, b, 1.0));
  const double q00 = IP * phi, pa = IP * (sa - b), pb = IP * (sb - a), q10 = fma(-a, q00, pa), q01 = fma(-b, q00, pb);
  const double q11 = fma(0.5 * IP, kap, -fma(b, pa, fma(a, pb, -a * b * q00)));
  const double h = 0.5 * fma(kap, q00, -fma(a, q10, b * q01));
  const double q20 = fma(-a, q10, h), q02 = fma(-b, q01, h);
  const double q12 = (1.0 / 3.0) * fma(kap, q10, -fma(4.0 * b, q11, a * q20));
  const double q21 = (1.0 / 3.0) * fma(kap, q01, -fma(4.0 * a, q11, b * q02));
  const double t = 0.5 * fma(kap, q11, -fma(a, q21, b * q12));
  const double q31 = fma(-a, q21, t), q13 = fma(-b, q12, t);
  const double q30 = fma(2.0, fma(b, q11, q12), -a * q20);
  const double q22 = 0.25 * fma(kap, q20, -fma(5.0 * b, q21, a * q30));
  const double D41 = 0.6 * fma(kap, q21, -fma(a, q31, b * q22)), D14 = 0.6 * fma(kap, q12, -fma(b, q13, a * q22));
  const double E23 = (2.0 / 3.0) * D41, E32 = (2.0 / 3.0) * D14;
  const double q41 = fma(-a, q31, D41), q23 = fma(-b, q22, E23), q32 = fma(-a, q22, E32);
  const double F = 0.5 * fma(kap, q22, -fma(a, q32, b * q23)), Gs = (1.0 / 3.0) * fma(kap, q31, -fma(a, q41, b * q32));
  const double c11 = fma(a, q11, q21), c12 = fma(a, q12, q22), s11 = fma(b, q11, q12), s21 = fma(b, q21, q22);
  const double one[4] = {q11, q21, q12, q22}, c[4] = {c11, t, c12, E32}, sn[4] = {s11, s21, t, E23};
  const double cc[4] = {fma(a, c11, t), fma(a, t, D41), fma(a, c12, E32), fma(a, E32, F)};
  const double z[4] = {fma(a, s11, s21), fma(a, s21, fma(b, q31, q32)), fma(a, t, E23), fma(a, E23, Gs)};
#pragma unroll
  for (int k = 0; k < 4; k++) {
    T.one[k] = one[k];
    T.c[k] = c[k];
    T.s[k] = sn[k];
    T.Z[k] = z[k];
    T.K[k] = fma(2.0, cc[k], -0.5 * one[k]);
    T.V[k] = one[k] - T.K[k];
  }
}
__device__ __forceinline__ void quarter_sums_d(const double g[4], const double w0[4], const double w1[4],
                                               const double w2[4], double &m0, double &m1, double &m2) {
#pragma unroll
  for (int k = 0; k < 4; k++) {
    m0 = fma(g[k], w0[k], m0);
    m1 = fma(g[k], w1[k], m1);
    m2 = fma(g[k], w2[k], m2);
  }
}

__device__ __forceinline__ const double *rec_at(const Grid &g, const double *recs, int ci, int cj) {
  return recs + REC64 * cell_index(g, ci, cj);
}

// the jumps across an edge midpoint's own line (p, u, v), the same for both
// time levels; seen from the other side the coefficients of X^2 change sign
struct LineJumps64 {
  double d[3][2][3];
};
template <int K>
__device__ __forceinline__ void line_jumps_d(const Grid &g, const double *recs, int i, int j, LineJumps64 &J) {
  if (K == VTX) return;
  const double *r = rec_at(g, recs, K == XE ? i - 1 : i, K == YE ? j - 1 : j), *o = rec_at(g, recs, i, j);
  jumps_d<K == YE>(coef_d(r, 3), coef_d(o, 3), 1.0, J.d[0]);
  jumps_d<K == YE>(coef_d(r, 1), coef_d(o, 1), 1.0, J.d[1]);
  jumps_d<K == YE>(coef_d(r, 2), coef_d(o, 2), 1.0, J.d[2]);
}

// EG2 of the cpq reconstruction at node (K, i, j), linearised about ul,
// relative to the reference state Kr; false if the Mach-cone base leaves the
// node's block of cells (the CFL bound of the linearisation state fails).
template <int K>
__device__ __forceinline__ bool eg2_d(const Grid &g, const Phys64 &ph, const double *recs, int i, int j,
                                      const double Kr[4], const double ul[4], double tau, const LineJumps64 &J,
                                      double out[4]) {
  if (!(ul[0] > 0.0 && ul[3] > 0.0 && tau > 0.0)) {
    for (int v = 0; v < NV; v++) out[v] = nan("");
    return true;
  }
  const double irp = 1.0 / ul[0], cp2 = ph.gam * ul[3] * irp, icp = rsqrt(cp2), cp = cp2 * icp;
  const double R = cp * tau, ut = ul[1] * tau, vt = ul[2] * tau;
  bool inside;
  {
    const double ex = fabs(ut) + R, ey = fabs(vt) + R;
    const double lx = (K == YE) ? 0.5 * ph.dx : ph.dx, ly = (K == XE) ? 0.5 * ph.dy : ph.dy;
    inside = !(ex > lx || ey > ly);
  }
  const double rx = R * ph.idx, ry = R * ph.idy;
  const bool nx_ = K != YE && ul[1] < 0.0, ny_ = K != XE && ul[2] < 0.0;
  const double fx = nx_ ? -1.0 : 1.0, fy = ny_ ? -1.0 : 1.0;
  const double ax = fabs(ul[1]) * icp, by = fabs(ul[2]) * icp;
  // reference cell (side -- of the reflected frame) and those across the lines
  const int ir = (K == YE) ? i : i - (nx_ ? 0 : 1), jr = (K == XE) ? j : j - (ny_ ? 0 : 1);
  const int io = (K == YE) ? i : i - (nx_ ? 1 : 0), jo = (K == XE) ? j : j - (ny_ ? 1 : 0);
  const double *rr = rec_at(g, recs, ir, jr);
  const double *rX = rec_at(g, recs, io, jr), *rY = rec_at(g, recs, ir, jo), *rQ = rec_at(g, recs, io, jo);
  const Circle64 C{fma(-ut, ph.idx, (K == YE) ? 0.0 : 0.5 * fx), fma(-vt, ph.idy, (K == XE) ? 0.0 : 0.5 * fy),
                   fx * rx, fy * ry, rx * rx, ry * ry};
  double Sp[3], Su[3], Sv[3], dpP, unused;
  circle_sums_d<0>(coef_d(rr, 3), __ldg(rr + M00_64 + 3) - Kr[3], C, Sp, dpP);
  circle_sums_d<1>(coef_d(rr, 1), __ldg(rr + M00_64 + 1) - Kr[1], C, Su, unused);
  circle_sums_d<2>(coef_d(rr, 2), __ldg(rr + M00_64 + 2) - Kr[2], C, Sv, unused);
  double alx = 0.0, snx = 0.0, aly = 0.0, sny = 0.0, d[2][3];
  if (K != YE && ax < 1.0) {
    alx = acos(ax);
    snx = sqrt(fma(-ax, ax, 1.0));
    Half64 H;
    half_table_d(ax, snx, alx, rx, K == XE ? fx * C.rx2 : C.rx2, H);
    if (K == VTX) jumps_d<false>(coef_d(rr, 3), coef_d(rX, 3), fx, d);
    half_sums_d<0>(K == VTX ? d : J.d[0], C.y0, C.ry, C.ry2, H, Sp[0], Sp[1], Sp[2]);
    if (K == VTX) jumps_d<false>(coef_d(rr, 1), coef_d(rX, 1), fx, d);
    half_sums_d<1>(K == VTX ? d : J.d[1], C.y0, C.ry, C.ry2, H, Su[0], Su[1], Su[2]);
    if (K == VTX) jumps_d<false>(coef_d(rr, 2), coef_d(rX, 2), fx, d);
    half_sums_d<2>(K == VTX ? d : J.d[2], C.y0, C.ry, C.ry2, H, Sv[0], Sv[1], Sv[2]);
  }
  if (K != XE && by < 1.0) {
    aly = acos(by);
    sny = sqrt(fma(-by, by, 1.0));
    Half64 H;
    half_table_d(by, sny, aly, ry, K == YE ? fy * C.ry2 : C.ry2, H);
    if (K == VTX) jumps_d<true>(coef_d(rr, 3), coef_d(rY, 3), fy, d);
    half_sums_d<0>(K == VTX ? d : J.d[0], C.x0, C.rx, C.rx2, H, Sp[0], Sp[2], Sp[1]);
    if (K == VTX) jumps_d<true>(coef_d(rr, 2), coef_d(rY, 2), fy, d);
    half_sums_d<1>(K == VTX ? d : J.d[2], C.x0, C.rx, C.rx2, H, Sv[0], Sv[1], Sv[2]);
    if (K == VTX) jumps_d<true>(coef_d(rr, 1), coef_d(rY, 1), fy, d);
    half_sums_d<2>(K == VTX ? d : J.d[1], C.x0, C.rx, C.rx2, H, Su[0], Su[1], Su[2]);
  }
  if (K == VTX && fma(ax, ax, by * by) < 1.0) {
    Quarter64 T;
    quarter_moments_d(ax, by, snx, sny, alx + aly - 0.5 * PI_D, T);
    const double rxy = rx * ry;
    auto crossing = [&](int v, double gq[4]) {
      const Coef64 m = coef_d(rr, v), x = coef_d(rX, v), y = coef_d(rY, v), q = coef_d(rQ, v);
      const double l1 = fma(fx, x.m11 - m.m11, -(x.m21 + m.m21)), l2 = fma(fx, x.m12 - m.m12, -(x.m22 + m.m22));
      const double u1 = fma(fx, q.m11 - y.m11, -(q.m21 + y.m21)), u2 = fma(fx, q.m12 - y.m12, -(q.m22 + y.m22));
      const double k1 = x.m21 - m.m21, k2 = x.m22 - m.m22, w1 = q.m21 - y.m21, w2 = q.m22 - y.m22;
      gq[0] = rxy * fma(fy, u1 - l1, -(u2 + l2));
      gq[1] = rxy * rx * fma(fy, w1 - k1, -(w2 + k2));
      gq[2] = rxy * ry * (u2 - l2);
      gq[3] = rxy * rxy * (w2 - k2);
    };
    double gq[4];
    crossing(3, gq);
    quarter_sums_d(gq, T.one, T.c, T.s, Sp[0], Sp[1], Sp[2]);
    crossing(1, gq);
    quarter_sums_d(gq, T.c, T.K, T.Z, Su[0], Su[1], Su[2]);
    crossing(2, gq);
    quarter_sums_d(gq, T.s, T.V, T.Z, Sv[0], Sv[1], Sv[2]);
  }
  // sums odd in cos change sign with fx, odd in sin with fy, back in the grid frame
  const double irc = icp * irp, icp2 = icp * icp, fxy = 2.0 * fx * fy;
  const double z = fma(-ul[0] * cp, fma(fx, Su[0], fy * Sv[0]), Sp[0]);
  const double drP = eval_at_d(coef_d(rr, 0), __ldg(rr + M00_64) - Kr[0], C.x0, C.y0);
  out[0] = Kr[0] + drP + icp2 * fma(-2.0, dpP, z);
  out[1] = Kr[1] + fma(-fx * irc, Sp[1], fma(fxy, Sv[2], Su[1]));
  out[2] = Kr[2] + fma(-fy * irc, Sp[2], fma(fxy, Su[2], Sv[1]));
  out[3] = Kr[3] + (z - dpP);
  return inside;
}

// Corollary 1: T such that C = tau^2/2 T, from centred differences of
// neighbouring point values or cell-centre values (the record's m00)
template <int K>
__device__ void correction_d(const Grid &g, const Step64 &S, int i, int j, const double U[4], double T[4]) {
  double Ux[4], Uy[4];
  const double idx = S.ph.idx, idy = S.ph.idy;
  for (int v = 0; v < NV; v++) {
    if (K == VTX) {
      Ux[v] = (S.n0[YE][at(g, v, i, j)] - S.n0[YE][at(g, v, i - 1, j)]) * idx;
      Uy[v] = (S.n0[XE][at(g, v, i, j)] - S.n0[XE][at(g, v, i, j - 1)]) * idy;
    } else if (K == XE) {
      Ux[v] = (rec_at(g, S.recs, i, j)[M00_64 + v] - rec_at(g, S.recs, i - 1, j)[M00_64 + v]) * idx;
      Uy[v] = (S.n0[VTX][at(g, v, i, j + 1)] - S.n0[VTX][at(g, v, i, j)]) * idy;
    } else {
      Ux[v] = (S.n0[VTX][at(g, v, i + 1, j)] - S.n0[VTX][at(g, v, i, j)]) * idx;
      Uy[v] = (rec_at(g, S.recs, i, j)[M00_64 + v] - rec_at(g, S.recs, i, j - 1)[M00_64 + v]) * idy;
    }
  }
  const double r = U[0], u = U[1], v = U[2], p = U[3], gm = S.ph.gam, ir = 1.0 / r;
  const double rx = Ux[0], ux = Ux[1], vx = Ux[2], px = Ux[3];
  const double ry = Uy[0], uy = Uy[1], vy = Uy[2], py = Uy[3];
  const double f1 = ux * ux + uy * vx, f2 = uy * vx + vy * vy;
  const double g1 = px * (gm * (ux + vy) + ux) + py * vx;
  const double g2 = py * (gm * (ux + vy) + vy) + px * uy;
  const double h1 = (rx * px + ry * py) * ir, h2 = (rx * u + ry * v) * ir * ir;
  T[0] = r * (f1 + f2) + u * (rx * (2.0 * ux + vy) + ry * vx) + v * (rx * uy + ry * (ux + 2.0 * vy)) - h1;
  T[1] = u * f1 + v * uy * (ux + vy) + g1 * ir - px * h2;
  T[2] = v * f2 + u * vx * (ux + vy) + g2 * ir - py * h2;
  T[3] = u * g1 + v * g2 + gm * p * (f1 + f2 - h1 * ir);
}

// averaged linearisation state, eq. (Un+1/2): Ubar of the cells around the node
template <int K>
__device__ void lin_avg_d(const Grid &g, const double *recs, int i, int j, double ul[4]) {
  for (int v = 0; v < NV; v++) {
    if (K == VTX)
      ul[v] = 0.25 * (rec_at(g, recs, i - 1, j - 1)[UBAR_64 + v] + rec_at(g, recs, i, j - 1)[UBAR_64 + v] +
                      rec_at(g, recs, i - 1, j)[UBAR_64 + v] + rec_at(g, recs, i, j)[UBAR_64 + v]);
    else if (K == XE)
      ul[v] = 0.5 * (rec_at(g, recs, i - 1, j)[UBAR_64 + v] + rec_at(g, recs, i, j)[UBAR_64 + v]);
    else
      ul[v] = 0.5 * (rec_at(g, recs, i, j - 1)[UBAR_64 + v] + rec_at(g, recs, i, j)[UBAR_64 + v]);
  }
}

__device__ void st4d_node(double *p, const Grid &g, int K, int i, int j, const double U[4]) {
  st4d(p, g, i, j, U);
  const bool dx_ = (K != YE) && g.per_x && i == 0, dy_ = (K != XE) && g.per_y && j == 0;
  if (dx_) st4d(p, g, g.nx, j, U);
  if (dy_) st4d(p, g, i, g.ny, U);
  if (dx_ && dy_) st4d(p, g, g.nx, g.ny, U);
}

// both time levels of node (K, i, j) (Alg. 1 without the Sec. 3 limiters)
template <int K>
__device__ __forceinline__ void node64(const Step64 &S, int i, int j, bool &cfl_bad, bool &nonfinite) {
  const Grid &g = S.g;
  double U0[4], T[4] = {0.0, 0.0, 0.0, 0.0}, ul[4], res[4];
  ld4d(g, S.n0[K], i, j, U0);
  if (S.correction) correction_d<K>(g, S, i, j, U0, T);
  const bool alg1 = S.lin_mode == 2;
  if (S.lin_mode != 0) {
    // (Alg. 1: level 0 of the loop below turns this into EG2's value over dt/4)
    for (int v = 0; v < NV; v++) ul[v] = U0[v];
  } else {
    const bool wx = (K != YE) && ((i == 0 && g.bc[0] == BC_REFLECTING) || (i == g.nx && g.bc[1] == BC_REFLECTING));
    const bool wy = (K != XE) && ((j == 0 && g.bc[2] == BC_REFLECTING) || (j == g.ny && g.bc[3] == BC_REFLECTING));
    if (wx || wy) {
      for (int v = 0; v < NV; v++) ul[v] = U0[v];
      if (wx) ul[1] = 0.0;
      if (wy) ul[2] = 0.0;
    } else {
      lin_avg_d<K>(g, S.recs, i, j, ul);
    }
  }
  LineJumps64 J;
  line_jumps_d<K>(g, S.recs, i, j, J);
#pragma unroll 1
  for (int lev = alg1 ? 0 : 1; lev <= 2; lev++) {
    const double tau = lev == 0 ? 0.25 * S.dt : (lev == 1 ? 0.5 * S.dt : S.dt);
    cfl_bad |= !eg2_d<K>(g, S.ph, S.recs, i, j, U0, ul, tau, J, res);
    if (lev > 0) {
      for (int v = 0; v < NV; v++) {
        res[v] = fma(0.5 * tau * tau, T[v], res[v]);
        nonfinite |= !isfinite(res[v]);
      }
      st4d_node(lev == 1 ? S.n1[K] : S.n2[K], g, K, i, j, res);
    }
    for (int v = 0; v < NV; v++) ul[v] = res[v];
  }
}

// all nodes in one launch: blocks [0, nb[0]) take vertices, the longest, then
// x-edge and y-edge midpoints, so that the kinds fill one another's tail
constexpr int NODE64_THREADS = 128;
__global__ void __launch_bounds__(NODE64_THREADS, 2) node64_kernel(Step64 S, int nbv, int nbx) {
  const Grid &g = S.g;
  const int b = blockIdx.x, kind = b < nbv ? VTX : (b < nbv + nbx ? XE : YE);
  const long long e = (long long)(b - (kind == VTX ? 0 : (kind == XE ? nbv : nbv + nbx))) * NODE64_THREADS + threadIdx.x;
  const int ni = kind == YE ? g.nx : g.nxv, nj = kind == XE ? g.ny : g.nyv;
  if (e >= (long long)ni * nj) return;
  const int i = (int)(e % ni), j = (int)(e / ni);
  bool cfl_bad = false, nonfinite = false;
  if (kind == VTX) node64<VTX>(S, i, j, cfl_bad, nonfinite);
  else if (kind == XE) node64<XE>(S, i, j, cfl_bad, nonfinite);
  else node64<YE>(S, i, j, cfl_bad, nonfinite);
  const int st = (cfl_bad ? ST_CFL : 0) | (nonfinite ? ST_NONFINITE : 0);
  if (st) atomicOr(S.status, st);
}

// records of cells -1 .. nx, -1 .. ny
__global__ void record64_kernel(Step64 S) {
  const Grid &g = S.g;
  const int w = g.nx + 2, h = g.ny + 2;
  const long long n = (long long)w * h;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
    const int ci = (int)(e % w) - 1, cj = (int)(e / w) - 1;
    build_record(g, S.ph.gam, S.avg, S.n0[VTX], S.n0[XE], S.n0[YE], ci, cj, S.recs + REC64 * cell_index(g, ci, cj));
  }
}

// f (dir 0) or g (dir 1) at primitive U
__device__ __forceinline__ void phys_flux_d(const double U[4], double gm1i, int dir, double F[4]) {
  const double r = U[0], u = U[1], v = U[2], p = U[3];
  const double un = dir == 0 ? u : v;
  const double E = p * gm1i + 0.5 * r * (u * u + v * v);
  F[0] = r * un;
  F[1] = r * u * un + (dir == 0 ? p : 0.0);
  F[2] = r * v * un + (dir == 1 ? p : 0.0);
  F[3] = un * (E + p);
}
struct Flux64 {
  Grid g;
  Phys64 ph;
  const double *n[3][3];  // [level][kind]
  double *avg;
  double lx, ly;  // dt/dx, dt/dy
  int *status;
};
// Simpson fluxes of eq. (F) and eq. (2dfvm) on a tile of F64_X x F64_Y cells:
// each node's flux is integrated in time once (weights 1, 4, 1 over the three
// levels), each face flux formed once from its three nodes (1, 4, 1) / 36, so
// the two cells sharing a face subtract the same number.  The FP64 pipe bounds
// it (84 %): 12 flux evaluations a cell instead of the 36 of a thread per cell
// that forms its four faces from scratch (46 -> 26 us at 192^2).
constexpr int F64_X = 32, F64_Y = 4, F64_THREADS = 160;
__device__ __forceinline__ void time_flux_d(const Flux64 &A, int kind, int i, int j, bool fx, bool gy, double gm1i,
                                            double F[4], double Gf[4]) {
#pragma unroll
  for (int v = 0; v < NV; v++) F[v] = Gf[v] = 0.0;
#pragma unroll
  for (int l = 0; l < 3; l++) {
    double U[4], f[4];
    ld4d(A.g, A.n[l][kind], i, j, U);
    const double w = l == 1 ? 4.0 : 1.0;
    if (fx) {
      phys_flux_d(U, gm1i, 0, f);
#pragma unroll
      for (int v = 0; v < NV; v++) F[v] = fma(w, f[v], F[v]);
    }
    if (gy) {
      phys_flux_d(U, gm1i, 1, f);
#pragma unroll
      for (int v = 0; v < NV; v++) Gf[v] = fma(w, f[v], Gf[v]);
    }
  }
}
__global__ void __launch_bounds__(F64_THREADS) flux64_kernel(Flux64 A) {
  __shared__ double vf[NV][F64_Y + 1][F64_X + 1], vg[NV][F64_Y + 1][F64_X + 1];
  __shared__ double xf[NV][F64_Y][F64_X + 1], yg[NV][F64_Y + 1][F64_X];
  const Grid &g = A.g;
  // (tiles on the x axis of the launch grid alone: ny has no limit of its own)
  const int tx = (g.nx + F64_X - 1) / F64_X, i0 = (int)(blockIdx.x % tx) * F64_X, j0 = (int)(blockIdx.x / tx) * F64_Y;
  const double gm1i = 1.0 / (A.ph.gam - 1.0);
  for (int k = threadIdx.x; k < (F64_X + 1) * (F64_Y + 1); k += F64_THREADS) {
    const int a = k % (F64_X + 1), b = k / (F64_X + 1), i = i0 + a, j = j0 + b;
    double F[4], Gf[4];
    if (i <= g.nx && j <= g.ny) {
      time_flux_d(A, VTX, i, j, true, true, gm1i, F, Gf);
#pragma unroll
      for (int v = 0; v < NV; v++) {
        vf[v][b][a] = F[v];
        vg[v][b][a] = Gf[v];
      }
    }
    if (b < F64_Y && i <= g.nx && j < g.ny) {
      time_flux_d(A, XE, i, j, true, false, gm1i, F, Gf);
#pragma unroll
      for (int v = 0; v < NV; v++) xf[v][b][a] = F[v];
    }
    if (a < F64_X && i < g.nx && j <= g.ny) {
      time_flux_d(A, YE, i, j, false, true, gm1i, F, Gf);
#pragma unroll
      for (int v = 0; v < NV; v++) yg[v][b][a] = Gf[v];
    }
  }
  __syncthreads();
  const int a = threadIdx.x % F64_X, b = threadIdx.x / F64_X, i = i0 + a, j = j0 + b;
  if (b >= F64_Y || i >= g.nx || j >= g.ny) return;
  double Q[4];
#pragma unroll
  for (int v = 0; v < NV; v++) {
    const double FL = (vf[v][b][a] + 4.0 * xf[v][b][a] + vf[v][b + 1][a]) * (1.0 / 36.0);
    const double FR = (vf[v][b][a + 1] + 4.0 * xf[v][b][a + 1] + vf[v][b + 1][a + 1]) * (1.0 / 36.0);
    const double GB = (vg[v][b][a] + 4.0 * yg[v][b][a] + vg[v][b][a + 1]) * (1.0 / 36.0);
    const double GT = (vg[v][b + 1][a] + 4.0 * yg[v][b + 1][a] + vg[v][b + 1][a + 1]) * (1.0 / 36.0);
    const long long k = at(g, v, i, j);
    Q[v] = A.avg[k] - (A.lx * (FR - FL) + A.ly * (GT - GB));
    A.avg[k] = Q[v];
  }
  double U[4];
  c2p_d(Q, A.ph.gam - 1.0, U);
  const bool finite = isfinite(Q[0]) && isfinite(Q[1]) && isfinite(Q[2]) && isfinite(Q[3]);
  const int st = !finite ? ST_NONFINITE : ((U[0] > 0.0 && U[3] > 0.0) ? 0 : ST_AVG_NONPOS);
  if (st) atomicOr(A.status, st);
}

// max over the averages and the owned point values of max(|u|, |v|) + c, as
// the bits of a positive double (which order like the values); bad set if a
// value is not admissible
__global__ void speed64_kernel(Grid g, double gam, const double *avg, const double *vtx, const double *xe, const double *ye,
                               unsigned long long *out, int *bad) {
  const long long nc = (long long)g.nx * g.ny, nv = (long long)g.nxv * g.nyv;
  const long long nxe = (long long)g.nxv * g.ny, nye = (long long)g.nx * g.nyv;
  const long long total = nc + nv + nxe + nye;
  double m = 0.0;
  bool b = false;
  for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < total;
       k += (long long)gridDim.x * blockDim.x) {
    long long r = k;
    double U[4];
    if (r < nc) {
      double Q[4];
      ld4d(g, avg, (int)(r % g.nx), (int)(r / g.nx), Q);
      c2p_d(Q, gam - 1.0, U);
    } else {
      const double *p;
      int ni;
      if ((r -= nc) < nv) {
        p = vtx;
        ni = g.nxv;
      } else if ((r -= nv) < nxe) {
        p = xe;
        ni = g.nxv;
      } else {
        r -= nxe;
        p = ye;
        ni = g.nx;
      }
      ld4d(g, p, (int)(r % ni), (int)(r / ni), U);
    }
    if (!(U[0] > 0.0 && U[3] > 0.0) || !isfinite(U[1]) || !isfinite(U[2])) {
      b = true;
      continue;
    }
    m = fmax(m, fmax(fabs(U[1]), fabs(U[2])) + sqrt(gam * U[3] / U[0]));
  }
  for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
  b = __any_sync(0xffffffffu, b);
  if ((threadIdx.x & 31) == 0) {
    atomicMax(out, (unsigned long long)__double_as_longlong(m));
    if (b) atomicOr(bad, 1);
  }
}

// per-block FP64 sums of the averages (fixed order within a block), then
// their fixed-order sum by one block
constexpr int TOT64_BLOCKS = 128;
__global__ void totals64_kernel(Grid g, const double *avg, double *partials) {
  __shared__ double sm[4][256];
  double acc[4] = {0.0, 0.0, 0.0, 0.0};
  const long long n = (long long)g.nx * g.ny;
  for (long long e = blockIdx.x * 256LL + threadIdx.x; e < n; e += 256LL * gridDim.x) {
    const int i = (int)(e % g.nx), j = (int)(e / g.nx);
    for (int v = 0; v < NV; v++) acc[v] += avg[at(g, v, i, j)];
  }
  for (int v = 0; v < NV; v++) sm[v][threadIdx.x] = acc[v];
  __syncthreads();
  for (int s = 128; s > 0; s >>= 1) {
    if (threadIdx.x < s)
      for (int v = 0; v < NV; v++) sm[v][threadIdx.x] += sm[v][threadIdx.x + s];
    __syncthreads();
  }
  if (threadIdx.x < 4) partials[blockIdx.x * 4 + threadIdx.x] = sm[threadIdx.x][0];
}
__global__ void totals64_final(const double *partials, int nblk, double area, double *out) {
  if (threadIdx.x < 4) {
    double s = 0.0;
    for (int b = 0; b < nblk; b++) s += partials[b * 4 + threadIdx.x];
    out[threadIdx.x] = s * area;
  }
}

// compact [4][nj][ni] <-> padded planes
__global__ void pack64_kernel(Grid g, const double *src, double *dst, int ni, int nj, int to_padded) {
  const long long n = 4LL * ni * nj;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
    const int i = (int)(e % ni), j = (int)((e / ni) % nj), v = (int)(e / ((long long)ni * nj));
    if (to_padded) dst[at(g, v, i, j)] = src[e];
    else dst[e] = src[at(g, v, i, j)];
  }
}

inline int blocks_for(long long n) {
  long long b = (n + 255) / 256;
  return (int)(b < 1 ? 1 : (b > 65536 ? 65536 : b));
}

}  // namespace

cudaError_t launch_step64(const Step64 &S, double lamx, double lamy, cudaStream_t s) {
  const Grid &g = S.g;
  record64_kernel<<<blocks_for((long long)(g.nx + 2) * (g.ny + 2)), 256, 0, s>>>(S);
  const auto nb = [](long long n) { return (unsigned)((n + NODE64_THREADS - 1) / NODE64_THREADS); };
  const unsigned nbv = nb((long long)g.nxv * g.nyv), nbx = nb((long long)g.nxv * g.ny), nby = nb((long long)g.nx * g.nyv);
  node64_kernel<<<nbv + nbx + nby, NODE64_THREADS, 0, s>>>(S, (int)nbv, (int)nbx);
  Flux64 F;
  F.g = g;
  F.ph = S.ph;
  for (int k = 0; k < 3; k++) {
    F.n[0][k] = S.n0[k];
    F.n[1][k] = S.n1[k];
    F.n[2][k] = S.n2[k];
  }
  F.avg = const_cast<double *>(S.avg);
  F.lx = lamx;
  F.ly = lamy;
  F.status = S.status;
  flux64_kernel<<<(unsigned)((g.nx + F64_X - 1) / F64_X) * ((g.ny + F64_Y - 1) / F64_Y), F64_THREADS, 0, s>>>(F);
  return cudaGetLastError();
}

cudaError_t launch_speed64(const Grid &g, double gam, const double *avg, const double *const n[3],
                           unsigned long long *out, int *bad, cudaStream_t s) {
  cudaMemsetAsync(out, 0, sizeof(unsigned long long), s);
  cudaMemsetAsync(bad, 0, sizeof(int), s);
  speed64_kernel<<<1024, 256, 0, s>>>(g, gam, avg, n[VTX], n[XE], n[YE], out, bad);
  return cudaGetLastError();
}

cudaError_t launch_totals64(const Grid &g, const double *avg, double *partials, double area, double *out,
                            cudaStream_t s) {
  totals64_kernel<<<TOT64_BLOCKS, 256, 0, s>>>(g, avg, partials);
  totals64_final<<<1, 32, 0, s>>>(partials, TOT64_BLOCKS, area, out);
  return cudaGetLastError();
}

cudaError_t launch_pack64(const Grid &g, const double *src, double *dst, int ni, int nj, bool to_padded,
                          cudaStream_t s) {
  pack64_kernel<<<blocks_for(4LL * ni * nj), 256, 0, s>>>(g, src, dst, ni, nj, to_padded ? 1 : 0);
  return cudaGetLastError();
}

AF_BOUNDS_READER(bounds_fp64)

}  // namespace af
