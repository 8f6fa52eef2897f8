// af_pointvalue.cuh -- point values at t^{n+1/2} and t^{n+1} (Alg. 1 steps 1
// and 2, with eq. (Un+1/2), eq. (1stStep), Alg. 2 and Alg. 3), with the cell
// prep of Sec. 2 fused in: the device code, compiled by two units.
// af_pointvalue.cu holds the plain instantiations; af_pointvalue_shock.cu
// (AF_PV_SHOCK defined) those with the Sec. 3 switches for discontinuous data,
// which sum EG2 in another form (af_eg2_arc.cuh) from another record layout.
//
// A block owns a TX x TY tile of cells; its threads (one per cell) each
// update the three nodes the cell owns: the vertex (i-1/2, j-1/2), the x-edge
// midpoint (i-1/2, j) and the y-edge midpoint (i, j-1/2).
//
// Prologue: for every cell of the tile and a one-cell halo the block forms
// the cell prep (Q_c by inverting Simpson's rule, U_c = C2P(Q_c), Ubar by
// Simpson's rule over the primitive point values, or optionally the primitive
// state of the cell average) and stores, per variable, the cell's biquadratic
// reconstruction as monomial coefficients about the cell centre in shared
// memory, plus Ubar.
//
// Node update: for each time level the node's EG2 operator (eq. (EG2)) is
// evaluated on that reconstruction.  The Mach-cone base is a circle of radius
// c' tau around P' = node - u' tau; it crosses the grid lines through the
// node at cos(theta) = u'/c' and sin(theta) = v'/c'.  The reconstruction on it
// is the reference cell's polynomial plus truncated powers of the distances
// from the grid lines (see "EG2 arc sums in the truncated-power form" below);
// every integral is taken exactly, without a crossing sort.  All data are
// taken relative to the node's own t^n value, which the operators reproduce
// exactly, so FP32 keeps its relative accuracy in the perturbations.
#pragma once
#include <type_traits>

#include "af_common.cuh"
#include "af_kernels.h"

namespace af {

namespace {

// keeps the loads on either side in order: the compiler otherwise moves the next
// stage's record loads up over the current one's arithmetic and holds them in
// registers (4096^2 vortex: 2.45 ms without, 2.43 with)
__device__ __forceinline__ void keep_order() { asm volatile("" ::: "memory"); }

constexpr float PI_F = 3.14159265358979f;
constexpr float INV_PI = 0.318309886183791f;
constexpr float INV_2PI = 0.159154943091895f;

// The divisions and square roots on the EG2 / EG1 / correction path use the
// hardware approximations (__fdividef and rsqrtf, a few ulp) instead of the
// correctly rounded sequences: they sit on the dependency chain that starts
// every evaluation (c' -> 1/c' -> the half-circle tables), and the kernel is
// bound by latency.  sqrt(t) for t >= 0 from the reciprocal square root (0 at
// t = 0):
__device__ __forceinline__ float sqrt_nn(float t) { return t > 0.0f ? t * rsqrtf(t) : 0.0f; }

// A tile is TX x TY cells: TX = 32 (one warp along x) and TY rows, TY one
// of the heights in tile_heights (the batched path picks one by timing).
constexpr int TX = 32;
constexpr int HX = TX + 2;                   // with a one-cell halo on each side
#ifdef AF_PV_SHOCK
// Cell records in shared memory: per cell 4 variables x (9 monomial coefficients
// and 3 pad) = 48 floats, then Ubar (4); 13 float4, an odd number: consecutive
// cells' 128-bit accesses meet no bank conflicts
constexpr int CELL_F = 52, UBAR_OFF = 48;
#else
// Cell records in shared memory, row by row: first the row's Ubar (HX cells, 4
// floats each), then the records of its HX - 1 cells that node updates read:
// per cell 4 variables x 8 monomial coefficients and the four values m00, 36
// floats (9 float4, an odd number: consecutive cells' 128-bit accesses meet no
// bank conflicts).  76.5 KB for an 8-row tile and its raw data.
constexpr int CELL_F = 36, M00_OFF = 32;
constexpr int ROW_F = HX * 4 + (HX - 1) * CELL_F;
#endif
// Raw t^n data of a tile, staged by TMA: for each of the node arrays (vertex,
// x-edge, y-edge) and the cell averages a box of RAW_W x (TY + 3) points x 4
// variables.  The box starts 4 points left of the first halo point so that
// its x coordinate is a multiple of 4 floats (16 bytes), and 1 row below.
constexpr int RAW_W = TX + 8;
template <int TY>
struct Tile {
  static constexpr int HY = TY + 2;
#ifdef AF_PV_SHOCK
  static constexpr int REC_FLOATS = HX * HY * CELL_F;
#else
  static constexpr int REC_FLOATS = (HY - 1) * ROW_F + HX * 4;
#endif
  static constexpr int RAW_H = TY + 3;
  static constexpr int RAW_ARR = RAW_W * RAW_H * NV;  // floats per array
  static constexpr int RAW_FLOATS = 4 * RAW_ARR;
  static constexpr unsigned RAW_BYTES = RAW_FLOATS * 4u;
  static constexpr int SMEM_BYTES = (RAW_FLOATS + REC_FLOATS) * 4 + 128;  // + alignment slack
  // with node fluxes: 5 floats a thread, component-major (a node's
  // t^{n+1/2} value between the two levels, the running wave-speed maximum)
  static constexpr int SCR_FLOATS = 5 * TX * TY;
  static constexpr int SMEM_NF_BYTES = SMEM_BYTES + SCR_FLOATS * 4;
};
enum { RAW_VTX = 0, RAW_XE = 1, RAW_YE = 2, RAW_AVG = 3 };

using Args = PointValueArgs;

// staged t^n value of array arr, variable v, at grid index (i, j), for the
// tile with origin (i0, j0)
template <int TY>
__device__ __forceinline__ float raw_at(const float *raw, int arr, int v, int i, int j, int i0, int j0) {
#ifdef AF_CHECK_BOUNDS
  if (!bounds_ok(arr >= 0 && arr < 4 && v >= 0 && v < NV && j - j0 + 1 >= 0 && j - j0 + 1 < Tile<TY>::RAW_H &&
                     i - i0 + 4 >= 0 && i - i0 + 4 < RAW_W,
                 BD_BOX))
    return raw[0];
#endif
  return raw[((arr * NV + v) * Tile<TY>::RAW_H + (j - j0 + 1)) * RAW_W + (i - i0 + 4)];
}
template <int TY>
__device__ __forceinline__ void raw4(const float *raw, int arr, int i, int j, int i0, int j0, float U[4]) {
#pragma unroll
  for (int v = 0; v < NV; v++) U[v] = raw_at<TY>(raw, arr, v, i, j, i0, j0);
}

__device__ __forceinline__ float ld(const Args &A, const float *p, int v, int i, int j) {
  return p[at(A.g, v, i, j)];
}
__device__ __forceinline__ void ld4(const Args &A, const float *p, int i, int j, float U[4]) {
#pragma unroll
  for (int v = 0; v < NV; v++) U[v] = ld(A, p, v, i, j);
}

__device__ __forceinline__ float4 pack4(const float U[4]) { return make_float4(U[0], U[1], U[2], U[3]); }
__device__ __forceinline__ void unpack4(float4 w, float U[4]) {
  U[0] = w.x;
  U[1] = w.y;
  U[2] = w.z;
  U[3] = w.w;
}

#ifdef AF_CHECK_BOUNDS
// rows of cell records the running kernel's tile holds (checking builds)
__shared__ int rec_rows;
#endif
#ifdef AF_PV_SHOCK
// shared-memory record of tile-local cell (a, b), a in [0, HX), b in [0, HY)
__device__ __forceinline__ const float *cell_rec(const float *sm, int a, int b) {
#ifdef AF_CHECK_BOUNDS
  if (!bounds_ok(a >= 0 && a < HX && b >= 0 && b < rec_rows, BD_RECORD)) return sm;
#endif
  return sm + (b * HX + a) * CELL_F;
}
#else
// shared-memory record of tile-local cell (a, b), a in [0, HX - 1), b in [0, HY - 1)
__device__ __forceinline__ const float *cell_rec(const float *sm, int a, int b) {
#ifdef AF_CHECK_BOUNDS
  if (!bounds_ok(a >= 0 && a < HX - 1 && b >= 0 && b < rec_rows - 1, BD_RECORD)) return sm;
#endif
  return sm + b * ROW_F + HX * 4 + a * CELL_F;
}
// U_c (the monomials m00 of the four variables) of a record
__device__ __forceinline__ float4 cell_m00(const float *rec) {
  return reinterpret_cast<const float4 *>(rec + M00_OFF)[0];
}
// Ubar of tile-local cell (a, b), a in [0, HX), b in [0, HY)
__device__ __forceinline__ const float *cell_ubar(const float *sm, int a, int b) {
#ifdef AF_CHECK_BOUNDS
  if (!bounds_ok(a >= 0 && a < HX && b >= 0 && b < rec_rows, BD_RECORD)) return sm;
#endif
  return sm + b * ROW_F + a * 4;
}
#endif

// ----------------------------------------------------------------- prologue
// nodal values f[k][l] at local (k/2, l/2) -> coefficients m[a][b] of
// x^a y^b with x, y in [-1/2, 1/2] about the cell centre
__device__ __forceinline__ void to_monomial(const float f[3][3], float m[3][3]) {
  float r[3][3];  // r[a][l]: along x for each row l
#pragma unroll
  for (int l = 0; l < 3; l++) {
    r[0][l] = f[1][l];
    r[1][l] = f[2][l] - f[0][l];
    r[2][l] = 2.0f * (f[0][l] + f[2][l]) - 4.0f * f[1][l];
  }
#pragma unroll
  for (int a = 0; a < 3; a++) {
    m[a][0] = r[a][1];
    m[a][1] = r[a][2] - r[a][0];
    m[a][2] = 2.0f * (r[a][0] + r[a][2]) - 4.0f * r[a][1];
  }
}

// prep of cell (ci, cj) from the staged tile: its Ubar and its record
template <int TY>
__device__ __forceinline__ void build_cell(const Grid &g, const float *raw, int i0, int j0, int ci, int cj,
                                           float *ub, float *rec) {
  float N[8][4];  // corners (ll, lr, ul, ur), then edges (left, right, bottom, top)
  raw4<TY>(raw, RAW_VTX, ci, cj, i0, j0, N[0]);
  raw4<TY>(raw, RAW_VTX, ci + 1, cj, i0, j0, N[1]);
  raw4<TY>(raw, RAW_VTX, ci, cj + 1, i0, j0, N[2]);
  raw4<TY>(raw, RAW_VTX, ci + 1, cj + 1, i0, j0, N[3]);
  raw4<TY>(raw, RAW_XE, ci, cj, i0, j0, N[4]);
  raw4<TY>(raw, RAW_XE, ci + 1, cj, i0, j0, N[5]);
  raw4<TY>(raw, RAW_YE, ci, cj, i0, j0, N[6]);
  raw4<TY>(raw, RAW_YE, ci, cj + 1, i0, j0, N[7]);
  float Qa[4], Uc[4], Ub[4];
#pragma unroll
  for (int v = 0; v < NV; v++) Qa[v] = raw_at<TY>(raw, RAW_AVG, v, ci, cj, i0, j0);
  cell_prep(N, Qa, g.gamma, g.ubar_c2p, Uc, Ub);
  *reinterpret_cast<float4 *>(ub) = make_float4(Ub[0], Ub[1], Ub[2], Ub[3]);
#ifdef AF_PV_SHOCK
#pragma unroll
  for (int v = 0; v < NV; v++) {
    const float f[3][3] = {{N[0][v], N[4][v], N[2][v]}, {N[6][v], Uc[v], N[7][v]}, {N[1][v], N[5][v], N[3][v]}};
    float m[3][3];
    to_monomial(f, m);
    float4 *r4 = reinterpret_cast<float4 *>(rec + 12 * v);
    r4[0] = make_float4(m[0][0], m[0][1], m[0][2], m[1][0]);
    r4[1] = make_float4(m[1][1], m[1][2], m[2][0], m[2][1]);
    r4[2] = make_float4(m[2][2], 0.0f, 0.0f, 0.0f);
  }
#else
  float4 *r4 = reinterpret_cast<float4 *>(rec);
#pragma unroll
  for (int v = 0; v < NV; v++) {
    const float f[3][3] = {{N[0][v], N[4][v], N[2][v]}, {N[6][v], Uc[v], N[7][v]}, {N[1][v], N[5][v], N[3][v]}};
    float m[3][3];
    to_monomial(f, m);
    r4[2 * v] = make_float4(m[1][0], m[2][0], m[0][1], m[0][2]);
    r4[2 * v + 1] = make_float4(m[1][1], m[1][2], m[2][1], m[2][2]);
  }
  r4[M00_OFF / 4] = make_float4(Uc[0], Uc[1], Uc[2], Uc[3]);
#endif
}

#ifndef AF_PV_SHOCK
// ---- EG2 arc sums in the truncated-power form of the reconstruction
// In the frame reflected so that u', v' >= 0 (cos -> fx cos, sin -> fy sin),
// with X = rx (cos - a), Y = ry (sin - b) the coordinates relative to the node
// on the Mach circle (a = |u'|/c', b = |v'|/c'), the reconstruction around a
// vertex is
//   q = q_ref + [X > 0] Dx + [Y > 0] Dy + [X > 0, Y > 0] Dxy,
// q_ref the biquadratic of the cell on side -- (it holds P') and
//   Dx = X d1(y) + X^2 d2(y),  Dy = Y d1(x) + Y^2 d2(x),
//   Dxy = X Y (g11 + g21 X + g12 Y + g22 X Y):
// q is continuous across a grid line, so the difference of the two cells
// vanishes on it, and only the jumps of the normal derivatives (6 numbers a
// line, 4 for the crossing) enter instead of 9 coefficients a cell.  An edge
// midpoint has one line: q_ref + [X > 0] Dx.  The integrals of cos^m sin^n
// times q_ref over the whole circle are constants; Dx is integrated over
// {cos > a} = (-acos a, acos a), where with
//   L_m = int (cos - a)^m,  N_m = int (cos - a)^m sin^2
// the end-point terms vanish and
//   m L_m = (m-1) (1 - a^2) L_(m-2) - (2m-1) a L_(m-1),
//   m N_(m-1) = L_(m+1) + a L_m = int cos (cos - a)^m;
// Dy likewise with the roles of cos and sin exchanged, and Dxy over the arc
// (asin b, acos a) (empty unless a^2 + b^2 < 1) from two identities of the
// same kind (quarter_moments).  All sums are taken divided by pi.
//
// The stages (circle, X, Y, crossing) each build their own small table and run
// over p, u and v, reading the records again, so that one table is live at a
// time; the terms in X and X^2 go together through the packed FP32x2
// instructions.  Bound by issue and latency at 16 warps an SM (128
// registers): 3735 thread instructions a cell at 66 % of the issue slots.  The
// earlier form took differences of all 9 coefficients of each cell on the
// circle with two half tables and an arc table live together (4990
// instructions).  Measured on 8-row tiles, 4096^2 vortex moving / at rest
// (crossings at no / every vertex): 3.05 / 3.32 -> 2.37 / 2.53 ms; Alg. 1
// linearisation at 2048^2 1.16 -> 0.85 ms.  80 or 96 registers (24 or 20 warps) spill to a local memory
// that the L1 beside the shared memory cannot hold: 2.97 and 2.88 ms.

__device__ __forceinline__ float2 pair(float x) { return make_float2(x, x); }

// Taylor coefficients t of q(x) = a0 + a1 x + a2 x^2 at x0 (the last is a2)
__device__ __forceinline__ void taylor(float a0, float a1, float a2, float x0, float &t0, float &t1) {
  const float t = fmaf(a2, x0, a1);
  t0 = fmaf(t, x0, a0);
  t1 = fmaf(a2, x0, t);
}
__device__ __forceinline__ float horner(float a0, float a1, float a2, float x0) {
  return fmaf(fmaf(a2, x0, a1), x0, a0);
}

// sums over the circle, divided by pi, with the reflected cos and sin:
// p: int p, int p cos, int p sin; u: int u cos, int u (2 cos^2 - 1/2),
// int u sin cos; v: int v sin, int v (2 sin^2 - 1/2), int v sin cos
struct Sums {
  float p[3], u[3], v[3];
};
__device__ __forceinline__ float total(float2 a) { return a.x + a.y; }
__device__ __forceinline__ void taylor2(float2 a0, float2 a1, float2 a2, float x0, float2 &t0, float2 &t1) {
  const float2 t = __ffma2_rn(a2, pair(x0), a1);
  t0 = __ffma2_rn(t, pair(x0), a0);
  t1 = __ffma2_rn(a2, pair(x0), t);
}

// a cell's coefficients of one variable: m[i][e] of x^i y^e (m00 apart)
struct Coef {
  float4 lin, mix;  // (m10, m20, m01, m02), (m11, m12, m21, m22)
};
__device__ __forceinline__ Coef coef(const float *rec, int v) {
  const float4 *r = reinterpret_cast<const float4 *>(rec) + 2 * v;
  return Coef{r[0], r[1]};
}

// the circle x = x0 + rx cos, y = y0 + ry sin in the reference cell's centred
// units (rx, ry carry the reflection signs), and the factors of the sums
struct Circle {
  float x0, y0, rx, ry, rx2, ry2;
};

// whole-circle sums of q_ref (value m00 - K at the cell centre): its Taylor
// coefficients at P' times the circle's constant integrals; only those that
// the variable's sums use
template <int VAR>
__device__ __forceinline__ void circle_sums(const Coef &m, float m00, const Circle &c, float s[3], float &centre) {
  // x first (p, u) or y first (v): r[i][e] of (first axis about P')^i
  // (second)^e, then t[i][e] about P' in both
  constexpr bool YF = VAR == 2;
  const float f0 = YF ? c.y0 : c.x0, s0 = YF ? c.x0 : c.y0;
  const float m20 = YF ? m.lin.w : m.lin.y, m21 = YF ? m.mix.y : m.mix.z;
  float r00, r10, r01, r11, r02, r12;
  taylor(m00, YF ? m.lin.z : m.lin.x, m20, f0, r00, r10);
  taylor(YF ? m.lin.x : m.lin.z, m.mix.x, m21, f0, r01, r11);
  taylor(YF ? m.lin.y : m.lin.w, YF ? m.mix.z : m.mix.y, m.mix.w, f0, r02, r12);
  float t00, t01, t10, t11;
  taylor(r00, r01, r02, s0, t00, t01);
  taylor(r10, r11, r12, s0, t10, t11);
  const float t20 = horner(m20, m21, m.mix.w, s0);
  const float rf = YF ? c.ry : c.rx, rs = YF ? c.rx : c.ry, rf2 = YF ? c.ry2 : c.rx2, rs2 = YF ? c.rx2 : c.ry2;
  centre = t00;
  if (VAR == 0) {
    const float t21 = fmaf(2.0f * s0, m.mix.w, m21);
    s[0] = fmaf(2.0f, t00, fmaf(rf2, fmaf(0.25f * rs2, m.mix.w, t20), rs2 * r02));
    s[1] = rf * fmaf(0.25f * rs2, r12, t10);
    s[2] = rs * fmaf(0.25f * rf2, t21, t01);
  } else {
    s[0] = rf * fmaf(0.25f * rs2, r12, t10);
    s[1] = fmaf(rf2, fmaf(0.125f * rs2, m.mix.w, t20), t00);
    s[2] = (0.25f * rf) * (rs * t11);
  }
}

// value of (cell polynomial - K) at (x0, y0); m00 already relative to K
__device__ __forceinline__ float eval_at(const Coef &m, float m00, float x0, float y0) {
  const float e0 = fmaf(fmaf(m.lin.y, x0, m.lin.x), x0, m00);
  const float e1 = fmaf(fmaf(m.mix.z, x0, m.mix.x), x0, m.lin.z);
  const float e2 = fmaf(fmaf(m.mix.w, x0, m.mix.y), x0, m.lin.w);
  return fmaf(fmaf(e2, y0, e1), y0, e0);
}

// moments over {cos > a} divided by pi: [k] for X (k = 0) and X^2 (k = 1), the
// weights 1, cos (c), 2 cos^2 - 1/2 (K), 2 sin^2 - 1/2 (V); the second row of
// each times sin^2.  r, r2: the factors of X and X^2.
struct HalfTable {
  float2 one[2], c[2], K[2], V[2];  // [times sin^2], the pair (X, X^2)
};
// a = |normal velocity| / c' (clamped to 1), s = sin(acos a), al = acos a.
// With W_m = int (cos - a)^m sin^4 the same integration by parts gives
//   N_1 = (2/3) s^3 - a N_0,  (m+3) N_(m+1) = m (1 - a^2) N_(m-1) - (2m+3) a N_m,
//   m W_(m-1) = 3 (N_(m+1) + a N_m) = 3 int cos (cos - a)^m sin^2,
// and the weights are 2 cos^2 - 1/2 = 3/2 - 2 sin^2, 2 sin^2 - 1/2.
__device__ __forceinline__ void half_table(float a, float s, float al, float r, float r2, HalfTable &H) {
  const float q = s * s;
  const float L0 = (2.0f * INV_PI) * al, L1 = (2.0f * INV_PI) * fmaf(-a, al, s);
  const float L2 = 0.5f * fmaf(q, L0, -3.0f * (a * L1));
  const float N0 = fmaf(a, L1, L2);
  const float N1 = fmaf((2.0f * INV_PI / 3.0f) * q, s, -a * N0);
  const float N2 = 0.25f * fmaf(q, N0, -5.0f * (a * N1));
  const float N3 = fmaf(0.4f * q, N1, -1.4f * (a * N2));
  const float N4 = fmaf(0.5f * q, N2, -1.5f * (a * N3));
  const float CN1 = fmaf(a, N1, N2), CN2 = fmaf(a, N2, N3), CN3 = fmaf(a, N3, N4);
  const float2 rr = make_float2(r, r2);
  H.one[0] = __fmul2_rn(rr, make_float2(L1, L2));
  H.one[1] = __fmul2_rn(rr, make_float2(N1, N2));
  H.c[0] = __fmul2_rn(rr, make_float2(N0, 2.0f * N1));
  H.c[1] = __fmul2_rn(rr, make_float2(CN1, CN2));
  const float2 W = __fmul2_rn(rr, make_float2(3.0f * CN2, 2.0f * CN3));  // 2 int X^k sin^4
  H.K[0] = __ffma2_rn(pair(1.5f), H.one[0], __fmul2_rn(pair(-2.0f), H.one[1]));
  H.K[1] = __ffma2_rn(pair(-1.0f), W, __fmul2_rn(pair(1.5f), H.one[1]));
  H.V[0] = __ffma2_rn(pair(-1.0f), H.K[0], H.one[0]);
  H.V[1] = __ffma2_rn(pair(-0.5f), H.one[1], W);
}

// jumps across a grid line: the derivatives' coefficients along the line
// (tangential powers 0, 1, 2), cell-centred; YL: the line is horizontal
// (x and y change roles); f the reflection sign of the normal axis
template <bool YL>
__device__ __forceinline__ void jumps(const Coef &R, const Coef &O, float f, float2 d[3]) {
  const float r1[3] = {YL ? R.lin.z : R.lin.x, R.mix.x, YL ? R.mix.z : R.mix.y};
  const float r2[3] = {YL ? R.lin.w : R.lin.y, YL ? R.mix.y : R.mix.z, R.mix.w};
  const float o1[3] = {YL ? O.lin.z : O.lin.x, O.mix.x, YL ? O.mix.z : O.mix.y};
  const float o2[3] = {YL ? O.lin.w : O.lin.y, YL ? O.mix.y : O.mix.z, O.mix.w};
#pragma unroll
  for (int n = 0; n < 3; n++) d[n] = make_float2(fmaf(f, o1[n] - r1[n], -(o2[n] + r2[n])), o2[n] - r2[n]);
}

// adds the half-circle sums of Dx (or Dy) of one variable: t0, rt, rt2 the
// circle along the line (tangential coordinate t = t0 + rt sin); VAR 0: p;
// 1: the velocity normal to the line; 2: the tangential one.  m in the frame
// of the line: p: 1, cos, sin; normal: cos, 2 cos^2 - 1/2, sin cos;
// tangential: sin, 2 sin^2 - 1/2, sin cos
template <int VAR>
__device__ __forceinline__ void half_sums(const float2 d[3], float t0, float rt, float rt2, const HalfTable &H,
                                          float &m0, float &m1, float &m2) {
  float2 e0, e1, a, b, c;
  taylor2(d[0], d[1], d[2], t0, e0, e1);
  e1 = __fmul2_rn(e1, pair(rt));
  const float2 e2 = __fmul2_rn(d[2], pair(rt2));
  if (VAR == 0) {
    a = __ffma2_rn(e0, H.one[0], __fmul2_rn(e2, H.one[1]));
    b = __ffma2_rn(e0, H.c[0], __fmul2_rn(e2, H.c[1]));
    c = __fmul2_rn(e1, H.one[1]);
  } else if (VAR == 1) {
    a = __ffma2_rn(e0, H.c[0], __fmul2_rn(e2, H.c[1]));
    b = __ffma2_rn(e0, H.K[0], __fmul2_rn(e2, H.K[1]));
    c = __fmul2_rn(e1, H.c[1]);
  } else {
    a = __fmul2_rn(e1, H.one[1]);
    b = __ffma2_rn(e0, H.V[0], __fmul2_rn(e2, H.V[1]));
    c = __fmul2_rn(e1, H.c[1]);
  }
  m0 += total(a);
  m1 += total(b);
  m2 += total(c);
}

// moments over the quarter (asin b, acos a), divided by pi, with c = cos,
// s = sin: entries XY, X^2 Y, X Y^2, X^2 Y^2 without the radii.  With
// q_mn = int (c - a)^m (s - b)^n, kap = 1 - a^2 - b^2 and both factors
// vanishing at an end point each, d[(c-a)^m (s-b)^n] and c^2 + s^2 = 1 give
//   m (q_(m-1,n+1) + b q_(m-1,n)) = n (q_(m+1,n-1) + a q_(m,n-1)),
//   q_(m+2,n) + 2 a q_(m+1,n) + q_(m,n+2) + 2 b q_(m,n+1) = kap q_mn.
struct QuarterTable {
  float2 one[2], c[2], s[2], K[2], V[2], Z[2];  // (XY, X^2 Y), (X Y^2, X^2 Y^2)
};
__device__ __forceinline__ void quarter_moments(float a, float b, float sa, float sb, float phi, QuarterTable &T) {
  const float kap = fmaf(-a, a, fmaf(-b, b, 1.0f));
  const float q00 = INV_PI * phi, q10 = fmaf(-a, q00, INV_PI * (sa - b)), q01 = fmaf(-b, q00, INV_PI * (sb - a));
  // q11 = int cos sin - b int cos - a int sin + a b phi
  const float q11 = fmaf(INV_PI * 0.5f, kap, -fmaf(INV_PI * b, sa - b, fmaf(a, INV_PI * (sb - a), -a * b * q00)));
  const float h = 0.5f * fmaf(kap, q00, -fmaf(a, q10, b * q01));
  const float q20 = fmaf(-a, q10, h), q02 = fmaf(-b, q01, h);
  const float q12 = (1.0f / 3.0f) * fmaf(kap, q10, -fmaf(4.0f * b, q11, a * q20));
  const float q21 = (1.0f / 3.0f) * fmaf(kap, q01, -fmaf(4.0f * a, q11, b * q02));
  const float t = 0.5f * fmaf(kap, q11, -fmaf(a, q21, b * q12));  // int c X^2 Y = int s X Y^2
  const float q31 = fmaf(-a, q21, t), q13 = fmaf(-b, q12, t);
  const float q30 = fmaf(2.0f, fmaf(b, q11, q12), -a * q20);
  const float q22 = 0.25f * fmaf(kap, q20, -fmaf(5.0f * b, q21, a * q30));
  const float D41 = 0.6f * fmaf(kap, q21, -fmaf(a, q31, b * q22));  // int c X^3 Y
  const float D14 = 0.6f * fmaf(kap, q12, -fmaf(b, q13, a * q22));  // int s X Y^3
  const float E23 = (2.0f / 3.0f) * D41, E32 = (2.0f / 3.0f) * D14;  // int s X^2 Y^2, int c X^2 Y^2
  const float q41 = fmaf(-a, q31, D41), q23 = fmaf(-b, q22, E23), q32 = fmaf(-a, q22, E32);
  const float F = 0.5f * fmaf(kap, q22, -fmaf(a, q32, b * q23));                // int c X^3 Y^2
  const float Gs = (1.0f / 3.0f) * fmaf(kap, q31, -fmaf(a, q41, b * q32));      // int s X^3 Y^2
  T.one[0] = make_float2(q11, q21);
  T.one[1] = make_float2(q12, q22);
  const float c11 = fmaf(a, q11, q21), c12 = fmaf(a, q12, q22), s11 = fmaf(b, q11, q12), s21 = fmaf(b, q21, q22);
  T.c[0] = make_float2(c11, t);
  T.c[1] = make_float2(c12, E32);
  T.s[0] = make_float2(s11, s21);
  T.s[1] = make_float2(t, E23);
  const float2 cc[2] = {make_float2(fmaf(a, c11, t), fmaf(a, t, D41)), make_float2(fmaf(a, c12, E32), fmaf(a, E32, F))};
  T.Z[0] = make_float2(fmaf(a, s11, s21), fmaf(a, s21, fmaf(b, q31, q32)));
  T.Z[1] = make_float2(fmaf(a, t, E23), fmaf(a, E23, Gs));
#pragma unroll
  for (int k = 0; k < 2; k++) {
    T.K[k] = __ffma2_rn(pair(2.0f), cc[k], __fmul2_rn(pair(-0.5f), T.one[k]));
    T.V[k] = __ffma2_rn(pair(-1.0f), T.K[k], T.one[k]);
  }
}
// adds the sums of Dxy with coefficients g (radii folded in)
__device__ __forceinline__ void quarter_sums(const float2 g[2], const float2 w0[2], const float2 w1[2],
                                             const float2 w2[2], float &m0, float &m1, float &m2) {
  m0 += total(__ffma2_rn(g[0], w0[0], __fmul2_rn(g[1], w0[1])));
  m1 += total(__ffma2_rn(g[0], w1[0], __fmul2_rn(g[1], w1[1])));
  m2 += total(__ffma2_rn(g[0], w2[0], __fmul2_rn(g[1], w2[1])));
}

// the jumps across an edge midpoint's own line, between the cells below / left
// (reference) and above / right of it: the same for both time levels.  Seen
// from the other side (f = -1) d1 is the same and d2 changes sign.
struct LineJumps {
  float2 p[3], u[3], v[3];
};
template <int K>
__device__ __forceinline__ void line_jumps(const float *sm, int li, int lj, LineJumps &J) {
  if (K == VTX) return;
  const float *r = cell_rec(sm, K == YE ? li + 1 : li, K == XE ? lj + 1 : lj), *o = cell_rec(sm, li + 1, lj + 1);
  jumps<K == YE>(coef(r, 3), coef(o, 3), 1.0f, J.p);
  jumps<K == YE>(coef(r, 1), coef(o, 1), 1.0f, J.u);
  jumps<K == YE>(coef(r, 2), coef(o, 2), 1.0f, J.v);
}

// EG2 of the cpq reconstruction at node (K, li, lj) of the tile, linearised
// about ul, relative to the reference state Kr.  Returns false if the Mach
// cone base leaves the node's block of cells (the CFL bound of the
// linearisation state fails; the value is then not an EG2 value).
template <int K>
__device__ __forceinline__ bool eg2(const Grid &g, const float *sm, int li, int lj, const float Kr[4],
                                    const float ul[4], float tau, const LineJumps &J, float out[4]) {
  // an inadmissible linearisation state gives NaN outputs: c' becomes NaN and
  // every sum with it, so that no branch splits the evaluation
  const bool good = ul[0] > 0.0f && ul[3] > 0.0f && tau > 0.0f;
  const float cp2 = good ? __fdividef(g.gamma * ul[3], ul[0]) : __int_as_float(0x7fc00000);
  const float icp = rsqrtf(cp2), cp = cp2 * icp;
  const float R = cp * tau;
  bool inside;
  {
    const float ex = fabsf(ul[1]) * tau + R, ey = fabsf(ul[2]) * tau + R;
    const float lx = (K == YE) ? 0.5f * g.dx : g.dx, ly = (K == XE) ? 0.5f * g.dy : g.dy;
    inside = !(ex > lx || ey > ly);
  }
  const float rx = R * g.idx, ry = R * g.idy, rx2 = rx * rx, ry2 = ry * ry;
  // reflection signs (u', v' >= 0 in the reflected frame)
  const bool nx_ = K != YE && ul[1] < 0.0f, ny_ = K != XE && ul[2] < 0.0f;
  const float fx = nx_ ? -1.0f : 1.0f, fy = ny_ ? -1.0f : 1.0f;
  const float ax = fabsf(ul[1] * icp), by = fabsf(ul[2] * icp);
  const float frx = fx * rx, fry = fy * ry;
  // cells by side of the reflected frame: reference --, across the vertical
  // line (X side), across the horizontal line (Y side); P' in the
  // reference cell's centred units
  const int ar = (K == YE) ? li + 1 : li + (nx_ ? 1 : 0), br = (K == XE) ? lj + 1 : lj + (ny_ ? 1 : 0);
  const int ao = (K == YE) ? ar : li + (nx_ ? 0 : 1), bo = (K == XE) ? br : lj + (ny_ ? 0 : 1);
  const float *rr = cell_rec(sm, ar, br);
  const float x0 = fmaf(-ul[1] * tau, g.idx, (K == YE) ? 0.0f : 0.5f * fx);
  const float y0 = fmaf(-ul[2] * tau, g.idy, (K == XE) ? 0.0f : 0.5f * fy);

  Sums S;
  float drP, dpP, unused;
  const float4 m00 = cell_m00(rr);
  // the signed radii carry the reflection: the sums are those of the
  // reflected cos and sin
  const Circle C{x0, y0, frx, fry, rx2, ry2};
  drP = eval_at(coef(rr, 0), m00.x - Kr[0], x0, y0);
  circle_sums<0>(coef(rr, 3), m00.w - Kr[3], C, S.p, dpP);
  keep_order();
  circle_sums<1>(coef(rr, 1), m00.y - Kr[1], C, S.u, unused);
  keep_order();
  circle_sums<2>(coef(rr, 2), m00.z - Kr[2], C, S.v, unused);
  keep_order();

  float alx = 0.0f, snx = 0.0f, aly = 0.0f, sny = 0.0f;
  float2 d[3];
  if (K != YE) {
    const float a = fminf(ax, 1.0f);
    alx = acosf(a);
    snx = sqrt_nn(fmaf(-a, a, 1.0f));
    HalfTable H;
    if (K == XE) {
      half_table(a, snx, alx, rx, fx * rx2, H);
      half_sums<0>(J.p, y0, fry, ry2, H, S.p[0], S.p[1], S.p[2]);
      half_sums<1>(J.u, y0, fry, ry2, H, S.u[0], S.u[1], S.u[2]);
      half_sums<2>(J.v, y0, fry, ry2, H, S.v[0], S.v[1], S.v[2]);
    } else {
      half_table(a, snx, alx, rx, rx2, H);
      const float *ro = cell_rec(sm, ao, br);
      jumps<false>(coef(rr, 3), coef(ro, 3), fx, d);
      half_sums<0>(d, y0, fry, ry2, H, S.p[0], S.p[1], S.p[2]);
      keep_order();
      jumps<false>(coef(rr, 1), coef(ro, 1), fx, d);
      half_sums<1>(d, y0, fry, ry2, H, S.u[0], S.u[1], S.u[2]);
      keep_order();
      jumps<false>(coef(rr, 2), coef(ro, 2), fx, d);
      half_sums<2>(d, y0, fry, ry2, H, S.v[0], S.v[1], S.v[2]);
      keep_order();
    }
  }
  if (K != XE) {
    const float b = fminf(by, 1.0f);
    aly = acosf(b);
    sny = sqrt_nn(fmaf(-b, b, 1.0f));
    HalfTable H;
    if (K == YE) {
      half_table(b, sny, aly, ry, fy * ry2, H);
      half_sums<0>(J.p, x0, frx, rx2, H, S.p[0], S.p[2], S.p[1]);
      half_sums<1>(J.v, x0, frx, rx2, H, S.v[0], S.v[1], S.v[2]);
      half_sums<2>(J.u, x0, frx, rx2, H, S.u[0], S.u[1], S.u[2]);
    } else {
      half_table(b, sny, aly, ry, ry2, H);
      const float *ro = cell_rec(sm, ar, bo);
      jumps<true>(coef(rr, 3), coef(ro, 3), fy, d);
      half_sums<0>(d, x0, frx, rx2, H, S.p[0], S.p[2], S.p[1]);
      keep_order();
      jumps<true>(coef(rr, 2), coef(ro, 2), fy, d);
      half_sums<1>(d, x0, frx, rx2, H, S.v[0], S.v[1], S.v[2]);
      keep_order();
      jumps<true>(coef(rr, 1), coef(ro, 1), fy, d);
      half_sums<2>(d, x0, frx, rx2, H, S.u[0], S.u[1], S.u[2]);
      keep_order();
    }
  }
  if (K == VTX && ax < 1.0f && by < 1.0f && fmaf(ax, ax, by * by) < 1.0f) {
    QuarterTable T;
    quarter_moments(ax, by, snx, sny, alx + aly - 0.5f * PI_F, T);
    const float *rX = cell_rec(sm, ao, br), *rY = cell_rec(sm, ar, bo), *rQ = cell_rec(sm, ao, bo);
    const float rxy = rx * ry;
    auto crossing = [&](int v, float2 gq[2]) {
      // mixed coefficients (m11, m12, m21, m22) of the four cells: jumps
      // across the vertical line below and above, then of those across the
      // horizontal one
      const float4 m = reinterpret_cast<const float4 *>(rr)[2 * v + 1], mx = reinterpret_cast<const float4 *>(rX)[2 * v + 1];
      const float4 my = reinterpret_cast<const float4 *>(rY)[2 * v + 1], mq = reinterpret_cast<const float4 *>(rQ)[2 * v + 1];
      const float l1 = fmaf(fx, mx.x - m.x, -(mx.z + m.z)), l2 = fmaf(fx, mx.y - m.y, -(mx.w + m.w));
      const float u1 = fmaf(fx, mq.x - my.x, -(mq.z + my.z)), u2 = fmaf(fx, mq.y - my.y, -(mq.w + my.w));
      const float k1 = mx.z - m.z, k2 = mx.w - m.w, w1 = mq.z - my.z, w2 = mq.w - my.w;
      gq[0] = make_float2(rxy * fmaf(fy, u1 - l1, -(u2 + l2)), rxy * rx * fmaf(fy, w1 - k1, -(w2 + k2)));
      gq[1] = make_float2(rxy * ry * (u2 - l2), rxy * rxy * (w2 - k2));
    };
    float2 gq[2];
    crossing(3, gq);
    quarter_sums(gq, T.one, T.c, T.s, S.p[0], S.p[1], S.p[2]);
    keep_order();
    crossing(1, gq);
    quarter_sums(gq, T.c, T.K, T.Z, S.u[0], S.u[1], S.u[2]);
    keep_order();
    crossing(2, gq);
    quarter_sums(gq, T.s, T.V, T.Z, S.v[0], S.v[1], S.v[2]);
    keep_order();
  }
  // sums odd in cos change sign with fx, odd in sin with fy, back in the grid
  // frame; div = int (u cos + v sin)
  const float irc = __fdividef(icp, ul[0]), icp2 = icp * icp;
  const float z = fmaf(-ul[0] * cp, fmaf(fx, S.u[0], fy * S.v[0]), S.p[0]);
  const float fxy = 2.0f * fx * fy;
  out[0] = fmaf(icp2, fmaf(-2.0f, dpP, z), Kr[0] + drP);
  out[1] = Kr[1] + fmaf(-fx * irc, S.p[1], fmaf(fxy, S.v[2], S.u[1]));
  out[2] = Kr[2] + fmaf(-fy * irc, S.p[2], fmaf(fxy, S.u[2], S.v[1]));
  out[3] = Kr[3] + (z - dpP);
  return inside;
}

#endif  // !AF_PV_SHOCK

// tile-local cell indices of the cells around node (K, i, j)
template <int K>
__device__ __forceinline__ void arc_cell(int li, int lj, int right, int top, int &a, int &b) {
  a = (K == YE) ? li + 1 : li + right;
  b = (K == XE) ? lj + 1 : lj + top;
}

#ifdef AF_PV_SHOCK
#include "af_eg2_arc.cuh"
#endif

// ---------------------------------------------------------------- Alg. 3 parts
#ifdef AF_PV_SHOCK
__device__ __forceinline__ float4 ubar4(const float *sm, int a, int b) {
  return reinterpret_cast<const float4 *>(cell_rec(sm, a, b) + UBAR_OFF)[0];
}
// U_c (the monomial m00) of variable v of tile-local cell (a, b)
__device__ __forceinline__ float centre(const float *sm, int a, int b, int v) {
  return reinterpret_cast<const float4 *>(cell_rec(sm, a, b) + 12 * v)[0].x;
}
#else
__device__ __forceinline__ float4 ubar4(const float *sm, int a, int b) {
  return reinterpret_cast<const float4 *>(cell_ubar(sm, a, b))[0];
}
#endif

// EG1 (Sec. 3.3) on piecewise-constant primitive averages, relative to Kr
template <int K>
__device__ __forceinline__ void eg1_pc(const Grid &g, const float *sm, int li, int lj, const float *Kr,
                                    const float *ul, float tau, float *out) {
  if (!(ul[0] > 0.0f && ul[3] > 0.0f && tau > 0.0f)) {
    for (int v = 0; v < NV; v++) out[v] = __int_as_float(0x7fc00000);
    return;
  }
  const float cp2 = __fdividef(g.gamma * ul[3], ul[0]), icp = rsqrtf(cp2), cp = cp2 * icp;
  const float am = ul[1] * icp, bm = ul[2] * icp;
  // the arc sums by inclusion-exclusion, as for EG2 (see "EG2 arc sums by
  // inclusion-exclusion"): with constant data per cell only cos^m sin^n,
  // m + n <= 2, enter; whole circle (1, cos^2, sin^2) = (2 pi, pi, pi); the
  // X half-circle (-al, al) and the Y half-circle (asin b, pi - asin b) give
  // theirs in closed form, zero for a line the circle misses; the quarter arc
  // X and Y from its end points
  const float fx = (K != YE && ul[1] < 0.0f) ? -1.0f : 1.0f, fy = (K != XE && ul[2] < 0.0f) ? -1.0f : 1.0f;
  const float ax = fminf(fabsf(am), 1.0f), by = fminf(fabsf(bm), 1.0f);
  const float alx = acosf(ax), snx = sqrt_nn(fmaf(-ax, ax, 1.0f));
  const float aly = acosf(by), sny = sqrt_nn(fmaf(-by, by, 1.0f));
  // [J00, J10, J01, J20, J11, J02] of each set, reflected frame
  const float X[6] = {2.0f * alx, 2.0f * snx, 0.0f, fmaf(ax, snx, alx), 0.0f, fmaf(-ax, snx, alx)};
  const float Y[6] = {2.0f * aly, 0.0f, 2.0f * sny, fmaf(-by, sny, aly), 0.0f, fmaf(by, sny, aly)};
  float Q[6] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
  if (K == VTX && fmaf(ax, ax, by * by) < 1.0f) {
    // from (cos, sin) = (sny, by) at pi/2 - aly to (ax, snx) at alx
    Q[0] = alx + aly - 0.5f * PI_F;
    Q[1] = snx - by;
    Q[2] = sny - ax;
    Q[3] = 0.5f * (ax * snx - sny * by + Q[0]);
    Q[4] = 0.5f * (snx * snx - by * by);
    Q[5] = Q[0] - Q[3];
  }
  // cell values relative to Kr by side (px, py) of the reflected frame
  auto dval = [&](int px, int py, float d[4]) {
    const int right = px ? (fx > 0.0f) : (fx < 0.0f), top = py ? (fy > 0.0f) : (fy < 0.0f);
    int a, b;
    arc_cell<K>(li, lj, right, top, a, b);
    const float4 w = ubar4(sm, a, b);
    d[0] = w.x - Kr[0];
    d[1] = w.y - Kr[1];
    d[2] = w.z - Kr[2];
    d[3] = w.w - Kr[3];
  };
  // M[w][v] = sum over the cells' arcs of d_v J_w
  float M[6][4], d0[4], dx[4], dy[4], dq[4];
  dval(0, 0, d0);
#pragma unroll
  for (int v = 0; v < NV; v++) {
    M[0][v] = 2.0f * PI_F * d0[v];
    M[1][v] = M[2][v] = M[4][v] = 0.0f;
    M[3][v] = M[5][v] = PI_F * d0[v];
  }
  if (K != YE) {
    dval(1, 0, dx);
#pragma unroll
    for (int v = 0; v < NV; v++) {
      const float e = dx[v] - d0[v];
#pragma unroll
      for (int w = 0; w < 6; w++) M[w][v] = fmaf(e, X[w], M[w][v]);
    }
  }
  if (K != XE) {
    dval(0, 1, dy);
#pragma unroll
    for (int v = 0; v < NV; v++) {
      const float e = dy[v] - d0[v];
#pragma unroll
      for (int w = 0; w < 6; w++) M[w][v] = fmaf(e, Y[w], M[w][v]);
    }
  }
  if (K == VTX) {
    dval(1, 1, dq);
#pragma unroll
    for (int v = 0; v < NV; v++) {
      const float e = dq[v] - dx[v] - dy[v] + d0[v];
#pragma unroll
      for (int w = 0; w < 6; w++) M[w][v] = fmaf(e, Q[w], M[w][v]);
    }
  }
  // back to the grid frame: odd in cos changes sign with fx, odd in sin with fy
  const float P0 = M[0][3], P10 = fx * M[1][3], P01 = fy * M[2][3];
  const float UC = fx * M[1][1], VS = fy * M[2][2], U20 = M[3][1], U00 = M[0][1], U11 = fx * fy * M[4][1];
  const float V11 = fx * fy * M[4][2], V02 = M[5][2], V00 = M[0][2];
  // value at P'; on a grid line the mean of the cells whose closure holds it
  float dP[4] = {0, 0, 0, 0};
  {
    const int xa = (K == YE) ? 0 : (ul[1] < 0.0f ? 1 : 0), xb = (K == YE) ? 0 : (ul[1] > 0.0f ? 0 : 1);
    const int ya = (K == XE) ? 0 : (ul[2] < 0.0f ? 1 : 0), yb = (K == XE) ? 0 : (ul[2] > 0.0f ? 0 : 1);
    int cnt = 0;
    for (int rr = xa; rr <= xb; rr++)
      for (int tt = ya; tt <= yb; tt++) {
        int a, b;
        arc_cell<K>(li, lj, rr, tt, a, b);
        const float4 w = ubar4(sm, a, b);
        dP[0] += w.x - Kr[0];
        dP[1] += w.y - Kr[1];
        dP[2] += w.z - Kr[2];
        dP[3] += w.w - Kr[3];
        cnt++;
      }
    const float ic = 1.0f / (float)cnt;
    for (int v = 0; v < NV; v++) dP[v] *= ic;
  }
  const float rp = ul[0], rc = rp * cp, icp2 = icp * icp;
  out[0] = Kr[0] + dP[0] - dP[3] * icp2 + INV_2PI * (P0 * icp2 - 2.0f * rp * icp * (UC + VS));
  out[1] = Kr[1] + 0.5f * dP[1] + INV_2PI * (-2.0f * P10 / rc + 3.0f * U20 - U00 + 3.0f * V11);
  out[2] = Kr[2] + 0.5f * dP[2] + INV_2PI * (-2.0f * P01 / rc + 3.0f * U11 + 3.0f * V02 - V00);
  out[3] = Kr[3] + INV_2PI * (P0 - 2.0f * rc * (UC + VS));
}

__device__ __forceinline__ void rusanov(const float *L, const float *R, float gam, int dir,
                                        float *F) {
  const float gm1i = 1.0f / (gam - 1.0f);
  float QL[4], QR[4];
  p2c(L, gm1i, QL);
  p2c(R, gm1i, QR);
  float uL = L[1 + dir], uR = R[1 + dir];
  float aL = fabsf(uL) + sqrtf(gam * L[3] / L[0]), aR = fabsf(uR) + sqrtf(gam * R[3] / R[0]);
  float al = fmaxf(aL, aR);
  float FL[4] = {QL[0] * uL, QL[1] * uL, QL[2] * uL, uL * (QL[3] + L[3])};
  float FR[4] = {QR[0] * uR, QR[1] * uR, QR[2] * uR, uR * (QR[3] + R[3])};
  FL[1 + dir] += L[3];
  FR[1 + dir] += R[3];
  for (int v = 0; v < NV; v++) F[v] = 0.5f * (FL[v] + FR[v]) - 0.5f * al * (QR[v] - QL[v]);
}

// Lax-Friedrichs update of a point value from the same-type point values one
// mesh width away (Alg. 3, last resort), converted back to primitive form
template <int K>
__device__ __noinline__ float4 lf_node(const Args &A, int i, int j, float tau) {
  const Grid &g = A.g;
  const float *a = A.n0[K];
  float U0[4], W[4], E[4], S[4], N[4], FW[4], FE[4], GS[4], GN[4], Q[4];
  ld4(A, a, i, j, U0);
  ld4(A, a, i - 1, j, W);
  ld4(A, a, i + 1, j, E);
  ld4(A, a, i, j - 1, S);
  ld4(A, a, i, j + 1, N);
  rusanov(W, U0, g.gamma, 0, FW);
  rusanov(U0, E, g.gamma, 0, FE);
  rusanov(S, U0, g.gamma, 1, GS);
  rusanov(U0, N, g.gamma, 1, GN);
  p2c(U0, 1.0f / (g.gamma - 1.0f), Q);
  const float lx = tau * g.idx, ly = tau * g.idy;
  for (int v = 0; v < NV; v++) Q[v] = Q[v] - lx * (FE[v] - FW[v]) - ly * (GN[v] - GS[v]);
  float out[4];
  c2p(Q, g.gamma - 1.0f, out);
  return pack4(out);
}

// averaged linearisation state, eq. (Un+1/2)
template <int K>
__device__ __forceinline__ void lin_avg(const float *sm, int li, int lj, float ul[4]) {
  const int a = li + 1, b = lj + 1;
  float4 s;
  if (K == VTX) {
    const float4 q0 = ubar4(sm, a - 1, b - 1), q1 = ubar4(sm, a, b - 1), q2 = ubar4(sm, a - 1, b), q3 = ubar4(sm, a, b);
    s = make_float4(0.25f * (q0.x + q1.x + q2.x + q3.x), 0.25f * (q0.y + q1.y + q2.y + q3.y),
                    0.25f * (q0.z + q1.z + q2.z + q3.z), 0.25f * (q0.w + q1.w + q2.w + q3.w));
  } else {
    const float4 q0 = (K == XE) ? ubar4(sm, a - 1, b) : ubar4(sm, a, b - 1), q1 = ubar4(sm, a, b);
    s = make_float4(0.5f * (q0.x + q1.x), 0.5f * (q0.y + q1.y), 0.5f * (q0.z + q1.z), 0.5f * (q0.w + q1.w));
  }
  ul[0] = s.x;
  ul[1] = s.y;
  ul[2] = s.z;
  ul[3] = s.w;
}

// Alg. 3 for one time level: EG1 on pc data with the averaged linearisation,
// else Lax-Friedrichs, else the node's t^n value Kr (the high-order value
// failed).  The calls behind which the rare paths sit take and return values,
// never addresses: an array whose address is passed lives in local memory for
// the whole kernel, taken path or not.  The events met here are counted with
// atomics (they are rare).
template <int K>
__device__ __noinline__ float4 limit(const Args &A, const float *sm, int i, int j, int li, int lj, float tau,
                                     float4 Kr4) {
  const float Kr[4] = {Kr4.x, Kr4.y, Kr4.z, Kr4.w};
  if (A.force_lo != 2) {
    float ul[4], lo[4];
    lin_avg<K>(sm, li, lj, ul);
    eg1_pc<K>(A.g, sm, li, lj, Kr, ul, tau, lo);
    atomicAdd(&A.counters[CNT_EG1], 1ull);
    if (admissible(lo)) return pack4(lo);
  }
  const float4 lf4 = lf_node<K>(A, i, j, tau);
  const float lf[4] = {lf4.x, lf4.y, lf4.z, lf4.w};
  atomicAdd(&A.counters[CNT_LF], 1ull);
  if (admissible(lf)) return lf4;
  atomicAdd(&A.counters[CNT_KEPT], 1ull);
  atomicOr(A.status, ST_KEPT);
  return Kr4;
}

// node bounds (with the option on): rho and p within [NB_ETA min, max / NB_ETA]
// of the node's own t^n value U0 and the primitive averages of its cells
constexpr float NB_ETA = 0.1f;
template <int K>
__device__ __noinline__ bool in_node_bounds(const float *sm, int li, int lj, float4 U0, float4 U) {
  const int a = li + 1, b = lj + 1;
  float rlo = U0.x, rhi = U0.x, plo = U0.w, phi = U0.w;
  const int ncell = K == VTX ? 4 : 2;
  for (int q = 0; q < ncell; q++) {
    const int ca = K == VTX ? a - 1 + (q & 1) : (K == XE ? a - 1 + q : a);
    const int cb = K == VTX ? b - 1 + (q >> 1) : (K == XE ? b : b - 1 + q);
    const float4 w = ubar4(sm, ca, cb);
    rlo = fminf(rlo, w.x);
    rhi = fmaxf(rhi, w.x);
    plo = fminf(plo, w.w);
    phi = fmaxf(phi, w.w);
  }
  return U.x >= NB_ETA * rlo && U.x <= rhi / NB_ETA && U.w >= NB_ETA * plo && U.w <= phi / NB_ETA;
}

// the blend's low-order value: EG1 on pc data inline (it is short and
// branch-free), the rest of Alg. 3's chain behind a call only if that fails
template <int K>
__device__ __forceinline__ void blend_low(const Args &A, const float *sm, int i, int j, int li, int lj, float tau,
                                          const float *Kr, float *res, unsigned *cnt) {
  if (A.force_lo != 2) {
    float ul[4], lo[4];
    lin_avg<K>(sm, li, lj, ul);
    eg1_pc<K>(A.g, sm, li, lj, Kr, ul, tau, lo);
    if (admissible(lo)) {
      cnt[CNT_EG1]++;
#pragma unroll
      for (int v = 0; v < NV; v++) res[v] = lo[v];
      return;
    }
  }
  unpack4(limit<K>(A, sm, i, j, li, lj, tau, pack4(Kr)), res);
}

// Alg. 2 indicator of the vertex at tile-local cell corner (a, b): the
// primitive averages of cells (a-1, b-1), (a, b-1), (a-1, b), (a, b)
__device__ __forceinline__ bool tsw_vertex(const float *sm, float gam, int a, int b) {
  float u[4], v[4], c[4];
  const int ca[4] = {a - 1, a, a - 1, a}, cb[4] = {b - 1, b - 1, b, b};  // LL, RL, LU, RU
#pragma unroll
  for (int q = 0; q < 4; q++) {
    const float4 w = ubar4(sm, ca[q], cb[q]);
    u[q] = w.y;
    v[q] = w.z;
    c[q] = sqrtf(gam * w.w / w.x);
  }
  bool f = false;
#pragma unroll
  for (int sg = -1; sg <= 1; sg += 2) {
    f = f || (u[2] + sg * c[2] > 0.0f && u[3] + sg * c[3] < 0.0f) ||
        (u[0] + sg * c[0] > 0.0f && u[1] + sg * c[1] < 0.0f) ||
        (v[0] + sg * c[0] > 0.0f && v[2] + sg * c[2] < 0.0f) ||
        (v[1] + sg * c[1] > 0.0f && v[3] + sg * c[3] < 0.0f);
  }
  return f;
}

// Corollary 1: T such that C = tau^2/2 T, from centred differences of
// neighbouring point values or cell-centre values (U_c = monomial m00)
template <int K, int TY>
__device__ __forceinline__ void correction(const Grid &g, const float *sm, const float *raw, int i, int j,
                                           int i0, int j0, const float U[4], float T[4]) {
  float Ux[4], Uy[4];
  const int a = i - i0 + 1, b = j - j0 + 1;
  float Cp[4], Cm[4];  // U_c on either side of the edge
  if (K != VTX) {
    const int ma = K == XE ? a - 1 : a, mb = K == XE ? b : b - 1;
#ifdef AF_PV_SHOCK
#pragma unroll
    for (int v = 0; v < NV; v++) {
      Cp[v] = centre(sm, a, b, v);
      Cm[v] = centre(sm, ma, mb, v);
    }
#else
    unpack4(cell_m00(cell_rec(sm, a, b)), Cp);
    unpack4(cell_m00(cell_rec(sm, ma, mb)), Cm);
#endif
  }
#pragma unroll
  for (int v = 0; v < NV; v++) {
    if (K == VTX) {
      Ux[v] = (raw_at<TY>(raw, RAW_YE, v, i, j, i0, j0) - raw_at<TY>(raw, RAW_YE, v, i - 1, j, i0, j0)) * g.idx;
      Uy[v] = (raw_at<TY>(raw, RAW_XE, v, i, j, i0, j0) - raw_at<TY>(raw, RAW_XE, v, i, j - 1, i0, j0)) * g.idy;
    } else if (K == XE) {
      Ux[v] = (Cp[v] - Cm[v]) * g.idx;
      Uy[v] = (raw_at<TY>(raw, RAW_VTX, v, i, j + 1, i0, j0) - raw_at<TY>(raw, RAW_VTX, v, i, j, i0, j0)) * g.idy;
    } else {
      Ux[v] = (raw_at<TY>(raw, RAW_VTX, v, i + 1, j, i0, j0) - raw_at<TY>(raw, RAW_VTX, v, i, j, i0, j0)) * g.idx;
      Uy[v] = (Cp[v] - Cm[v]) * g.idy;
    }
  }
  const float r = U[0], u = U[1], v = U[2], p = U[3], gm = g.gamma, ir = __fdividef(1.0f, r);
  const float rx = Ux[0], ux = Ux[1], vx = Ux[2], px = Ux[3];
  const float ry = Uy[0], uy = Uy[1], vy = Uy[2], py = Uy[3];
  const float f1 = ux * ux + uy * vx, f2 = uy * vx + vy * vy;
  const float g1 = px * (gm * (ux + vy) + ux) + py * vx;
  const float g2 = py * (gm * (ux + vy) + vy) + px * uy;
  const float h1 = (rx * px + ry * py) * ir, h2 = (rx * u + ry * v) * ir * ir;
  T[0] = r * (f1 + f2) + u * (rx * (2.0f * ux + vy) + ry * vx) + v * (rx * uy + ry * (ux + 2.0f * vy)) - h1;
  T[1] = u * f1 + v * uy * (ux + vy) + g1 * ir - px * h2;
  T[2] = v * f2 + u * vx * (ux + vy) + g2 * ir - py * h2;
  T[3] = u * g1 + v * g2 + gm * p * (f1 + f2 - h1 * ir);
}

__device__ __forceinline__ void st4(float *p, const Grid &g, int i, int j, const float U[4]) {
#pragma unroll
  for (int v = 0; v < NV; v++) p[at(g, v, i, j)] = U[v];
}
// store a value of node (K, i, j) and, on periodic axes, its duplicates (the
// duplicated last node line equals the first)
template <int K>
__device__ __forceinline__ void st4_node(float *p, const Grid &g, int i, int j, const float U[4]) {
  st4(p, g, i, j, U);
  const bool dx_ = (K != YE) && g.per_x && i == 0, dy_ = (K != XE) && g.per_y && j == 0;
  if (dx_) st4(p, g, g.nx, j, U);
  if (dy_) st4(p, g, i, g.ny, U);
  if (dx_ && dy_) st4(p, g, g.nx, g.ny, U);
}

// Instantiations of the node update, so that the code and the registers of each
// carry no more than its runs need: PV_LEAN the plain method with the Alg. 3
// limiter (linearisation about the averages or the node value, the correction);
// PV_FULL also Alg. 1's linearisation and the masks of the surrogate's fallback;
// PV_SHOCK also the switches for discontinuous data (Alg. 2, the Sec. 3.4 blend,
// node bounds) and the test hooks, with EG2 in the form of af_eg2_arc.cuh;
// PV_NF and PV_NF_SHOCK also write node fluxes.  pv_class picks.
enum { PV_LEAN = 0, PV_FULL = 1, PV_SHOCK = 2, PV_NF = 3, PV_NF_SHOCK = 4 };
__host__ __device__ inline int pv_class(const PointValueArgs &A) {
  const bool shock = A.tsw || A.theta[0] || A.node_bounds || A.force_lo;
  if (A.nflux[0]) return shock ? PV_NF_SHOCK : PV_NF;
  if (shock) return PV_SHOCK;
  return A.lin_mode == 2 || A.mask[0] || A.mask[1] || A.mask[2] || A.tile_flag ? PV_FULL : PV_LEAN;
}

// Simpson in time of eq. (F) at a node, for the flux kernel, once both levels
// are known: f(U^n) + 4 f(U^{n+1/2}) + f(U^{n+1}) (f for vertices and x-edges,
// g for vertices and y-edges; U^{n+1/2} kept in the thread's scratch, slots
// 0..3) into the node-flux arrays, and the new value's wave speed into the
// running maximum (slot 4; infinity for a value that is not admissible)
template <int K, int TY>
__device__ __forceinline__ void node_flux(const Args &A, int i, int j, const float U0[4], const float U1[4],
                                          float *scr) {
  const Grid &g = A.g;
  const float gm1i = 1.0f / (g.gamma - 1.0f);
  constexpr int NT = TX * TY;
  float Uh[4];
#pragma unroll
  for (int v = 0; v < NV; v++) Uh[v] = scr[v * NT];
#pragma unroll
  for (int dir = 0; dir < 2; dir++) {
    if ((dir == 0 && K == YE) || (dir == 1 && K == XE)) continue;
    float F[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    add_time_flux(U0, gm1i, dir, 1.0f, F);
    add_time_flux(Uh, gm1i, dir, 4.0f, F);
    add_time_flux(U1, gm1i, dir, 1.0f, F);
    st4_node<K>(A.nflux[K == VTX ? dir : (K == XE ? 2 : 3)], g, i, j, F);
  }
  bool bad = false;
  const float w = wave_speed(U1, g.gamma, bad);
  scr[4 * NT] = fmaxf(scr[4 * NT], bad ? __int_as_float(0x7f800000) : w);
}

// both time levels of node (K, i, j), tile-local (li, lj)
template <int K, int TY, int FT>
__device__ __forceinline__ void node_update(const Args &A, const float *sm, const float *raw, int i0, int j0,
                                            int i, int j, int li, int lj, unsigned cnt[4], bool &cfl_bad,
                                            bool &nonfinite, float *scr) {
  constexpr bool SHOCK = FT == PV_SHOCK || FT == PV_NF_SHOCK, NF = FT >= PV_NF, FULL = FT != PV_LEAN;
  const Grid &g = A.g;
  const int ni = (K == YE) ? g.nx : g.nxv, nj = (K == XE) ? g.ny : g.nyv;
  if (i >= ni || j >= nj) return;
  if (FULL && A.mask[K] && !A.mask[K][(long long)(j + OY) * g.P + (i + OX)]) return;
  float U0[4], T[4] = {0.0f, 0.0f, 0.0f, 0.0f};
  raw4<TY>(raw, K == VTX ? RAW_VTX : (K == XE ? RAW_XE : RAW_YE), i, j, i0, j0, U0);
  if (A.correction) correction<K, TY>(g, sm, raw, i, j, i0, j0, U0, T);

  float ul[4], res[4];
  // linearisation state of the half step
  if (A.lin_mode == 1) {
#pragma unroll
    for (int v = 0; v < NV; v++) ul[v] = U0[v];
  } else if (FULL && A.lin_mode == 2) {
#ifdef AF_PV_SHOCK
    cfl_bad |= !eg2_arc<K>(g, sm, li, lj, U0, U0, 0.25f * A.dt, ul);
#else
    // Alg. 1: level 0 of the loop below turns this into EG2's value over dt/4
#pragma unroll
    for (int v = 0; v < NV; v++) ul[v] = U0[v];
#endif
  } else {
    const bool wx = (K != YE) && ((i == 0 && g.bc[0] == BC_REFLECTING) || (i == g.nx && g.bc[1] == BC_REFLECTING));
    const bool wy = (K != XE) && ((j == 0 && g.bc[2] == BC_REFLECTING) || (j == g.ny && g.bc[3] == BC_REFLECTING));
    if (wx || wy) {
#pragma unroll
      for (int v = 0; v < NV; v++) ul[v] = U0[v];
      if (wx) ul[1] = 0.0f;
      if (wy) ul[2] = 0.0f;
    } else {
      lin_avg<K>(sm, li, lj, ul);
    }
  }
  // Sec. 3.4 blend weight (the same for both levels; from the t^n averages)
  float th = 1.0f;
  if (SHOCK && A.theta[0]) {
    if (K == XE) th = A.theta[0][at(g, 0, i, j)];
    else if (K == YE) th = A.theta[1][at(g, 0, i, j)];
    else
      th = fminf(fminf(A.theta[0][at(g, 0, i, j)], A.theta[0][at(g, 0, i, j - 1)]),
                 fminf(A.theta[1][at(g, 0, i, j)], A.theta[1][at(g, 0, i - 1, j)]));
  }
  bool sw = false;
  if (SHOCK && A.tsw) {
    const int a = li + 1, b = lj + 1;
    if (K == VTX) sw = tsw_vertex(sm, g.gamma, a, b);
    else if (K == XE) sw = tsw_vertex(sm, g.gamma, a, b) || tsw_vertex(sm, g.gamma, a, b + 1);
    else sw = tsw_vertex(sm, g.gamma, a, b) || tsw_vertex(sm, g.gamma, a + 1, b);
    if (K == VTX && sw) cnt[CNT_TSW]++;
  }

#ifndef AF_PV_SHOCK
  LineJumps J;
  line_jumps<K>(sm, li, lj, J);
#endif
#pragma unroll 1
  for (int lev = FULL && !SHOCK && A.lin_mode == 2 ? 0 : 1; lev <= 2; lev++) {
    const float tau = lev == 1 ? 0.5f * A.dt : (FULL && !SHOCK && lev == 0 ? 0.25f * A.dt : A.dt);
    if (lev == 2) {
      if (SHOCK && sw) {
        lin_avg<K>(sm, li, lj, ul);
      } else {
#pragma unroll
        for (int v = 0; v < NV; v++) ul[v] = res[v];
      }
    }
    float ho[4];
    bool inb;
#ifdef AF_PV_SHOCK
    inb = eg2_arc<K>(g, sm, li, lj, U0, ul, tau, ho);
#else
    inb = eg2<K>(g, sm, li, lj, U0, ul, tau, J, ho);
#endif
    cfl_bad |= !inb;
    if (FULL && !SHOCK && lev == 0) {
#pragma unroll
      for (int v = 0; v < NV; v++) ul[v] = ho[v];
      continue;
    }
    const float ht = 0.5f * tau * tau;
#pragma unroll
    for (int v = 0; v < NV; v++) ho[v] = fmaf(ht, T[v], ho[v]);
    // Alg. 3 (a value from a Mach cone outside the block counts as not
    // admissible, and, with the option, one outside the node's bounds)
    bool ok = inb && admissible(ho);
    if (SHOCK && ok && A.node_bounds) ok = in_node_bounds<K>(sm, li, lj, pack4(U0), pack4(ho));
    if ((SHOCK && A.force_lo) || (A.limiter && !ok)) {
      unpack4(limit<K>(A, sm, i, j, li, lj, tau, pack4(U0)), res);
    } else {
#pragma unroll
      for (int v = 0; v < NV; v++) res[v] = ho[v];
    }
    if (SHOCK && 1.0f - th >= 1e-6f) {
      // blend with the low-order value of Alg. 3's chain (EG1 on pc data,
      // else Lax-Friedrichs, else the t^n value): both ends admissible
      float lo[4];
      blend_low<K>(A, sm, i, j, li, lj, tau, U0, lo, cnt);
#pragma unroll
      for (int v = 0; v < NV; v++) res[v] = th * res[v] + (1.0f - th) * lo[v];
    }
#pragma unroll
    for (int v = 0; v < NV; v++) nonfinite |= (SHOCK || !ok) && !isfinite(res[v]);  // (an ok value is finite; a blend with it need not be)
    if (NF && lev == 1) {
#pragma unroll
      for (int v = 0; v < NV; v++) scr[v * (TX * TY)] = res[v];
    }
    if (!NF || lev == 2 || A.write_half) st4_node<K>(lev == 1 ? A.n1[K] : A.n2[K], g, i, j, res);
  }
  if (NF) node_flux<K, TY>(A, i, j, U0, res, scr);
}

// prologue: the block builds the records of the tile's cells and its halo on
// the low sides, (TX+1) x (TY+1); only cells -1..nx, -1..ny can be referenced
// by owned nodes, the others are skipped.  The last column and row of the halo
// (cells i0 + TX, j0 + TY) are read only by Alg. 2's indicator at the tile's last
// edge nodes: built with Alg. 2 only (340 instead of 297 records at TY = 8).
#ifdef AF_PV_SHOCK
template <int TY, int W, int H>
__device__ __forceinline__ void build_records(const Args &A, const float *raw, float *sm, int i0, int j0, int tid) {
  for (int k = tid; k < W * H; k += TX * TY) {
    const int a = k % W, b = k / W, ci = i0 - 1 + a, cj = j0 - 1 + b;
    if (ci <= A.g.nx && cj <= A.g.ny) {
      float *rec = const_cast<float *>(cell_rec(sm, a, b));
      build_cell<TY>(A.g, raw, i0, j0, ci, cj, rec + UBAR_OFF, rec);
    }
  }
}
template <int TY>
__device__ __forceinline__ void tile_prologue(const Args &A, const float *raw, float *sm, int i0, int j0,
                                              int tid) {
  if (A.tsw) build_records<TY, HX, Tile<TY>::HY>(A, raw, sm, i0, j0, tid);
  else build_records<TY, HX - 1, Tile<TY>::HY - 1>(A, raw, sm, i0, j0, tid);
}
#else
template <int TY>
__device__ __forceinline__ void tile_prologue(const Args &A, const float *raw, float *sm, int i0, int j0,
                                              int tid) {
  constexpr int W = HX - 1, H = Tile<TY>::HY - 1;
  for (int k = tid; k < W * H; k += TX * TY) {
    const int a = k % W, b = k / W, ci = i0 - 1 + a, cj = j0 - 1 + b;
    if (ci <= A.g.nx && cj <= A.g.ny)
      build_cell<TY>(A.g, raw, i0, j0, ci, cj, const_cast<float *>(cell_ubar(sm, a, b)),
                     const_cast<float *>(cell_rec(sm, a, b)));
  }
}
#endif

// the block's maximum wave speed of the new point values (node-flux
// instantiation: each thread's running maximum in scratch slot 4) into
// A.speed, one atomic a block
template <int TY>
__device__ __forceinline__ void block_speed(const Args &A, const float *scr, int tid) {
  __shared__ float wmax[TX * TY / 32];
  __shared__ int wbad[TX * TY / 32];
  float smax = scr[4 * TX * TY];
  const bool sbad = isinf(smax);
  smax = sbad ? 0.0f : smax;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) smax = fmaxf(smax, __shfl_xor_sync(0xffffffffu, smax, o));
  const bool anybad = __any_sync(0xffffffffu, sbad);
  if ((tid & 31) == 0) {
    wmax[tid >> 5] = smax;
    wbad[tid >> 5] = anybad;
  }
  __syncthreads();
  if (tid == 0) {
    float m = 0.0f;
    int b = 0;
    for (int w = 0; w < TX * TY / 32; w++) {
      m = fmaxf(m, wmax[w]);
      b |= wbad[w];
    }
    atomicMax(A.speed, __float_as_uint(m));  // positive floats order like their bit patterns
    if (b) atomicOr(A.speed_bad, 1);
  }
}

// node updates of the cell (i0 + tx, j0 + ty), of one kind or (kind < 0) all; NF: the instantiation that
// writes node fluxes (separate, so that the plain kernel carries none of it)
template <int TY, int FT>
__device__ __forceinline__ void tile_nodes(const Args &A, const float *sm, const float *raw, int i0, int j0,
                                           int tx, int ty, float *scr, int kind) {
  constexpr bool NF = FT >= PV_NF;
  unsigned cnt[4] = {0, 0, 0, 0};
  bool cfl_bad = false, nonfinite = false;
  const int i = i0 + tx, j = j0 + ty;
  constexpr int NT = TX * TY;
  if (NF) scr[4 * NT] = 0.0f;
  if (kind < 0 || kind == VTX) node_update<VTX, TY, FT>(A, sm, raw, i0, j0, i, j, tx, ty, cnt, cfl_bad, nonfinite, scr);
  if (kind < 0 || kind == XE) node_update<XE, TY, FT>(A, sm, raw, i0, j0, i, j, tx, ty, cnt, cfl_bad, nonfinite, scr);
  if (kind < 0 || kind == YE) node_update<YE, TY, FT>(A, sm, raw, i0, j0, i, j, tx, ty, cnt, cfl_bad, nonfinite, scr);
  if (NF) block_speed<TY>(A, scr, ty * TX + tx);
  // (the limiter reports its own kept values and Lax-Friedrichs fall-backs)
  const int st = (cfl_bad ? ST_CFL : 0) | (nonfinite ? ST_NONFINITE : 0);
  if (st) atomicOr(A.status, st);
#pragma unroll
  for (int k = 0; k < 4; k++)
    if (cnt[k]) atomicAdd(&A.counters[k], (unsigned long long)cnt[k]);
}

// ---------------------------------------------------------------- TMA staging
__device__ __forceinline__ unsigned smem_addr(const void *p) {
  return static_cast<unsigned>(__cvta_generic_to_shared(p));
}

// one thread: arm the barrier with the byte count and issue the four box
// loads (no_copy: the timeout test hook, which arms it and issues nothing)
template <int TY>
__device__ __forceinline__ void tile_fetch(const TileMaps &T, float *raw, unsigned long long *bar, int i0,
                                           int j0, int no_copy) {
  const unsigned b = smem_addr(bar);
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(b) : "memory");
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(b), "r"(Tile<TY>::RAW_BYTES) : "memory");
  if (no_copy) return;
  // box origin: column i0 (grid index i0 - 4), row j0 + 1 (grid index j0 - 1), variable 0
  const int x = i0, y = j0 + OY - 1;
  const CUtensorMap *maps[4] = {&T.vtx, &T.xe, &T.ye, &T.avg};
#pragma unroll
  for (int a = 0; a < 4; a++) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(smem_addr(raw + a * Tile<TY>::RAW_ARR)),
        "l"(reinterpret_cast<unsigned long long>(maps[a])), "r"(x), "r"(y), "r"(0), "r"(b)
        : "memory");
  }
}

// bounded wait for phase 0 of the barrier; false on time-out
__device__ __forceinline__ bool tile_wait(unsigned long long *bar, unsigned limit) {
  const unsigned b = smem_addr(bar);
  for (unsigned it = 0; it < limit; it++) {
    unsigned done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], 0;\n selp.u32 %0, 1, 0, p;\n}"
        : "=r"(done)
        : "r"(b)
        : "memory");
    if (done) return true;
  }
  return false;
}

// one tile: stage the t^n box, build the cell records, update the nodes
template <int TY, int FT>
__device__ __forceinline__ void tile_body(const Args &A, const TileMaps &T, float *raw, unsigned long long *bar,
                                          int i0, int j0, int kind) {
  float *sm = raw + Tile<TY>::RAW_FLOATS;
  const int tid = threadIdx.y * TX + threadIdx.x;
#ifdef AF_CHECK_BOUNDS
  if (tid == 0) rec_rows = Tile<TY>::HY;
#endif
  if (tid == 0) tile_fetch<TY>(T, raw, bar, i0, j0, A.test_no_copy);
  __syncthreads();
  const bool landed = tile_wait(bar, A.wait_limit);
  if (!__syncthreads_and(landed)) {
    // the copy did not land in time: report it (the host then refuses further
    // steps of the handle) and leave the tile alone.  The block's shared
    // memory stays allocated until its last thread exits, so thread 0 first
    // waits kDrainFactor times longer for the copy to land; if even that runs
    // out, the block exits with its copy unfinished.  Under the test hook no
    // copy was issued and nothing is in flight.
    if (tid == 0) {
      atomicOr(A.status, ST_TIMEOUT);
      if (!landed && !A.test_no_copy) tile_wait(bar, kDrainFactor * A.wait_limit);
    }
    return;
  }
  tile_prologue<TY>(A, raw, sm, i0, j0, tid);
  __syncthreads();
  tile_nodes<TY, FT>(A, sm, raw, i0, j0, threadIdx.x, threadIdx.y, sm + Tile<TY>::REC_FLOATS + tid, kind);
}

// TMA destinations must start on 128-byte boundaries
__device__ __forceinline__ float *tile_smem(float4 *smem4) {
  return reinterpret_cast<float *>((reinterpret_cast<size_t>(smem4) + 127) & ~size_t(127));
}

// Blocks per SM that the register budget is sized for: two for 8 rows (128
// registers a thread, 16 warps), one for 16 rows, four for 4 rows (the same 16
// warps; with five blocks the 96 registers spill: 2.88 against 2.39 ms at
// 4096^2).
template <int TY>
constexpr int min_blocks() {
  return TY == 4 ? 4 : (TY == 8 ? 2 : 1);
}

// L2 prefetch of the tile that the block PREFETCH_AHEAD places later in
// launch order takes, so that its TMA copy finds the data in L2.  304 is a wave of
// the 8-row kernels (two blocks an SM), for which it was chosen (with their former
// sums 12.96 -> 12.87 ms at 8192^2).  Half a wave of the plain 4-row kernel, which it
// costs 0.4 %: 9.13 against 9.09 ms without it and 9.13 at a whole wave, 608.
constexpr unsigned PREFETCH_AHEAD = 304;
template <int TY>
__device__ __forceinline__ void tile_prefetch_l2(const TileMaps &T) {
  const unsigned lin = blockIdx.y * gridDim.x + blockIdx.x + PREFETCH_AHEAD;
  if (lin >= gridDim.x * gridDim.y) return;
  const int x = (lin % gridDim.x) * TX, y = (lin / gridDim.x) * TY + OY - 1;
  const CUtensorMap *maps[4] = {&T.vtx, &T.xe, &T.ye, &T.avg};
#pragma unroll
  for (int a = 0; a < 4; a++)
    asm volatile("cp.async.bulk.prefetch.tensor.3d.L2.global.tile [%0, {%1, %2, %3}];" ::"l"(
                     reinterpret_cast<unsigned long long>(maps[a])),
                 "r"(x), "r"(y), "r"(0)
                 : "memory");
}

template <int TY, int FT>
__global__ void __launch_bounds__(TX *TY, min_blocks<TY>()) pointvalue_kernel(Args A, const __grid_constant__ TileMaps T) {
  extern __shared__ float4 smem4[];
  __shared__ alignas(8) unsigned long long bar;
  pdl_start();
  pdl_wait();
  if (A.clear_speed && threadIdx.x == 0 && threadIdx.y == 0 && blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0) {
    *A.clear_speed = 0u;
    *A.clear_bad = 0;
  }
  if (FT != PV_LEAN && A.tile_flag && !A.tile_flag[blockIdx.y * gridDim.x + blockIdx.x]) return;
  if (threadIdx.x == 0 && threadIdx.y == 0) tile_prefetch_l2<TY>(T);
  tile_body<TY, FT>(A, T, tile_smem(smem4), &bar, blockIdx.x * TX, blockIdx.y * TY,
                    FT != PV_SHOCK && FT != PV_NF_SHOCK && gridDim.z > 1 ? (int)blockIdx.z : -1);
}

// Batched form: block b takes tile B.tiles[b] = (instance, i0, j0) and the
// instance's arguments and descriptors for the buffer now holding its t^n;
// instances that have stopped are skipped.
template <int TY, int FT>
__global__ void __launch_bounds__(TX *TY, min_blocks<TY>()) pointvalue_batch_kernel(PointValueBatch B) {
  extern __shared__ float4 smem4[];
  __shared__ alignas(8) unsigned long long bar;
  const int4 t = B.tiles[blockIdx.x];
  const BatchCtl &c = B.ctl[t.x];
  if (!c.active) return;
  // the instance's arguments are read in place (the step's dt is in them):
  // read-only, so the compiler may load a field again where a copy in shared
  // memory held it in a register (half the spills)
  const Args *__restrict__ A = B.args + 2 * t.x + c.cur;
  tile_body<TY, FT>(*A, B.maps[2 * t.x + c.cur], tile_smem(smem4), &bar, t.y, t.z, -1);
}

}  // namespace

}  // namespace af
