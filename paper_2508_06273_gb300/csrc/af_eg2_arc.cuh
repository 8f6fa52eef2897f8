// af_eg2_arc.cuh -- EG2 summed from the circle coefficients of the cells around a
// node (part of af_pointvalue.cuh, on its records for shock units).  The runs with the
// Sec. 3 switches for discontinuous data (Alg. 2, the Sec. 3.4 blend, node
// bounds) keep this form and its order of summation: their solutions amplify a
// difference in the last place by up to 1e6 in ten steps (seeded four-quadrant
// problems of 64^2 to 512^2: 3 of 12 ensembles differ by more than 1e-4 after
// one unit in the last place on the inputs), so a form that rounds otherwise
// gives other trajectories, though none less accurate.  The truncated-power form of
// af_pointvalue.cuh, which every other run takes, is 19 % faster here.
#pragma once

// J[m][n] = int_{t0}^{t1} cos^m sin^n for m, n <= 4, m + n <= 6
__device__ __forceinline__ void jtable(float t0, float c0, float s0, float t1, float c1, float s1,
                                       float J[5][5]) {
  float c0s = c0 * c0, c1s = c1 * c1, c0c = c0s * c0, c1c = c1s * c1;
  float s0s = s0 * s0, s1s = s1 * s1, s0c = s0s * s0, s1c = s1s * s1;
  float s0q = s0s * s0s, s1q = s1s * s1s;
  float Ds = s1 - s0, Dc = c1 - c0, Ds2 = s1s - s0s;
  float Dcs = c1 * s1 - c0 * s0, Dc2s = c1s * s1 - c0s * s0, Dc3s = c1c * s1 - c0c * s0;
  float Dcs2 = c1 * s1s - c0 * s0s, Dc2s2 = c1s * s1s - c0s * s0s, Dc3s2 = c1c * s1s - c0c * s0s;
  float Dcs3 = c1 * s1c - c0 * s0c, Dc2s3 = c1s * s1c - c0s * s0c, Dc3s3 = c1c * s1c - c0c * s0c;
  float Dcs4 = c1 * s1q - c0 * s0q, Dc2s4 = c1s * s1q - c0s * s0q;
  float Dcs5 = c1 * s1q * s1 - c0 * s0q * s0;
  J[0][0] = t1 - t0;
  J[1][0] = Ds;
  J[0][1] = -Dc;
  J[1][1] = 0.5f * Ds2;
  J[2][0] = 0.5f * (Dcs + J[0][0]);
  J[3][0] = (Dc2s + 2.0f * J[1][0]) * (1.0f / 3.0f);
  J[4][0] = 0.25f * (Dc3s + 3.0f * J[2][0]);
  J[2][1] = (Dcs2 + J[0][1]) * (1.0f / 3.0f);
  J[3][1] = 0.25f * (Dc2s2 + 2.0f * J[1][1]);
  J[4][1] = 0.2f * (Dc3s2 + 3.0f * J[2][1]);
  J[0][2] = 0.5f * (J[0][0] - Dcs);
  J[1][2] = (J[1][0] - Dc2s) * (1.0f / 3.0f);
  J[2][2] = 0.25f * (Dcs3 + J[0][2]);
  J[3][2] = 0.2f * (Dc2s3 + 2.0f * J[1][2]);
  J[4][2] = (Dc3s3 + 3.0f * J[2][2]) * (1.0f / 6.0f);
  J[0][3] = (2.0f * J[0][1] - Dcs2) * (1.0f / 3.0f);
  J[1][3] = 0.25f * (2.0f * J[1][1] - Dc2s2);
  J[2][3] = 0.2f * (Dcs4 + J[0][3]);
  J[3][3] = (Dc2s4 + 2.0f * J[1][3]) * (1.0f / 6.0f);
  J[0][4] = 0.25f * (3.0f * J[0][2] - Dcs3);
  J[1][4] = 0.2f * (3.0f * J[1][2] - Dc2s3);
  J[2][4] = (Dcs5 + J[0][4]) * (1.0f / 6.0f);
}

// Taylor shift of q(x) = a0 + a1 x + a2 x^2 to x = x0 + r c:  q = b0 + b1 c + b2 c^2
__device__ __forceinline__ void shift(float a0, float a1, float a2, float x0, float r, float r2,
                                      float &b0, float &b1, float &b2) {
  const float t = fmaf(a2, x0, a1);
  b0 = fmaf(t, x0, a0);
  b1 = fmaf(a2, x0, t) * r;
  b2 = a2 * r2;
}

// coefficients b[a][e] of cos^a sin^e of (cell polynomial - K) on the circle
// x = x0 + rx cos, y = y0 + ry sin (cell-centred units)
__device__ __forceinline__ void circle_coef(const float *rec, float K, float x0, float y0, float rx,
                                            float rx2, float ry, float ry2, float b[3][3]) {
  const float4 p0 = reinterpret_cast<const float4 *>(rec)[0];
  const float4 p1 = reinterpret_cast<const float4 *>(rec)[1];
  const float m22 = reinterpret_cast<const float4 *>(rec)[2].x;
  // m[a][e]: x^a y^e;  p0 = (m00, m01, m02, m10), p1 = (m11, m12, m20, m21)
  float q[3][3];  // q[a][e]: cos^a y^e
  shift(p0.x - K, p0.w, p1.z, x0, rx, rx2, q[0][0], q[1][0], q[2][0]);
  shift(p0.y, p1.x, p1.w, x0, rx, rx2, q[0][1], q[1][1], q[2][1]);
  shift(p0.z, p1.y, m22, x0, rx, rx2, q[0][2], q[1][2], q[2][2]);
#pragma unroll
  for (int a = 0; a < 3; a++) shift(q[a][0], q[a][1], q[a][2], y0, ry, ry2, b[a][0], b[a][1], b[a][2]);
}

// value of (cell polynomial - K) at (x0, y0)
__device__ __forceinline__ float eval_at(const float *rec, float K, float x0, float y0) {
  const float4 p0 = reinterpret_cast<const float4 *>(rec)[0];
  const float4 p1 = reinterpret_cast<const float4 *>(rec)[1];
  const float m22 = reinterpret_cast<const float4 *>(rec)[2].x;
  const float e0 = fmaf(fmaf(p1.z, x0, p0.w), x0, p0.x - K);
  const float e1 = fmaf(fmaf(p1.w, x0, p1.x), x0, p0.y);
  const float e2 = fmaf(fmaf(m22, x0, p1.y), x0, p0.z);
  return fmaf(fmaf(e2, y0, e1), y0, e0);
}

// ---- EG2 arc sums by inclusion-exclusion
// In the frame reflected so that u', v' >= 0 (cos -> fx cos, sin -> fy sin),
// the grid lines through the node split the circle into the sides
// X = {cos > a} (a = |u'|/c') and Y = {sin > b} (b = |v'|/c'): X is the arc
// (-acos a, acos a), Y the arc (asin b, pi - asin b), and X and Y meet in the
// single arc (asin b, acos a) when a^2 + b^2 < 1, else not at all.  With b_q
// the circle coefficients of the cell on side q (++, +-, -+, --), the sum
// over the cells' arcs of int b_q w is
//   int_circle b_-- w + int_X (b_+- - b_--) w + int_Y (b_-+ - b_--) w
//   + int_(X and Y) (b_++ - b_+- - b_-+ + b_--) w,
// exactly (inclusion-exclusion of the four quadrants).  Over the whole circle
// only even powers of both cos and sin integrate to non-zero values; over X
// (symmetric about 0) only even powers of sin, over Y (symmetric about
// pi/2) only even powers of cos.  An edge-midpoint node (one grid line) keeps
// the first two terms (XE) or the first and third (YE).

// H[m][n] = int_{-al}^{al} cos^m sin^n for n even (al = acos a, s = sin al):
// twice the integrals from 0, by the recurrences of jtable with the start
// point (1, 0); the entries m <= 4, n <= 4, m + n <= 6 the moments use
__device__ __forceinline__ void half_table(float a, float s, float al, float H[5][5]) {
  const float s2 = s * s, s3 = s2 * s, a2 = a * a, a3 = a2 * a;
  const float as = a * s, as3 = a * s3;
  const float I20 = 0.5f * (as + al), I02 = 0.5f * (al - as), I12 = s3 * (1.0f / 3.0f);
  const float I22 = 0.25f * (as3 + I02), I04 = 0.25f * (3.0f * I02 - as3);
  H[0][0] = 2.0f * al;
  H[1][0] = 2.0f * s;
  H[2][0] = 2.0f * I20;
  H[3][0] = (2.0f / 3.0f) * (a2 * s + 2.0f * s);
  H[4][0] = 0.5f * (a3 * s + 3.0f * I20);
  H[0][2] = 2.0f * I02;
  H[1][2] = 2.0f * I12;
  H[2][2] = 2.0f * I22;
  H[3][2] = 0.4f * (a2 * s3 + 2.0f * I12);
  H[4][2] = (1.0f / 3.0f) * (a3 * s3 + 3.0f * I22);
  H[0][4] = 2.0f * I04;
  H[1][4] = 0.4f * (3.0f * I12 - a2 * s3);
  H[2][4] = (1.0f / 3.0f) * (as3 * s2 + I04);
}

// int over the whole circle of cos^m sin^n for the (m, n) the moments use
// (zero unless m and n are even)
__host__ __device__ constexpr float jfull(int m, int n) {
  return ((m & 1) || (n & 1)) ? 0.0f
         : (m == 0 && n == 0) ? 2.0f * PI_F
         : (m + n == 2) ? PI_F
         : (m == 2 && n == 2) ? 0.25f * PI_F
         : (m + n == 4) ? 0.75f * PI_F
         : (m + n == 6 && m != 0 && n != 0) ? 0.125f * PI_F
         : 0.0f;
}

// table kinds: full arc table, X-side table H (odd n vanish), Y-side table
// (odd m vanish; stored transposed, H[n][m]), whole circle (constants)
enum { TB_ARC = 0, TB_X = 1, TB_Y = 2, TB_CIRCLE = 3 };

// acc + sum_{i,e <= 2} b[i][e] T(i + DI, e + DE), skipping the entries the
// table's symmetry makes zero
template <int DI, int DE, int KIND>
__device__ __forceinline__ float contract(const float b[3][3], const float T[5][5], float acc) {
#pragma unroll
  for (int i = 0; i < 3; i++)
#pragma unroll
    for (int e = 0; e < 3; e++) {
      const int m = i + DI, n = e + DE;
      if (KIND == TB_X && (n & 1)) continue;
      if (KIND == TB_Y && (m & 1)) continue;
      if (KIND == TB_CIRCLE && ((m | n) & 1)) continue;
      const float t = KIND == TB_CIRCLE ? jfull(m, n) : (KIND == TB_Y ? T[n][m] : T[m][n]);
      acc = fmaf(b[i][e], t, acc);
    }
  return acc;
}

// the EG2 moments of one variable against one table: p (VAR 0): int p,
// int p cos, int p sin; u (1): int u cos, int u cos^2, int u, int u sin cos;
// v (2): int v sin, int v sin^2, int v, int v sin cos
template <int VAR, int KIND>
__device__ __forceinline__ void moments(const float b[3][3], const float T[5][5], float acc[4]) {
  if (VAR == 0) {
    acc[0] = contract<0, 0, KIND>(b, T, acc[0]);
    acc[1] = contract<1, 0, KIND>(b, T, acc[1]);
    acc[2] = contract<0, 1, KIND>(b, T, acc[2]);
  } else if (VAR == 1) {
    acc[0] = contract<1, 0, KIND>(b, T, acc[0]);
    acc[1] = contract<2, 0, KIND>(b, T, acc[1]);
    acc[2] = contract<0, 0, KIND>(b, T, acc[2]);
    acc[3] = contract<1, 1, KIND>(b, T, acc[3]);
  } else {
    acc[0] = contract<0, 1, KIND>(b, T, acc[0]);
    acc[1] = contract<0, 2, KIND>(b, T, acc[1]);
    acc[2] = contract<0, 0, KIND>(b, T, acc[2]);
    acc[3] = contract<1, 1, KIND>(b, T, acc[3]);
  }
}

// node position in the cell-centred units of that cell, before the shift by -u' tau
template <int K>
__device__ __forceinline__ void node_in_cell(int right, int top, float &xn, float &yn) {
  xn = (K == YE) ? 0.0f : (right ? -0.5f : 0.5f);
  yn = (K == XE) ? 0.0f : (top ? -0.5f : 0.5f);
}

// EG2 of the cpq reconstruction at node (K, li, lj) of the tile, linearised
// about ul, relative to the reference state Kr.  Returns false if the Mach
// cone base leaves the node's block of cells (the CFL bound of the
// linearisation state fails; the value is then not an EG2 value).
template <int K>
__device__ __forceinline__ bool eg2_arc(const Grid &g, const float *sm, int li, int lj, const float Kr[4],
                                    const float ul_in[4], float tau, float out[4]) {
  // an inadmissible linearisation state gives NaN outputs; the arithmetic
  // runs on a harmless substitute so that no branch splits the evaluation
  const bool good = ul_in[0] > 0.0f && ul_in[3] > 0.0f && tau > 0.0f;
  const float ul[4] = {good ? ul_in[0] : 1.0f, good ? ul_in[1] : 0.0f, good ? ul_in[2] : 0.0f,
                       good ? ul_in[3] : 1.0f};
  const float cp2 = __fdividef(g.gamma * ul[3], ul[0]), icp = rsqrtf(cp2), cp = cp2 * icp;
  const float R = cp * tau;
  const float am = ul[1] * icp, bm = ul[2] * icp;
  bool inside;
  {
    const float ex = fabsf(ul[1]) * tau + R, ey = fabsf(ul[2]) * tau + R;
    const float lx = (K == YE) ? 0.5f * g.dx : g.dx, ly = (K == XE) ? 0.5f * g.dy : g.dy;
    inside = !(ex > lx || ey > ly);
  }
  const float rx = R * g.idx, ry = R * g.idy, rx2 = rx * rx, ry2 = ry * ry;
  const float sx = ul[1] * tau * g.idx, sy = ul[2] * tau * g.idy;

  // reflection signs (u', v' >= 0 in the reflected frame) and the sides met
  const float fx = (K != YE && ul[1] < 0.0f) ? -1.0f : 1.0f, fy = (K != XE && ul[2] < 0.0f) ? -1.0f : 1.0f;
  const float ax = fabsf(am), by = fabsf(bm);
  // a line the circle does not cross gives a half table of zeros (al = 0,
  // sin al = 0), so the X and Y stages run without branches
  constexpr bool hx = K != YE, hy = K != XE;
  const bool hq = K == VTX && ax < 1.0f && by < 1.0f && fmaf(ax, ax, by * by) < 1.0f;
  float Tx[5][5], Ty[5][5], Jq[5][5];
  float alx = 0.0f, snx = 0.0f, aly = 0.0f, sny = 0.0f;
  if (hx) {
    const float a = fminf(ax, 1.0f);
    alx = acosf(a);
    snx = sqrt_nn(fmaf(-a, a, 1.0f));
    half_table(a, snx, alx, Tx);
  }
  if (hy) {
    const float b = fminf(by, 1.0f);
    aly = acosf(b);
    sny = sqrt_nn(fmaf(-b, b, 1.0f));
    half_table(b, sny, aly, Ty);
  }
  // X and Y meet in (asin b, acos a): (cos, sin) = (sin aly, b) to (a, sin alx)
  if (hq) jtable(0.5f * PI_F - aly, sny, by, alx, ax, snx, Jq);
  const float frx = fx * rx, fry = fy * ry;

  // circle coefficients of variable (record offset off, reference Kv) of
  // the cell on side (px, py) (1: the + side) of the reflected frame
  auto side = [&](int px, int py, int off, float Kv, float q[3][3]) {
    const int right = px ? (fx > 0.0f) : (fx < 0.0f), top = py ? (fy > 0.0f) : (fy < 0.0f);
    int a, b;
    arc_cell<K>(li, lj, right, top, a, b);
    float xn, yn;
    node_in_cell<K>(right, top, xn, yn);
    circle_coef(cell_rec(sm, a, b) + off, Kv, xn - sx, yn - sy, frx, rx2, fry, ry2, q);
  };
  // all moments of one variable: b_-- over the circle, then the differences
  // over X, Y and their intersection
  auto var_moments = [&](auto var_tag, int off, float Kv, float acc[4]) {
    constexpr int VAR = decltype(var_tag)::value;
    float b0[3][3], S[3][3], d[3][3];
    side(0, 0, off, Kv, b0);
    moments<VAR, TB_CIRCLE>(b0, Tx, acc);
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
      for (int e = 0; e < 3; e++) S[i][e] = b0[i][e];
    if (hx) {
      side(1, 0, off, Kv, d);
#pragma unroll
      for (int i = 0; i < 3; i++)
#pragma unroll
        for (int e = 0; e < 3; e++) {
          S[i][e] -= d[i][e];
          d[i][e] -= b0[i][e];
        }
      moments<VAR, TB_X>(d, Tx, acc);
    }
    if (hy) {
      side(0, 1, off, Kv, d);
#pragma unroll
      for (int i = 0; i < 3; i++)
#pragma unroll
        for (int e = 0; e < 3; e++) {
          S[i][e] -= d[i][e];
          d[i][e] -= b0[i][e];
        }
      moments<VAR, TB_Y>(d, Ty, acc);
    }
    if (hq) {
      side(1, 1, off, Kv, d);
#pragma unroll
      for (int i = 0; i < 3; i++)
#pragma unroll
        for (int e = 0; e < 3; e++) d[i][e] += S[i][e];
      moments<VAR, TB_ARC>(d, Jq, acc);
    }
  };
  // the moments enter the result as soon as each variable is done (moments
  // odd in cos change sign with fx, odd in sin with fy, back in the grid frame)
  const float rp = ul[0], rc = rp * cp, irc = __fdividef(icp, rp), icp2 = icp * icp, rpi = rp * icp;
  float o[4], M[4] = {0.0f, 0.0f, 0.0f, 0.0f};
  var_moments(std::integral_constant<int, 0>(), 36, Kr[3], M);  // p0, pc, ps
  o[0] = M[0] * icp2;
  o[1] = -fx * M[1] * irc;
  o[2] = -fy * M[2] * irc;
  o[3] = M[0];
  M[0] = M[1] = M[2] = M[3] = 0.0f;
  var_moments(std::integral_constant<int, 1>(), 12, Kr[1], M);  // uc, u2, u0, usc
  const float uc = fx * M[0];
  o[0] = fmaf(-rpi, uc, o[0]);
  o[3] = fmaf(-rc, uc, o[3]);
  o[1] += 2.0f * M[1] - 0.5f * M[2];
  o[2] += 2.0f * fx * fy * M[3];
  M[0] = M[1] = M[2] = M[3] = 0.0f;
  var_moments(std::integral_constant<int, 2>(), 24, Kr[2], M);  // vs, v2, v0, vsc
  const float vs = fy * M[0];
  o[0] = fmaf(-rpi, vs, o[0]);
  o[3] = fmaf(-rc, vs, o[3]);
  o[2] += 2.0f * M[1] - 0.5f * M[2];
  o[1] += 2.0f * fx * fy * M[3];
  // rho and p at P' (the cell on side --: its closure holds P')
  float drP, dpP;
  {
    const int right = fx < 0.0f, top = fy < 0.0f;
    int a, b;
    arc_cell<K>(li, lj, right, top, a, b);
    const float *rec = cell_rec(sm, a, b);
    float xn, yn;
    node_in_cell<K>(right, top, xn, yn);
    drP = eval_at(rec, Kr[0], xn - sx, yn - sy);
    dpP = eval_at(rec + 36, Kr[3], xn - sx, yn - sy);
  }
  out[0] = Kr[0] + drP - 2.0f * dpP * icp2 + INV_PI * o[0];
  out[1] = Kr[1] + INV_PI * o[1];
  out[2] = Kr[2] + INV_PI * o[2];
  out[3] = Kr[3] - dpP + INV_PI * o[3];
  if (!good) {
#pragma unroll
    for (int v = 0; v < NV; v++) out[v] = __int_as_float(0x7fc00000);
    return true;
  }
  return inside;
}

