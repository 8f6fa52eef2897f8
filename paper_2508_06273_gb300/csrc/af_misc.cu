// af_misc.cu -- ghost cells (Sec. 4.3), reductions and layout conversion
// kernels.
#include "af_common.cuh"
#include "af_ghost.cuh"
#include "af_kernels.h"

namespace af {

namespace {

struct GhostArgs {
  Grid g;
  float *a[5];  // avg_hi, avg_lo, vtx, xe, ye
};

__global__ void ghost_kernel(GhostArgs A) {
  const int arr = blockIdx.y;
  const GhostRange R(A.g, arr);
  for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < R.total; k += gridDim.x * blockDim.x)
    ghost_entry(A.g, R, A.a[arr], arr, k);
}

// FP64 path: averages (no low word) and node arrays
__global__ void ghost64_kernel(Grid g, double *avg, double *vtx, double *xe, double *ye) {
  const int arr = blockIdx.y;
  if (arr == 1) return;
  double *p = arr == 0 ? avg : (arr == 2 ? vtx : (arr == 3 ? xe : ye));
  const GhostRange R(g, arr);
  for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < R.total; k += gridDim.x * blockDim.x)
    ghost_entry(g, R, p, arr, k);
}

// batched: block b fills chunk B.chunks[b] = (instance, array, first entry)
// (a list of exactly the blocks that have work, where a grid sized for the
// largest instance left most blocks of the small ones empty)
__global__ void __launch_bounds__(GHOST_CHUNK) ghost_batch_kernel(GhostBatch B) {
  const int4 c = B.chunks[blockIdx.x];
  const int inst = c.x, arr = c.y;
  if (!B.ctl[inst].active) return;
  const Grid &g = B.grids[inst];
  const GhostRange R(g, arr);
  float *p = B.arrays[(2 * inst + B.ctl[inst].cur) * 5 + arr];
  const int k = c.z + threadIdx.x;
  if (k < R.total) ghost_entry(g, R, p, arr, k);
}

// ---- Sec. 3.4 shock indicator: theta = exp(-phi1 phi2) per edge midpoint,
// phi1 the larger normalised second difference of the averaged pressure on
// either side of the edge, phi2 = 2^(max |u_n| + c of its two cells), the
// "bar" quantities from the primitive cell averages Ubar.
struct TnArrays {
  const float *avg, *vtx, *xe, *ye;
};
__device__ __forceinline__ float d2ratio(float a, float b, float c) {
  return fabsf((a - 2.0f * b + c) / (a + 2.0f * b + c));
}
// A block computes 32 x 8 entries: entry (a, b), a <= nx + 1, b <= ny + 1, is the
// x-edge (a - 1/2, b - 1) for a < nxv, b - 1 in -1 .. ny, and the y-edge
// (a - 1, b - 1/2) for a - 1 in -1 .. nx, b < nyv: the edges of every owned vertex
// (a vertex takes the minimum of its 4 edges).  The pressures and signal speeds of
// the tile's cells and of the two or one around it are formed once in shared
// memory, 1.5 cells an entry, where each entry formed its own eight: 105 -> 72
// us at 2048^2 (4 Riemann steps at 600^2 796 -> 779).
constexpr int TH_W = 32, TH_H = 8, TH_CW = TH_W + 3, TH_CH = TH_H + 3;
struct ThetaSmem {
  float p[TH_CH][TH_CW], s[2][TH_CH][TH_CW];  // pressure; |u| + c, |v| + c
};
__device__ __forceinline__ void theta_tile(const Grid &g, const TnArrays &t, float *tx, float *ty, int a0, int b0,
                                           ThetaSmem &S) {
  for (int k = threadIdx.y * TH_W + threadIdx.x; k < TH_CW * TH_CH; k += TH_W * TH_H) {
    const int ci = k % TH_CW, cj = k / TH_CW, i = a0 - 2 + ci, j = b0 - 2 + cj;
    const bool for_x = i <= g.nxv && j >= -1 && j <= g.ny, for_y = i >= -1 && i <= g.nx && j <= g.nyv;
    if (!for_x && !for_y) continue;
    float U[4];
    cell_ubar_global(g, t.avg, t.vtx, t.xe, t.ye, i, j, U);
    const float c = sqrtf(g.gamma * U[3] / U[0]);
    S.p[cj][ci] = U[3];
    S.s[0][cj][ci] = fabsf(U[1]) + c;
    S.s[1][cj][ci] = fabsf(U[2]) + c;
  }
  __syncthreads();
  const int x = threadIdx.x, y = threadIdx.y, a = a0 + x, b = b0 + y;
  auto theta = [&](int dir, int ci, int cj, int di, int dj) {  // of cells n = 0 .. 3 from (ci, cj) on
    const float m2 = S.p[cj][ci], m1 = S.p[cj + dj][ci + di], p0 = S.p[cj + 2 * dj][ci + 2 * di],
                p1 = S.p[cj + 3 * dj][ci + 3 * di];
    const float phi1 = fmaxf(d2ratio(p1, p0, m1), d2ratio(p0, m1, m2));
    return expf(-phi1 * exp2f(fmaxf(S.s[dir][cj + 2 * dj][ci + 2 * di], S.s[dir][cj + dj][ci + di])));
  };
  if (a < g.nxv && b <= g.ny + 1) tx[at(g, 0, a, b - 1)] = theta(0, x, y + 1, 1, 0);
  if (a <= g.nx + 1 && b < g.nyv) ty[at(g, 0, a - 1, b)] = theta(1, x + 1, y, 0, 1);
}
__global__ void __launch_bounds__(TH_W *TH_H) shock_theta_kernel(Grid g, TnArrays t, float *tx, float *ty) {
  __shared__ ThetaSmem S;
  theta_tile(g, t, tx, ty, blockIdx.x * TH_W, blockIdx.y * TH_H, S);
}
// batched: block k takes tile tiles[k] = (instance, a0, b0) of 32 x 8 entries
// (tiles only for the instances with the blend on); the instance's arrays
// (averages hi, lo, then the three node arrays) for its current t^n buffer
__global__ void __launch_bounds__(TH_W *TH_H) shock_theta_batch_kernel(const int4 *tiles, const BatchCtl *ctl,
                                                                       const Grid *grids, const float *const *arrays,
                                                                       float *const *theta) {
  __shared__ ThetaSmem S;
  const int4 tl = tiles[blockIdx.x];
  const int inst = tl.x;
  if (!ctl[inst].active || !theta[2 * inst]) return;
  const float *const *arr = arrays + (2 * inst + ctl[inst].cur) * 5;
  const TnArrays t = {arr[0], arr[2], arr[3], arr[4]};
  theta_tile(grids[inst], t, theta[2 * inst], theta[2 * inst + 1], tl.y, tl.z, S);
}

// Per-instance dt for the coming step from the wave speed of the current
// state (CFL condition, Sec. 2): dt = cfl * min(dx, dy) / speed, clipped so
// that the step ends at t_end.  An instance stops at t_end, or when its
// state has no finite positive wave speed (flagged ST_STOPPED).  The flip of
// the t^n buffer of the previous step is applied first; the speed is zeroed
// for the coming step's flux kernel, which refills it.
__global__ void batch_dt_kernel(BatchCtl *ctl, int n, double *hist, int hist_cap, int mode, PointValueArgs *pv) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) return;
  BatchCtl &c = ctl[k];
  if (mode != DT_PROBE && c.stepped) {
    c.cur ^= 1;
    c.stepped = 0;
  }
  if (mode == DT_SETTLE) return;
  double dt = 0.0;
  int go = 0;
  if (c.active) {
    const float sp = __uint_as_float(c.speed);
    const double left = c.t_end - c.t;
    if (c.speed_bad || !(sp > 0.0f) || !isfinite(sp)) {
      if (mode == DT_STEP) {
        c.active = 0;
        c.status |= ST_STOPPED;
      }
    } else if (isfinite(c.t_end) && !(left > 1e-12 * fabs(c.t_end))) {
      if (mode == DT_STEP) c.active = 0;
    } else {
      dt = c.cfl * c.h / (double)sp;
      if (dt >= left) dt = left;
      go = 1;
    }
  }
  c.dt = (float)dt;
  if (pv) pv[2 * k].dt = pv[2 * k + 1].dt = c.dt;
  const double lx = dt / c.dx, ly = dt / c.dy;
  c.lxh = (float)lx;
  c.lxl = (float)(lx - (double)c.lxh);
  c.lyh = (float)ly;
  c.lyl = (float)(ly - (double)c.lyh);
  if (mode == DT_PROBE) return;
  if (go) {
    if (hist && c.steps < hist_cap) hist[(long long)c.steps * n + k] = dt;
    c.t += dt;
    c.steps += 1;
    c.stepped = 1;
    c.speed = 0u;
    c.speed_bad = 0;
  }
}

__global__ void export_words_kernel(unsigned *a, unsigned *b, int clear_a, unsigned *dst) {
  if (threadIdx.x != 0) return;
  volatile unsigned *d = dst;
  d[0] = *a;
  d[1] = b ? *b : 0u;
  if (clear_a) *a = 0u;
  __threadfence_system();
}

// order-preserving unsigned key of a float (atomicMin on keys is a min on
// the floats; -0 and +0 get neighbouring keys)
__device__ __forceinline__ unsigned float_key(float f) {
  const unsigned u = __float_as_uint(f);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// Block b sums rows b, b + nblk, ... in a fixed order; the last block to finish
// sums the blocks' sums, in a fixed order too, into mapped host memory.  A read
// of this, of the minima or of the wave speed is bound by latency on all but the
// largest grids: it takes one launch and a wait, where it took memsets, a second
// launch and a device-to-host copy (8 steps on 211 x 149 cells with all of a log's
// reads each: 1065 -> 760 us).
__global__ void __launch_bounds__(TOTALS_BLOCKS) totals_kernel(Grid g, const float *__restrict__ hi,
                                                               const float *__restrict__ lo, double *partials,
                                                               unsigned *ticket, double *host) {
  __shared__ double sm[4][TOTALS_BLOCKS];
  __shared__ bool last;
  double acc[4] = {0, 0, 0, 0};
  for (int j = blockIdx.x; j < g.ny; j += gridDim.x)
    for (int i = threadIdx.x; i < g.nx; i += blockDim.x)
#pragma unroll
      for (int v = 0; v < NV; v++) acc[v] += (double)hi[at(g, v, i, j)] + (double)lo[at(g, v, i, j)];
  auto block_sum = [&] {
#pragma unroll
    for (int v = 0; v < NV; v++) sm[v][threadIdx.x] = acc[v];
    __syncthreads();
    for (int s = TOTALS_BLOCKS / 2; s > 0; s >>= 1) {
      if (threadIdx.x < s)
#pragma unroll
        for (int v = 0; v < NV; v++) sm[v][threadIdx.x] += sm[v][threadIdx.x + s];
      __syncthreads();
    }
  };
  block_sum();
  if (threadIdx.x < NV) {
    partials[blockIdx.x * NV + threadIdx.x] = sm[threadIdx.x][0];
    __threadfence();
  }
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(ticket, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
#pragma unroll
  for (int v = 0; v < NV; v++) acc[v] = __ldcg(partials + threadIdx.x * NV + v);
  block_sum();
  if (threadIdx.x < NV) {
    ((volatile double *)host)[threadIdx.x] = sm[threadIdx.x][0];
    __threadfence_system();
  }
  if (threadIdx.x == 0) *ticket = 0;
}

__global__ void export_counters_kernel(const unsigned long long *c, unsigned long long *host) {
  if (threadIdx.x < 4) ((volatile unsigned long long *)host)[threadIdx.x] = c[threadIdx.x];
  __threadfence_system();
}

__global__ void pack_kernel(Grid g, const float *__restrict__ src, float *dst, int ni, int nj,
                            int to_padded) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y * blockDim.y + threadIdx.y;
  if (i >= ni || j >= nj) return;
#pragma unroll
  for (int v = 0; v < NV; v++) {
    const long long e = ((long long)v * nj + j) * ni + i;
    if (to_padded)
      dst[at(g, v, i, j)] = src[e];
    else
      dst[e] = src[at(g, v, i, j)];
  }
}

// ---- whole states: 32 x 32 points of one of the four arrays a block (blocks
// [first[w], first[w + 1]) take array w), 4 rows and all variables a thread, so
// that 16 loads are in flight; one launch moves a state where packing array by
// array, clearing the low words, the ghost fill and the wave speed were nine.
constexpr int ST_W = 32, ST_H = 32, ST_ROWS = 4;
struct StateTiles {
  unsigned first[5];
  int tx[4];
};
__device__ __forceinline__ void state_tile(const StateTiles &T, int &w, int &i0, int &j0) {
  unsigned b = blockIdx.x;
  w = b < T.first[1] ? 0 : (b < T.first[2] ? 1 : (b < T.first[3] ? 2 : 3));
  b -= T.first[w];
  i0 = (int)(b % T.tx[w]) * ST_W;
  j0 = (int)(b / T.tx[w]) * ST_H;
}

struct LoadArgs {
  Grid g;
  StateTiles T;
  const float *ext[4];
  float *pad[4], *lo;
  int *status, *speed_bad;
  unsigned *speed, *host_speed, *ticket;
};
__global__ void __launch_bounds__(ST_W *ST_H / ST_ROWS) load_state_kernel(const __grid_constant__ LoadArgs A) {
  const Grid &g = A.g;
  int w, i0, j0;
  state_tile(A.T, w, i0, j0);
  const int arr = w == 0 ? 0 : w + 1;  // as in GhostRange (1: the low words)
  const GhostRange R(g, arr);
  const int ni = g.nx + R.nodex, nj = g.ny + R.nodey;
  const int i = i0 - OX + (int)threadIdx.x;  // (so that a warp's stores fill aligned lines)
  const bool ion = i >= -G && i < R.hix;
  float smax = 0.0f;
  bool bad = false;
  if (blockIdx.x == 0 && threadIdx.x == 0 && threadIdx.y == 0) *A.status = 0;
  float x[ST_ROWS][4];
#pragma unroll
  for (int r = 0; r < ST_ROWS; r++) {
    const int j = j0 - G + (int)threadIdx.y + r * (ST_H / ST_ROWS);
    bool fx = false, fy = false;
    // (threads beyond the padded extents read an interior point and store nothing)
    const int si = ion ? ghost_src(i, g.nx, R.ownx, R.nodex, g.per_x, g.bc[0], g.bc[1], fx) : 0;
    const int sj = j < R.hiy ? ghost_src(j, g.ny, R.owny, R.nodey, g.per_y, g.bc[2], g.bc[3], fy) : 0;
    const float *src = A.ext[w] + (long long)sj * ni + si;
#pragma unroll
    for (int v = 0; v < NV; v++) x[r][v] = __ldg(src + (long long)v * ni * nj);
    const int xside = i < 0 ? 0 : (i >= R.ownx ? 1 : -1), yside = j < 0 ? 2 : (j >= R.owny ? 3 : -1);
    const bool xin = !g.per_x && xside >= 0 && g.bc[xside] == BC_INFLOW;
    const bool yin = !g.per_y && yside >= 0 && g.bc[yside] == BC_INFLOW;
    if (xin || yin) {
      float U[4];
#pragma unroll
      for (int v = 0; v < NV; v++) U[v] = g.inflow[yin ? yside : xside][v];
      if (!yin && fy) U[2] = -U[2];
      if (arr == 0) p2c(U, 1.0f / (g.gamma - 1.0f), x[r]);
      else
#pragma unroll
        for (int v = 0; v < NV; v++) x[r][v] = U[v];
    } else {
      if (fx) x[r][1] = -x[r][1];
      if (fy) x[r][2] = -x[r][2];
    }
  }
#pragma unroll
  for (int r = 0; r < ST_ROWS; r++) {
    const int j = j0 - G + (int)threadIdx.y + r * (ST_H / ST_ROWS);
    if (!ion || j >= R.hiy) continue;
#pragma unroll
    for (int v = 0; v < NV; v++) {
      const long long e = at(g, v, i, j);
      A.pad[w][e] = x[r][v];
      if (arr == 0) A.lo[e] = 0.0f;
    }
    if (i >= 0 && j >= 0 && i < R.ownx && j < R.owny) {
      float U[4];
      if (arr == 0) c2p(x[r], g.gamma - 1.0f, U);
      smax = fmaxf(smax, wave_speed(arr == 0 ? U : x[r], g.gamma, bad));
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) smax = fmaxf(smax, __shfl_xor_sync(0xffffffffu, smax, o));
  __shared__ float wmax[ST_H / ST_ROWS];
  const int anybad = __syncthreads_or(bad);
  if (threadIdx.x == 0) wmax[threadIdx.y] = smax;
  __syncthreads();
  if (threadIdx.x == 0 && threadIdx.y == 0) {
    for (int k = 1; k < ST_H / ST_ROWS; k++) smax = fmaxf(smax, wmax[k]);
    atomicMax(A.speed, __float_as_uint(smax));
    if (anybad) atomicOr(A.speed_bad, 1);
    if (!A.host_speed) return;
    __threadfence();
    if (atomicAdd(A.ticket, 1u) == gridDim.x - 1) {
      __threadfence();
      volatile unsigned *h = A.host_speed;
      h[0] = atomicMax(A.speed, 0u);
      h[1] = (unsigned)atomicOr(A.speed_bad, 0);
      *A.ticket = 0;
      __threadfence_system();
    }
  }
}

struct StoreArgs {
  Grid g;
  StateTiles T;
  const float *pad[4];
  float *ext[4];
};
__global__ void __launch_bounds__(ST_W *ST_H / ST_ROWS) store_state_kernel(const __grid_constant__ StoreArgs A) {
  const Grid &g = A.g;
  int w, i0, j0;
  state_tile(A.T, w, i0, j0);
  const int ni = g.nx + (w == 1 || w == 2), nj = g.ny + (w == 1 || w == 3);
  const int i = i0 + (int)threadIdx.x;
  if (i >= ni) return;
  float x[ST_ROWS][4];
#pragma unroll
  for (int r = 0; r < ST_ROWS; r++) {
    const int j = min(j0 + (int)threadIdx.y + r * (ST_H / ST_ROWS), nj - 1);
#pragma unroll
    for (int v = 0; v < NV; v++) x[r][v] = __ldg(A.pad[w] + at(g, v, i, j));
  }
#pragma unroll
  for (int r = 0; r < ST_ROWS; r++) {
    const int j = j0 + (int)threadIdx.y + r * (ST_H / ST_ROWS);
    if (j >= nj) continue;
#pragma unroll
    for (int v = 0; v < NV; v++) A.ext[w][((long long)v * nj + j) * ni + i] = x[r][v];
  }
}

// Reductions over a whole state (averages in primitive form and owned point
// values), tile by tile as above: MIN: the minimum density and pressure (as
// ordered keys); else the maximum wave speed.  part[block] = (value, value or 0,
// bad); the last block reduces the blocks' and writes the result to mapped host
// memory and, for the speed, to the device words.
struct ReduceArgs {
  Grid g;
  StateTiles T;
  const float *pad[4];
  unsigned *part, *ticket, *host;
  unsigned *speed;
  int *speed_bad;
};
constexpr int RED_THREADS = ST_W * ST_H / ST_ROWS;
template <bool MIN>
__global__ void __launch_bounds__(RED_THREADS) reduce_state_kernel(const __grid_constant__ ReduceArgs A) {
  const Grid &g = A.g;
  unsigned k0 = MIN ? ~0u : 0u, k1 = k0;  // keys of rho and p, or the speed's bits
  float m = 0.0f;
  bool bad = false;
  for (unsigned t = blockIdx.x; t < A.T.first[4]; t += gridDim.x) {
    unsigned b = t;
    const int w = b < A.T.first[1] ? 0 : (b < A.T.first[2] ? 1 : (b < A.T.first[3] ? 2 : 3));
    b -= A.T.first[w];
    const int ni = w == 1 || w == 2 ? g.nxv : g.nx, nj = w == 1 || w == 3 ? g.nyv : g.ny;
    const int i = (int)(b % A.T.tx[w]) * ST_W + (int)threadIdx.x, j0 = (int)(b / A.T.tx[w]) * ST_H + (int)threadIdx.y;
    if (i >= ni) continue;
    float x[ST_ROWS][4];
#pragma unroll
    for (int r = 0; r < ST_ROWS; r++) {
      const int j = min(j0 + r * (ST_H / ST_ROWS), nj - 1);  // (a row beyond the last repeats it)
#pragma unroll
      for (int v = 0; v < NV; v++) x[r][v] = __ldg(A.pad[w] + at(g, v, i, j));
    }
#pragma unroll
    for (int r = 0; r < ST_ROWS; r++) {
      float U[4] = {x[r][0], x[r][1], x[r][2], x[r][3]};
      if (w == 0) c2p(x[r], g.gamma - 1.0f, U);
      if (MIN) {
        bad |= !(isfinite(U[0]) && isfinite(U[1]) && isfinite(U[2]) && isfinite(U[3]));
        k0 = min(k0, float_key(U[0]));
        k1 = min(k1, float_key(U[3]));
      } else {
        m = fmaxf(m, wave_speed(U, g.gamma, bad));
      }
    }
  }
  if (!MIN) k0 = __float_as_uint(m);
  __shared__ unsigned s0[RED_THREADS / 32], s1[RED_THREADS / 32];
  __shared__ bool last;
  const int tid = threadIdx.y * ST_W + threadIdx.x;
  auto block_reduce = [&](unsigned &a, unsigned &b, bool f) {
    a = MIN ? __reduce_min_sync(0xffffffffu, a) : __reduce_max_sync(0xffffffffu, a);
    b = MIN ? __reduce_min_sync(0xffffffffu, b) : 0u;
    if ((tid & 31) == 0) {
      s0[tid >> 5] = a;
      s1[tid >> 5] = b;
    }
    const bool any = __syncthreads_or(f) != 0;
    for (int w = 0; w < RED_THREADS / 32; w++) {
      a = MIN ? min(a, s0[w]) : max(a, s0[w]);
      b = MIN ? min(b, s1[w]) : 0u;
    }
    return any;
  };
  const bool any = block_reduce(k0, k1, bad);
  if (tid == 0) {
    A.part[3 * blockIdx.x] = k0;
    A.part[3 * blockIdx.x + 1] = k1;
    A.part[3 * blockIdx.x + 2] = any;
    __threadfence();
    last = atomicAdd(A.ticket, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  bool f = false;
  k0 = k1 = MIN ? ~0u : 0u;
  for (unsigned q = tid; q < gridDim.x; q += RED_THREADS) {
    const unsigned a = __ldcg(A.part + 3 * q), b = __ldcg(A.part + 3 * q + 1);
    k0 = MIN ? min(k0, a) : max(k0, a);
    k1 = MIN ? min(k1, b) : 0u;
    f |= __ldcg(A.part + 3 * q + 2) != 0u;
  }
  const bool flag = block_reduce(k0, k1, f);
  if (tid == 0) {
    volatile unsigned *h = A.host;
    h[0] = k0;
    h[1] = MIN ? k1 : (unsigned)flag;
    if (MIN) h[2] = flag;
    if (!MIN) {
      *A.speed = k0;
      *A.speed_bad = flag;
    }
    *A.ticket = 0;
    __threadfence_system();
  }
}

// periodic duplicate lines of the three node arrays (blockIdx.z; y: variable)
struct CheckArgs {
  Grid g;
  const float *ext[4];
  unsigned *bad, *speed;
  int *speed_bad;
};
__global__ void check_state_kernel(const __grid_constant__ CheckArgs A) {
  const Grid &g = A.g;
  const int k = blockIdx.x * blockDim.x + threadIdx.x, v = blockIdx.y, w = 1 + blockIdx.z;
  if (k == 0 && v == 0 && w == 1) {
    *A.speed = 0u;
    *A.speed_bad = 0;
  }
  const int nodex = w == 1 || w == 2, nodey = w == 1 || w == 3, ni = g.nx + nodex, nj = g.ny + nodey;
  const float *p = A.ext[w] + (long long)v * ni * nj;
  bool bad = false;
  if (g.per_x && nodex && k < nj) bad |= !(p[(long long)k * ni + ni - 1] == p[(long long)k * ni]);
  if (g.per_y && nodey && k < ni) bad |= !(p[(long long)(nj - 1) * ni + k] == p[k]);
  if (bad) {
    *(volatile unsigned *)A.bad = 1u;
    __threadfence_system();
  }
}

__global__ void check_dup_kernel(const float *__restrict__ a, int ni, int nj, int dup_x, int dup_y,
                                 int *bad) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  const int v = blockIdx.y;
  const float *p = a + (long long)v * ni * nj;
  if (dup_x && k < nj && !(p[(long long)k * ni + ni - 1] == p[(long long)k * ni])) atomicOr(bad, 1);
  if (dup_y && k < ni && !(p[(long long)(nj - 1) * ni + k] == p[k])) atomicOr(bad, 1);
}

}  // namespace

cudaError_t launch_ghost_fill64(const Grid &g, double *avg, double *const n[3], cudaStream_t s) {
  const long long per = 2LL * (g.nx + g.ny + 2 * G + 2) * (2 * G + 1);
  int blocks = (int)((per + 255) / 256);
  if (blocks < 1) blocks = 1;
  ghost64_kernel<<<dim3(blocks, 5), 256, 0, s>>>(g, avg, n[VTX], n[XE], n[YE]);
  return cudaGetLastError();
}

cudaError_t launch_ghost_fill(const Grid &g, float *avg_hi, float *avg_lo, const NodeSet &n,
                              cudaStream_t s) {
  GhostArgs A;
  A.g = g;
  A.a[0] = avg_hi;
  A.a[1] = avg_lo;
  A.a[2] = n.k[VTX];
  A.a[3] = n.k[XE];
  A.a[4] = n.k[YE];
  const long long per = 2LL * (g.nx + g.ny + 2 * G + 2) * (2 * G + 1);
  int blocks = (int)((per + 255) / 256);
  if (blocks < 1) blocks = 1;
  ghost_kernel<<<dim3(blocks, 5), 256, 0, s>>>(A);
  return cudaGetLastError();
}

long long ghost_total(const Grid &g, int arr) { return GhostRange(g, arr).total; }

cudaError_t launch_ghost_batch(const GhostBatch &B, int nchunks, cudaStream_t s) {
  if (nchunks <= 0) return cudaSuccess;
  ghost_batch_kernel<<<nchunks, GHOST_CHUNK, 0, s>>>(B);
  return cudaGetLastError();
}

cudaError_t launch_shock_theta(const Grid &g, const float *avg_hi, const NodeSet &n0, float *tx, float *ty,
                               cudaStream_t s) {
  dim3 blk(TH_W, TH_H), grd((g.nx + 2 + TH_W - 1) / TH_W, (g.ny + 2 + TH_H - 1) / TH_H);
  const TnArrays t = {avg_hi, n0.k[VTX], n0.k[XE], n0.k[YE]};
  shock_theta_kernel<<<grd, blk, 0, s>>>(g, t, tx, ty);
  return cudaGetLastError();
}

cudaError_t launch_shock_theta_batch(const int4 *tiles, int ntiles, const BatchCtl *ctl, const Grid *grids,
                                     const float *const *arrays, float *const *theta, cudaStream_t s) {
  if (ntiles <= 0) return cudaSuccess;
  shock_theta_batch_kernel<<<ntiles, dim3(32, 8), 0, s>>>(tiles, ctl, grids, arrays, theta);
  return cudaGetLastError();
}

cudaError_t launch_batch_dt(BatchCtl *ctl, int n, double *hist, int hist_cap, int mode, PointValueArgs *pv_args,
                            cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  batch_dt_kernel<<<(n + 127) / 128, 128, 0, s>>>(ctl, n, hist, hist_cap, mode, pv_args);
  return cudaGetLastError();
}

cudaError_t launch_export_words(unsigned *a, unsigned *b, int clear_a, unsigned *dst, cudaStream_t s) {
  export_words_kernel<<<1, 32, 0, s>>>(a, b, clear_a, dst);
  return cudaGetLastError();
}

// tiles of the four arrays of extents ni x nj (0: left out)
static StateTiles state_tiles(const int ni[4], const int nj[4]) {
  StateTiles T;
  T.first[0] = 0;
  for (int w = 0; w < 4; w++) {
    T.tx[w] = ni[w] > 0 ? (ni[w] + ST_W - 1) / ST_W : 1;
    T.first[w + 1] = T.first[w] + (ni[w] > 0 ? (unsigned)T.tx[w] * ((nj[w] + ST_H - 1) / ST_H) : 0u);
  }
  return T;
}

static ReduceArgs reduce_args(const Grid &g, const float *avg_hi, const NodeSet &n, double *scratch, unsigned *host,
                              unsigned *ticket) {
  ReduceArgs A;
  A.g = g;
  const int ni[4] = {g.nx, g.nxv, g.nxv, g.nx}, nj[4] = {g.ny, g.nyv, g.ny, g.nyv};
  A.T = state_tiles(ni, nj);
  A.pad[0] = avg_hi;
  for (int k = 0; k < 3; k++) A.pad[1 + k] = n.k[k];
  A.part = reinterpret_cast<unsigned *>(scratch);
  A.ticket = ticket;
  A.host = host;
  A.speed = nullptr;
  A.speed_bad = nullptr;
  return A;
}
// (as many blocks as the scratch has room for three words of each)
constexpr unsigned RED_BLOCKS = TOTALS_BLOCKS * NV * 2 / 3;
cudaError_t launch_max_speed(const Grid &g, const float *avg_hi, const NodeSet &n, double *scratch, unsigned *out_bits,
                             int *bad, unsigned *host, unsigned *ticket, cudaStream_t s) {
  ReduceArgs A = reduce_args(g, avg_hi, n, scratch, host, ticket);
  A.speed = out_bits;
  A.speed_bad = bad;
  const unsigned blocks = A.T.first[4] < RED_BLOCKS ? A.T.first[4] : RED_BLOCKS;
  reduce_state_kernel<false><<<blocks, dim3(ST_W, ST_H / ST_ROWS), 0, s>>>(A);
  return cudaGetLastError();
}
cudaError_t launch_state_min(const Grid &g, const float *avg_hi, const NodeSet &n, double *scratch, unsigned *host,
                             unsigned *ticket, cudaStream_t s) {
  const ReduceArgs A = reduce_args(g, avg_hi, n, scratch, host, ticket);
  const unsigned blocks = A.T.first[4] < RED_BLOCKS ? A.T.first[4] : RED_BLOCKS;
  reduce_state_kernel<true><<<blocks, dim3(ST_W, ST_H / ST_ROWS), 0, s>>>(A);
  return cudaGetLastError();
}
cudaError_t launch_totals(const Grid &g, const float *avg_hi, const float *avg_lo, double *partials, double *host,
                          unsigned *ticket, cudaStream_t s) {
  totals_kernel<<<TOTALS_BLOCKS, TOTALS_BLOCKS, 0, s>>>(g, avg_hi, avg_lo, partials, ticket, host);
  return cudaGetLastError();
}
cudaError_t launch_export_counters(const unsigned long long *c, unsigned long long *host, cudaStream_t s) {
  export_counters_kernel<<<1, 32, 0, s>>>(c, host);
  return cudaGetLastError();
}

cudaError_t launch_check_state(const Grid &g, const float *const ext[4], unsigned *bad, unsigned *speed, int *speed_bad,
                               cudaStream_t s) {
  CheckArgs A;
  A.g = g;
  for (int w = 0; w < 4; w++) A.ext[w] = ext[w];
  A.bad = bad;
  A.speed = speed;
  A.speed_bad = speed_bad;
  const int n = (g.nx > g.ny ? g.nx : g.ny) + 1;
  check_state_kernel<<<dim3((n + 255) / 256, NV, 3), 256, 0, s>>>(A);
  return cudaGetLastError();
}

cudaError_t launch_load_state(const Grid &g, const StateArrays &a, float *avg_lo, int *status, unsigned *speed,
                              int *speed_bad, unsigned *host_speed, unsigned *ticket, cudaStream_t s) {
  LoadArgs A;
  A.g = g;
  int ni[4], nj[4];
  for (int w = 0; w < 4; w++) {
    const GhostRange R(g, w == 0 ? 0 : w + 1);
    ni[w] = a.ext[w] ? R.hix + OX : 0;
    nj[w] = R.hiy + G;
    A.ext[w] = a.ext[w];
    A.pad[w] = a.pad[w];
  }
  A.T = state_tiles(ni, nj);
  A.lo = avg_lo;
  A.status = status;
  A.speed = speed;
  A.speed_bad = speed_bad;
  A.host_speed = host_speed;
  A.ticket = ticket;
  load_state_kernel<<<A.T.first[4], dim3(ST_W, ST_H / ST_ROWS), 0, s>>>(A);
  return cudaGetLastError();
}

cudaError_t launch_store_state(const Grid &g, const float *const pad[4], float *const ext[4], cudaStream_t s) {
  StoreArgs A;
  A.g = g;
  int ni[4], nj[4];
  for (int w = 0; w < 4; w++) {
    const bool on = ext[w] && pad[w];
    ni[w] = on ? g.nx + (w == 1 || w == 2) : 0;
    nj[w] = on ? g.ny + (w == 1 || w == 3) : 0;
    A.pad[w] = pad[w];
    A.ext[w] = ext[w];
  }
  A.T = state_tiles(ni, nj);
  if (A.T.first[4] == 0) return cudaSuccess;
  store_state_kernel<<<A.T.first[4], dim3(ST_W, ST_H / ST_ROWS), 0, s>>>(A);
  return cudaGetLastError();
}

cudaError_t launch_pack(const Grid &g, const float *src, float *dst, int ni, int nj, bool to_padded,
                        cudaStream_t s) {
  dim3 blk(32, 8), grd((ni + 31) / 32, (nj + 7) / 8);
  pack_kernel<<<grd, blk, 0, s>>>(g, src, dst, ni, nj, to_padded ? 1 : 0);
  return cudaGetLastError();
}

cudaError_t launch_check_dup(const float *ext, int ni, int nj, int dup_x, int dup_y, int *bad,
                             cudaStream_t s) {
  int n = ni > nj ? ni : nj;
  check_dup_kernel<<<dim3((n + 255) / 256, NV), 256, 0, s>>>(ext, ni, nj, dup_x, dup_y, bad);
  return cudaGetLastError();
}

AF_BOUNDS_READER(bounds_misc)

}  // namespace af
