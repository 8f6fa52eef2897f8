// af_ghost.cuh -- ghost entries of the padded arrays (Sec. 4.3): their source
// along each axis, their enumeration and their values, and the images of an
// interior cell among them.
#pragma once
#include <type_traits>

#include "af_common.cuh"

namespace af {

// Source index of a ghost entry along one axis.  Periodic: wrap.  Outflow:
// mirror copy of the interior.  Solid wall: the same mirror, with the normal
// velocity negated (flip).  node: the array sits on grid lines along the axis.
__device__ __forceinline__ int ghost_src(int i, int n, int own, int node, int per, int blo,
                                         int bhi, bool &flip) {
  if (i >= 0 && i < own) return i;
  if (per) {
    int r = i % n;
    return r < 0 ? r + n : r;
  }
  if (i < 0) {
    flip = (blo == BC_REFLECTING);
    return node ? -i : -1 - i;
  }
  flip = (bhi == BC_REFLECTING);
  return node ? 2 * n - i : 2 * n - 1 - i;
}

// entries of array arr (0..4) in ghost order; total is their number
struct GhostRange {
  int nodex, nodey, ownx, owny, hix, hiy, wext, nb, nt, nl, wr, total;
  __host__ __device__ GhostRange(const Grid &g, int arr) {
    nodex = (arr == 2 || arr == 3);
    nodey = (arr == 2 || arr == 4);
    ownx = nodex ? g.nxv : g.nx;
    owny = nodey ? g.nyv : g.ny;
    hix = nodex ? g.nx + G + 1 : g.nx + G;
    hiy = nodey ? g.ny + G + 1 : g.ny + G;
    wext = hix + G;
    nb = G * wext;
    nt = (hiy - owny) * wext;
    nl = owny * G;
    wr = hix - ownx;
    total = nb + nt + nl + owny * wr;
  }
};

// ghost entry k of array arr (0 averages hi, 1 averages lo, 2..4 node
// arrays): copy from its source, flipping the normal velocity at walls; on
// an inflow side the side's state (conservative for the averages, zero low
// word).  A corner entry takes the y side's rule applied to the x side's
// value, as two passes (x, then y) would give.  SKIP_DUP leaves out the
// duplicated last node line of a periodic axis (the point-value kernel stores
// it with the first line, and others may be reading it).
template <typename T, bool SKIP_DUP = false>
__device__ __forceinline__ void ghost_entry(const Grid &g, const GhostRange &R, T *p, int arr, int k) {
  int i, j, r = k;
  if (r < R.nb) {
    j = -G + r / R.wext;
    i = -G + r % R.wext;
  } else if ((r -= R.nb) < R.nt) {
    j = R.owny + r / R.wext;
    i = -G + r % R.wext;
  } else if ((r -= R.nt) < R.nl) {
    j = r / G;
    i = -G + r % G;
  } else {
    r -= R.nl;
    j = r / R.wr;
    i = R.ownx + r % R.wr;
  }
  if (SKIP_DUP && i >= 0 && j >= 0 && i < g.nx + R.nodex && j < g.ny + R.nodey) return;
  bool fx = false, fy = false;
  const int si = ghost_src(i, g.nx, R.ownx, R.nodex, g.per_x, g.bc[0], g.bc[1], fx);
  const int sj = ghost_src(j, g.ny, R.owny, R.nodey, g.per_y, g.bc[2], g.bc[3], fy);
  const int xside = i < 0 ? 0 : (i >= R.ownx ? 1 : -1), yside = j < 0 ? 2 : (j >= R.owny ? 3 : -1);
  const bool xin = !g.per_x && xside >= 0 && g.bc[xside] == BC_INFLOW;
  const bool yin = !g.per_y && yside >= 0 && g.bc[yside] == BC_INFLOW;
  if constexpr (std::is_same<T, float>::value) {  // (the FP64 path has no inflow sides)
  if (xin || yin) {
    float U[4];
#pragma unroll
    for (int v = 0; v < NV; v++) U[v] = g.inflow[yin ? yside : xside][v];
    if (!yin && fy) U[2] = -U[2];
    float Q[4];
    if (arr == 0) p2c(U, 1.0f / (g.gamma - 1.0f), Q);
#pragma unroll
    for (int v = 0; v < NV; v++) p[at(g, v, i, j)] = arr == 0 ? Q[v] : (arr == 1 ? 0.0f : U[v]);
    return;
  }
  }
#pragma unroll
  for (int v = 0; v < NV; v++) {
    T x = p[at(g, v, si, sj)];
    if ((v == 1 && fx) || (v == 2 && fy)) x = -x;
    p[at(g, v, i, j)] = x;
  }
}

// The ghost images of interior cell (i, j) of the averages: calls
// put(i', j', flip the x momentum, flip the y momentum) for every ghost entry
// whose source it is.  Entries of an inflow side hold its constant state and
// have no source.  (G ghost layers, so only cells within G of a side have any.)
template <typename Put>
__device__ __forceinline__ void cell_images(const Grid &g, int i, int j, Put put) {
  static_assert(G == 2, "at most two images an axis");
  // positions 0: the cell itself, then its images along the axis (count n)
  auto axis = [](int i, int n, int per, int blo, int bhi, int pos[3], bool flip[3]) {
    int c = 1;
    pos[0] = i;
    flip[0] = false;
    if (i < G && (per || blo != BC_INFLOW)) {
      pos[c] = per ? i + n : -1 - i;
      flip[c++] = !per && blo == BC_REFLECTING;
    }
    if (i >= n - G && (per || bhi != BC_INFLOW)) {
      pos[c] = per ? i - n : 2 * n - 1 - i;
      flip[c++] = !per && bhi == BC_REFLECTING;
    }
    return c;
  };
  int px[3], py[3];
  bool fx[3], fy[3];
  const int nx = axis(i, g.nx, g.per_x, g.bc[0], g.bc[1], px, fx), ny = axis(j, g.ny, g.per_y, g.bc[2], g.bc[3], py, fy);
#pragma unroll
  for (int b = 0; b < 3; b++)
#pragma unroll
    for (int a = 0; a < 3; a++)
      if (a < nx && b < ny && a + b > 0) put(px[a], py[b], fx[a], fy[b]);
}

}  // namespace af
