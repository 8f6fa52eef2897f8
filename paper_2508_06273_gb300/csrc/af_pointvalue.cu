// af_pointvalue.cu -- point values: the plain instantiations (the code is in
// af_pointvalue.cuh), the TMA descriptors and the launchers.
#include "af_pointvalue.cuh"

namespace af {

cudaError_t make_tile_maps(const Grid &g, float *vtx, float *xe, float *ye, float *avg, int tile_h,
                           TileMaps *out) {
  static PFN_cuTensorMapEncodeTiled_v12000 encode = nullptr;
  if (!encode) {
    void *fn = nullptr;
    cudaDriverEntryPointQueryResult q;
    cudaError_t e = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q);
    if (e != cudaSuccess) return e;
    if (q != cudaDriverEntryPointSuccess || !fn) return cudaErrorSymbolNotFound;
    encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
  }
  if (tile_h == TILE_SPLIT) tile_h = 4;
  if (tile_h != 4 && tile_h != 8 && tile_h != 16) return cudaErrorInvalidValue;
  // planes of P x H floats, 4 variables: 3-D tensors (x, row, variable)
  const cuuint64_t dims[3] = {(cuuint64_t)g.P, (cuuint64_t)g.H, (cuuint64_t)NV};
  const cuuint64_t strides[2] = {(cuuint64_t)g.P * 4u, (cuuint64_t)g.plane * 4u};
  const cuuint32_t box[3] = {(cuuint32_t)RAW_W, (cuuint32_t)(tile_h + 3), (cuuint32_t)NV};
  const cuuint32_t estr[3] = {1, 1, 1};
  float *base[4] = {vtx, xe, ye, avg};
  CUtensorMap *dst[4] = {&out->vtx, &out->xe, &out->ye, &out->avg};
  for (int k = 0; k < 4; k++) {
    if ((reinterpret_cast<size_t>(base[k]) & 15) != 0 || (strides[0] & 15) != 0 || (strides[1] & 15) != 0 ||
        (RAW_W * 4) % 16 != 0)
      return cudaErrorInvalidValue;
    CUresult r = encode(dst[k], CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, base[k], dims, strides, box, estr,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                        CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return cudaErrorInvalidValue;
  }
  return cudaSuccess;
}

cudaError_t prepare_pointvalue() {
  cudaError_t e = cudaSuccess;
  auto attr = [&](const void *f, int bytes) {
    if (e == cudaSuccess) e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  };
  auto height = [&](auto ty) {
    constexpr int TY = decltype(ty)::value;
    attr((const void *)pointvalue_kernel<TY, PV_LEAN>, Tile<TY>::SMEM_BYTES);
    attr((const void *)pointvalue_kernel<TY, PV_FULL>, Tile<TY>::SMEM_BYTES);
    attr((const void *)pointvalue_kernel<TY, PV_NF>, Tile<TY>::SMEM_NF_BYTES);
    attr((const void *)pointvalue_batch_kernel<TY, PV_LEAN>, Tile<TY>::SMEM_BYTES);
    attr((const void *)pointvalue_batch_kernel<TY, PV_FULL>, Tile<TY>::SMEM_BYTES);
  };
  height(std::integral_constant<int, 4>());
  height(std::integral_constant<int, 8>());
  height(std::integral_constant<int, 16>());
  if (e == cudaSuccess) e = prepare_pointvalue_shock();
  return e;
}

// tiles cover the owned nodes: up to nxv x nyv (vertex lines n + 1 on a
// non-periodic axis); every box x coordinate is a multiple of TX floats; the
// node-flux instantiation (with its scratch) only when node fluxes are
// written, the lean one whenever no option it leaves out is set
// (split: one node kind a block, three blocks a tile)
template <int TY>
static cudaError_t launch_h(const Args &A, const TileMaps &maps, bool split, cudaStream_t s) {
  const Grid &g = A.g;
  const dim3 grd((g.nxv + TX - 1) / TX, (g.nyv + TY - 1) / TY, split ? 3 : 1), blk(TX, TY);
  switch (pv_class(A)) {
    case PV_NF: return launch_pdl(pointvalue_kernel<TY, PV_NF>, dim3(grd.x, grd.y), blk, Tile<TY>::SMEM_NF_BYTES, s, A, maps);
    case PV_LEAN: return launch_pdl(pointvalue_kernel<TY, PV_LEAN>, grd, blk, Tile<TY>::SMEM_BYTES, s, A, maps);
    case PV_FULL: return launch_pdl(pointvalue_kernel<TY, PV_FULL>, grd, blk, Tile<TY>::SMEM_BYTES, s, A, maps);
    default: return launch_pointvalue_shock(A, maps, TY, s);
  }
}
static cudaError_t launch_single(const Args &A, const TileMaps &maps, int tile_h, cudaStream_t s) {
  switch (tile_h) {
    case TILE_SPLIT: return launch_h<4>(A, maps, true, s);
    case 4: return launch_h<4>(A, maps, false, s);
    case 16: return launch_h<16>(A, maps, false, s);
    default: return launch_h<8>(A, maps, false, s);
  }
}

cudaError_t launch_pointvalue(const Grid &g, const NodeSet &n0, const float *avg_hi, const TileMaps &maps,
                              const NodeSet &n1, const NodeSet &n2, float dt, const Options &o,
                              int *status, unsigned long long *counters, const float *const theta[2],
                              int tile_h, const NodeFluxOut *nf, unsigned *clear_speed, int *clear_bad,
                              cudaStream_t s) {
  Args A = pointvalue_args(g, n0, avg_hi, n1, n2, o, status, counters);
  A.dt = dt;
  A.theta[0] = theta[0];
  A.theta[1] = theta[1];
  A.clear_speed = clear_speed;
  A.clear_bad = clear_bad;
  if (nf) {
    for (int q = 0; q < 4; q++) A.nflux[q] = nf->q[q];
    A.speed = nf->speed;
    A.speed_bad = nf->speed_bad;
    A.write_half = nf->write_half;
  }
  return launch_single(A, maps, tile_h, s);
}

cudaError_t launch_pointvalue_masked(const Grid &g, const NodeSet &n0, const float *avg_hi, const TileMaps &maps,
                                     const NodeSet &n1, const NodeSet &n2, float dt, const Options &o, int *status,
                                     unsigned long long *counters, const unsigned char *const mask[3],
                                     const int *tile_flag, const float *const theta[2], int tile_h,
                                     unsigned *clear_speed, int *clear_bad, cudaStream_t s) {
  Args A = pointvalue_args(g, n0, avg_hi, n1, n2, o, status, counters);
  A.dt = dt;
  A.theta[0] = theta[0];
  A.theta[1] = theta[1];
  A.clear_speed = clear_speed;
  A.clear_bad = clear_bad;
  for (int k = 0; k < 3; k++) A.mask[k] = mask[k];
  A.tile_flag = tile_flag;
  return launch_single(A, maps, tile_h, s);
}

int batch_class(const PointValueArgs &A) { return pv_class(A); }

template <int TY>
static void launch_batch_h(const PointValueBatch &B, int c, int ntiles, cudaStream_t s) {
  const dim3 blk(TX, TY);
  if (c == PV_LEAN) pointvalue_batch_kernel<TY, PV_LEAN><<<ntiles, blk, Tile<TY>::SMEM_BYTES, s>>>(B);
  else if (c == PV_FULL) pointvalue_batch_kernel<TY, PV_FULL><<<ntiles, blk, Tile<TY>::SMEM_BYTES, s>>>(B);
  else launch_pointvalue_shock_batch(B, ntiles, TY, s);
}
cudaError_t launch_pointvalue_batch(const PointValueBatch &B, const int ntiles[PV_CLASSES],
                                    const int tile_h[PV_CLASSES], cudaStream_t s) {
  static_assert(PV_LEAN == 0 && PV_FULL == 1 && PV_SHOCK == 2 && PV_CLASSES == 3, "order of the tile list");
  PointValueBatch L = B;
  for (int c = 0; c < PV_CLASSES; L.tiles += ntiles[c++]) {
    if (ntiles[c] == 0) continue;
    switch (tile_h[c]) {
      case 4: launch_batch_h<4>(L, c, ntiles[c], s); break;
      case 8: launch_batch_h<8>(L, c, ntiles[c], s); break;
      case 16: launch_batch_h<16>(L, c, ntiles[c], s); break;
      default: return cudaErrorInvalidValue;
    }
  }
  return cudaGetLastError();
}

AF_BOUNDS_READER(bounds_pointvalue)

}  // namespace af
