// af_pointvalue_shock.cu -- point values: the instantiations with the switches for
// discontinuous data (PV_SHOCK, PV_NF_SHOCK of af_pointvalue.cuh).
#define AF_PV_SHOCK
#include "af_pointvalue.cuh"

namespace af {

cudaError_t prepare_pointvalue_shock() {
  cudaError_t e = cudaSuccess;
  auto attr = [&](const void *f, int bytes) {
    if (e == cudaSuccess) e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  };
  auto height = [&](auto ty) {
    constexpr int TY = decltype(ty)::value;
    attr((const void *)pointvalue_kernel<TY, PV_SHOCK>, Tile<TY>::SMEM_BYTES);
    attr((const void *)pointvalue_kernel<TY, PV_NF_SHOCK>, Tile<TY>::SMEM_NF_BYTES);
    attr((const void *)pointvalue_batch_kernel<TY, PV_SHOCK>, Tile<TY>::SMEM_BYTES);
  };
  height(std::integral_constant<int, 4>());
  height(std::integral_constant<int, 8>());
  height(std::integral_constant<int, 16>());
  return e;
}

template <int TY>
static cudaError_t launch_h(const PointValueArgs &A, const TileMaps &maps, cudaStream_t s) {
  const Grid &g = A.g;
  const dim3 grd((g.nxv + TX - 1) / TX, (g.nyv + TY - 1) / TY), blk(TX, TY);
  if (A.nflux[0]) return launch_pdl(pointvalue_kernel<TY, PV_NF_SHOCK>, grd, blk, Tile<TY>::SMEM_NF_BYTES, s, A, maps);
  return launch_pdl(pointvalue_kernel<TY, PV_SHOCK>, grd, blk, Tile<TY>::SMEM_BYTES, s, A, maps);
}
cudaError_t launch_pointvalue_shock(const PointValueArgs &A, const TileMaps &maps, int tile_h, cudaStream_t s) {
  return tile_h == 4 ? launch_h<4>(A, maps, s) : (tile_h == 16 ? launch_h<16>(A, maps, s) : launch_h<8>(A, maps, s));
}

template <int TY>
static void launch_batch_h(const PointValueBatch &B, int ntiles, cudaStream_t s) {
  pointvalue_batch_kernel<TY, PV_SHOCK><<<ntiles, dim3(TX, TY), Tile<TY>::SMEM_BYTES, s>>>(B);
}
void launch_pointvalue_shock_batch(const PointValueBatch &B, int ntiles, int tile_h, cudaStream_t s) {
  if (tile_h == 4) launch_batch_h<4>(B, ntiles, s);
  else if (tile_h == 16) launch_batch_h<16>(B, ntiles, s);
  else launch_batch_h<8>(B, ntiles, s);
}

AF_BOUNDS_READER(bounds_pointvalue_shock)

}  // namespace af
