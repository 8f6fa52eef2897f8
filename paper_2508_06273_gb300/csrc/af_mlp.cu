// af_mlp.cu -- the surrogate network's parameters and its training on the
// GPU: forward and backward on the tcgen05 tensor cores (FP32 accumulation),
// MSE loss, and Adam (Kingma & Ba 2015) on FP32 master weights.
//
// One training step on a minibatch of B rows (B a multiple of 8):
//   Z1 = X W1^T + b1, H1 = gelu(Z1), ..., Y = H3 W4^T + b4     (forward)
//   dY = 2 (Y - T) / (8 B) on the 8 used outputs                (MSE loss)
//   dH3 = dY W4, dZ3 = dH3 gelu'(Z3), dH2 = dZ3 W3, ...         (backward)
//   dW4 = dY^T H3, dW3 = dZ3^T H2, ..., dW1 = dZ1^T X           (weights)
// in three launches: network_kernel takes 128 rows a CTA from the gather to
// dZ1 with Z1, Z2, Z3 and dH in the 512 columns of tensor memory and every
// weight (and transpose) in shared memory; weight_grad_kernel contracts the
// transposes it left over the batch; adam_kernel adds the partial products and
// updates the weights and their BF16 copies.  All sums have a fixed order.
// Measured at B = 4096 in calls of 24 steps: 420 -> 47 us a step (26 launches
// before, 11 of them products of 38 us whose row-per-thread epilogues wrote 4 bytes
// a sector); in calls of 200 steps 42.5.
#include <cmath>
#include <cstdio>
#include <cstring>
#include <new>
#include <vector>

#include "../../include/af.h"
#include "af_common.cuh"
#include "af_kernels.h"
#include "af_mlp.h"
#include "af_tc.cuh"

using namespace af;
using namespace af::mlp;

namespace {

__host__ __device__ __forceinline__ uint64_t mix64(uint64_t x) {  // splitmix64 finaliser
  x += 0x9E3779B97F4A7C15ull;
  x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
  x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
  return x ^ (x >> 31);
}
__device__ __forceinline__ float uniform01(uint64_t h) {  // (0, 1]
  return ((float)(h >> 40) + 1.0f) * (1.0f / 16777216.0f);
}

// He-normal weights (Box-Muller on counter-based uniforms), zero biases,
// the last layer scaled by 0.1 and its unused rows zero; unit scales
__global__ void init_kernel(float *p, uint64_t seed) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= NPARAM) return;
  float fan = 0.0f, mul = 1.0f;
  bool zero = false;
  if (k < OFF_B1) fan = NIN;
  else if (k < OFF_W2) zero = true;
  else if (k < OFF_B2) fan = NH;
  else if (k < OFF_W3) zero = true;
  else if (k < OFF_B3) fan = NH;
  else if (k < OFF_W4) zero = true;
  else if (k < OFF_B4) {
    fan = NH;
    mul = 0.1f;
    zero = (k - OFF_W4) / NH >= NOUT;
  } else if (k < NTRAIN) zero = true;
  if (k >= NTRAIN) {
    p[k] = 1.0f;
    return;
  }
  if (zero) {
    p[k] = 0.0f;
    return;
  }
  const float u1 = uniform01(mix64(seed ^ (2ull * k))), u2 = uniform01(mix64(seed ^ (2ull * k + 1)));
  const float g = sqrtf(-2.0f * logf(u1)) * cosf(6.283185307f * u2);
  p[k] = g * sqrtf(2.0f / fan) * mul;
}

// BF16 copies of trained parameter k (none for a bias): row-major, for the
// surrogate's kernels, and in the layout of network_kernel's shared memory,
// where two bulk copies put them (the weights; then the transposes of W2, W3, W4)
__device__ __forceinline__ void store_copies(int k, float w, __nv_bfloat16 *wb, unsigned char *core) {
  int off, rows, cols, base;
  if (k < OFF_B1) {
    off = OFF_W1; rows = NH; cols = NIN; base = WB_W1;
  } else if (k >= OFF_W2 && k < OFF_B2) {
    off = OFF_W2; rows = NH; cols = NH; base = WB_W2;
  } else if (k >= OFF_W3 && k < OFF_B3) {
    off = OFF_W3; rows = NH; cols = NH; base = WB_W3;
  } else if (k >= OFF_W4 && k < OFF_B4) {
    off = OFF_W4; rows = NOUT_PAD; cols = NH; base = WB_W4;
  } else {
    return;
  }
  const int e = k - off, r = e / cols, c = e % cols;
  const __nv_bfloat16 b = __float2bfloat16_rn(w);
  wb[base + e] = b;
  *reinterpret_cast<__nv_bfloat16 *>(core + 2 * base + tc::chunk_offset(rows, r, c)) = b;
  if (base != WB_W1) *reinterpret_cast<__nv_bfloat16 *>(core + 2 * (NWB + base - WB_W2) + tc::chunk_offset(cols, c, r)) = b;
}
__global__ void refresh_kernel(const float *p, __nv_bfloat16 *wb, unsigned char *core) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k < NTRAIN) store_copies(k, p[k], wb, core);
}

// ---- forward and backward of a tile of 128 rows
// 16 warps: warp w reads tensor-memory lanes (rows) 32 (w % 4) .. + 31 and, of
// a 128-column accumulator, columns 32 (w / 4) .. + 31, so that the epilogues
// (GELU, its derivative, the transposed stores) are spread over all warps.  The
// chain gather -> 4 layers -> loss -> 3 layers back is serial; what bounds it is
// the latency of its seven MMA-and-epilogue stages (about 3 us each, 30 us cold
// from launch to end for any batch up to 152 tiles), not the tensor rate.
constexpr int TROWS = 128, NET_THREADS = 512;
constexpr unsigned S_W1 = 0, S_W2 = S_W1 + NH * NIN * 2, S_W3 = S_W2 + NH * NH * 2, S_W4 = S_W3 + NH * NH * 2;
constexpr unsigned S_ACT = S_W4 + NOUT_PAD * NH * 2;  // the layer's input: X, H or dZ (128 x 128)
constexpr unsigned S_F32 = S_ACT + TROWS * NH * 2;    // biases, scales, bias-gradient slots, loss slots
constexpr int NBIAS_G = 3 * NH + NOUT_PAD;            // bias gradients: b1, b2, b3, b4
constexpr int F_BIAS = 0, F_INS = F_BIAS + NBIAS_G, F_OUTS = F_INS + NIN, F_DB = F_OUTS + NOUT,
              F_LOSS = F_DB + 4 * NBIAS_G, F_TOTAL = F_LOSS + 4 * 2;  // the loss slots are doubles
static_assert(S_F32 % 8 == 0 && F_LOSS % 2 == 0, "alignment of the loss slots");
constexpr unsigned S_BACK = (S_F32 + F_TOTAL * 4 + 127) & ~127u;  // backward only: W2^T, W3^T, W4^T, dY
constexpr unsigned S_W2T = S_BACK, S_W3T = S_W2T + NH * NH * 2, S_W4T = S_W3T + NH * NH * 2,
                   S_DY = S_W4T + NOUT_PAD * NH * 2;
constexpr unsigned NET_SMEM_FWD = S_BACK, NET_SMEM = S_DY + TROWS * NOUT_PAD * 2;
static_assert(NET_SMEM <= 227 * 1024, "shared memory");
constexpr unsigned CORE_FWD = 2 * NWB, CORE_BYTES = CORE_FWD + 2 * (NWB - WB_W2);
static_assert(S_ACT - S_W1 == CORE_FWD && S_DY - S_W2T == CORE_BYTES - CORE_FWD, "layout of the weight copies");
constexpr unsigned MLP_WAIT = 1u << 20;  // polls of an MMA barrier before a CTA gives up
constexpr int PART_B = NBIAS_G + 2;      // a CTA's partial row: bias gradients, its loss as a double

struct NetArgs {
  const float *X, *T;  // samples; T null: forward only
  float *Yout;         // forward only: n x 8 outputs, scaled
  const float *p;
  const unsigned char *core;  // weights in the shared-memory layout
  int n, B, nvalid;  // samples, rows of the batch (a multiple of 8), rows that count
  uint64_t seed;     // 0: row r is sample r
  long long step;
  __nv_bfloat16 *XT, *HT[3], *dZT[3], *dYT;  // transposes, leading dimension B
  float *partB;                              // [gridDim.x][PART_B]
  int *err;
};

// `bytes` (a multiple of 16) of global memory into shared memory, completing on bar
__device__ __forceinline__ void bulk_copy(void *dst, const void *src, unsigned bytes, unsigned long long *bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   tc::smem_u32(dst)),
               "l"(src), "r"(bytes), "r"(tc::smem_u32(bar))
               : "memory");
}

// D (tmem) = A (128 x Kd) W^T (N x Kd): one elected thread
__device__ __forceinline__ void issue(unsigned tmem, unsigned a_s, unsigned w_s, int Kd, int N,
                                      unsigned long long *bar) {
  const uint32_t idesc = tc::make_idesc(TROWS, N);
  const unsigned lboA = TROWS * 16, lboW = (unsigned)N * 16;
  for (int k = 0; k < Kd / 16; k++)
    tc::mma_bf16(tmem, tc::make_desc(a_s + 2 * k * lboA, lboA, 128), tc::make_desc(w_s + 2 * k * lboW, lboW, 128),
                 idesc, k > 0 ? 1 : 0);
  tc::mma_commit(bar);
}

// one stage: the tile's operand is in shared memory; MMAs, then a bounded
// wait with a block-uniform outcome
__device__ __forceinline__ bool stage(unsigned tmem, unsigned a_s, unsigned w_s, int Kd, int N,
                                      unsigned long long *bar, unsigned &phase) {
  tc::fence_async_smem();
  tc::fence_before_sync();
  __syncthreads();
  if (threadIdx.x == 0) {
    tc::fence_after_sync();
    issue(tmem, a_s, w_s, Kd, N, bar);
  }
  const bool ok = __syncthreads_and(tc::bar_wait(bar, phase, MLP_WAIT)) != 0;
  phase ^= 1;
  tc::fence_after_sync();
  return ok;
}

// 32 values of row `row` at columns cb .. cb + 31: BF16 into the operand buffer
// and, if T is given, transposed into T (leading dimension B)
__device__ __forceinline__ void put_row(unsigned char *act, __nv_bfloat16 *T, int B, int grow, int row, int cb,
                                        const float v[32], bool in_batch) {
  __nv_bfloat16 h[32];
#pragma unroll
  for (int j = 0; j < 32; j++) h[j] = __float2bfloat16_rn(v[j]);
#pragma unroll
  for (int q = 0; q < 4; q++) {
    unsigned w[4];
#pragma unroll
    for (int e = 0; e < 4; e++)
      w[e] = (unsigned)__bfloat16_as_ushort(h[8 * q + 2 * e]) | ((unsigned)__bfloat16_as_ushort(h[8 * q + 2 * e + 1]) << 16);
    *reinterpret_cast<uint4 *>(act + tc::chunk_offset(TROWS, row, cb + 8 * q)) = make_uint4(w[0], w[1], w[2], w[3]);
  }
  if (T && in_batch) {
#pragma unroll
    for (int j = 0; j < 32; j++) T[(long long)(cb + j) * B + grow] = h[j];
  }
}

// sums over the warp's 32 lanes of 32 values each: lane c gets the sum of v[c]
__device__ __forceinline__ float column_sums(float v[32], int lane) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int j = 0; j < o; j++) {
      const float give = up ? v[j] : v[j + o], keep = up ? v[j + o] : v[j];
      v[j] = keep + __shfl_xor_sync(0xffffffffu, give, o);
    }
  }
  return v[0];
}

template <bool TRAIN>
__global__ void __launch_bounds__(NET_THREADS, 1) network_kernel(NetArgs A) {
  extern __shared__ __align__(128) unsigned char nsm[];
  __shared__ alignas(8) unsigned long long bar, wbar;
  __shared__ unsigned tslot;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int row = 32 * (warp & 3) + lane, cb = 32 * (warp >> 2);
  float *f = reinterpret_cast<float *>(nsm + S_F32);
  double *loss = reinterpret_cast<double *>(f + F_LOSS);  // by row group, over all tiles of the CTA
  float *db = f + F_DB + (warp & 3) * NBIAS_G;  // this row group's slots; a column belongs to one warp of it
  unsigned char *act = nsm + S_ACT;
  pdl_start();
  if (warp == 0) tc::tmem_alloc(&tslot, 512);
  pdl_wait();
  if (tid == 0) {
    tc::bar_init(&bar, 1);
    tc::bar_init(&wbar, 1);
    // the weights, while the first tile is gathered
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(tc::smem_u32(&wbar)),
                 "r"(TRAIN ? CORE_BYTES : CORE_FWD)
                 : "memory");
    bulk_copy(nsm + S_W1, A.core, CORE_FWD, &wbar);
    if (TRAIN) bulk_copy(nsm + S_W2T, A.core + CORE_FWD, CORE_BYTES - CORE_FWD, &wbar);
  }
  for (int k = tid; k < F_TOTAL; k += NET_THREADS) {
    float x = 0.0f;
    if (k < NH) x = A.p[OFF_B1 + k];
    else if (k < 2 * NH) x = A.p[OFF_B2 + k - NH];
    else if (k < 3 * NH) x = A.p[OFF_B3 + k - 2 * NH];
    else if (k < F_INS) x = A.p[OFF_B4 + k - 3 * NH];
    else if (k < F_DB) x = A.p[OFF_INS + k - F_INS];  // input scales, then output scales
    f[k] = x;
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const unsigned tmem = tslot, tlane = tmem + ((unsigned)(32 * (warp & 3)) << 16);
  const unsigned act_s = tc::smem_u32(act), base_s = tc::smem_u32(nsm);
  unsigned phase = 0;
  bool ok = true, loaded = false;
  const int ntiles = (A.B + TROWS - 1) / TROWS;
  for (int tile = blockIdx.x; tile < ntiles && ok; tile += gridDim.x) {
    const int r0 = tile * TROWS;
    const auto sample = [&](int r) {
      return A.seed ? (long long)(mix64(A.seed ^ mix64((uint64_t)A.step * 1315423911ull + r)) % A.n) : (long long)r;
    };
    {
      // four threads a row, 16 inputs each, in the epilogues' mapping
      const int c0 = 16 * (warp >> 2), r = r0 + row;
      float x[16];
#pragma unroll
      for (int j = 0; j < 16; j++) x[j] = 0.0f;
      if (r < A.nvalid) {
        const float *src = A.X + sample(r) * NIN + c0;
        if (reinterpret_cast<size_t>(A.X) & 15) {  // rows are 256 bytes: the first decides for all
#pragma unroll
          for (int j = 0; j < 16; j++) x[j] = __ldg(src + j);
        } else {
#pragma unroll
          for (int q = 0; q < 4; q++) {
            const float4 w = __ldg(reinterpret_cast<const float4 *>(src) + q);
            x[4 * q] = w.x;
            x[4 * q + 1] = w.y;
            x[4 * q + 2] = w.z;
            x[4 * q + 3] = w.w;
          }
        }
#pragma unroll
        for (int j = 0; j < 16; j++) x[j] *= f[F_INS + c0 + j];
      }
#pragma unroll
      for (int q = 0; q < 2; q++) {
        unsigned w[4];
#pragma unroll
        for (int e = 0; e < 4; e++) {
          const __nv_bfloat162 b = __floats2bfloat162_rn(x[8 * q + 2 * e], x[8 * q + 2 * e + 1]);
          w[e] = *reinterpret_cast<const unsigned *>(&b);
        }
        *reinterpret_cast<uint4 *>(act + tc::chunk_offset(TROWS, row, c0 + 8 * q)) = make_uint4(w[0], w[1], w[2], w[3]);
      }
      if (TRAIN && r < A.B) {
#pragma unroll
        for (int j = 0; j < 16; j++) A.XT[(long long)(c0 + j) * A.B + r] = __float2bfloat16_rn(x[j]);
      }
    }
    const int grow = r0 + row;
    const bool in_batch = grow < A.B;
    if (!loaded) loaded = ok = __syncthreads_and(tc::bar_wait(&wbar, 0, MLP_WAIT)) != 0;
#pragma unroll 1
    for (int l = 0; l < 3 && ok; l++) {
      ok = stage(tmem + 128 * l, act_s, base_s + (l == 0 ? S_W1 : (l == 1 ? S_W2 : S_W3)), l == 0 ? NIN : NH, NH, &bar,
                 phase);
      if (!ok) break;
      float v[32];
      tc::tmem_ld32(tlane + 128 * l + cb, v);
#pragma unroll
      for (int j = 0; j < 32; j++) v[j] = gelu(v[j] + f[F_BIAS + l * NH + cb + j]);
      put_row(act, TRAIN ? A.HT[l] : nullptr, A.B, grow, row, cb, v, in_batch);
    }
    if (ok) ok = stage(tmem + 384, act_s, base_s + S_W4, NH, NOUT_PAD, &bar, phase);
    if (!ok) break;
    if (warp < 4) {
      float y[32];
      tc::tmem_ld32(tlane + 384, y);
      if (!TRAIN) {
        if (grow < A.nvalid)
#pragma unroll
          for (int k = 0; k < NOUT; k++)
            A.Yout[(long long)grow * NOUT + k] = (y[k] + f[F_BIAS + 3 * NH + k]) * f[F_OUTS + k];
      } else {
        float d[NOUT_PAD], l = 0.0f;
#pragma unroll
        for (int k = 0; k < NOUT_PAD; k++) d[k] = 0.0f;
        if (grow < A.nvalid) {
          const float *t = A.T + sample(grow) * NOUT;
#pragma unroll
          for (int k = 0; k < NOUT; k++) {
            const float e = y[k] + f[F_BIAS + 3 * NH + k] - t[k] / f[F_OUTS + k];
            l += e * e;
            d[k] = 2.0f * e / (float)(NOUT * (long long)A.nvalid);
          }
        }
        unsigned char *dy = nsm + S_DY;
        unsigned w[8];
#pragma unroll
        for (int e = 0; e < 8; e++) {
          const __nv_bfloat162 b = __floats2bfloat162_rn(d[2 * e], d[2 * e + 1]);
          w[e] = *reinterpret_cast<const unsigned *>(&b);
        }
        *reinterpret_cast<uint4 *>(dy + tc::chunk_offset(TROWS, row, 0)) = make_uint4(w[0], w[1], w[2], w[3]);
        *reinterpret_cast<uint4 *>(dy + tc::chunk_offset(TROWS, row, 8)) = make_uint4(w[4], w[5], w[6], w[7]);
        if (in_batch)
#pragma unroll
          for (int k = 0; k < NOUT_PAD; k++) A.dYT[(long long)k * A.B + grow] = __float2bfloat16_rn(d[k]);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          l += __shfl_xor_sync(0xffffffffu, l, o);
#pragma unroll
          for (int k = 0; k < NOUT; k++) d[k] += __shfl_xor_sync(0xffffffffu, d[k], o);
        }
        if (lane == 0) {
          loss[warp] += l;
#pragma unroll
          for (int k = 0; k < NOUT; k++) db[3 * NH + k] += d[k];
        }
      }
    }
    if (TRAIN) {
      // back through the layers: dH into columns 384 .. 511, dZ = dH gelu'(Z)
#pragma unroll 1
      for (int l = 2; l >= 0 && ok; l--) {
        ok = l == 2 ? stage(tmem + 384, tc::smem_u32(nsm + S_DY), base_s + S_W4T, NOUT_PAD, NH, &bar, phase)
                    : stage(tmem + 384, act_s, base_s + (l == 1 ? S_W3T : S_W2T), NH, NH, &bar, phase);
        if (!ok) break;
        float z[32], v[32];
        tc::tmem_ld32(tlane + 128 * l + cb, z);
        tc::tmem_ld32(tlane + 384 + cb, v);
#pragma unroll
        for (int j = 0; j < 32; j++) v[j] = in_batch ? v[j] * gelu_grad(z[j] + f[F_BIAS + l * NH + cb + j]) : 0.0f;
        put_row(act, A.dZT[l], A.B, grow, row, cb, v, in_batch);
        db[l * NH + cb + lane] += column_sums(v, lane);
      }
    }
    // the next tile's gather overwrites the operand buffer and its MMAs the
    // accumulators: every read of this tile's must be done
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
  }
  if (!ok) {
    // the weights' copies or the MMAs did not complete in time: record it and
    // give them one more bounded wait before the memory is released
    if (tid == 0) atomicOr(A.err, 1);
    if (!loaded) tc::bar_wait(&wbar, 0, MLP_WAIT);
    else tc::bar_wait(&bar, phase ^ 1, MLP_WAIT);
  }
  if (TRAIN) {
    float *out = A.partB + (long long)blockIdx.x * PART_B;
    for (int k = tid; k < NBIAS_G; k += NET_THREADS) {
      const float *d = f + F_DB + k;
      out[k] = (d[0] + d[NBIAS_G]) + (d[2 * NBIAS_G] + d[3 * NBIAS_G]);
    }
    if (tid == 0) {
      const double l = (loss[0] + loss[1]) + (loss[2] + loss[3]);
      *reinterpret_cast<double *>(out + NBIAS_G) = l / (double)(NOUT * (long long)A.nvalid);
    }
  }
  tc::fence_before_sync();
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc(tmem, 512);
}

// ---- weight gradients: dW_l = dZ_l^T H_(l-1) over the batch, layer blockIdx.y,
// batch rows [blockIdx.x * per, + per) x 256, the partial product into
// partW[blockIdx.x].  A 256-row step's operands (two of 64 KB) are loaded with
// all loads in flight and contracted by 16 MMAs: 12.8 us (cold) for B = 4096,
// where the four products took four launches of 38 us, their results added by
// scattered atomics.  128-row steps are no faster at 4096 and 17 % slower a
// training step at 16384 (twice the partial products).  At most WG_CHAIN steps (512
// rows) are summed in tensor memory; a split of more adds its chains in registers,
// so that the small terms of a large batch are not lost one by one beside a large
// partial sum.
constexpr int WG_THREADS = 256, WG_STEP = 256, WG_CHAIN = 2;
constexpr unsigned WG_OP = NH * WG_STEP * 2, WG_SMEM = 2 * WG_OP + 1024;
struct WgradArgs {
  const __nv_bfloat16 *A[4], *Bm[4];  // per layer: dZ^T (or dY^T), the input's transpose
  int M[4], N[4], off[4];             // rows, columns, place in the parameters
  float *partW;                       // [gridDim.x][NTRAIN]
  int B, per;
  int *err;
};
// rows [0, R) (zero from `rows` on) of a row-major R x B array, columns k0 ..
// k0 + 255 (zero from B on), into the K-major core layout of R rows
__device__ __forceinline__ void load_step(unsigned char *dst, const __nv_bfloat16 *X, int rows, int R, int B, int k0) {
  static_assert(WG_THREADS == WG_STEP && NH % 8 == 0, "8 rows of WG_STEP / 8 pieces a round");
  const int r0 = threadIdx.x & 7, kv = threadIdx.x >> 3, k = k0 + 8 * kv;
  // (the loads first: plain ones, of the launch before, do not pass the stores)
  uint4 v[NH / 8];
#pragma unroll
  for (int q = 0; q < NH / 8; q++) {
    const int r = r0 + 8 * q;
    v[q] = make_uint4(0u, 0u, 0u, 0u);
    if (r < rows && k < B) v[q] = *reinterpret_cast<const uint4 *>(X + (long long)r * B + k);
  }
#pragma unroll
  for (int q = 0; q < NH / 8; q++)
    if (8 * q < R) *reinterpret_cast<uint4 *>(dst + tc::chunk_offset(R, r0 + 8 * q, 8 * kv)) = v[q];
}
__global__ void __launch_bounds__(WG_THREADS, 1) weight_grad_kernel(WgradArgs a) {
  extern __shared__ __align__(128) unsigned char wsm[];
  __shared__ alignas(8) unsigned long long bar;
  __shared__ unsigned tslot;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, l = blockIdx.y;
  const int M = a.M[l], N = a.N[l];
  unsigned char *sA = wsm, *sB = wsm + WG_OP;
  pdl_start();
  if (warp == 0) tc::tmem_alloc(&tslot, 128);
  if (tid == 0) tc::bar_init(&bar, 1);
  pdl_wait();
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const unsigned tmem = tslot;
  const uint32_t idesc = tc::make_idesc(NH, N);
  const unsigned lboA = NH * 16, lboB = (unsigned)N * 16;
  unsigned phase = 0;
  bool ok = true;
  const int c0 = blockIdx.x * a.per, c1 = min((a.B + WG_STEP - 1) / WG_STEP, c0 + a.per);
  // this thread's row, columns cb0 .. + 31 and cb0 + 64 .. + 95
  const int row = 32 * (warp & 3) + lane, cb0 = 32 * (warp >> 2);
  float acc[2][32] = {};
  for (int c = c0; c < c1 && ok; c++) {
    load_step(sA, a.A[l], M, NH, a.B, c * WG_STEP);
    load_step(sB, a.Bm[l], N, N, a.B, c * WG_STEP);
    tc::fence_async_smem();
    __syncthreads();
    if (tid == 0) {
      tc::fence_after_sync();
      const unsigned ba = tc::smem_u32(sA), bb = tc::smem_u32(sB);
#pragma unroll
      for (int k = 0; k < WG_STEP / 16; k++)
        tc::mma_bf16(tmem, tc::make_desc(ba + 2 * k * lboA, lboA, 128), tc::make_desc(bb + 2 * k * lboB, lboB, 128),
                     idesc, ((c - c0) % WG_CHAIN > 0 || k > 0) ? 1 : 0);
      tc::mma_commit(&bar);
    }
    ok = __syncthreads_and(tc::bar_wait(&bar, phase, MLP_WAIT)) != 0;
    phase ^= 1;
    if (ok && ((c - c0) % WG_CHAIN == WG_CHAIN - 1 || c == c1 - 1)) {  // the chain ends
      tc::fence_after_sync();
#pragma unroll
      for (int h = 0; h < 2; h++) {
        if (cb0 + 64 * h >= N) break;
        float v[32];
        tc::tmem_ld32(tmem + ((unsigned)(32 * (warp & 3)) << 16) + (unsigned)(cb0 + 64 * h), v);
#pragma unroll
        for (int j = 0; j < 32; j++) acc[h][j] += v[j];
      }
      tc::fence_before_sync();  // before the next chain's MMAs, issued after a __syncthreads
    }
  }
  if (!ok) {
    if (tid == 0) atomicOr(a.err, 1);
    tc::bar_wait(&bar, phase ^ 1, MLP_WAIT);
  } else {
    float *out = a.partW + (long long)blockIdx.x * NTRAIN + a.off[l] + row * N + cb0;
    if (row < M)
#pragma unroll
      for (int h = 0; h < 2; h++) {
        if (cb0 + 64 * h >= N) break;
        const float *v = acc[h];
#pragma unroll
        for (int q = 0; q < 8; q++)
          reinterpret_cast<float4 *>(out + 64 * h)[q] = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
      }
  }
  tc::fence_before_sync();
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc(tmem, 128);
}

// gradient of parameter k from the partial sums: weights over the splits of
// weight_grad_kernel, biases over the CTAs of network_kernel
struct Partials {
  const float *partW, *partB;
  int nW, nB;
};
__device__ __forceinline__ float gradient(const Partials &P, int k) {
  int b = -1;
  if (k >= OFF_B4) b = 3 * NH + k - OFF_B4;
  else if (k >= OFF_B3 && k < OFF_W4) b = 2 * NH + k - OFF_B3;
  else if (k >= OFF_B2 && k < OFF_W3) b = NH + k - OFF_B2;
  else if (k >= OFF_B1 && k < OFF_W2) b = k - OFF_B1;
  const float *p = b < 0 ? P.partW + k : P.partB + b;
  const int n = b < 0 ? P.nW : P.nB, stride = b < 0 ? NTRAIN : PART_B;
  float s = 0.0f;
  // all of up to 32 loads in flight; partial sums beyond
  for (int q0 = 0; q0 < n; q0 += 32) {
    float x[32];
#pragma unroll
    for (int q = 0; q < 32; q++) x[q] = q0 + q < n ? p[(long long)(q0 + q) * stride] : 0.0f;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
      for (int q = 0; q < o; q++) x[q] += x[q + o];
    s += x[0];
  }
  return s;
}
// the batch's loss, by the first warp of a block of its own
__device__ __forceinline__ void sum_loss(const Partials &P, double *loss) {
  const int lane = threadIdx.x;
  if (lane >= 32) return;
  double s = 0.0;
  for (int q = lane; q < P.nB; q += 32) s += *reinterpret_cast<const double *>(P.partB + (long long)q * PART_B + NBIAS_G);
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) *loss = s;
}
// blocks of gradient_kernel and adam_kernel: the parameters, then one for the loss
constexpr int PAR_THREADS = 128, PAR_BLOCKS = (NTRAIN + PAR_THREADS - 1) / PAR_THREADS;
__global__ void gradient_kernel(Partials P, float *g, double *loss) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (blockIdx.x == PAR_BLOCKS) sum_loss(P, loss);
  else if (k < NTRAIN) g[k] = gradient(P, k);
}

// Adam on parameter k, and its BF16 copies
__global__ void adam_kernel(Partials P, float *p, float *m, float *v, __nv_bfloat16 *wb, unsigned char *core, float lr,
                            float b1, float b2, float eps, float c1, float c2, double *loss) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  pdl_start();
  pdl_wait();
  if (blockIdx.x == PAR_BLOCKS) sum_loss(P, loss);
  if (k >= NTRAIN) return;
  const float gk = gradient(P, k);
  const float mk = b1 * m[k] + (1.0f - b1) * gk;
  const float vk = b2 * v[k] + (1.0f - b2) * gk * gk;
  m[k] = mk;
  v[k] = vk;
  const float w = p[k] - lr * (mk / c1) / (sqrtf(vk / c2) + eps);
  p[k] = w;
  store_copies(k, w, wb, core);
}

// root mean square of each column of a row-major (n x cols) array
__global__ void colrms_kernel(const float *A, long long n, int cols, double *out) {
  const int c = blockIdx.y;
  double s = 0.0;
  for (long long r = blockIdx.x * (long long)blockDim.x + threadIdx.x; r < n; r += (long long)gridDim.x * blockDim.x) {
    const double a = A[r * cols + c];
    s += a * a;
  }
  __shared__ double sm[256];
  sm[threadIdx.x] = s;
  __syncthreads();
  for (int k = blockDim.x / 2; k > 0; k >>= 1) {
    if (threadIdx.x < k) sm[threadIdx.x] += sm[threadIdx.x + k];
    __syncthreads();
  }
  if (threadIdx.x == 0) atomicAdd(out + c, sm[0]);
}

int mfail(int code, const char *msg) { return set_error(code, msg); }
int mcuda(cudaError_t e, const char *where) {
  cudaGetLastError();  // reported here: not once more by the check after a later launch
  char m[400];
  std::snprintf(m, sizeof(m), "%s: %s", where, cudaGetErrorString(e));
  return set_error(AF_ERR_CUDA, m);
}
#define MCK(call, where)                              \
  do {                                                \
    cudaError_t e_ = (call);                          \
    if (e_ != cudaSuccess) return mcuda(e_, where);   \
  } while (0)

struct MDev {
  int old = -1;
  explicit MDev(int d) {
    if (cudaGetDevice(&old) == cudaSuccess && old != d) cudaSetDevice(d);
    else old = -1;
  }
  ~MDev() {
    if (old >= 0) cudaSetDevice(old);
  }
};

int refresh(af_mlp *m, cudaStream_t s) {
  refresh_kernel<<<(NTRAIN + 255) / 256, 256, 0, s>>>(m->params, m->wb, m->core);
  MCK(cudaGetLastError(), "af_mlp: refresh");
  return AF_OK;
}

constexpr int MAX_SPLITS = 32;  // of weight_grad_kernel over the batch

// training scratch for B rows (B a multiple of 8) and a loss history of `steps`
int ensure_cap(af_mlp *m, int B, int steps) {
  if (m->cap >= B && m->hist_cap >= steps) return AF_OK;
  if (B < m->cap) B = m->cap;
  if (steps < m->hist_cap) steps = m->hist_cap;
  if (m->scratch) cudaFree(m->scratch);
  m->scratch = nullptr;
  m->cap = m->hist_cap = -1;  // nothing held: should the allocation fail, the next call of any size allocates
  const size_t b16 = sizeof(__nv_bfloat16), f32 = sizeof(float);
  const size_t sizes[] = {(size_t)B * NIN * b16,      3 * (size_t)B * NH * b16,      3 * (size_t)B * NH * b16,  // XT, HT, dZT
                          (size_t)B * NOUT_PAD * b16, MAX_SPLITS * (size_t)NTRAIN * f32,                       // dYT, partW
                          (size_t)m->sms * PART_B * f32, sizeof(double) * (size_t)(steps + 1), 64};            // partB, loss, err
  size_t total = 0;
  for (size_t z : sizes) total += (z + 255) & ~size_t(255);
  MCK(cudaMalloc(&m->scratch, total), "af_mlp: cudaMalloc(scratch)");
  char *q = (char *)m->scratch;
  auto take = [&](size_t z) {
    char *r = q;
    q += (z + 255) & ~size_t(255);
    return r;
  };
  m->XT = (__nv_bfloat16 *)take(sizes[0]);
  m->HT = (__nv_bfloat16 *)take(sizes[1]);
  m->dZT = (__nv_bfloat16 *)take(sizes[2]);
  m->dYT = (__nv_bfloat16 *)take(sizes[3]);
  m->partW = (float *)take(sizes[4]);
  m->partB = (float *)take(sizes[5]);
  m->loss = (double *)take(sizes[6]);
  m->err = (int *)take(sizes[7]);
  m->cap = B;
  m->hist_cap = steps;
  return AF_OK;
}

int prepare_network() {
  MCK(cudaFuncSetAttribute(network_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, NET_SMEM), "af_mlp: attributes");
  MCK(cudaFuncSetAttribute(network_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, NET_SMEM_FWD), "af_mlp: attributes");
  MCK(cudaFuncSetAttribute(weight_grad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, WG_SMEM), "af_mlp: attributes");
  return AF_OK;
}

NetArgs net_args(af_mlp *m, const float *X, const float *T, float *Y, int n, int B, int nvalid, uint64_t seed,
                 long long step) {
  NetArgs A;
  A.X = X;
  A.T = T;
  A.Yout = Y;
  A.p = m->params;
  A.core = m->core;
  A.n = n;
  A.B = B;
  A.nvalid = nvalid;
  A.seed = seed;
  A.step = step;
  A.XT = m->XT;
  for (int l = 0; l < 3; l++) {
    A.HT[l] = m->HT + (size_t)l * B * NH;
    A.dZT[l] = m->dZT + (size_t)l * B * NH;
  }
  A.dYT = m->dYT;
  A.partB = m->partB;
  A.err = m->err;
  return A;
}

// forward and backward of B rows (nvalid of them real); P: the partial sums of
// the loss's gradient
int loss_partials(af_mlp *m, const float *X, const float *T, int n, int B, int nvalid, uint64_t seed, long long step,
                  Partials &P, cudaStream_t s) {
  const NetArgs A = net_args(m, X, T, nullptr, n, B, nvalid, seed, step);
  const int tiles = (B + TROWS - 1) / TROWS;
  P.nB = tiles < m->sms ? tiles : m->sms;
  // (a step's three launches each begin while the one before ends: 54 -> 47 us a
  // step of 4096 samples)
  MCK(launch_pdl(network_kernel<true>, dim3(P.nB), dim3(NET_THREADS), NET_SMEM, s, A), "af_mlp: network");
  WgradArgs G;
  const int M[4] = {NH, NH, NH, NOUT_PAD}, N[4] = {NIN, NH, NH, NH}, off[4] = {OFF_W1, OFF_W2, OFF_W3, OFF_W4};
  for (int l = 0; l < 4; l++) {
    G.A[l] = l < 3 ? A.dZT[l] : A.dYT;
    G.Bm[l] = l > 0 ? A.HT[l - 1] : A.XT;
    G.M[l] = M[l];
    G.N[l] = N[l];
    G.off[l] = off[l];
  }
  G.partW = m->partW;
  G.B = B;
  G.err = m->err;
  const int steps = (B + WG_STEP - 1) / WG_STEP;
  G.per = (steps + MAX_SPLITS - 1) / MAX_SPLITS;
  P.nW = (steps + G.per - 1) / G.per;
  MCK(launch_pdl(weight_grad_kernel, dim3(P.nW, 4), dim3(WG_THREADS), WG_SMEM, s, G), "af_mlp: weight gradients");
  P.partW = m->partW;
  P.partB = m->partB;
  return AF_OK;
}

int check_err(af_mlp *m, cudaStream_t s) {
  int e = 0;
  MCK(cudaMemcpyAsync(&e, m->err, sizeof(int), cudaMemcpyDeviceToHost, s), "af_mlp: err");
  MCK(cudaStreamSynchronize(s), "af_mlp: sync");
  if (e) return mfail(AF_ERR_CUDA, "af_mlp: a tensor-core wait timed out");
  return AF_OK;
}

void free_mlp(af_mlp *m) {
  cudaFree(m->params);
  cudaFree(m->grads);
  cudaFree(m->adam_m);
  cudaFree(m->adam_v);
  cudaFree(m->wb);
  cudaFree(m->core);
  if (m->scratch) cudaFree(m->scratch);
  delete m;
}

}  // namespace

extern "C" {

af_mlp *af_mlp_create(uint64_t seed) {
  af_mlp *m = new (std::nothrow) af_mlp();
  if (!m) {
    mfail(AF_ERR_ALLOC, "af_mlp_create: out of host memory");
    return nullptr;
  }
  cudaGetDevice(&m->device);
  if (prepare_network() != AF_OK) {
    delete m;
    return nullptr;
  }
  cudaError_t e = cudaDeviceGetAttribute(&m->sms, cudaDevAttrMultiProcessorCount, m->device);
  if (e == cudaSuccess) e = cudaMalloc(&m->params, sizeof(float) * NPARAM);
  if (e == cudaSuccess) e = cudaMalloc(&m->grads, sizeof(float) * NTRAIN);
  if (e == cudaSuccess) e = cudaMalloc(&m->adam_m, sizeof(float) * NTRAIN);
  if (e == cudaSuccess) e = cudaMalloc(&m->adam_v, sizeof(float) * NTRAIN);
  if (e == cudaSuccess) e = cudaMalloc(&m->wb, sizeof(__nv_bfloat16) * NWB);
  if (e == cudaSuccess) e = cudaMalloc(&m->core, CORE_BYTES);
  if (e == cudaSuccess) e = cudaMemset(m->adam_m, 0, sizeof(float) * NTRAIN);
  if (e == cudaSuccess) e = cudaMemset(m->adam_v, 0, sizeof(float) * NTRAIN);
  if (e != cudaSuccess) {
    mcuda(e, "af_mlp_create");
    free_mlp(m);
    return nullptr;
  }
  init_kernel<<<(NPARAM + 255) / 256, 256>>>(m->params, seed);
  if (refresh(m, nullptr) != AF_OK || cudaDeviceSynchronize() != cudaSuccess) {
    free_mlp(m);
    return nullptr;
  }
  return m;
}

void af_mlp_destroy(af_mlp *m) {
  if (!m) return;
  MDev d(m->device);
  cudaDeviceSynchronize();
  free_mlp(m);
}

int af_mlp_set_params(af_mlp *m, const float *host) {
  if (!m || !host) return mfail(AF_ERR_ARG, "af_mlp_set_params: null argument");
  MDev d(m->device);
  MCK(cudaMemcpy(m->params, host, sizeof(float) * NPARAM, cudaMemcpyHostToDevice), "af_mlp_set_params");
  MCK(cudaMemset(m->adam_m, 0, sizeof(float) * NTRAIN), "af_mlp_set_params");
  MCK(cudaMemset(m->adam_v, 0, sizeof(float) * NTRAIN), "af_mlp_set_params");
  m->adam_t = 0;
  int rc = refresh(m, nullptr);
  if (rc) return rc;
  MCK(cudaDeviceSynchronize(), "af_mlp_set_params");
  return AF_OK;
}

int af_mlp_get_params(af_mlp *m, float *host) {
  if (!m || !host) return mfail(AF_ERR_ARG, "af_mlp_get_params: null argument");
  MDev d(m->device);
  MCK(cudaDeviceSynchronize(), "af_mlp_get_params");
  MCK(cudaMemcpy(host, m->params, sizeof(float) * NPARAM, cudaMemcpyDeviceToHost), "af_mlp_get_params");
  return AF_OK;
}

int af_mlp_fit_scales(af_mlp *m, const float *X, const float *T, long long n) {
  if (!m || !X || !T || n <= 0) return mfail(AF_ERR_ARG, "af_mlp_fit_scales: bad arguments");
  MDev d(m->device);
  double *acc = nullptr;
  MCK(cudaMalloc(&acc, sizeof(double) * (NIN + NOUT)), "af_mlp_fit_scales");
  cudaMemset(acc, 0, sizeof(double) * (NIN + NOUT));
  colrms_kernel<<<dim3(64, NIN), 256>>>(X, n, NIN, acc);
  colrms_kernel<<<dim3(64, NOUT), 256>>>(T, n, NOUT, acc + NIN);
  double h[NIN + NOUT];
  cudaError_t e = cudaMemcpy(h, acc, sizeof(h), cudaMemcpyDeviceToHost);
  cudaFree(acc);
  MCK(e, "af_mlp_fit_scales");
  float sc[NIN + NOUT];
  for (int k = 0; k < NIN; k++) {
    const double r = std::sqrt(h[k] / (double)n);
    sc[k] = r > 1e-12 ? (float)(1.0 / r) : 0.0f;  // an input that is always 0 stays 0
  }
  for (int k = 0; k < NOUT; k++) {
    const double r = std::sqrt(h[NIN + k] / (double)n);
    sc[NIN + k] = r > 1e-30 ? (float)r : 1.0f;
  }
  MCK(cudaMemcpy(m->params + OFF_INS, sc, sizeof(sc), cudaMemcpyHostToDevice), "af_mlp_fit_scales");
  return AF_OK;
}

int af_mlp_forward(af_mlp *m, const float *X, float *Y, int n, void *stream) {
  if (!m || !X || !Y || n <= 0) return mfail(AF_ERR_ARG, "af_mlp_forward: bad arguments");
  MDev d(m->device);
  cudaStream_t s = (cudaStream_t)stream;
  const int B = (n + 7) & ~7, tiles = (B + TROWS - 1) / TROWS;
  int rc = ensure_cap(m, 0, 0);
  if (rc) return rc;
  MCK(cudaMemsetAsync(m->err, 0, sizeof(int), s), "af_mlp_forward");
  network_kernel<false><<<tiles < m->sms ? tiles : m->sms, NET_THREADS, NET_SMEM_FWD, s>>>(
      net_args(m, X, nullptr, Y, n, B, n, 0, 0));
  MCK(cudaGetLastError(), "af_mlp_forward");
  return check_err(m, s);
}

int af_mlp_loss_grad(af_mlp *m, const float *X, const float *T, int n, double *loss, float *grads) {
  if (!m || !X || !T || n <= 0) return mfail(AF_ERR_ARG, "af_mlp_loss_grad: bad arguments");
  MDev d(m->device);
  cudaStream_t s = nullptr;
  const int B = (n + 7) & ~7;
  int rc = ensure_cap(m, B, 0);
  if (rc) return rc;
  MCK(cudaMemsetAsync(m->err, 0, sizeof(int), s), "af_mlp_loss_grad");
  Partials P;
  if ((rc = loss_partials(m, X, T, n, B, n, 0, 0, P, s))) return rc;
  gradient_kernel<<<PAR_BLOCKS + 1, PAR_THREADS, 0, s>>>(P, m->grads, m->loss);
  MCK(cudaGetLastError(), "af_mlp_loss_grad");
  if ((rc = check_err(m, s))) return rc;
  if (loss) MCK(cudaMemcpy(loss, m->loss, sizeof(double), cudaMemcpyDeviceToHost), "af_mlp_loss_grad");
  if (grads) MCK(cudaMemcpy(grads, m->grads, sizeof(float) * NTRAIN, cudaMemcpyDeviceToHost), "af_mlp_loss_grad");
  return AF_OK;
}

int af_mlp_train(af_mlp *m, const float *X, const float *T, long long n, int steps, int batch, double lr,
                 uint64_t seed, float *loss_hist) {
  if (!m || !X || !T || n <= 0 || steps < 0 || batch < 8 || (batch & 7) || !(lr > 0) || seed == 0)
    return mfail(AF_ERR_ARG, "af_mlp_train: bad arguments (batch a multiple of 8, lr > 0, seed != 0)");
  MDev d(m->device);
  cudaStream_t s = nullptr;
  int rc = ensure_cap(m, batch, steps);
  if (rc) return rc;
  MCK(cudaMemsetAsync(m->err, 0, sizeof(int), s), "af_mlp_train");
  const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
  for (int k = 0; k < steps && rc == AF_OK; k++) {
    m->adam_t += 1;
    const float c1 = 1.0f - std::pow(b1, (float)m->adam_t), c2 = 1.0f - std::pow(b2, (float)m->adam_t);
    Partials P;
    if ((rc = loss_partials(m, X, T, (int)(n > 0x7fffffff ? 0x7fffffff : n), batch, batch, seed, m->adam_t, P, s))) break;
    const cudaError_t e =
        launch_pdl(adam_kernel, dim3(PAR_BLOCKS + 1), dim3(PAR_THREADS), 0, s, P, m->params, m->adam_m, m->adam_v, m->wb,
                   m->core, (float)lr, b1, b2, eps, c1, c2, m->loss + k);
    if (e != cudaSuccess) rc = mcuda(e, "af_mlp_train");
  }
  if (rc == AF_OK) rc = check_err(m, s);
  if (rc == AF_OK && loss_hist && steps > 0) {
    std::vector<double> h(steps);
    cudaError_t e = cudaMemcpy(h.data(), m->loss, sizeof(double) * steps, cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) rc = mcuda(e, "af_mlp_train");
    for (int k = 0; k < steps; k++) loss_hist[k] = (float)h[k];
  }
  return rc;
}

}  // extern "C"
