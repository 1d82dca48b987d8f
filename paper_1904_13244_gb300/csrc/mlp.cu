// Learned surrogate of the compressed Bloch model (K8): an MLP 3 -> H -> H -> H -> R
// from (ln T1, ln T2, B1) to the coefficients of the echo time course in the plan's
// time basis, with its derivatives in ln T1 and ln T2 by forward-mode tangents.
//
// Network (tanh hidden layers, linear output, per-coefficient output scale):
//     u = ((ln T1 - mu1)/s1, (ln T2 - mu2)/s2, (B1 - mu3)/s3)
//     a_l = tanh(W_l a_{l-1} + b_l),   c = scale * (W_4 a_3 + b_4)
// A tanh layer maps a tangent t to (1 - a^2) (W t); the tangents of u along ln T1 and
// ln T2 are (1/s1, 0, 0) and (0, 1/s2, 0).  So a batch of B samples runs as M = 3B rows
// (values, ln T1 tangents, ln T2 tangents) through every layer: one BF16 tcgen05 GEMM
// per layer shared by the value and both tangent streams, float32 accumulation, the
// activation and the tangent scaling in its epilogue.
//
// Training minimises the Sobolev loss
//     L = 1/B sum_b sum_r [(c - c*)^2 + lam ((dc1 - dc1*)^2 + (dc2 - dc2*)^2)] / scale_r^2
// with a hand-written backward pass: through s_k = (1 - a^2) z_k the value
// pre-activation receives (g_a - 2 a sum_k g_sk z_k)(1 - a^2) and each tangent
// pre-activation g_sk (1 - a^2); weight gradients are GEMMs of the gradient rows with
// the layer inputs over all 3B rows, input gradients GEMMs with the transposed weights.
// Inference and training share one fused layer kernel (mlp_layer_persistent_kernel): its
// epilogue sees the three streams of one (sample, feature) together and applies the
// activation (forward), the loss (output layer) or the way back through the activation
// (backward), so no GEMM result makes a trip through memory of its own.  Every weight
// gradient comes from one launch (mlp_dw_kernel), the biases' from the row tiles' column
// sums (mlp_grad_sum_kernel): nothing is added atomically, so a gradient is bitwise
// reproducible.  Adam keeps float32 master weights and refreshes the BF16 copies
// (row-major and transposed) used by the GEMMs.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <random>
#include <vector>

#include <cuda_bf16.h>

#include "internal.cuh"
#include "mlp.cuh"
#include "reduce.cuh"
#include "tc_prims.cuh"

namespace mrstat {
namespace {

inline int pad8(int k) { return (k + 7) / 8 * 8; }

// Layer 0's BF16 input rows for training: columns 0..2 the normalised (ln T1, ln T2, B1),
// then the two tangents' rows; columns 3..7 zero.
__global__ void mlp_input_kernel(const float* __restrict__ lnT, const float* __restrict__ b1, int B, float mu1,
                                 float s1, float mu2, float s2, float mu3, float s3, __nv_bfloat16* __restrict__ X0) {
  red::pdl_trigger();
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= B) return;
  const float bb = b1 != nullptr ? b1[b] : 1.f;
  const float u[3] = {(lnT[b] - mu1) / s1, (lnT[B + b] - mu2) / s2, (bb - mu3) / s3};
  __align__(16) __nv_bfloat16 o[3][8];
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    o[0][k] = __float2bfloat16_rn(k < 3 ? u[k] : 0.f);
    o[1][k] = __float2bfloat16_rn(k == 0 ? 1.f / s1 : 0.f);
    o[2][k] = __float2bfloat16_rn(k == 1 ? 1.f / s2 : 0.f);
  }
#pragma unroll
  for (int k = 0; k < 3; ++k)
    *reinterpret_cast<uint4*>(X0 + ((size_t)k * B + b) * 8) = *reinterpret_cast<const uint4*>(o[k]);
}

// Adam on one layer (weights [out][in] then bias [out]) and refresh of its BF16 copies
__global__ void mlp_adam_kernel(float* __restrict__ theta, float* __restrict__ m, float* __restrict__ v,
                                const float* __restrict__ g, int out, int in, float lr, float b1, float b2, float eps,
                                float c1, float c2, __nv_bfloat16* __restrict__ W, int ldw,
                                __nv_bfloat16* __restrict__ WT, int ldwt) {
  const int total = out * in + out;
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < total; e += gridDim.x * blockDim.x) {
    const float gi = g[e];
    const float mi = b1 * m[e] + (1.f - b1) * gi;
    const float vi = b2 * v[e] + (1.f - b2) * gi * gi;
    m[e] = mi;
    v[e] = vi;
    const float w = theta[e] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    theta[e] = w;
    if (e < out * in) {
      const int o = e / in, i = e - o * in;
      W[(size_t)o * ldw + i] = __float2bfloat16_rn(w);
      WT[(size_t)i * ldwt + o] = __float2bfloat16_rn(w);
    }
  }
}

// BF16 copies of one layer's weights from the float32 master (after set_params)
__global__ void mlp_cast_kernel(const float* __restrict__ theta, int out, int in, __nv_bfloat16* __restrict__ W,
                                int ldw, __nv_bfloat16* __restrict__ WT, int ldwt) {
  const int total = out * in;
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < total; e += gridDim.x * blockDim.x) {
    const int o = e / in, i = e - o * in;
    const __nv_bfloat16 w = __float2bfloat16_rn(theta[e]);
    W[(size_t)o * ldw + i] = w;
    WT[(size_t)i * ldwt + o] = w;
  }
}

// ---------------------------------------------------------------------------
// The layer kernel of inference and training (LayerMode).  Per K chunk TMA brings the three
// 128-row tiles of the layer input (value rows b, ln T1 tangent rows B + b, ln T2 tangent rows
// 2B + b) and one weight tile; one thread issues three tcgen05.mma per K step into three TMEM
// accumulators, so the epilogue sees z, z1, z2 of the same (sample, feature) and applies the
// layer there.  Inference:
//   hidden: a = tanh(z + bias), s_k = (1 - a^2) z_k, written as the next layer's BF16 input;
//   output: pred[k][r][b] = scale_r (z_k + [k = 0] bias_r), coalesced along the samples.
// Its pre-activations never reach global memory, and its hidden-layer tanh is the hardware
// tanh.approx.f32 (relative error about 2^-11, below the BF16 rounding of the values it
// produces).  Training takes tanhf and keeps a, z1, z2 in float32 for the way back, which the
// same kernel goes with the transposed weights.
//
__device__ __forceinline__ float tanh_fast(float x) {
  float y;
  asm("tanh.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// Persistent kernel: one CTA per SM walks the (128-row tile, 64-column tile) pairs, n
// fastest, so the CTAs working on one row tile at a time share its three input tiles
// through L2.  Warp 0 issues the TMA loads (three input
// tiles and the weight tile per 64-wide K chunk) into a ring of stages, warp 1 issues the
// three MMAs per K step into one of two TMEM accumulator sets (3 x 64 columns each), and
// sixteen epilogue warps (four per TMEM lane quarter, one 16-column chunk each: enough
// warps to hide the latency of the per-element work) run the epilogue of tile i while the
// MMAs of tile i + 1 proceed: bias and tanh, the tangent scaling 1 - a^2, BF16, 32-byte stores
// straight to the next layer's input rows (or, for the last layer, the scaled outputs).
// Every wait is bounded; a CTA that gives up sets err and drains its copies in flight.
// ---------------------------------------------------------------------------
// Layer 0 (three inputs: ln T1, ln T2, B1) on the CUDA cores, straight from the
// parameters: the same BF16-rounded inputs and weights and float32 sums as a tensor-core
// layer, then the hidden-layer epilogue, written as layer 1's BF16 input rows (value,
// ln T1 tangent, ln T2 tangent).  Thread per (sample, 8 features): consecutive threads
// take consecutive feature groups of one sample, so the 16-byte stores of a warp fill
// whole rows; the block's copy of the weights and biases sits in shared memory as
// [input][feature within group][group], which the lanes of a warp read without bank
// conflicts.  N <= 256 features (groups <= 32), N a multiple of 8.
constexpr int kFirstMaxGroups = 32;
__global__ void __launch_bounds__(256)
mlp_first_layer_kernel(const float* __restrict__ lnT, const float* __restrict__ b1, int B, float mu1, float s1,
                       float mu2, float s2, float mu3, float s3, const __nv_bfloat16* __restrict__ W0, int ldw,
                       const float* __restrict__ bias, int N, __nv_bfloat16* __restrict__ xn, int ldn) {
  __shared__ float ws[4][8][kFirstMaxGroups];
  const int groups = N / 8;
  for (int n = threadIdx.x; n < N; n += blockDim.x) {
    const int g = n >> 3, j = n & 7;
    ws[0][j][g] = __bfloat162float(W0[(size_t)n * ldw]);
    ws[1][j][g] = __bfloat162float(W0[(size_t)n * ldw + 1]);
    ws[2][j][g] = __bfloat162float(W0[(size_t)n * ldw + 2]);
    ws[3][j][g] = bias[n];
  }
  __syncthreads();
  const float d1 = __bfloat162float(__float2bfloat16_rn(1.f / s1));
  const float d2 = __bfloat162float(__float2bfloat16_rn(1.f / s2));
  const int total = B * groups;
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < total; e += gridDim.x * blockDim.x) {
    const int b = e / groups, g = e - b * groups;
    const float bb = b1 != nullptr ? b1[b] : 1.f;
    const float u0 = __bfloat162float(__float2bfloat16_rn((lnT[b] - mu1) / s1));
    const float u1 = __bfloat162float(__float2bfloat16_rn((lnT[B + b] - mu2) / s2));
    const float u2 = __bfloat162float(__float2bfloat16_rn((bb - mu3) / s3));
    __align__(16) __nv_bfloat16 o0[8], o1[8], o2[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const float w0 = ws[0][j][g], w1 = ws[1][j][g], w2 = ws[2][j][g];
      const float z = fmaf(w2, u2, fmaf(w1, u1, w0 * u0));
      const float a = tanh_fast(z + ws[3][j][g]);
      const float dd = 1.f - a * a;
      o0[j] = __float2bfloat16_rn(a);
      o1[j] = __float2bfloat16_rn(dd * (w0 * d1));
      o2[j] = __float2bfloat16_rn(dd * (w1 * d2));
    }
    const size_t row = (size_t)b * ldn + 8 * g, plane = (size_t)B * ldn;
    *reinterpret_cast<uint4*>(xn + row) = *reinterpret_cast<const uint4*>(o0);
    *reinterpret_cast<uint4*>(xn + plane + row) = *reinterpret_cast<const uint4*>(o1);
    *reinterpret_cast<uint4*>(xn + 2 * plane + row) = *reinterpret_cast<const uint4*>(o2);
  }
}

constexpr int kPerStages = 3;
struct PerShape {
  static constexpr int BN = 64;
  static constexpr uint32_t kA = tc::BM * tc::BK * 2;  // one 128-row input tile
  static constexpr uint32_t kB = BN * tc::BK * 2;      // one 64-row weight tile
  static constexpr uint32_t kStage = 3 * kA + kB;
  static constexpr uint32_t kTmemCols = 512;           // 2 sets x 3 streams x 64 columns
  static constexpr size_t kSmem = (size_t)kPerStages * kStage + 1024 + 256;
};

constexpr int kPerEpiWarps = 16;  // four per TMEM lane quarter, one 16-column chunk each
constexpr int kPerThreads = 64 + 32 * kPerEpiWarps;

// What the epilogue of a layer does with the three accumulators z, z1, z2 of a (sample,
// feature): inference (hidden, output), training forward (hidden: also keeps a, z1, z2 in
// float32; output: the loss and the gradient rows) and training backward (the accumulators
// are dL/d(layer output); back through the layer's tanh, and for layer 0 its weight
// gradient's sums instead of gradient rows).
enum LayerMode { kInferHidden, kInferLast, kTrainHidden, kTrainLast, kBack, kBackFirst };

struct LayerIo {
  const float* bias = nullptr;       // [N]
  __nv_bfloat16* xn = nullptr;       // [3B][ldn]: next layer's input rows, or the gradient rows
  int ldn = 0;
  const float* scale = nullptr;      // [R] output scale
  float* pred = nullptr;             // [3][R][B] (inference)
  float* za = nullptr;               // [3][B][N] a, z1, z2 of the layer (training)
  const float* target = nullptr;     // [3][R][B]
  float lam = 0.f;
  float* colpart = nullptr;          // [4 row tiles][sums][N] sums over 32 rows each (1 sum; kBackFirst 6)
  double* losspart = nullptr;        // [4 row tiles][column chunks of 8]
  const float* lnT = nullptr;        // kBackFirst: layer 0's inputs
  const float* b1 = nullptr;
  float norm[6] = {0.f, 1.f, 0.f, 1.f, 1.f, 1.f};
};

// Sums of K columns over a warp's 32 rows by halving exchanges (K + log2(32 / K) - 1
// shuffles); lane l returns the sum of column l K / 32.
template <int K>
__device__ __forceinline__ float warp_columns(float (&v)[K], int lane) {
#pragma unroll
  for (int n = K, off = 16; n > 1; n >>= 1, off >>= 1) {
    const bool up = lane & off;
#pragma unroll
    for (int i = 0; i < n / 2; ++i) {
      const float send = up ? v[i] : v[i + n / 2];
      const float keep = up ? v[i + n / 2] : v[i];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, send, off);
    }
  }
  float t = v[0];
#pragma unroll
  for (int off = 16 / K; off > 0; off >>= 1) t += __shfl_xor_sync(0xffffffffu, t, off);
  return t;
}

// K BF16 values of one row to columns col.. of a row-major matrix with leading dimension ld
// (ld and col are multiples of 8 elements), the columns past ld left out
template <int K>
__device__ __forceinline__ void store_row(__nv_bfloat16* row, int col, int ld, const __nv_bfloat16 (&o)[K]) {
#pragma unroll
  for (int j = 0; j < K; j += 8)
    if (col + j < ld) *reinterpret_cast<uint4*>(row + col + j) = *reinterpret_cast<const uint4*>(o + j);
}

template <int MODE>
__global__ void __launch_bounds__(kPerThreads, 1)
mlp_layer_persistent_kernel(const __grid_constant__ CUtensorMap tx, const __grid_constant__ CUtensorMap tw, int B,
                            int N, int K, const __grid_constant__ LayerIo io, int* __restrict__ err) {
  using namespace tc;
  using PS = PerShape;
  constexpr int BN = PS::BN;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + kPerStages * PS::kStage);
  uint64_t* empty = full + kPerStages;
  uint64_t* accf = empty + kPerStages;
  uint64_t* acce = accf + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acce + 2);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int n_tiles = (N + BN - 1) / BN;
  const int tiles = ((B + BM - 1) / BM) * n_tiles;
  const int nk = (K + BK - 1) / BK;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kPerStages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(&accf[a], 1);
      mbar_init(&acce[a], kPerEpiWarps);  // one arrival per epilogue warp
    }
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) tmem_alloc<PS::kTmemCols>(tmem_slot);
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = *tmem_slot;
  red::pdl_trigger();
  red::pdl_wait();  // the input rows come from the previous launch

  int issued = 0;
  if (warp == 0) {
    if (lane == 0) {
      int g = 0;
      bool go = true;
      for (int t = blockIdx.x; t < tiles && go; t += gridDim.x) {
        const int b0 = (t / n_tiles) * BM, n0 = (t % n_tiles) * BN;
        for (int c = 0; c < nk; ++c, ++g) {
          const int s = g % kPerStages;
          const uint32_t use = (uint32_t)(g / kPerStages);
          if (g >= kPerStages && !mbar_wait(&empty[s], (use - 1) & 1u, abort_flag)) {
            go = false;
            break;
          }
          uint8_t* st = smem + s * PS::kStage;
          mbar_expect_tx(&full[s], PS::kStage);
          tma_load_2d(&tx, &full[s], st, c * BK, b0);
          tma_load_2d(&tx, &full[s], st + PS::kA, c * BK, B + b0);
          tma_load_2d(&tx, &full[s], st + 2 * PS::kA, c * BK, 2 * B + b0);
          tma_load_2d(&tw, &full[s], st + 3 * PS::kA, c * BK, n0);
          issued = g + 1;
        }
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      constexpr uint32_t idesc = make_idesc(BM, BN);
      int g = 0, i = 0;
      bool go = true;
      for (int t = blockIdx.x; t < tiles && go; t += gridDim.x, ++i) {
        const int acc = i & 1;
        if (i >= 2 && !mbar_wait(&acce[acc], (uint32_t)((i >> 1) - 1) & 1u, abort_flag)) break;
        fence_after();
        const uint32_t d = tmem + (uint32_t)(acc * 3 * BN);
        for (int c = 0; c < nk; ++c, ++g) {
          const int s = g % kPerStages;
          if (!mbar_wait(&full[s], (uint32_t)(g / kPerStages) & 1u, abort_flag)) {
            go = false;
            break;
          }
          fence_after();
          const uint8_t* st = smem + s * PS::kStage;
          const uint64_t d0 = sdesc_sw128(st), d1 = sdesc_sw128(st + PS::kA), d2 = sdesc_sw128(st + 2 * PS::kA);
          const uint64_t dw = sdesc_sw128(st + 3 * PS::kA);
#pragma unroll
          for (int k = 0; k < BK / 16; ++k) {
            const uint64_t off = 2ull * k;
            const uint32_t accum = (c > 0 || k > 0) ? 1u : 0u;
            mma_bf16(d, d0 + off, dw + off, idesc, accum);
            mma_bf16(d + BN, d1 + off, dw + off, idesc, accum);
            mma_bf16(d + 2 * BN, d2 + off, dw + off, idesc, accum);
          }
          mma_commit(&empty[s]);
        }
        if (go) mma_commit(&accf[acc]);
      }
    }
  } else {
    const int q = warp & 3;              // TMEM lane quarter of this warp
    // its 16-column chunk of the tile (the output layer in training has at most 32 columns:
    // 8 each, so that all sixteen warps share them)
    constexpr int kCols = MODE == kTrainLast ? 8 : 16;
    const int cb = ((warp - 2) >> 2) * kCols;
    int i = 0;
    for (int t = blockIdx.x; t < tiles; t += gridDim.x, ++i) {
      const int acc = i & 1;
      const int b0 = (t / n_tiles) * BM, n0 = (t % n_tiles) * BN;
      const int b = b0 + q * 32 + lane;  // this lane's row (sample)
      float tg[3][8];  // the targets, loaded while the accumulators are formed
      if constexpr (MODE == kTrainLast) {
#pragma unroll
        for (int k = 0; k < 3; ++k)
#pragma unroll
          for (int j = 0; j < 8; ++j)
            tg[k][j] = b < B && cb + j < N ? io.target[(size_t)(k * N + cb + j) * B + b] : 0.f;
      }
      if (!mbar_wait(&accf[acc], (uint32_t)(i >> 1) & 1u, abort_flag)) break;
      __syncwarp();
      fence_after();
      const uint32_t trow = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(acc * 3 * BN);
      float v0[kCols], v1[kCols], v2[kCols];
      if constexpr (kCols == 16) {
        tmem_ld16(trow + (uint32_t)cb, v0);
        tmem_ld16(trow + (uint32_t)(BN + cb), v1);
        tmem_ld16(trow + (uint32_t)(2 * BN + cb), v2);
      } else {
        tmem_ld8(trow + (uint32_t)cb, v0);
        tmem_ld8(trow + (uint32_t)(BN + cb), v1);
        tmem_ld8(trow + (uint32_t)(2 * BN + cb), v2);
      }
      // this warp's part of the accumulator set is in registers: hand it back
      fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&acce[acc]);
      const int col = n0 + cb;  // this warp's first column
      const bool on = b < B;
      if constexpr (MODE == kInferLast) {
        if (!on) continue;
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          const int r = col + j;
          if (r < N) {
            const float sc = io.scale[r];
            io.pred[(size_t)r * B + b] = sc * (v0[j] + io.bias[r]);
            io.pred[(size_t)(N + r) * B + b] = sc * v1[j];
            io.pred[(size_t)(2 * N + r) * B + b] = sc * v2[j];
          }
        }
      } else if constexpr (MODE == kInferHidden) {
        if (!on) continue;
        __align__(16) __nv_bfloat16 o[3][16];
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          const int n = col + j;
          const float a = tanh_fast(v0[j] + (n < N ? io.bias[n] : 0.f));
          const float dd = 1.f - a * a;
          o[0][j] = __float2bfloat16_rn(a);
          o[1][j] = __float2bfloat16_rn(dd * v1[j]);
          o[2][j] = __float2bfloat16_rn(dd * v2[j]);
        }
#pragma unroll
        for (int k = 0; k < 3; ++k) store_row(io.xn + ((size_t)k * B + b) * io.ldn, col, io.ldn, o[k]);
      } else if constexpr (MODE == kTrainHidden) {
        if (!on) continue;  // N is the hidden width, a multiple of the 64-column tile
        __align__(16) __nv_bfloat16 o[3][16];
        float* za = io.za + (size_t)b * N + col;
        const size_t plane = (size_t)B * N;
#pragma unroll
        for (int g = 0; g < 4; ++g) {
          float av[4];
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int j = 4 * g + i;
            const float a = tanhf(v0[j] + io.bias[col + j]);
            const float d = 1.f - a * a;
            av[i] = a;
            o[0][j] = __float2bfloat16_rn(a);
            o[1][j] = __float2bfloat16_rn(d * v1[j]);
            o[2][j] = __float2bfloat16_rn(d * v2[j]);
          }
          *reinterpret_cast<float4*>(za + 4 * g) = make_float4(av[0], av[1], av[2], av[3]);
          *reinterpret_cast<float4*>(za + plane + 4 * g) = make_float4(v1[4 * g], v1[4 * g + 1], v1[4 * g + 2], v1[4 * g + 3]);
          *reinterpret_cast<float4*>(za + 2 * plane + 4 * g) =
              make_float4(v2[4 * g], v2[4 * g + 1], v2[4 * g + 2], v2[4 * g + 3]);
        }
#pragma unroll
        for (int k = 0; k < 3; ++k) store_row(io.xn + ((size_t)k * B + b) * io.ldn, col, io.ldn, o[k]);
      } else if constexpr (MODE == kTrainLast) {
        // predictions against the targets: the loss, the gradient rows with respect to the
        // output pre-activations and the output bias's column sums
        if (col >= N) continue;  // the same in every lane of the warp
        __align__(16) __nv_bfloat16 o[3][8];
        // the loss terms' sums, values and tangents, in float64 for its precision and range (3 us
        // of 174 at 4096 samples, three conversions and multiply-adds per output)
        double acc = 0.0, acct = 0.0;
        const float inv = 2.f / (float)B;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          float g0 = 0.f, g1 = 0.f, g2 = 0.f;
          if (col + j < N && on) {
            const float sc = io.scale[col + j];
            const float r0 = v0[j] + io.bias[col + j] - tg[0][j] / sc;
            const float r1 = v1[j] - tg[1][j] / sc;
            const float r2 = v2[j] - tg[2][j] / sc;
            acc = fma((double)r0, (double)r0, acc);
            acct = fma((double)r1, (double)r1, acct);
            acct = fma((double)r2, (double)r2, acct);
            g0 = inv * r0;
            g1 = inv * io.lam * r1;
            g2 = inv * io.lam * r2;
          }
          o[0][j] = __float2bfloat16_rn(g0);
          o[1][j] = __float2bfloat16_rn(g1);
          o[2][j] = __float2bfloat16_rn(g2);
          v0[j] = g0;
        }
        if (on) {
#pragma unroll
          for (int k = 0; k < 3; ++k) store_row(io.xn + ((size_t)k * B + b) * io.ldn, col, io.ldn, o[k]);
        }
        const size_t prow = (size_t)(b0 / BM) * 4 + q;
        const float sum = warp_columns(v0, lane);
        if ((lane & 3) == 0 && col + (lane >> 2) < N) io.colpart[prow * N + col + (lane >> 2)] = sum;
        acc = fma((double)io.lam, acct, acc);
#pragma unroll
        for (int of = 16; of > 0; of >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, of);
        if (lane == 0) io.losspart[prow * ((N + 7) / 8) + (col >> 3)] = acc;
      } else {
        // kBack, kBackFirst: v0, v1, v2 = dL/d(a, s1, s2) of a tanh layer
        __align__(16) __nv_bfloat16 o[3][16];
        const float* za = io.za + (size_t)(on ? b : 0) * N + col;
        const size_t plane = (size_t)B * N;
#pragma unroll
        for (int g = 0; g < 4; ++g) {
          const float4 a4 = *reinterpret_cast<const float4*>(za + 4 * g);
          const float4 p4 = *reinterpret_cast<const float4*>(za + plane + 4 * g);
          const float4 q4 = *reinterpret_cast<const float4*>(za + 2 * plane + 4 * g);
          const float av[4] = {a4.x, a4.y, a4.z, a4.w}, zv1[4] = {p4.x, p4.y, p4.z, p4.w},
                      zv2[4] = {q4.x, q4.y, q4.z, q4.w};
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int j = 4 * g + i;
            const float a = av[i], z1 = zv1[i], z2 = zv2[i];
            const float d = 1.f - a * a;
            const float ga = v0[j], g1 = v1[j], g2 = v2[j];
            const float gz1 = g1 * d, gz2 = g2 * d;
            const float gz = (ga - 2.f * a * (g1 * z1 + g2 * z2)) * d;
            o[0][j] = __float2bfloat16_rn(gz);
            o[1][j] = __float2bfloat16_rn(gz1);
            o[2][j] = __float2bfloat16_rn(gz2);
            v0[j] = on ? gz : 0.f;
          }
        }
        const size_t prow = (size_t)(b0 / BM) * 4 + q;
        constexpr int kSums = MODE == kBackFirst ? 6 : 1;
        float* cp = io.colpart + prow * kSums * N + col + (lane >> 1);
        const float sum = warp_columns(v0, lane);
        if ((lane & 1) == 0) cp[0] = sum;
        if constexpr (MODE == kBack) {
          if (on) {
#pragma unroll
            for (int k = 0; k < 3; ++k) store_row(io.xn + ((size_t)k * B + b) * io.ldn, col, io.ldn, o[k]);
          }
        } else {
          // layer 0's weight gradient: its inputs are three columns, so the sums over the
          // BF16 gradient rows times the BF16 inputs are formed here
          float u[3] = {0.f, 0.f, 0.f};
          if (on) {
            const float bb = io.b1 != nullptr ? io.b1[b] : 1.f;
            u[0] = __bfloat162float(__float2bfloat16_rn((io.lnT[b] - io.norm[0]) / io.norm[1]));
            u[1] = __bfloat162float(__float2bfloat16_rn((io.lnT[B + b] - io.norm[2]) / io.norm[3]));
            u[2] = __bfloat162float(__float2bfloat16_rn((bb - io.norm[4]) / io.norm[5]));
          }
#pragma unroll
          for (int k = 0; k < 5; ++k) {
#pragma unroll
            for (int j = 0; j < 16; ++j) {
              if (k < 3) v0[j] = __bfloat162float(o[0][j]) * u[k];
              else v0[j] = on ? __bfloat162float(o[k - 2][j]) : 0.f;
            }
            const float t = warp_columns(v0, lane);
            if ((lane & 1) == 0) cp[(size_t)(k + 1) * N] = t;
          }
        }
      }
    }
  }

  __syncwarp();
  if (threadIdx.x == 0 && *abort_flag) {
    atomicExch(err, 1);
    // let the copies this thread issued land before the CTA's shared memory goes away
    for (int g = issued > kPerStages ? issued - kPerStages : 0; g < issued; ++g) {
      int spins = 0;
      while (!mbar_try_wait(&full[g % kPerStages], (uint32_t)(g / kPerStages) & 1u) && ++spins < (1 << 16)) {
      }
    }
  }
  fence_before();
  __syncthreads();
  if (warp == 0) tmem_dealloc<PS::kTmemCols>(tmem);
}

// ---------------------------------------------------------------------------
// Weight gradient dW_l = GZ_l^T X_l of one layer (l = 1..3) over the 3B gradient and input
// rows: one CTA per 128 x 64 tile.  Both operands are read as they were written (rows = the
// GEMM's K): MN-major tiles of 64 rows, so no transposed copies exist.  Bound by the chain
// of dependent MMAs over the rows, about 75 ns per 16 rows at any tile size: 57 us at 4096
// samples (108 us from transposed K-major copies, 64-row chunks of 32 KB); the tensor pipe is
// active on 23 % of its SMs' cycles.  The rows are not split over CTAs by choice, not by need:
// a trial with sixteen parts took 13 us, but the tensor core's float32 accumulation rounds
// towards zero, so shorter chains change a gradient by 3e-5 relative (its error against
// float64 is 1e-3, from the BF16 operands).  The launch uses few SMs (8 at H = 256), so the
// three layers' gradients run on streams of their own beside the backward layers.
// ---------------------------------------------------------------------------
constexpr int kDwN = 64;                             // columns of a tile
constexpr int kDwStages = 8;
constexpr uint32_t kDwBox = 64 * tc::BK * 2;         // 64 rows x 64 columns
constexpr uint32_t kDwStage = 3 * kDwBox;            // two boxes of GZ, one of X
constexpr size_t kDwSmem = (size_t)kDwStages * kDwStage + 1024 + 256;

__global__ void __launch_bounds__(128, 1)
mlp_dw_kernel(const __grid_constant__ CUtensorMap tgz, const __grid_constant__ CUtensorMap tx, int rows, int out,
              int in, float* __restrict__ grad, int* __restrict__ err) {
  using namespace tc;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + kDwStages * kDwStage);
  uint64_t* empty = full + kDwStages;
  uint64_t* done = empty + kDwStages;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nt = in / kDwN;  // in is the hidden width, a multiple of 64
  const int m0 = (blockIdx.x / nt) * BM, n0 = (blockIdx.x % nt) * kDwN;
  const int nk = (rows + BK - 1) / BK;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kDwStages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    mbar_init(done, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) tmem_alloc<64>(tmem_slot);
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = *tmem_slot;

  int issued = 0;
  if (warp == 0 && lane == 0) {
    for (int g = 0; g < nk; ++g) {
      const int s = g % kDwStages;
      if (g >= kDwStages && !mbar_wait(&empty[s], (uint32_t)(g / kDwStages - 1) & 1u, abort_flag)) break;
      uint8_t* st = smem + s * kDwStage;
      mbar_expect_tx(&full[s], kDwStage);
      tma_load_2d(&tgz, &full[s], st, m0, g * BK);
      tma_load_2d(&tgz, &full[s], st + kDwBox, m0 + 64, g * BK);
      tma_load_2d(&tx, &full[s], st + 2 * kDwBox, n0, g * BK);
      issued = g + 1;
    }
  } else if (warp == 1 && lane == 0) {
    constexpr uint32_t idesc = make_idesc(BM, kDwN) | kIdescMnMajorA | kIdescMnMajorB;
    for (int g = 0; g < nk; ++g) {
      const int s = g % kDwStages;
      if (!mbar_wait(&full[s], (uint32_t)(g / kDwStages) & 1u, abort_flag)) break;
      fence_after();
      const uint8_t* st = smem + s * kDwStage;
      const uint64_t da = sdesc_sw128_mn(st, kDwBox), db = sdesc_sw128_mn(st + 2 * kDwBox, kDwBox);
#pragma unroll
      for (int k = 0; k < BK / 16; ++k)  // 16 rows of 128 bytes, in 16-byte units
        mma_bf16(tmem, da + 128ull * k, db + 128ull * k, idesc, (g > 0 || k > 0) ? 1u : 0u);
      mma_commit(&empty[s]);
    }
    mma_commit(done);
  }
  __syncwarp();
  const bool ok = mbar_wait(done, 0, abort_flag) && *abort_flag == 0;
  __syncwarp();
  fence_after();
  if (ok) {
    const int o = m0 + warp * 32 + lane;
    float* dst = grad + (int64_t)o * in + n0;
#pragma unroll
    for (int cb = 0; cb < kDwN; cb += 16) {
      float v[16];
      tmem_ld16(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)cb, v);
      if (o < out) {
#pragma unroll
        for (int j = 0; j < 16; j += 4)
          *reinterpret_cast<float4*>(dst + cb + j) = make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]);
      }
    }
  } else if (threadIdx.x == 0) {
    atomicExch(err, 1);
    // let the copies this thread issued land before the CTA's shared memory goes away
    for (int g = issued > kDwStages ? issued - kDwStages : 0; g < issued; ++g) {
      int spins = 0;
      while (!mbar_try_wait(&full[g % kDwStages], (uint32_t)(g / kDwStages) & 1u) && ++spins < (1 << 16)) {
      }
    }
  }
  fence_before();
  __syncthreads();
  if (warp == 0) tmem_dealloc<64>(tmem);
}

// The biases' and layer 0's gradient from the row tiles' column sums, in a fixed order (32
// columns per block, the tiles split over its warps: latency, not bytes, bounds it), and the loss (last block).
constexpr int kSumWarps = 16;
__global__ void __launch_bounds__(32 * kSumWarps)
mlp_grad_sum_kernel(const float* __restrict__ cp0, const float* __restrict__ cp1, const float* __restrict__ cp2,
                    const float* __restrict__ cp3, const double* __restrict__ losspart, int nloss, int prows, int H,
                    int R, int B, float d1, float d2, float* __restrict__ grad, double* __restrict__ loss) {
  const int64_t off1 = 4 * (int64_t)H, off2 = off1 + (int64_t)H * H + H, off3 = off2 + (int64_t)H * H + H;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  red::pdl_wait();
  __shared__ float ws[kSumWarps][6][32];
  if (blockIdx.x == gridDim.x - 1) {
    __shared__ double wd[kSumWarps];
    double s = 0.0;
    for (int i = threadIdx.x; i < nloss; i += 32 * kSumWarps) s += losspart[i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) wd[warp] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
      for (int k = 1; k < kSumWarps; ++k) s += wd[k];
      *loss = s / (double)B;
    }
    return;
  }
  const int c = blockIdx.x * 32 + lane;  // column: layer 0, 1, 2 (H each), 3 (R)
  const int l = c / H, n = c - l * H;
  const bool in = l < 3 || (l == 3 && n < R);
  const float* cp = l == 0 ? cp0 : l == 1 ? cp1 : l == 2 ? cp2 : cp3;
  const int sums = l == 0 ? 6 : 1, ld = l == 3 ? R : H;
  float s[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  if (in) {
#pragma unroll 4
    for (int p = warp; p < prows; p += kSumWarps)
#pragma unroll
      for (int k = 0; k < 6; ++k)
        if (k < sums) s[k] += cp[((size_t)p * sums + k) * ld + n];
  }
#pragma unroll
  for (int k = 0; k < 6; ++k) ws[warp][k][lane] = s[k];
  __syncthreads();
  if (warp != 0 || !in) return;
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    s[k] = 0.f;
#pragma unroll
    for (int w = 0; w < kSumWarps; ++w) s[k] += ws[w][k][lane];
  }
  if (l == 0) {
    grad[3 * H + n] = s[0];
    grad[3 * n] = fmaf(d1, s[4], s[1]);
    grad[3 * n + 1] = fmaf(d2, s[5], s[2]);
    grad[3 * n + 2] = s[3];
  } else {
    grad[l == 1 ? off2 - H + n : l == 2 ? off3 - H + n : off3 + (int64_t)R * H + n] = s[0];
  }
}

int blocks_for(int64_t n, int t = 256) {
  int64_t b = (n + t - 1) / t;
  return (int)(b < 1 ? 1 : (b > 8192 ? 8192 : b));
}

}  // namespace

// ---------------------------------------------------------------------------
Mlp::~Mlp() {
  release_batch();
  free_weights();
  if (stat) cudaFree(stat);
  if (stat_host) cudaFreeHost(stat_host);
  for (int k = 0; k < 3; ++k) {
    if (side[k]) cudaStreamDestroy(side[k]);
    if (ev_fork[k]) cudaEventDestroy(ev_fork[k]);
    if (ev_join[k]) cudaEventDestroy(ev_join[k]);
  }
}

void Mlp::free_weights() {
  void* ptrs[] = {theta, adam_m, adam_v, grad, scale_dev};
  for (void* q : ptrs)
    if (q) cudaFree(q);
  for (int l = 0; l < 4; ++l) {
    if (Wb[l]) cudaFree(Wb[l]);
    if (WTb[l]) cudaFree(WTb[l]);
    Wb[l] = WTb[l] = nullptr;
  }
  theta = adam_m = adam_v = grad = scale_dev = nullptr;
}

void Mlp::release_batch() {
  for (int l = 0; l < 4; ++l) {
    void* ptrs[] = {X[l], ZA[l], GZ[l], colpart[l]};
    for (void* q : ptrs)
      if (q) cudaFree(q);
    X[l] = GZ[l] = nullptr;
    ZA[l] = colpart[l] = nullptr;
  }
  if (losspart) cudaFree(losspart);
  losspart = nullptr;
  cap = 0;
  maps_b = -1;
}

int Mlp::setup(int h, int r, uint64_t seed) {
  H = h;
  R = r;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device) != cudaSuccess || sms < 1) sms = 1;
  const int dims[5] = {3, H, H, H, R};
  np = 0;
  for (int l = 0; l < 4; ++l) {
    in[l] = dims[l];
    out[l] = dims[l + 1];
    off[l] = np;
    np += (int64_t)out[l] * in[l] + out[l];
  }
  cudaError_t e = cudaSuccess;
  auto chk = [&](cudaError_t q) {
    if (e == cudaSuccess) e = q;
  };
  chk(cudaMalloc(&theta, np * sizeof(float)));
  chk(cudaMalloc(&adam_m, np * sizeof(float)));
  chk(cudaMalloc(&adam_v, np * sizeof(float)));
  chk(cudaMalloc(&grad, np * sizeof(float)));
  chk(cudaMalloc(&scale_dev, R * sizeof(float)));
  chk(cudaMalloc(&stat, 2 * sizeof(double)));
  chk(cudaMallocHost(&stat_host, 2 * sizeof(double)));
  if (e == cudaSuccess) chk(cudaMemset(stat, 0, 2 * sizeof(double)));
  for (int k = 0; k < 3; ++k) {
    chk(cudaStreamCreateWithFlags(&side[k], cudaStreamNonBlocking));
    chk(cudaEventCreateWithFlags(&ev_fork[k], cudaEventDisableTiming));
    chk(cudaEventCreateWithFlags(&ev_join[k], cudaEventDisableTiming));
  }
  loss_dev = stat;
  dev_err = reinterpret_cast<int*>(stat + 1);
  for (int l = 0; l < 4; ++l) {
    chk(cudaMalloc(&Wb[l], (size_t)out[l] * pad8(in[l]) * 2));
    chk(cudaMalloc(&WTb[l], (size_t)in[l] * pad8(out[l]) * 2));
    if (e == cudaSuccess) {
      chk(cudaMemset(Wb[l], 0, (size_t)out[l] * pad8(in[l]) * 2));
      chk(cudaMemset(WTb[l], 0, (size_t)in[l] * pad8(out[l]) * 2));
      chk(make_bf16_tmap(&wmap64[l], Wb[l], out[l], in[l], pad8(in[l]), PerShape::BN));
      chk(make_bf16_tmap(&wtmap64[l], WTb[l], in[l], out[l], pad8(out[l]), PerShape::BN));
    }
  }
  if (e != cudaSuccess) return cuda_fail(e, "surrogate allocation");
  // Glorot-uniform weights, zero biases, unit output scale
  std::vector<float> th(np, 0.f), sc(R, 1.f);
  std::mt19937_64 rng(seed);
  for (int l = 0; l < 4; ++l) {
    const float lim = std::sqrt(6.f / (float)(in[l] + out[l]));
    std::uniform_real_distribution<float> U(-lim, lim);
    for (int64_t k = 0; k < (int64_t)out[l] * in[l]; ++k) th[off[l] + k] = U(rng);
  }
  chk(cudaMemcpy(scale_dev, sc.data(), R * sizeof(float), cudaMemcpyHostToDevice));
  scale_host = sc;
  chk(cudaMemset(adam_m, 0, np * sizeof(float)));
  chk(cudaMemset(adam_v, 0, np * sizeof(float)));
  if (e != cudaSuccess) return cuda_fail(e, "surrogate init");
  return set_params(th.data(), nullptr);
}

int Mlp::set_params(const float* host, cudaStream_t st) {
  cudaError_t e = cudaMemcpy(theta, host, np * sizeof(float), cudaMemcpyHostToDevice);
  for (int l = 0; l < 4 && e == cudaSuccess; ++l) {
    mlp_cast_kernel<<<blocks_for((int64_t)out[l] * in[l]), 256, 0, st>>>(theta + off[l], out[l], in[l], Wb[l],
                                                                        pad8(in[l]), WTb[l], pad8(out[l]));
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  step = 0;
  return e == cudaSuccess ? MRSTAT_OK : cuda_fail(e, "surrogate parameters");
}

// (re)allocates the activation buffers for up to B samples and encodes the tensor maps
int Mlp::ensure_batch(int B, bool train) {
  if (B > cap || (train && !have_train_buffers)) {
    release_batch();
    const int Mc = 3 * B;
    const size_t prows = 4 * (size_t)((B + tc::BM - 1) / tc::BM);
    cudaError_t e = cudaSuccess;
    auto chk = [&](cudaError_t q) {
      if (e == cudaSuccess) e = q;
    };
    for (int l = 0; l < 4; ++l) {
      chk(cudaMalloc(&X[l], (size_t)Mc * pad8(in[l]) * 2));
      if (train) {
        if (l < 3) chk(cudaMalloc(&ZA[l], (size_t)Mc * out[l] * sizeof(float)));
        if (l > 0) chk(cudaMalloc(&GZ[l], (size_t)Mc * pad8(out[l]) * 2));
        chk(cudaMalloc(&colpart[l], prows * (l == 0 ? 6 : 1) * out[l] * sizeof(float)));
      }
    }
    if (train) {
      chk(cudaMalloc(&losspart, prows * ((R + 7) / 8) * sizeof(double)));
    }
    for (int l = 0; l < 4 && e == cudaSuccess; ++l) {
      chk(cudaMemset(X[l], 0, (size_t)Mc * pad8(in[l]) * 2));
      if (train && l > 0) chk(cudaMemset(GZ[l], 0, (size_t)Mc * pad8(out[l]) * 2));
    }
    if (e != cudaSuccess) {
      release_batch();
      return cuda_fail(e, "surrogate batch buffers");
    }
    cap = B;
    have_train_buffers = train;
  }
  if (maps_b != B || maps_train != train) {
    const int Mc = 3 * B;
    cudaError_t e = cudaSuccess;
    for (int l = 0; l < 4 && e == cudaSuccess; ++l) {
      e = make_bf16_tmap(&xmap[l], X[l], Mc, in[l], pad8(in[l]), tc::BM);
      if (!train || l == 0) continue;
      if (e == cudaSuccess) e = make_bf16_tmap(&gzmap[l], GZ[l], Mc, out[l], pad8(out[l]), tc::BM);
      // 64-row boxes, the rows as the GEMM's K (the weight gradients)
      if (e == cudaSuccess) e = make_bf16_tmap(&xmap_k[l], X[l], Mc, in[l], pad8(in[l]), tc::BK);
      if (e == cudaSuccess) e = make_bf16_tmap(&gzmap_k[l], GZ[l], Mc, out[l], pad8(out[l]), tc::BK);
    }
    if (e != cudaSuccess) return cuda_fail(e, "surrogate tensor maps");
    maps_b = B;
    maps_train = train;
  }
  return MRSTAT_OK;
}

template <int MODE>
static cudaError_t launch_layer(const CUtensorMap& x, const CUtensorMap& w, int B, int N, int K, const LayerIo& io,
                                int sms, int* err, cudaStream_t st) {
  const size_t sm = PerShape::kSmem;
  cudaError_t e = cudaFuncSetAttribute(mlp_layer_persistent_kernel<MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)sm);
  if (e != cudaSuccess) return e;
  const int tiles = ((B + tc::BM - 1) / tc::BM) * ((N + PerShape::BN - 1) / PerShape::BN);
  // programmatic dependent launch: the set-up overlaps the previous layer's tail
  return launch_pdl(mlp_layer_persistent_kernel<MODE>, dim3(std::max(1, std::min(tiles, sms))), dim3(kPerThreads), sm, st,
                    x, w, B, N, K, io, err);
}

// Loss and gradient of one batch into loss_dev and grad: the input rows, four forward
// layers (the last with the loss), three backward layers, the weight gradients and the sums.
int Mlp::loss_gradient(const float* lnT, const float* b1, const float* target, int B, cudaStream_t st) {
  mlp_input_kernel<<<blocks_for(B), 256, 0, st>>>(lnT, b1, B, norm[0], norm[1], norm[2], norm[3], norm[4], norm[5],
                                                  X[0]);
  cudaError_t e = cudaGetLastError();
  LayerIo io;
  io.scale = scale_dev;
  io.target = target;
  io.lam = lam;
  io.losspart = losspart;
  io.lnT = lnT;
  io.b1 = b1;
  for (int k = 0; k < 6; ++k) io.norm[k] = norm[k];
  for (int l = 0; l < 4 && e == cudaSuccess; ++l) {
    io.bias = theta + off[l] + (int64_t)out[l] * in[l];
    io.za = ZA[l];
    io.xn = l < 3 ? X[l + 1] : GZ[3];
    io.ldn = l < 3 ? pad8(in[l + 1]) : pad8(out[3]);
    io.colpart = colpart[l];
    e = l < 3 ? launch_layer<kTrainHidden>(xmap[l], wmap64[l], B, out[l], in[l], io, sms, dev_err, st)
              : launch_layer<kTrainLast>(xmap[l], wmap64[l], B, out[l], in[l], io, sms, dev_err, st);
  }
  // dL/dX_l = GZ_l W_l, then back through layer l - 1's tanh.  dW_3 and dW_2 run on streams
  // of their own as soon as their gradient rows stand, dW_1 on the caller's beside the last
  // backward layer (side 2); everything is joined below.
  auto dw = [&](int l, cudaStream_t s) {
    const int tiles = ((out[l] + tc::BM - 1) / tc::BM) * (in[l] / kDwN);
    mlp_dw_kernel<<<tiles, 128, kDwSmem, s>>>(gzmap_k[l], xmap_k[l], 3 * B, out[l], in[l], grad + off[l], dev_err);
    return cudaGetLastError();
  };
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(mlp_dw_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kDwSmem);
  int forked = 0;  // side streams with work on them
  auto fork = [&](int k) {
    cudaError_t r = cudaEventRecord(ev_fork[k], st);
    if (r == cudaSuccess) r = cudaStreamWaitEvent(side[k], ev_fork[k], 0);
    if (r == cudaSuccess) forked = k + 1;
    return r;
  };
  for (int l = 3; l > 0 && e == cudaSuccess; --l) {
    const int lp = l - 1;
    io.za = ZA[lp];
    io.xn = GZ[lp];  // not kept for layer 0
    io.ldn = pad8(out[lp]);
    io.colpart = colpart[lp];
    e = fork(3 - l);
    if (e != cudaSuccess) break;
    if (lp > 0) {
      e = dw(l, side[3 - l]);
      if (e == cudaSuccess)
        e = launch_layer<kBack>(gzmap[l], wtmap64[l], B, in[l], out[l], io, sms, dev_err, st);
    } else {
      e = launch_layer<kBackFirst>(gzmap[l], wtmap64[l], B, in[l], out[l], io, sms, dev_err, side[2]);
      if (e == cudaSuccess) {
        // layer 0's tangent inputs as the GEMM operand holds them
        const float d1 = host_bf16_to_float(host_bf16(1.f / norm[1]));
        const float d2 = host_bf16_to_float(host_bf16(1.f / norm[3]));
        const int prows = 4 * ((B + tc::BM - 1) / tc::BM);
        e = launch_pdl(mlp_grad_sum_kernel, dim3((3 * H + R + 31) / 32 + 1), dim3(32 * kSumWarps), 0, side[2],
                       colpart[0], colpart[1], colpart[2], colpart[3], losspart, prows * ((R + 7) / 8), prows, H, R, B,
                       d1, d2, grad, loss_dev);
      }
      if (e == cudaSuccess) e = dw(1, st);
    }
  }
  // join, also after an error: the caller's stream owns the buffers
  for (int k = 0; k < forked; ++k) {
    cudaError_t r = cudaEventRecord(ev_join[k], side[k]);
    if (r == cudaSuccess) r = cudaStreamWaitEvent(st, ev_join[k], 0);
    if (e == cudaSuccess) e = r;
  }
  return e == cudaSuccess ? MRSTAT_OK : cuda_fail(e, "surrogate gradient");
}

int Mlp::adam(float lr, cudaStream_t st) {
  ++step;
  const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
  const float c1 = 1.f - std::pow(b1, (float)step), c2 = 1.f - std::pow(b2, (float)step);
  cudaError_t e = cudaSuccess;
  for (int l = 0; l < 4 && e == cudaSuccess; ++l) {
    mlp_adam_kernel<<<blocks_for((int64_t)out[l] * in[l] + out[l]), 256, 0, st>>>(
        theta + off[l], adam_m + off[l], adam_v + off[l], grad + off[l], out[l], in[l], lr, b1, b2, eps, c1, c2, Wb[l],
        pad8(in[l]), WTb[l], pad8(out[l]));
    e = cudaGetLastError();
  }
  return e == cudaSuccess ? MRSTAT_OK : cuda_fail(e, "surrogate Adam step");
}


// Inference: layer 0 on the CUDA cores, then one persistent fused tensor-core kernel per
// layer (no pre-activation buffers).
int Mlp::infer_fused(const float* lnT, const float* b1, int B, float* pred, cudaStream_t st) {
  {
    const int groups = out[0] / 8;  // hidden width 64, 128 or 256
    mlp_first_layer_kernel<<<blocks_for((int64_t)B * groups), 256, 0, st>>>(
        lnT, b1, B, norm[0], norm[1], norm[2], norm[3], norm[4], norm[5], Wb[0], pad8(in[0]),
        theta + off[0] + (int64_t)out[0] * in[0], out[0], X[1], pad8(in[1]));
  }
  cudaError_t e = cudaGetLastError();
  LayerIo io;
  io.scale = scale_dev;
  io.pred = pred;
  for (int l = 1; l < 4 && e == cudaSuccess; ++l) {
    io.bias = theta + off[l] + (int64_t)out[l] * in[l];
    io.xn = l < 3 ? X[l + 1] : nullptr;
    io.ldn = l < 3 ? pad8(in[l + 1]) : 0;
    e = l < 3 ? launch_layer<kInferHidden>(xmap[l], wmap64[l], B, out[l], in[l], io, sms, dev_err, st)
              : launch_layer<kInferLast>(xmap[l], wmap64[l], B, out[l], in[l], io, sms, dev_err, st);
  }
  return e == cudaSuccess ? MRSTAT_OK : cuda_fail(e, "surrogate inference");
}

int mlp_infer(Mlp* m, const float* lnT, const float* b1, int n, float* coef, cudaStream_t st) {
  int s = m->ensure_batch(n, false);
  if (s == MRSTAT_OK) s = m->infer_fused(lnT, b1, n, coef, st);
  return s;
}

}  // namespace mrstat

// ---------------------------------------------------------------------------
// C entry points
// ---------------------------------------------------------------------------
using namespace mrstat;

struct mrstat_mlp : public Mlp {};

extern "C" {

int mrstat_mlp_create(const mrstat_mlp_config* cfg, mrstat_mlp** out) {
  if (out == nullptr || cfg == nullptr) return fail(MRSTAT_ERR_INVALID_ARG, "NULL config or out");
  *out = nullptr;
  if ((cfg->hidden != 64 && cfg->hidden != 128 && cfg->hidden != 256) || cfg->rank < 1 || cfg->rank > kMaxRank)
    return fail(MRSTAT_ERR_INVALID_ARG, "hidden %d (64, 128 or 256) or rank %d (1..32) not supported", cfg->hidden,
                cfg->rank);
  for (int k = 1; k < 6; k += 2)
    if (!(cfg->norm[k] > 0)) return fail(MRSTAT_ERR_INVALID_ARG, "normalisation scales must be positive");
  mrstat_mlp* m = new mrstat_mlp();
  if (cudaGetDevice(&m->device) != cudaSuccess) {
    delete m;
    return fail(MRSTAT_ERR_CUDA, "no CUDA device");
  }
  for (int k = 0; k < 6; ++k) m->norm[k] = cfg->norm[k];
  m->lam = cfg->sobolev_weight;
  const int s = m->setup(cfg->hidden, cfg->rank, cfg->seed);
  if (s != MRSTAT_OK) {
    delete m;
    return s;
  }
  *out = m;
  return MRSTAT_OK;
}

int mrstat_mlp_destroy(mrstat_mlp* m) {
  if (m == nullptr) return MRSTAT_OK;
  DeviceGuard g(m->device);
  cudaDeviceSynchronize();
  delete m;
  return MRSTAT_OK;
}

int64_t mrstat_mlp_num_params(const mrstat_mlp* m) { return m ? m->np : 0; }

int mrstat_mlp_set_output_scale(mrstat_mlp* m, const float* scale) {
  if (m == nullptr || scale == nullptr) return fail(MRSTAT_ERR_INVALID_ARG, "NULL argument");
  for (int r = 0; r < m->R; ++r)
    if (!(scale[r] > 0)) return fail(MRSTAT_ERR_INVALID_ARG, "output scales must be positive");
  DeviceGuard g(m->device);
  m->scale_host.assign(scale, scale + m->R);
  cudaError_t e = cudaMemcpy(m->scale_dev, scale, m->R * sizeof(float), cudaMemcpyHostToDevice);
  return e == cudaSuccess ? MRSTAT_OK : cuda_fail(e, "output scale");
}

int mrstat_mlp_get_params(mrstat_mlp* m, float* host) {
  if (m == nullptr || host == nullptr) return fail(MRSTAT_ERR_INVALID_ARG, "NULL argument");
  DeviceGuard g(m->device);
  cudaError_t e = cudaDeviceSynchronize();
  if (e == cudaSuccess) e = cudaMemcpy(host, m->theta, m->np * sizeof(float), cudaMemcpyDeviceToHost);
  return e == cudaSuccess ? MRSTAT_OK : cuda_fail(e, "get parameters");
}

int mrstat_mlp_set_params(mrstat_mlp* m, const float* host) {
  if (m == nullptr || host == nullptr) return fail(MRSTAT_ERR_INVALID_ARG, "NULL argument");
  DeviceGuard g(m->device);
  cudaDeviceSynchronize();
  return m->set_params(host, nullptr);
}

int mrstat_mlp_infer(mrstat_mlp* m, const float* lnT, const float* b1, int32_t n, float* coef, void* stream) {
  MRSTAT_ABI_RANGE();
  if (m == nullptr || lnT == nullptr || coef == nullptr || n < 1)
    return fail(MRSTAT_ERR_INVALID_ARG, "bad argument to mrstat_mlp_infer");
  DeviceGuard g(m->device);
  return mlp_infer(m, lnT, b1, n, coef, reinterpret_cast<cudaStream_t>(stream));
}

int mrstat_mlp_train_step(mrstat_mlp* m, const float* lnT, const float* b1, const float* target, int32_t B, float lr,
                          double* loss_out, void* stream) {
  MRSTAT_ABI_RANGE();
  if (m == nullptr || lnT == nullptr || target == nullptr || B < 1 || !(lr >= 0))
    return fail(MRSTAT_ERR_INVALID_ARG, "bad argument to mrstat_mlp_train_step");
  DeviceGuard g(m->device);
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  int s = m->ensure_batch(B, true);
  if (s == MRSTAT_OK) s = m->loss_gradient(lnT, b1, target, B, st);
  if (s == MRSTAT_OK && lr > 0) s = m->adam(lr, st);
  if (s == MRSTAT_OK && loss_out != nullptr) {
    cudaError_t e = cudaMemcpyAsync(loss_out, m->loss_dev, sizeof(double), cudaMemcpyDeviceToDevice, st);
    if (e != cudaSuccess) s = cuda_fail(e, "loss copy");
  }
  return s;
}

int mrstat_mlp_loss_grad(mrstat_mlp* m, const float* lnT, const float* b1, const float* target, int32_t B,
                         double* loss_host, float* grad, void* stream) {
  MRSTAT_ABI_RANGE();
  if (m == nullptr || lnT == nullptr || target == nullptr || B < 1)
    return fail(MRSTAT_ERR_INVALID_ARG, "bad argument to mrstat_mlp_loss_grad");
  DeviceGuard g(m->device);
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  int s = m->ensure_batch(B, true);
  if (s == MRSTAT_OK) s = m->loss_gradient(lnT, b1, target, B, st);
  if (s != MRSTAT_OK) return s;
  cudaError_t e = cudaSuccess;
  if (grad) e = cudaMemcpyAsync(grad, m->grad, m->np * sizeof(float), cudaMemcpyDeviceToDevice, st);
  // the loss and the error flag in one copy and one wait
  if (e == cudaSuccess) e = cudaMemcpyAsync(m->stat_host, m->stat, 2 * sizeof(double), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return cuda_fail(e, "surrogate gradient");
  if (loss_host) *loss_host = m->stat_host[0];
  int herr = 0;
  std::memcpy(&herr, m->stat_host + 1, sizeof(int));
  if (herr) {
    cudaMemset(m->dev_err, 0, sizeof(int));
    return fail(MRSTAT_ERR_TIMEOUT, "a tensor-core kernel gave up waiting on its pipeline barriers");
  }
  return MRSTAT_OK;
}

}  // extern "C"
