// Point-wise MLP of the learned density warm start (not in the paper): 9
// features per interface node -- the history projection psi_F, its residual
// r_F and the right-hand side g^n, each divided by its root mean square over
// the nodes, then the node and its unit normal -- through 4 hidden layers of
// width 128 with SiLU to one output o; the initial density is
// psi_L = psi_F + 2 gamma r_F + rms(r_F) (s_out o + m_out).  bfloat16 weights
// and activations, float32 accumulation on the tensor cores (wmma bf16
// 16x16x16 fragments), float32 master weights with Adam.  The network only
// supplies GMRES's initial guess; the solver tolerance still fixes the
// converged density.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <mma.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "internal.cuh"

using bf16 = __nv_bfloat16;

namespace kfbi {
namespace {

constexpr int NIN = 9, KIN = 16, WID = 128, NL = 5;  // 4 hidden + output
constexpr int TILE = 64;

struct Offsets {
  size_t w[NL], b[NL], total;
  Offsets() {
    const int in[NL] = {NIN, WID, WID, WID, WID};
    const int out[NL] = {WID, WID, WID, WID, 1};
    size_t o = 0;
    for (int l = 0; l < NL; ++l) {
      w[l] = o;
      o += (size_t)in[l] * out[l];
      b[l] = o;
      o += out[l];
    }
    total = o;
  }
};

__device__ __forceinline__ float silu_f(float z) { return z / (1.0f + expf(-z)); }
__device__ __forceinline__ float dsilu_f(float z) {
  const float s = 1.0f / (1.0f + expf(-z));
  return s * (1.0f + z * (1.0f - s));
}

// Weight gradients dW_l += d_l^T A_{l-1} of the four hidden layers in one
// launch (bf16 operands, float32 accumulation and atomics; A_{-1} = X).  A
// block owns a 64 x 64 tile of one layer's product over `kch` rows: the row
// sum is a serial chain of 16-row products, so it is split into about one
// block per SM and layer (16 blocks of 1024 rows each took 107 us a layer at
// 4096 rows).
struct WeightGrad {
  const bf16 *d[4], *A[4];  // delta [Bp][128], activation [Bp][lda]
  float* g[4];              // [128][n]
};
__global__ void __launch_bounds__(128) k_weight_grad(WeightGrad P, int K, int kch, int splits) {
  using namespace nvcuda;
  const int l = blockIdx.z / splits, split = blockIdx.z % splits;
  const int lda = l == 0 ? KIN : WID, n = l == 0 ? NIN : WID, N = l == 0 ? KIN : WID;
  const int warp = threadIdx.x >> 5, wy = warp >> 1, wx = warp & 1;
  const int m0 = blockIdx.y * TILE + wy * 32, n0 = blockIdx.x * TILE + wx * 32;
  if (n0 >= N) return;
  const bf16 *D = P.d[l], *A = P.A[l];
  const int k0 = split * kch, k1 = min(K, k0 + kch);
  wmma::fragment<wmma::accumulator, 16, 16, 16, float> acc[2][2];
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 2; ++j) wmma::fill_fragment(acc[i][j], 0.0f);
#pragma unroll 2
  for (int k = k0; k < k1; k += 16) {
    wmma::fragment<wmma::matrix_a, 16, 16, 16, bf16, wmma::col_major> fa[2];
    wmma::fragment<wmma::matrix_b, 16, 16, 16, bf16, wmma::row_major> fb[2];
#pragma unroll
    for (int i = 0; i < 2; ++i) wmma::load_matrix_sync(fa[i], D + (size_t)k * WID + m0 + i * 16, WID);
#pragma unroll
    for (int j = 0; j < 2; ++j)
      if (n0 + j * 16 < N) wmma::load_matrix_sync(fb[j], A + (size_t)k * lda + n0 + j * 16, lda);
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int j = 0; j < 2; ++j)
        if (n0 + j * 16 < N) wmma::mma_sync(acc[i][j], fa[i], fb[j], acc[i][j]);
  }
  __shared__ float stage[4][16 * 16];
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int mb = m0 + i * 16, nb = n0 + j * 16;
      if (nb >= N) continue;
      wmma::store_matrix_sync(stage[warp], acc[i][j], 16, wmma::mem_row_major);
      __syncwarp();
      for (int e = threadIdx.x & 31; e < 256; e += 32)
        if (nb + (e % 16) < n) atomicAdd(P.g[l] + (size_t)(mb + e / 16) * n + nb + (e % 16), stage[warp][e]);
      __syncwarp();
    }
}

// normalised bfloat16 features [Bp][16] from raw float32 features [B][9]
__global__ void k_feat_raw(const float* __restrict__ F, int B, int Bp, const float* __restrict__ norm, bf16* X) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= Bp * KIN) return;
  const int b = i / KIN, c = i % KIN;
  float v = 0.0f;
  if (b < B && c < NIN) v = (F[(size_t)b * NIN + c] - norm[c]) / norm[NIN + c];
  X[i] = __float2bfloat16_rn(v);
}

// raw input row of node b from the solver state: psi_F, r_F and g^n each
// scaled by the inverse root mean square rsqrt(sq[k] / B) (sq = their sums
// of squares over the B nodes), then the node and its unit normal
__device__ __forceinline__ void raw_features(const double* __restrict__ psiF, const double* __restrict__ rF,
                                             const double* __restrict__ g, const double* __restrict__ sq,
                                             const double* __restrict__ nodes, const double* __restrict__ normals,
                                             int B, int b, float* f) {
  const double s0 = rsqrt(fmax(sq[0] / B, 1e-300)), s1 = rsqrt(fmax(sq[1] / B, 1e-300)),
               s2 = rsqrt(fmax(sq[2] / B, 1e-300));
  f[0] = (float)(psiF[b] * s0);
  f[1] = (float)(rF[b] * s1);
  f[2] = (float)(g[b] * s2);
  for (int k = 0; k < 3; ++k) {
    f[3 + k] = (float)nodes[(size_t)b * 3 + k];
    f[6 + k] = (float)normals[(size_t)b * 3 + k];
  }
}

// normalised bfloat16 network input rows [Bp][16] from the solver state
__global__ void k_feat_proj(const double* __restrict__ psiF, const double* __restrict__ rF,
                            const double* __restrict__ g, const double* __restrict__ sq,
                            const double* __restrict__ nodes, const double* __restrict__ normals, int B, int Bp,
                            const float* __restrict__ norm, bf16* X) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= Bp) return;
  float f[NIN];
  if (b < B) raw_features(psiF, rF, g, sq, nodes, normals, B, b, f);
  for (int c = 0; c < KIN; ++c) {
    float v = 0.0f;
    if (b < B && c < NIN) v = (f[c] - norm[c]) / norm[NIN + c];
    X[(size_t)b * KIN + c] = __float2bfloat16_rn(v);
  }
}

// training rows of one solve: raw features F[b][9] (the rows the network
// reads at inference) and the target T[b] = (psi - psi_F - 2 gamma r_F) /
// rms(r_F), the correction of the projection start in units of rms(r_F)
__global__ void k_train_rows(const double* __restrict__ psi, const double* __restrict__ psiF,
                             const double* __restrict__ rF, const double* __restrict__ g,
                             const double* __restrict__ sq, const double* __restrict__ nodes,
                             const double* __restrict__ normals, int B, double two_gamma, float* __restrict__ F,
                             float* __restrict__ T) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= B) return;
  float f[NIN];
  raw_features(psiF, rF, g, sq, nodes, normals, B, b, f);
  for (int c = 0; c < NIN; ++c) F[(size_t)b * NIN + c] = f[c];
  const double s1 = rsqrt(fmax(sq[1] / B, 1e-300));
  T[b] = (float)((psi[b] - psiF[b] - two_gamma * rF[b]) * s1);
}

// normalisation moments of the training rows, one block per column (the 9
// features of F [n][9], then the targets T [n]): mean and sample standard
// deviation in float64, two passes (mean first, then the squared deviations);
// a spread below 1e-12 (features) or 1e-30 (target) becomes 1.  out[c] =
// mean, out[10 + c] = std.
__global__ void __launch_bounds__(256) k_moments(const float* __restrict__ F, const float* __restrict__ T, int n,
                                                 double* __restrict__ out) {
  const int c = blockIdx.x;
  __shared__ double red[256];
  auto value = [&](int i) -> double { return c < NIN ? (double)F[(size_t)i * NIN + c] : (double)T[i]; };
  auto block_sum = [&](double v) -> double {
    red[threadIdx.x] = v;
    __syncthreads();
    for (int s = 128; s > 0; s >>= 1) {
      if ((int)threadIdx.x < s) red[threadIdx.x] += red[threadIdx.x + s];
      __syncthreads();
    }
    const double t = red[0];
    __syncthreads();
    return t;
  };
  double acc = 0.0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) acc += value(i);
  const double mean = block_sum(acc) / n;
  acc = 0.0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    const double d = value(i) - mean;
    acc += d * d;
  }
  const double var = n > 1 ? block_sum(acc) / (n - 1) : 0.0;
  if (threadIdx.x == 0) {
    const double sd = sqrt(var);
    out[c] = mean;
    out[10 + c] = sd > (c < NIN ? 1e-12 : 1e-30) ? sd : 1.0;
  }
}

__global__ void k_adam(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m, float* __restrict__ v,
                       int n, float lr, float c1, float c2) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float gi = g[i];
  const float mi = 0.9f * m[i] + 0.1f * gi;
  const float vi = 0.999f * v[i] + 0.001f * gi * gi;
  m[i] = mi;
  v[i] = vi;
  p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + 1e-8f);
}

// bfloat16 weight copies (W0 padded from 9 to 16 input columns)
__global__ void k_refresh(const float* __restrict__ p, Offsets off, bf16* W0, bf16* W1, bf16* W2, bf16* W3, bf16* w4) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < WID * KIN) {
    const int r = i / KIN, c = i % KIN;
    W0[i] = __float2bfloat16_rn(c < NIN ? p[off.w[0] + (size_t)r * NIN + c] : 0.0f);
  }
  if (i < WID * WID) {
    W1[i] = __float2bfloat16_rn(p[off.w[1] + i]);
    W2[i] = __float2bfloat16_rn(p[off.w[2] + i]);
    W3[i] = __float2bfloat16_rn(p[off.w[3] + i]);
  }
  if (i < WID) w4[i] = __float2bfloat16_rn(p[off.w[4] + i]);
}

// psi_L = psi_F + 2 gamma r_F + rms(r_F) * (s_out o + m_out), the network
// output denormalised in float32
__global__ void k_predict(const double* __restrict__ psiF, const double* __restrict__ rF,
                          const double* __restrict__ sq, double two_gamma, const float* __restrict__ o,
                          const float* __restrict__ norm, double* out, int B) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b < B) {
    const double sr = sqrt(sq[1] / B);
    out[b] = psiF[b] + two_gamma * rF[b] + sr * (double)(norm[2 * NIN + 1] * o[b] + norm[2 * NIN]);
  }
}

// Inference of the whole network in one persistent kernel (training has
// k_mlp_step, which also keeps what the backward pass needs).  The bfloat16
// weights are staged in shared memory once per block; per tile of 64 rows
// each layer runs on the tensor cores from the tile's activations in shared
// memory, the float32 products go to a shared staging tile, and the epilogue
// adds the bias, applies SiLU and rounds to bfloat16 in place; the output
// layer is one warp dot product per row.
constexpr int IR = 64;                      // rows per tile
constexpr int LDW = WID + 8, LDX = KIN + 8;  // padded bf16 leading dimensions
constexpr int LDS = WID + 4;                 // padded float32 staging
constexpr size_t INFER_SMEM = (size_t)3 * WID * LDW * 2 + (size_t)WID * LDX * 2 + (size_t)IR * LDW * 2 +
                              (size_t)IR * LDX * 2 + (size_t)IR * LDS * 4 + (size_t)4 * WID * 4 + (size_t)WID * 4;

__global__ void __launch_bounds__(256, 1) k_mlp_infer(const bf16* __restrict__ X, int Bp, const bf16* __restrict__ W0,
                                                      const bf16* __restrict__ W1, const bf16* __restrict__ W2,
                                                      const bf16* __restrict__ W3, const bf16* __restrict__ w4,
                                                      const float* __restrict__ p, Offsets off, float* __restrict__ o) {
  using namespace nvcuda;
  extern __shared__ __align__(128) unsigned char sm_infer[];
  bf16* sW = reinterpret_cast<bf16*>(sm_infer);  // 3 x [WID][LDW], B[n][k]
  bf16* sW0 = sW + 3 * WID * LDW;                 // [WID][LDX]
  bf16* sA = sW0 + WID * LDX;                     // [IR][LDW]
  bf16* sX = sA + IR * LDW;                       // [IR][LDX]
  float* sZ = reinterpret_cast<float*>(sX + IR * LDX);  // [IR][LDS]
  float* sB = sZ + IR * LDS;                      // [4][WID]
  float* sw4 = sB + 4 * WID;                      // [WID]
  const int tid = threadIdx.x;
  const bf16* Wg[3] = {W1, W2, W3};
  for (int l = 0; l < 3; ++l)
    for (int i = tid; i < WID * WID / 8; i += blockDim.x) {
      const int n = i / (WID / 8), q = i % (WID / 8);
      *reinterpret_cast<uint4*>(sW + (size_t)l * WID * LDW + n * LDW + 8 * q) =
          *reinterpret_cast<const uint4*>(Wg[l] + (size_t)n * WID + 8 * q);
    }
  for (int i = tid; i < WID * KIN / 8; i += blockDim.x) {
    const int n = i / (KIN / 8), q = i % (KIN / 8);
    *reinterpret_cast<uint4*>(sW0 + n * LDX + 8 * q) = *reinterpret_cast<const uint4*>(W0 + (size_t)n * KIN + 8 * q);
  }
  for (int i = tid; i < 4 * WID; i += blockDim.x) sB[i] = p[off.b[i / WID] + i % WID];
  for (int i = tid; i < WID; i += blockDim.x) sw4[i] = __bfloat162float(w4[i]);
  const float b4 = p[off.b[4]];
  const int warp = tid >> 5, lane = tid & 31;
  const int rb = warp & 3, cb = (warp >> 2) * 4;  // 16-row block, four 16-column blocks
  for (int tile = blockIdx.x; tile < Bp / IR; tile += gridDim.x) {
    for (int i = tid; i < IR * KIN / 8; i += blockDim.x) {
      const int r = i / (KIN / 8), q = i % (KIN / 8);
      *reinterpret_cast<uint4*>(sX + r * LDX + 8 * q) =
          *reinterpret_cast<const uint4*>(X + ((size_t)tile * IR + r) * KIN + 8 * q);
    }
    __syncthreads();
    for (int l = 0; l < 4; ++l) {
      const bf16* Ain = l == 0 ? sX : sA;
      const int lda = l == 0 ? LDX : LDW, ldb = lda, K = l == 0 ? KIN : WID;
      const bf16* Bw = l == 0 ? sW0 : sW + (size_t)(l - 1) * WID * LDW;
      wmma::fragment<wmma::accumulator, 16, 16, 16, float> acc[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) wmma::fill_fragment(acc[j], 0.0f);
      for (int k0 = 0; k0 < K; k0 += 16) {
        wmma::fragment<wmma::matrix_a, 16, 16, 16, bf16, wmma::row_major> fa;
        wmma::load_matrix_sync(fa, Ain + rb * 16 * lda + k0, lda);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          wmma::fragment<wmma::matrix_b, 16, 16, 16, bf16, wmma::col_major> fb;
          wmma::load_matrix_sync(fb, Bw + (cb + j) * 16 * ldb + k0, ldb);
          wmma::mma_sync(acc[j], fa, fb, acc[j]);
        }
      }
#pragma unroll
      for (int j = 0; j < 4; ++j)
        wmma::store_matrix_sync(sZ + rb * 16 * LDS + (cb + j) * 16, acc[j], LDS, wmma::mem_row_major);
      __syncthreads();  // every warp has read its inputs and written its products
      for (int i = tid; i < IR * WID; i += blockDim.x) {
        const int r = i / WID, c = i % WID;
        sA[r * LDW + c] = __float2bfloat16_rn(silu_f(sZ[r * LDS + c] + sB[l * WID + c]));
      }
      __syncthreads();
    }
    for (int r = warp; r < IR; r += (int)(blockDim.x >> 5)) {
      float acc = 0.0f;
      for (int j = lane; j < WID; j += 32) acc += __bfloat162float(sA[r * LDW + j]) * sw4[j];
      for (int sft = 16; sft > 0; sft >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, sft);
      if (lane == 0) o[(size_t)tile * IR + r] = acc + b4;
    }
    __syncthreads();  // the next tile overwrites sX and sA
  }
}

// Forward and backward pass of a training batch but for the weight products,
// one launch: a block takes TR rows through the four hidden layers and, with
// targets, back through their deltas (both are row-wise), with the bfloat16
// weights and the current layer's operands in shared memory.  Pre-activations
// and activations go to memory once (the backward pass and the weight
// gradients read them); a column's sums over the block's rows (bias and
// output gradients) take one float32 atomic each.  As one launch per product
// and pointwise pass (22 launches of 3 to 22 us) the 4096-row gradient took
// 200 us.  Same products and summation order per element as k_mlp_infer.
constexpr int TR = 32;
constexpr size_t STEP_SMEM = (size_t)3 * WID * LDW * 2 + (size_t)WID * LDX * 2 + (size_t)TR * LDW * 2 +
                             (size_t)TR * LDX * 2 + (size_t)TR * LDS * 4 + (size_t)4 * WID * 4 + (size_t)2 * WID * 4 +
                             (size_t)TR * 4;
struct StepArgs {
  const float *F, *T;  // raw rows [B][9], raw targets [B] (null: forward only)
  const float* norm;
  int B;
  const bf16 *W0, *W[3], *w4;
  const float* p;
  Offsets off;
  bf16* X;
  float* Z[4];
  bf16 *A[4], *db[4];
  float *o, *d4, *g, *loss, *dump_d;
};

// a column's values of the two row halves to one atomic addition
__device__ __forceinline__ void column_add(float* g, float v, float* red) {
  const int j = threadIdx.x & (WID - 1);
  if (threadIdx.x >= WID) red[j] = v;
  __syncthreads();
  if (threadIdx.x < WID) atomicAdd(g + j, v + red[j]);
  __syncthreads();
}

__global__ void __launch_bounds__(256, 1) k_mlp_step(StepArgs P) {
  using namespace nvcuda;
  extern __shared__ __align__(128) unsigned char sm_step[];
  bf16* sW = reinterpret_cast<bf16*>(sm_step);  // 3 x [WID][LDW], W[n][k]
  bf16* sW0 = sW + 3 * WID * LDW;                // [WID][LDX]
  bf16* sA = sW0 + WID * LDX;                    // [TR][LDW] activations, then deltas
  bf16* sX = sA + TR * LDW;                      // [TR][LDX]
  float* sZ = reinterpret_cast<float*>(sX + TR * LDX);  // [TR][LDS]
  float* sB = sZ + TR * LDS;                     // [4][WID]
  float* sw4 = sB + 4 * WID;                     // [WID]
  float* red = sw4 + WID;                        // [WID]
  float* sd4 = red + WID;                        // [TR]
  const int tid = threadIdx.x, row0 = blockIdx.x * TR;
  for (int l = 0; l < 3; ++l)
    for (int i = tid; i < WID * WID / 8; i += blockDim.x) {
      const int n = i / (WID / 8), q = i % (WID / 8);
      *reinterpret_cast<uint4*>(sW + (size_t)l * WID * LDW + n * LDW + 8 * q) =
          *reinterpret_cast<const uint4*>(P.W[l] + (size_t)n * WID + 8 * q);
    }
  for (int i = tid; i < WID * KIN / 8; i += blockDim.x) {
    const int n = i / (KIN / 8), q = i % (KIN / 8);
    *reinterpret_cast<uint4*>(sW0 + n * LDX + 8 * q) = *reinterpret_cast<const uint4*>(P.W0 + (size_t)n * KIN + 8 * q);
  }
  for (int i = tid; i < 4 * WID; i += blockDim.x) sB[i] = P.p[P.off.b[i / WID] + i % WID];
  for (int i = tid; i < WID; i += blockDim.x) sw4[i] = __bfloat162float(P.w4[i]);
  for (int i = tid; i < TR * KIN; i += blockDim.x) {
    const int r = i / KIN, c = i % KIN, b = row0 + r;
    float v = 0.0f;
    if (b < P.B && c < NIN) v = (P.F[(size_t)b * NIN + c] - P.norm[c]) / P.norm[NIN + c];
    const bf16 x = __float2bfloat16_rn(v);
    sX[r * LDX + c] = x;
    P.X[(size_t)b * KIN + c] = x;
  }
  const int warp = tid >> 5, lane = tid & 31;
  const int rb = warp & 1, cb = (warp >> 1) * 2;  // 16-row block, two 16-column blocks
  const int col = tid & (WID - 1), r0 = tid >> 7;  // the pointwise passes: one column, every other row
  wmma::fragment<wmma::accumulator, 16, 16, 16, float> acc[2];
  auto store = [&]() {
#pragma unroll
    for (int j = 0; j < 2; ++j)
      wmma::store_matrix_sync(sZ + rb * 16 * LDS + (cb + j) * 16, acc[j], LDS, wmma::mem_row_major);
    __syncthreads();  // every warp has read its inputs and written its products
  };
  __syncthreads();
  for (int l = 0; l < 4; ++l) {
    const bf16* Ain = l == 0 ? sX : sA;
    const int lda = l == 0 ? LDX : LDW, K = l == 0 ? KIN : WID;
    const bf16* Bw = l == 0 ? sW0 : sW + (size_t)(l - 1) * WID * LDW;
#pragma unroll
    for (int j = 0; j < 2; ++j) wmma::fill_fragment(acc[j], 0.0f);
    for (int k0 = 0; k0 < K; k0 += 16) {
      wmma::fragment<wmma::matrix_a, 16, 16, 16, bf16, wmma::row_major> fa;
      wmma::load_matrix_sync(fa, Ain + rb * 16 * lda + k0, lda);
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        wmma::fragment<wmma::matrix_b, 16, 16, 16, bf16, wmma::col_major> fb;
        wmma::load_matrix_sync(fb, Bw + (cb + j) * 16 * lda + k0, lda);
        wmma::mma_sync(acc[j], fa, fb, acc[j]);
      }
    }
    store();
    const float bias = sB[l * WID + col];
    float* Z = P.Z[l] + (size_t)row0 * WID + col;
    bf16* A = P.A[l] + (size_t)row0 * WID + col;
#pragma unroll 4
    for (int r = r0; r < TR; r += 2) {
      const float z = sZ[r * LDS + col] + bias;
      const bf16 a = __float2bfloat16_rn(silu_f(z));
      Z[(size_t)r * WID] = z;
      A[(size_t)r * WID] = a;
      sA[r * LDW + col] = a;
    }
    __syncthreads();
  }
  // output, its delta and the loss
  const float b4 = P.p[P.off.b[4]];
  float sq = 0.0f;
  for (int r = warp; r < TR; r += 8) {
    float v = 0.0f;
    for (int j = lane; j < WID; j += 32) v += __bfloat162float(sA[r * LDW + j]) * sw4[j];
    for (int sft = 16; sft > 0; sft >>= 1) v += __shfl_xor_sync(0xffffffffu, v, sft);
    const int b = row0 + r;
    const float o = v + b4;
    if (lane == 0) P.o[b] = o;
    if (P.T != nullptr) {
      const float e = b < P.B ? o - (P.T[b] - P.norm[2 * NIN]) / P.norm[2 * NIN + 1] : 0.0f;
      sq += e * e;
      if (lane == 0) {
        sd4[r] = e / (float)P.B;
        P.d4[b] = sd4[r];
      }
    }
  }
  if (P.T == nullptr) return;
  if (lane == 0) atomicAdd(P.loss, sq);
  __syncthreads();
  if (warp == 0) {
    float v = sd4[lane];
    for (int sft = 16; sft > 0; sft >>= 1) v += __shfl_xor_sync(0xffffffffu, v, sft);
    if (lane == 0) atomicAdd(P.g + P.off.b[4], v);
  }
  // deltas of the hidden layers, last first (a thread reads back the
  // pre-activations it wrote)
  for (int l = 3; l >= 0; --l) {
    const float* Z = P.Z[l] + (size_t)row0 * WID + col;
    bf16* db = P.db[l] + (size_t)row0 * WID + col;
    float* dump = P.dump_d == nullptr ? nullptr : P.dump_d + ((size_t)(3 - l) * P.B + row0) * WID + col;
    float sb = 0.0f, sw = 0.0f;
#pragma unroll 4
    for (int r = r0; r < TR; r += 2) {
      float v;
      if (l == 3) {
        const float dq = __bfloat162float(__float2bfloat16_rn(sd4[r]));
        sw += dq * __bfloat162float(sA[r * LDW + col]);
        v = dq * sw4[col] * dsilu_f(Z[(size_t)r * WID]);
      } else {
        v = sZ[r * LDS + col] * dsilu_f(Z[(size_t)r * WID]);
      }
      sb += v;
      if (dump != nullptr && row0 + r < P.B) dump[(size_t)r * WID] = v;
      const bf16 q = __float2bfloat16_rn(v);
      db[(size_t)r * WID] = q;
      sA[r * LDW + col] = q;
    }
    if (l == 3) column_add(P.g + P.off.w[4], sw, red);
    column_add(P.g + P.off.b[l], sb, red);
    if (l == 0) break;
    // d_l W_l: W_l's rows are its outputs, so it is the row-major right factor
    const bf16* Bw = sW + (size_t)(l - 1) * WID * LDW;
#pragma unroll
    for (int j = 0; j < 2; ++j) wmma::fill_fragment(acc[j], 0.0f);
    for (int k0 = 0; k0 < WID; k0 += 16) {
      wmma::fragment<wmma::matrix_a, 16, 16, 16, bf16, wmma::row_major> fa;
      wmma::load_matrix_sync(fa, sA + rb * 16 * LDW + k0, LDW);
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        wmma::fragment<wmma::matrix_b, 16, 16, 16, bf16, wmma::row_major> fb;
        wmma::load_matrix_sync(fb, Bw + (size_t)k0 * LDW + (cb + j) * 16, LDW);
        wmma::mma_sync(acc[j], fa, fb, acc[j]);
      }
    }
    store();
  }
}

}  // namespace
}  // namespace kfbi

struct kfbi_mlp {
  kfbi::Offsets off;
  int bmax = 0, bpmax = 0;
  cudaStream_t stream = nullptr;
  float *p = nullptr, *g = nullptr, *m = nullptr, *v = nullptr, *norm = nullptr;
  bf16 *W0 = nullptr, *W[3] = {nullptr, nullptr, nullptr}, *w4 = nullptr;
  bf16* X = nullptr;
  bf16* A[4] = {nullptr, nullptr, nullptr, nullptr};
  float* Z[4] = {nullptr, nullptr, nullptr, nullptr};
  float *o = nullptr, *d4 = nullptr, *loss = nullptr;  // loss: the element after g
  bf16* db[4] = {nullptr, nullptr, nullptr, nullptr};
  float* dump_d = nullptr;   // kfbi_mlp_layers: per-layer deltas go here (else null)
  float* dump_d4 = nullptr;
  int step = 0;
  std::vector<void*> allocs;
};

namespace kfbi {
namespace {

template <typename T>
int malloc_mlp(kfbi_mlp* m, T** p, size_t n) {
  if (cudaMalloc((void**)p, sizeof(T) * (n ? n : 1)) != cudaSuccess) {
    set_error("cudaMalloc failed for the MLP workspace");
    return KFBI_ERR_OOM;
  }
  m->allocs.push_back((void*)*p);
  return KFBI_OK;
}

int blocks(size_t n, int bs) { return (int)((n + bs - 1) / bs); }

// opts a kernel into its dynamic shared memory, once per device (bit of done)
template <typename K>
int opt_in(K kernel, size_t smem, std::atomic<uint64_t>& done, const char* what) {
  int dev = 0;
  KFBI_CUDA(cudaGetDevice(&dev));
  const uint64_t bit = 1ull << (dev & 63);
  if (dev < 64 && (done.load() & bit) != 0) return KFBI_OK;
  if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) {
    cudaGetLastError();
    set_error("cudaFuncSetAttribute failed for the %s kernel", what);
    return KFBI_ERR_CUDA;
  }
  done.fetch_or(bit);
  return KFBI_OK;
}

// inference over rows already placed in m->X (Bp a multiple of 64): m->o
int mlp_infer_rows(kfbi_mlp* m, int Bp) {
  static std::atomic<uint64_t> opted{0};
  if (int rc = opt_in(k_mlp_infer, INFER_SMEM, opted, "inference")) return rc;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int tiles = Bp / IR;
  const int grid = tiles < sms ? tiles : sms;
  k_mlp_infer<<<grid, 256, INFER_SMEM, m->stream>>>(m->X, Bp, m->W0, m->W[0], m->W[1], m->W[2], m->w4, m->p, m->off,
                                                    m->o);
  KFBI_CHECK_LAUNCH();
  return KFBI_OK;
}

int mlp_prepare_raw(kfbi_mlp* m, const float* F, int B, int* Bp) {
  if (B < 1 || B > m->bmax) {
    set_error("batch %d outside 1..%d", B, m->bmax);
    return KFBI_ERR_ARG;
  }
  *Bp = (B + TILE - 1) / TILE * TILE;
  k_feat_raw<<<blocks((size_t)*Bp * KIN, 256), 256, 0, m->stream>>>(F, B, *Bp, m->norm, m->X);
  KFBI_CHECK_LAUNCH();
  return KFBI_OK;
}

// forward pass over raw rows F (leaves o, Z, A, X) and, with raw targets t,
// the gradients of 0.5 mean (o - t)^2 into m->g and the squared error sum
int mlp_step(kfbi_mlp* m, const float* F, const float* t, int B) {
  if (B < 1 || B > m->bmax) {
    set_error("batch %d outside 1..%d", B, m->bmax);
    return KFBI_ERR_ARG;
  }
  static std::atomic<uint64_t> opted{0};
  if (int rc = opt_in(k_mlp_step, STEP_SMEM, opted, "training")) return rc;
  cudaStream_t st = m->stream;
  const Offsets& off = m->off;
  const int Bp = (B + TILE - 1) / TILE * TILE;
  StepArgs P;
  P.F = F;
  P.T = t;
  P.norm = m->norm;
  P.B = B;
  P.W0 = m->W0;
  P.w4 = m->w4;
  P.p = m->p;
  P.off = off;
  P.X = m->X;
  P.o = m->o;
  P.d4 = m->d4;
  P.g = m->g;
  P.loss = m->loss;
  P.dump_d = m->dump_d;
  for (int l = 0; l < 3; ++l) P.W[l] = m->W[l];
  WeightGrad G;
  for (int l = 0; l < 4; ++l) {
    P.Z[l] = m->Z[l];
    P.A[l] = m->A[l];
    P.db[l] = m->db[l];
    G.d[l] = m->db[l];
    G.A[l] = l == 0 ? m->X : m->A[l - 1];
    G.g[l] = m->g + off.w[l];
  }
  if (t != nullptr) KFBI_CUDA(cudaMemsetAsync(m->g, 0, sizeof(float) * (off.total + 1), st));
  k_mlp_step<<<Bp / TR, 256, STEP_SMEM, st>>>(P);
  KFBI_CHECK_LAUNCH();
  if (t == nullptr) return KFBI_OK;
  if (m->dump_d4) KFBI_CUDA(cudaMemcpyAsync(m->dump_d4, m->d4, sizeof(float) * B, cudaMemcpyDeviceToDevice, st));
  const int tiles = (WID / TILE) * (WID / TILE);
  const int kch = std::max(TILE, blocks((size_t)Bp * tiles, 152 * TILE) * TILE), splits = blocks(Bp, kch);
  k_weight_grad<<<dim3(WID / TILE, WID / TILE, 4 * splits), 128, 0, st>>>(G, Bp, kch, splits);
  KFBI_CHECK_LAUNCH();
  return KFBI_OK;
}

int mlp_refresh(kfbi_mlp* m) {
  k_refresh<<<blocks(WID * WID, 256), 256, 0, m->stream>>>(m->p, m->off, m->W0, m->W[0], m->W[1], m->W[2], m->w4);
  KFBI_CHECK_LAUNCH();
  return KFBI_OK;
}

}  // namespace

// warm start used by bidomain_step: psi_L from the projection psi_F, its
// residual r_F and g (sq = their sums of squares) through the network
int mlp_warmstart(kfbi_mlp* m, cudaStream_t st, const double* psiF, const double* rF, const double* g,
                  const double* sq, const double* nodes, const double* normals, int M, double two_gamma,
                  double* out) {
  if (M > m->bmax) {
    set_error("warm start: %d nodes exceed the network's batch capacity %d", M, m->bmax);
    return KFBI_ERR_ARG;
  }
  cudaStream_t saved = m->stream;
  m->stream = st;
  const int Bp = (M + TILE - 1) / TILE * TILE;
  k_feat_proj<<<blocks(Bp, 128), 128, 0, st>>>(psiF, rF, g, sq, nodes, normals, M, Bp, m->norm, m->X);
  KFBI_CHECK_LAUNCH();
  int rc = mlp_infer_rows(m, Bp);
  if (rc == KFBI_OK) {
    k_predict<<<blocks(M, 256), 256, 0, st>>>(psiF, rF, sq, two_gamma, m->o, m->norm, out, M);
    KFBI_CHECK_LAUNCH();
  }
  m->stream = saved;
  return rc;
}

int launch_train_rows(cudaStream_t st, const double* psi, const double* psiF, const double* rF, const double* g,
                      const double* sq, const double* nodes, const double* normals, int M, double two_gamma, float* F,
                      float* T) {
  k_train_rows<<<blocks(M, 256), 256, 0, st>>>(psi, psiF, rF, g, sq, nodes, normals, M, two_gamma, F, T);
  KFBI_CHECK_LAUNCH();
  return KFBI_OK;
}

}  // namespace kfbi

using namespace kfbi;

extern "C" {

int kfbi_mlp_fit_norm(const float* F_dev, const float* T_dev, int n, void* stream, float* norm_host) {
  if (!F_dev || !T_dev || !norm_host || n < 1) {
    set_error("null argument or no rows");
    return KFBI_ERR_ARG;
  }
  cudaStream_t st = (cudaStream_t)stream;
  double* out = nullptr;
  KFBI_CUDA(cudaMalloc((void**)&out, sizeof(double) * 20));
  k_moments<<<NIN + 1, 256, 0, st>>>(F_dev, T_dev, n, out);
  double h[20];
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaMemcpyAsync(h, out, sizeof(h), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  cudaFree(out);
  if (e != cudaSuccess) {
    set_error("normalisation moments failed: %s", cudaGetErrorString(e));
    return KFBI_ERR_CUDA;
  }
  KFBI_COUNT(1);
  for (int c = 0; c < NIN; ++c) {
    norm_host[c] = (float)h[c];
    norm_host[NIN + c] = (float)h[10 + c];
  }
  norm_host[2 * NIN] = (float)h[NIN];
  norm_host[2 * NIN + 1] = (float)h[10 + NIN];
  return KFBI_OK;
}

int kfbi_mlp_create(const float* params_host, const float* norm_host, int max_batch, void* stream, kfbi_mlp** out) {
  if (!params_host || !norm_host || !out || max_batch < 1) {
    set_error("null argument or empty batch");
    return KFBI_ERR_ARG;
  }
  kfbi_mlp* m = new kfbi_mlp();
  m->stream = (cudaStream_t)stream;
  m->bmax = max_batch;
  m->bpmax = (max_batch + TILE - 1) / TILE * TILE;
  const size_t P = m->off.total, Bp = m->bpmax;
  int rc = 0;
  auto fail = [&](int code) {
    kfbi_mlp_destroy(m);
    return code;
  };
  if ((rc = malloc_mlp(m, &m->p, P)) || (rc = malloc_mlp(m, &m->g, P + 1)) || (rc = malloc_mlp(m, &m->m, P)) ||
      (rc = malloc_mlp(m, &m->v, P)) || (rc = malloc_mlp(m, &m->norm, 2 * NIN + 2)) ||
      (rc = malloc_mlp(m, &m->W0, WID * KIN)) || (rc = malloc_mlp(m, &m->w4, WID)) ||
      (rc = malloc_mlp(m, &m->X, Bp * KIN)) || (rc = malloc_mlp(m, &m->o, Bp)) || (rc = malloc_mlp(m, &m->d4, Bp)))
    return fail(rc);
  m->loss = m->g + P;
  for (int l = 0; l < 3; ++l)
    if ((rc = malloc_mlp(m, &m->W[l], WID * WID))) return fail(rc);
  for (int l = 0; l < 4; ++l)
    if ((rc = malloc_mlp(m, &m->A[l], Bp * WID)) || (rc = malloc_mlp(m, &m->Z[l], Bp * WID)) ||
        (rc = malloc_mlp(m, &m->db[l], Bp * WID)))
      return fail(rc);
  cudaStream_t st = m->stream;
  if (cudaMemcpyAsync(m->p, params_host, sizeof(float) * P, cudaMemcpyHostToDevice, st) != cudaSuccess ||
      cudaMemcpyAsync(m->norm, norm_host, sizeof(float) * (2 * NIN + 2), cudaMemcpyHostToDevice, st) != cudaSuccess ||
      cudaMemsetAsync(m->m, 0, sizeof(float) * P, st) != cudaSuccess ||
      cudaMemsetAsync(m->v, 0, sizeof(float) * P, st) != cudaSuccess) {
    set_error("MLP upload failed");
    return fail(KFBI_ERR_CUDA);
  }
  if ((rc = mlp_refresh(m))) return fail(rc);
  if (cudaStreamSynchronize(st) != cudaSuccess) {
    set_error("MLP setup failed");
    return fail(KFBI_ERR_CUDA);
  }
  *out = m;
  return KFBI_OK;
}

void kfbi_mlp_destroy(kfbi_mlp* m) {
  if (!m) return;
  cudaStreamSynchronize(m->stream);
  for (void* p : m->allocs) cudaFree(p);
  delete m;
}

int kfbi_mlp_num_params(void) { return (int)Offsets().total; }

int kfbi_mlp_get(kfbi_mlp* m, float* params_host) {
  if (!m || !params_host) {
    set_error("null argument");
    return KFBI_ERR_ARG;
  }
  KFBI_CUDA(cudaMemcpyAsync(params_host, m->p, sizeof(float) * m->off.total, cudaMemcpyDeviceToHost, m->stream));
  KFBI_CUDA(cudaStreamSynchronize(m->stream));
  return KFBI_OK;
}

int kfbi_mlp_forward(kfbi_mlp* m, const float* F_dev, int B, float* o_dev) {
  if (!m || !F_dev || !o_dev) {
    set_error("null argument");
    return KFBI_ERR_ARG;
  }
  int Bp, rc;
  if ((rc = mlp_prepare_raw(m, F_dev, B, &Bp))) return rc;
  if ((rc = mlp_infer_rows(m, Bp))) return rc;
  KFBI_CUDA(cudaMemcpyAsync(o_dev, m->o, sizeof(float) * B, cudaMemcpyDeviceToDevice, m->stream));
  return KFBI_OK;
}

int kfbi_mlp_grad(kfbi_mlp* m, const float* F_dev, const float* t_dev, int B, float* loss_host, float* grad_host) {
  if (!m || !F_dev || !t_dev) {
    set_error("null argument");
    return KFBI_ERR_ARG;
  }
  if (int rc = mlp_step(m, F_dev, t_dev, B)) return rc;
  float l = 0.0f;
  KFBI_CUDA(cudaMemcpyAsync(&l, m->loss, sizeof(float), cudaMemcpyDeviceToHost, m->stream));
  if (grad_host)
    KFBI_CUDA(cudaMemcpyAsync(grad_host, m->g, sizeof(float) * m->off.total, cudaMemcpyDeviceToHost, m->stream));
  KFBI_CUDA(cudaStreamSynchronize(m->stream));
  if (loss_host) *loss_host = 0.5f * l / (float)B;
  return KFBI_OK;
}

int kfbi_mlp_layers(kfbi_mlp* m, const float* F_dev, const float* T_dev, int B, float* z_dev, float* o_dev,
                    float* d_dev, float* d4_dev) {
  if (!m || !F_dev) {
    set_error("null argument");
    return KFBI_ERR_ARG;
  }
  cudaStream_t st = m->stream;
  m->dump_d = T_dev ? d_dev : nullptr;
  m->dump_d4 = T_dev ? d4_dev : nullptr;
  const int rc = mlp_step(m, F_dev, T_dev, B);
  m->dump_d = m->dump_d4 = nullptr;
  if (rc) return rc;
  if (z_dev)
    for (int l = 0; l < 4; ++l)
      KFBI_CUDA(cudaMemcpyAsync(z_dev + (size_t)l * B * WID, m->Z[l], sizeof(float) * B * WID,
                                cudaMemcpyDeviceToDevice, st));
  if (o_dev) KFBI_CUDA(cudaMemcpyAsync(o_dev, m->o, sizeof(float) * B, cudaMemcpyDeviceToDevice, st));
  KFBI_CUDA(cudaStreamSynchronize(st));
  return KFBI_OK;
}

int kfbi_mlp_train_step(kfbi_mlp* m, const float* F_dev, const float* t_dev, int B, float lr, float* loss_host) {
  int rc = kfbi_mlp_grad(m, F_dev, t_dev, B, loss_host, nullptr);
  if (rc) return rc;
  ++m->step;
  const float c1 = 1.0f - powf(0.9f, (float)m->step), c2 = 1.0f - powf(0.999f, (float)m->step);
  k_adam<<<blocks(m->off.total, 256), 256, 0, m->stream>>>(m->p, m->g, m->m, m->v, (int)m->off.total, lr, c1, c2);
  KFBI_CHECK_LAUNCH();
  return mlp_refresh(m);
}

}  // extern "C"
