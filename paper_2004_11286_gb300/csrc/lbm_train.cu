// lbm_train.cu -- training kernels of the learned Stefan-Maxwell closure:
// forward and backward passes of the network (two GELU layers of width 128
// and a linear output layer) for a mini-batch, the mean-squared loss over the
// 3M valid outputs, and the Adam update (Kingma & Ba 2015, Algorithm 1).
// FP32 master weights, packed W1 [H][F] | b1 [H] | W2 [H][H] | b2 [H] |
// W3 [O][H] | b3 [O]; the inference path uses a bf16 copy (lbm_mlp.cuh).
//
// The mini-batch gradient is two launches.  mlp_grad_kernel keeps all three
// weight matrices in shared memory (up to 119 KB) and carries a tile of rows
// through the whole network and back: the activations never leave the SM, and
// the weight gradients accumulate in registers over the block's tiles.
// grad_reduce_kernel adds the blocks' partial gradients in a fixed order.
// It is bound by the FP32 FMA and shared-memory pipes (2.5 MFMA per 32-row
// tile).  The former chain of 16 launches spent its time in the weight
// gradients, which it computed on 2 to 4 blocks walking all rows in series.
// Measured (GB300, M = 8, call to loss on the host): 76 against 1475 us at
// 4096 rows (67 against 1487 back to back), 505 against 48300 us at 100,000
// rows, 66 against 226 us at 256.  A handle's first call also allocates the
// blocks' partials (0.17 ms).
#include <cmath>

#include <cuda_runtime.h>

#include "lbm_train.h"

namespace lbm {

namespace {

constexpr int H = 128;          // hidden width
constexpr int GT = 256;         // threads of a gradient block
constexpr int LDH = H + 4;      // row strides in shared memory: 4 mod 32 words
                                // (or 20), so 16-byte reads of 8 consecutive rows
                                // fall in distinct banks

__device__ __forceinline__ float gelu_cdf(float x) { return 0.5f * (1.0f + erff(x * 0.70710678118654752f)); }

// Weight-gradient blocks write nw floats and one loss each.
__host__ __device__ constexpr int weight_count(int F, int O) { return H * F + H + H * H + H + O * H + O; }

template <int F, int O, int TR>
struct GradSmem {
  static constexpr int LDF = F + 4, LDO = O + 4;
  static constexpr int W1 = 0, W2 = W1 + H * LDF, W3 = W2 + H * LDH, X = W3 + O * LDH, A1 = X + TR * LDF,
                       D1 = A1 + TR * LDH, A2 = D1 + TR * LDH, D2 = A2 + TR * LDH, DO = D2 + TR * LDH,
                       FLOATS = DO + TR * LDO;
  static constexpr size_t BYTES = FLOATS * sizeof(float);
};

// acc[i][j] = sum_k A[r0 + i][k] W[lane + 32 j][k] (rows of both K-major):
// a warp's RW rows against 32 J columns; A reads are broadcasts.
template <int RW, int J, int K, int LDA, int LDW>
__device__ __forceinline__ void rows_times_wt(const float* A, const float* Wt, int lane, float (&acc)[RW][J]) {
#pragma unroll 4
  for (int k = 0; k < K; k += 4) {
    float4 a[RW], b[J];
#pragma unroll
    for (int i = 0; i < RW; ++i) a[i] = *reinterpret_cast<const float4*>(A + i * LDA + k);
#pragma unroll
    for (int j = 0; j < J; ++j) b[j] = *reinterpret_cast<const float4*>(Wt + (lane + 32 * j) * LDW + k);
#pragma unroll
    for (int i = 0; i < RW; ++i)
#pragma unroll
      for (int j = 0; j < J; ++j)
        acc[i][j] += a[i].x * b[j].x + a[i].y * b[j].y + a[i].z * b[j].z + a[i].w * b[j].w;
  }
}
// acc[i][j] = sum_k D[r0 + i][k] W[k][lane + 32 j].
template <int RW, int K, int LDD>
__device__ __forceinline__ void rows_times_w(const float* D, const float* W, int lane, float (&acc)[RW][4]) {
#pragma unroll 4
  for (int k = 0; k < K; k += 4) {
    float4 d[RW];
#pragma unroll
    for (int i = 0; i < RW; ++i) d[i] = *reinterpret_cast<const float4*>(D + i * LDD + k);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float* w = W + k * LDH + lane + 32 * j;
      const float w0 = w[0], w1 = w[LDH], w2 = w[2 * LDH], w3 = w[3 * LDH];
#pragma unroll
      for (int i = 0; i < RW; ++i) acc[i][j] += d[i].x * w0 + d[i].y * w1 + d[i].z * w2 + d[i].w * w3;
    }
  }
}

// Each block takes tiles of TR rows (blockIdx.x, + gridDim.x, ...): forward,
// loss, backward; weight gradients in registers (each thread an 8 x 8 patch
// of gW2 and its share of gW1, gW3 and the biases), written to part at the end.
template <int F, int O, int TR>
__global__ void __launch_bounds__(GT, 1)
mlp_grad_kernel(int rows, int valid, float scale, double inv, const float* __restrict__ w, const float* __restrict__ X,
                const float* __restrict__ T, float* __restrict__ part, double* __restrict__ loss_part) {
  using S = GradSmem<F, O, TR>;
  constexpr int RW = TR / (GT / 32);          // rows per warp
  extern __shared__ __align__(16) float sm[];
  __shared__ double sl[GT / 32];
  float *sW1 = sm + S::W1, *sW2 = sm + S::W2, *sW3 = sm + S::W3, *sX = sm + S::X, *sA1 = sm + S::A1,
        *sD1 = sm + S::D1, *sA2 = sm + S::A2, *sD2 = sm + S::D2, *sDO = sm + S::DO;
  const int tid = threadIdx.x, lane = tid & 31, r0 = (tid >> 5) * RW;
  const int tx = tid & 15, ty = tid >> 4;
  const float* W1 = w;
  const float* b1 = W1 + H * F;
  const float* W2 = b1 + H;
  const float* b2 = W2 + H * H;
  const float* W3 = b2 + H;
  const float* b3 = W3 + O * H;
  for (int e = tid; e < H * F / 4; e += GT)
    *reinterpret_cast<float4*>(sW1 + (4 * e / F) * S::LDF + 4 * e % F) = reinterpret_cast<const float4*>(W1)[e];
  for (int e = tid; e < H * H / 4; e += GT)
    *reinterpret_cast<float4*>(sW2 + (4 * e / H) * LDH + 4 * e % H) = reinterpret_cast<const float4*>(W2)[e];
  for (int e = tid; e < O * H / 4; e += GT)
    *reinterpret_cast<float4*>(sW3 + (4 * e / H) * LDH + 4 * e % H) = reinterpret_cast<const float4*>(W3)[e];
  float rb1[4], rb2[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) { rb1[j] = b1[lane + 32 * j]; rb2[j] = b2[lane + 32 * j]; }
  const int oc = lane % O;                    // O = 16: both half warps hold the same columns
  const float rb3 = b3[oc];
  constexpr int F16 = F / 16, O16 = O / 16;
  float g2[8][8] = {}, g1[8][F16] = {}, g3[O16][8] = {}, gb12 = 0.0f, gb3 = 0.0f;
  double loss = 0.0;
  const int ntiles = (rows - 1) / TR + 1;
  for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
    const long long row0 = (long long)t * TR;
    const int nr = rows - row0 < TR ? (int)(rows - row0) : TR;
    __syncthreads();                          // weights staged; the previous tile's operands free
    for (int e = tid; e < TR * F; e += GT) {
      const int r = e / F;
      sX[r * S::LDF + e % F] = r < nr ? X[row0 * F + e] : 0.0f;
    }
    __syncthreads();
    {
      float h[RW][4];
#pragma unroll
      for (int i = 0; i < RW; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) h[i][j] = rb1[j];
      rows_times_wt<RW, 4, F, S::LDF, S::LDF>(sX + r0 * S::LDF, sW1, lane, h);
#pragma unroll
      for (int i = 0; i < RW; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const float x = h[i][j], c = gelu_cdf(x);
          sA1[(r0 + i) * LDH + lane + 32 * j] = x * c;
          sD1[(r0 + i) * LDH + lane + 32 * j] = c + x * expf(-0.5f * x * x) * 0.39894228040143268f;
        }
      __syncwarp();                           // a warp reads only its own rows until the weight gradients
#pragma unroll
      for (int i = 0; i < RW; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) h[i][j] = rb2[j];
      rows_times_wt<RW, 4, H, LDH, LDH>(sA1 + r0 * LDH, sW2, lane, h);
#pragma unroll
      for (int i = 0; i < RW; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const float x = h[i][j], c = gelu_cdf(x);
          sA2[(r0 + i) * LDH + lane + 32 * j] = x * c;
          sD2[(r0 + i) * LDH + lane + 32 * j] = c + x * expf(-0.5f * x * x) * 0.39894228040143268f;
        }
      __syncwarp();
      float o[RW][1];
#pragma unroll
      for (int i = 0; i < RW; ++i) o[i][0] = rb3;
      rows_times_wt<RW, 1, H, LDH, LDH>(sA2 + r0 * LDH, sW3, oc, o);
#pragma unroll
      for (int i = 0; i < RW; ++i) {
        const int r = r0 + i;
        float d = 0.0f;
        if (r < nr && oc < valid) {
          const float e = o[i][0] - T[(row0 + r) * O + oc];
          d = scale * e;
          if (lane < O) loss += (double)e * e;
        }
        if (lane < O) sDO[r * S::LDO + oc] = d;
      }
      __syncwarp();
      // dh2 = (dout W3) gelu'(h2), dh1 = (dh2 W2) gelu'(h1), in the places of the derivatives
#pragma unroll
      for (int i = 0; i < RW; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) h[i][j] = 0.0f;
      rows_times_w<RW, O, S::LDO>(sDO + r0 * S::LDO, sW3, lane, h);
#pragma unroll
      for (int i = 0; i < RW; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) { sD2[(r0 + i) * LDH + lane + 32 * j] *= h[i][j]; h[i][j] = 0.0f; }
      __syncwarp();
      rows_times_w<RW, H, LDH>(sD2 + r0 * LDH, sW2, lane, h);
#pragma unroll
      for (int i = 0; i < RW; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) sD1[(r0 + i) * LDH + lane + 32 * j] *= h[i][j];
    }
    __syncthreads();
#pragma unroll 2
    for (int r = 0; r < TR; ++r) {
      float d[8], a[8];
      *reinterpret_cast<float4*>(d) = *reinterpret_cast<const float4*>(sD2 + r * LDH + ty * 8);
      *reinterpret_cast<float4*>(d + 4) = *reinterpret_cast<const float4*>(sD2 + r * LDH + ty * 8 + 4);
      *reinterpret_cast<float4*>(a) = *reinterpret_cast<const float4*>(sA1 + r * LDH + tx * 4);
      *reinterpret_cast<float4*>(a + 4) = *reinterpret_cast<const float4*>(sA1 + r * LDH + 64 + tx * 4);
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) g2[i][j] += d[i] * a[j];
      *reinterpret_cast<float4*>(d) = *reinterpret_cast<const float4*>(sD1 + r * LDH + ty * 8);
      *reinterpret_cast<float4*>(d + 4) = *reinterpret_cast<const float4*>(sD1 + r * LDH + ty * 8 + 4);
#pragma unroll
      for (int j = 0; j < F16; ++j) {
        const float x = sX[r * S::LDF + tx + 16 * j];
#pragma unroll
        for (int i = 0; i < 8; ++i) g1[i][j] += d[i] * x;
      }
      *reinterpret_cast<float4*>(a) = *reinterpret_cast<const float4*>(sA2 + r * LDH + tx * 4);
      *reinterpret_cast<float4*>(a + 4) = *reinterpret_cast<const float4*>(sA2 + r * LDH + 64 + tx * 4);
#pragma unroll
      for (int i = 0; i < O16; ++i) {
        const float e = sDO[r * S::LDO + ty * O16 + i];
#pragma unroll
        for (int j = 0; j < 8; ++j) g3[i][j] += e * a[j];
      }
      gb12 += tid < H ? sD1[r * LDH + tid] : sD2[r * LDH + tid - H];
      if (tid < O) gb3 += sDO[r * S::LDO + tid];
    }
  }
  float* pW1 = part + (long long)blockIdx.x * weight_count(F, O);
  float* pb1 = pW1 + H * F;
  float* pW2 = pb1 + H;
  float* pb2 = pW2 + H * H;
  float* pW3 = pb2 + H;
  float* pb3 = pW3 + O * H;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
#pragma unroll
    for (int j = 0; j < F16; ++j) pW1[(ty * 8 + i) * F + tx + 16 * j] = g1[i][j];
#pragma unroll
    for (int j = 0; j < 8; j += 4)
      *reinterpret_cast<float4*>(pW2 + (ty * 8 + i) * H + 16 * j + tx * 4) =
          make_float4(g2[i][j], g2[i][j + 1], g2[i][j + 2], g2[i][j + 3]);
  }
#pragma unroll
  for (int i = 0; i < O16; ++i)
#pragma unroll
    for (int j = 0; j < 8; j += 4)
      *reinterpret_cast<float4*>(pW3 + (ty * O16 + i) * H + 16 * j + tx * 4) =
          make_float4(g3[i][j], g3[i][j + 1], g3[i][j + 2], g3[i][j + 3]);
  if (tid < H) pb1[tid] = gb12; else pb2[tid - H] = gb12;
  if (tid < O) pb3[tid] = gb3;
  for (int o = 16; o > 0; o >>= 1) loss += __shfl_down_sync(0xffffffffu, loss, o);
  if (lane == 0) sl[tid >> 5] = loss;
  __syncthreads();
  if (tid == 0) {
    double s = 0.0;
    for (int k = 0; k < GT / 32; ++k) s += sl[k];
    loss_part[blockIdx.x] = s * inv;
  }
}

// g[e] = sum of the nb blocks' partial gradients, *loss that of their losses:
// eight slices of the blocks summed in parallel, then the slices in order.
constexpr int RX = 32, RY = 8;
__global__ void __launch_bounds__(RX * RY)
grad_reduce_kernel(const float* __restrict__ part, int nb, int nw, float* __restrict__ g,
                   const double* __restrict__ loss_part, double* __restrict__ loss) {
  __shared__ float sh[RY][RX];
  const int e = blockIdx.x * RX + threadIdx.x;
  float s = 0.0f;
  if (e < nw) {
#pragma unroll 4
    for (int b = threadIdx.y; b < nb; b += RY) s += part[(long long)b * nw + e];
  }
  sh[threadIdx.y][threadIdx.x] = s;
  __syncthreads();
  if (threadIdx.y == 0 && e < nw) {
    float t = 0.0f;
    for (int k = 0; k < RY; ++k) t += sh[k][threadIdx.x];
    g[e] = t;
  }
  if (blockIdx.x == 0 && threadIdx.y == 1) {
    double l = 0.0;
    for (int b = threadIdx.x; b < nb; b += RX) l += loss_part[b];
    for (int o = 16; o > 0; o >>= 1) l += __shfl_down_sync(0xffffffffu, l, o);
    if (threadIdx.x == 0) *loss = l;
  }
}

__global__ void adam_kernel(float* __restrict__ w, const float* __restrict__ g, float* __restrict__ m,
                            float* __restrict__ v, long long count, float lr, float c1, float c2) {
  const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= count) return;
  const float gi = g[e];
  const float mi = 0.9f * m[e] + 0.1f * gi;
  const float vi = 0.999f * v[e] + 0.001f * gi * gi;
  m[e] = mi;
  v[e] = vi;
  w[e] -= lr * (mi * c1) / (sqrtf(vi * c2) + 1e-8f);
}

inline unsigned blocks(long long n, int b) { return (unsigned)((n + b - 1) / b); }

template <int F, int O, int TR>
cudaError_t grad_launch(cudaStream_t s, int rows, int valid, const float* w, const float* X, const float* T,
                        const MlpScratch& z, float* g, double* d_loss) {
  constexpr size_t smem = GradSmem<F, O, TR>::BYTES;
  cudaError_t e = cudaFuncSetAttribute(mlp_grad_kernel<F, O, TR>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const int ntiles = (rows - 1) / TR + 1;
  const int nb = ntiles < z.blocks ? ntiles : z.blocks;
  const double inv = 1.0 / ((double)rows * valid);
  mlp_grad_kernel<F, O, TR><<<nb, GT, smem, s>>>(rows, valid, (float)(2.0 * inv), inv, w, X, T, z.part, z.loss);
  constexpr int nw = weight_count(F, O);
  grad_reduce_kernel<<<blocks(nw, RX), dim3(RX, RY), 0, s>>>(z.part, nb, nw, g, z.loss, d_loss);
  return cudaGetLastError();
}

}  // namespace

cudaError_t mlp_train_grad(cudaStream_t s, const MlpShape& sh, const float* w, const float* X, const float* T,
                           int rows, const MlpScratch& z, float* g, double* d_loss) {
  // Tiles of 16 rows where those of 32 would leave blocks without work.
  const bool small = rows <= 16LL * z.blocks;
#define LBM_GRAD(FF, OO)                                                                       \
  if (sh.F == FF && sh.O == OO)                                                                \
    return small ? grad_launch<FF, OO, 16>(s, rows, sh.valid, w, X, T, z, g, d_loss)           \
                 : grad_launch<FF, OO, 32>(s, rows, sh.valid, w, X, T, z, g, d_loss)
  LBM_GRAD(16, 16);      // M = 1..3
  LBM_GRAD(32, 16);      // M = 4, 5
  LBM_GRAD(48, 32);      // M = 6
  LBM_GRAD(64, 32);      // M = 7, 8
#undef LBM_GRAD
  return cudaErrorInvalidValue;
}

cudaError_t mlp_adam(cudaStream_t s, float* w, const float* g, float* m, float* v, long long count, float lr, int t) {
  const float c1 = 1.0f / (1.0f - (float)std::pow(0.9, t));
  const float c2 = 1.0f / (1.0f - (float)std::pow(0.999, t));
  adam_kernel<<<blocks(count, 256), 256, 0, s>>>(w, g, m, v, count, lr, c1, c2);
  return cudaGetLastError();
}

}  // namespace lbm
