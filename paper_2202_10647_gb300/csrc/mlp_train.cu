// mlp_train.cu -- training of the rate surrogate on the GPU: the loss and its
// gradient for a batch (forward pass, chain rule, batch reductions), the Adam
// update, and a plain (CUDA-core) forward pass used as the reference of the
// tensor-core inference.  Network and parameter layout: mlp_device.cuh.
//
//   loss  L = (1/(B K)) sum_b sum_k (y_bk - t_bk)^2
//   mlp_train_kernel  a block per tile of 64 samples: forward pass, backward
//                   pass and the tile's part of the gradient, all products as
//                   register tiles over shared memory.
//   mlp_grad_sum    sums the blocks' parts and losses in a fixed order
//                   (deterministic).
//   mlp_adam        Adam with bias-corrected moments.
// With ION_MLP_BF16 the forward pass rounds W2, W3, h1 and h2 to their
// bf16 pairs (split_round) and takes the SFU tanh, as the tensor-core
// inference does; the backward pass then treats the rounding as the identity
// (straight-through).
#include <algorithm>
#include <cmath>
#include <cstdint>

#include "ion_step.cuh"
#include "ionize.h"
#include "mlp_device.cuh"

namespace ion {
namespace mlp {
namespace {

constexpr int kThreads = 128;
// Samples of a training tile, and threads of its block: 16 x 16, each with 4
// samples x 4 units of every 64 x 64 product.
constexpr int kTile = 64;
constexpr int kTrainThreads = 256;
constexpr int kLd = kTile + 4;  // row length in shared memory

struct Parts {
  float* grad;  // [blocks][nparams]
  float* loss;  // [blocks]
};

size_t round256(size_t x) { return (x + 255) / 256 * 256; }

int64_t train_tiles(int64_t B) { return (B + kTile - 1) / kTile; }

// Room for one part per tile (the grid never exceeds the tiles) up to
// kMaxParts of them.
constexpr int kMaxParts = 256;
int64_t most_parts(int64_t B) { return std::min<int64_t>(train_tiles(B), kMaxParts); }

size_t ws_bytes(int K, int64_t B) {
  return round256(4 * (size_t)most_parts(B) * nparams(K)) + round256(4 * (size_t)most_parts(B));
}

Parts bind(void* ws, int K, int64_t B) {
  char* p = static_cast<char*>(ws);
  return {reinterpret_cast<float*>(p),
          reinterpret_cast<float*>(p + round256(4 * (size_t)most_parts(B) * nparams(K)))};
}

int fwd_blocks(int64_t B) { return (int)((B + kThreads - 1) / kThreads); }

// The network staged in shared memory; output rows k >= K are zero.
template <int KP>
struct Net {
  float W1[H], b1[H], b2[H];
  float W2[H * H];
  float W3[KP * H];
  float b3[KP];
};

template <int KP, bool Q>
__device__ __forceinline__ void stage(const float* __restrict__ P, int K, Net<KP>& n) {
  for (int i = threadIdx.x; i < H; i += blockDim.x) {
    n.W1[i] = P[off_W1() + i];
    n.b1[i] = P[off_b1() + i];
    n.b2[i] = P[off_b2() + i];
  }
  for (int i = threadIdx.x; i < H * H; i += blockDim.x) {
    const float w = P[off_W2() + i];
    n.W2[i] = Q ? split_round(w) : w;
  }
  for (int i = threadIdx.x; i < KP * H; i += blockDim.x) {
    const float w = i < K * H ? P[off_W3() + i] : 0.0f;
    n.W3[i] = Q ? split_round(w) : w;
  }
  for (int k = threadIdx.x; k < KP; k += blockDim.x) n.b3[k] = k < K ? P[off_b3(K) + k] : 0.0f;
}

// ---- training --------------------------------------------------------------
// Shared memory of a training block: the weights in both orders (a product
// reads its inner index first), and the tile's activations and their
// gradients as [unit][sample], which serves both the products over units (an
// inner index at a time) and those over samples (four samples at a time).
template <int KP>
struct Train {
  float W1[H], b1[H], b2[H], b3[KP];
  float W2[H][kLd], W2T[H][kLd];    // [o][i], [i][o]
  float W3[KP][kLd], W3T[H][KP];    // [k][o], [o][k]
  float h1[H][kLd], h2[H][kLd];     // [unit][sample]
  float d2[H][kLd];                 // dL/dz2
  float dy[KP][kLd];                // dL/dy
  float x[kTile];
  float red[kTrainThreads / 32];
};

// acc[a][b] += sum over c < n of A[c][4 ty + a] B[c][4 tx + b], c in order.
template <int n, int ldb>
__device__ __forceinline__ void tile_product(float (&acc)[4][4], const float (*A)[kLd],
                                             const float (*Bm)[ldb], int tx, int ty) {
#pragma unroll 8
  for (int c = 0; c < n; ++c) {
    const float4 u = *reinterpret_cast<const float4*>(&A[c][4 * ty]);
    const float4 w = *reinterpret_cast<const float4*>(&Bm[c][4 * tx]);
    const float ua[4] = {u.x, u.y, u.z, u.w}, wb[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int b = 0; b < 4; ++b) acc[a][b] = fmaf(ua[a], wb[b], acc[a][b]);
  }
}

// acc[a][b] += sum over the tile's samples s of A[ty + 16 a][s] B[tx + 16 b][s].
template <int NA>
__device__ __forceinline__ void sample_product(float (&acc)[NA][4], const float (*A)[kLd],
                                               const float (*Bm)[kLd], int tx, int ty) {
#pragma unroll 2
  for (int s = 0; s < kTile; s += 4) {
    float4 u[NA], w[4];
#pragma unroll
    for (int a = 0; a < NA; ++a) u[a] = *reinterpret_cast<const float4*>(&A[ty + 16 * a][s]);
#pragma unroll
    for (int b = 0; b < 4; ++b) w[b] = *reinterpret_cast<const float4*>(&Bm[tx + 16 * b][s]);
#pragma unroll
    for (int a = 0; a < NA; ++a)
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        acc[a][b] = fmaf(u[a].x, w[b].x, acc[a][b]);
        acc[a][b] = fmaf(u[a].y, w[b].y, acc[a][b]);
        acc[a][b] = fmaf(u[a].z, w[b].z, acc[a][b]);
        acc[a][b] = fmaf(u[a].w, w[b].w, acc[a][b]);
      }
  }
}

__device__ __forceinline__ void put4(float* p, float a, float b, float c, float d) {
  *reinterpret_cast<float4*>(p) = make_float4(a, b, c, d);
}

// Loss and gradient of the block's tiles.  The work is six small products
// (129 M multiply-adds for 8192 samples of a 64-64-18 network, 3.2 us at the
// FP32 rate of 152 SMs); one thread per sample left 64 blocks of 4 warps in
// a serial loop over units (41 + 40 us) and a gradient pass that read
// every activation 64 times (64 us).  A tile of 64 samples per block gives 128
// blocks their 8 warps, 16 accumulators per 2 shared-memory loads, keeps all
// activations on the chip, and takes each tanh once (the derivatives stay in
// registers until the backward pass).  Per sample every sum runs in the
// order of the serial loop.  18 us at that size, and 4 us to add the parts
// (latency: two warps per scheduler; the products issue in about 5 us).
template <int KP, bool Q>
__global__ void __launch_bounds__(kTrainThreads)
    mlp_train_kernel(const float* __restrict__ P, int K, const float* __restrict__ x,
                     const float* __restrict__ t, int B, float two_over_BK, Parts out) {
  constexpr int KJ = KP / 16;  // outputs per thread
  extern __shared__ __align__(16) unsigned char train_smem[];
  Train<KP>& S = *reinterpret_cast<Train<KP>*>(train_smem);
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  {
    // weights: a thread has column o of the transposes (no bank conflicts)
    for (int i = tid; i < H; i += kTrainThreads) {
      S.W1[i] = P[off_W1() + i];
      S.b1[i] = P[off_b1() + i];
      S.b2[i] = P[off_b2() + i];
    }
    for (int k = tid; k < KP; k += kTrainThreads) S.b3[k] = k < K ? P[off_b3(K) + k] : 0.0f;
    const int o = tid & 63, q = tid >> 6;
#pragma unroll
    for (int i = 16 * q; i < 16 * q + 16; ++i) {
      const float w = P[off_W2() + o * H + i];
      const float v = Q ? split_round(w) : w;
      S.W2[o][i] = v;
      S.W2T[i][o] = v;
    }
#pragma unroll
    for (int k = q; k < KP; k += 4) {
      const float w = k < K ? P[off_W3() + k * H + o] : 0.0f;
      const float v = Q ? split_round(w) : w;
      S.W3[k][o] = v;
      S.W3T[o][k] = v;
    }
  }
  float gW2[4][4], gW3[KJ][4], gw1[4], gb1[4], gb2[4], gb3[KJ], loss = 0.0f;
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    gw1[a] = gb1[a] = gb2[a] = 0.0f;
#pragma unroll
    for (int b = 0; b < 4; ++b) gW2[a][b] = 0.0f;
  }
#pragma unroll
  for (int a = 0; a < KJ; ++a) {
    gb3[a] = 0.0f;
#pragma unroll
    for (int b = 0; b < 4; ++b) gW3[a][b] = 0.0f;
  }

  for (int64_t s0 = (int64_t)blockIdx.x * kTile; s0 < B; s0 += (int64_t)gridDim.x * kTile) {
    const int n = (int)min((int64_t)kTile, B - s0);
    __syncthreads();  // the previous tile's products are done
    if (tid < kTile) S.x[tid] = tid < n ? x[s0 + tid] : 0.0f;
    __syncthreads();
    // layer 1: samples 4 ty + a, units 4 tx + b; g1, g2 the derivatives
    float g1[4][4], g2[4][4], acc[4][4];
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      const int i = 4 * tx + b;
      float h[4];
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        const float z = fmaf(S.W1[i], S.x[4 * ty + a], S.b1[i]);
        float th;
        h[a] = gelu<Q>(z, th);
        if (Q) h[a] = split_round(h[a]);
        g1[a][b] = gelu_grad(z, th);
        acc[a][b] = S.b2[i];
      }
      put4(&S.h1[i][4 * ty], h[0], h[1], h[2], h[3]);
    }
    __syncthreads();
    tile_product<H, kLd>(acc, S.h1, S.W2T, tx, ty);
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      float h[4];
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        float th;
        h[a] = gelu<Q>(acc[a][b], th);
        if (Q) h[a] = split_round(h[a]);
        g2[a][b] = gelu_grad(acc[a][b], th);
      }
      put4(&S.h2[4 * tx + b][4 * ty], h[0], h[1], h[2], h[3]);
    }
    __syncthreads();
    // outputs k = tx + 16 j of samples 4 ty + a, and dL/dy
    float y[4][KJ];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int j = 0; j < KJ; ++j) y[a][j] = S.b3[tx + 16 * j];
#pragma unroll 8
    for (int o = 0; o < H; ++o) {
      const float4 u = *reinterpret_cast<const float4*>(&S.h2[o][4 * ty]);
      const float ua[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
      for (int j = 0; j < KJ; ++j) {
        const float w = S.W3T[o][tx + 16 * j];
#pragma unroll
        for (int a = 0; a < 4; ++a) y[a][j] = fmaf(w, ua[a], y[a][j]);
      }
    }
#pragma unroll
    for (int j = 0; j < KJ; ++j) {
      const int k = tx + 16 * j;
      float d[4];
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        const bool on = 4 * ty + a < n && k < K;
        const float e = on ? y[a][j] - t[(s0 + 4 * ty + a) * K + k] : 0.0f;
        loss = fmaf(e, e, loss);
        d[a] = two_over_BK * e;
        gb3[j] += d[a];
      }
      put4(&S.dy[k][4 * ty], d[0], d[1], d[2], d[3]);
    }
    __syncthreads();
    // dL/dz2 = (dL/dy W3) g2
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int b = 0; b < 4; ++b) acc[a][b] = 0.0f;
    tile_product<KP, kLd>(acc, S.dy, S.W3, tx, ty);
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      float d[4];
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        d[a] = acc[a][b] * g2[a][b];
        gb2[b] += d[a];
        acc[a][b] = 0.0f;
      }
      put4(&S.d2[4 * tx + b][4 * ty], d[0], d[1], d[2], d[3]);
    }
    sample_product<KJ>(gW3, S.dy, S.h2, tx, ty);
    __syncthreads();
    // dL/dz1 = (dL/dz2 W2) g1
    tile_product<H, kLd>(acc, S.d2, S.W2, tx, ty);
#pragma unroll
    for (int b = 0; b < 4; ++b)
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        const float d = acc[a][b] * g1[a][b];
        gb1[b] += d;
        gw1[b] = fmaf(d, S.x[4 * ty + a], gw1[b]);
      }
    sample_product<4>(gW2, S.d2, S.h1, tx, ty);
  }

  // the block's part: the matrices from their owners, the vectors summed over
  // the 16 sample groups in order
  float* part = out.grad + (int64_t)blockIdx.x * nparams(K);
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) part[off_W2() + (ty + 16 * a) * H + tx + 16 * b] = gW2[a][b];
#pragma unroll
  for (int a = 0; a < KJ; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b)
      if (ty + 16 * a < K) part[off_W3() + (ty + 16 * a) * H + tx + 16 * b] = gW3[a][b];
  __syncthreads();
  float(*v)[kLd] = S.h1;  // rows: W1, b1, b2 x 16 groups, then b3 in S.h2
#pragma unroll
  for (int b = 0; b < 4; ++b) {
    v[ty][4 * tx + b] = gw1[b];
    v[16 + ty][4 * tx + b] = gb1[b];
    v[32 + ty][4 * tx + b] = gb2[b];
  }
#pragma unroll
  for (int j = 0; j < KJ; ++j) S.h2[ty][tx + 16 * j] = gb3[j];
#pragma unroll
  for (int s = 16; s > 0; s >>= 1) loss += __shfl_xor_sync(0xffffffffu, loss, s);
  if ((tid & 31) == 0) S.red[tid >> 5] = loss;
  __syncthreads();
  {
    const int which = tid >> 6, c = tid & 63;
    float s = 0.0f;
    const float(*r)[kLd] = which < 3 ? &v[16 * which] : &S.h2[0];
#pragma unroll
    for (int g = 0; g < 16; ++g) s += r[g][c];
    if (which == 0) part[off_W1() + c] = s;
    if (which == 1) part[off_b1() + c] = s;
    if (which == 2) part[off_b2() + c] = s;
    if (which == 3 && c < K) part[off_b3(K) + c] = s;
  }
  if (tid == 0) {
    float s = 0.0f;
#pragma unroll
    for (int w = 0; w < kTrainThreads / 32; ++w) s += S.red[w];
    out.loss[blockIdx.x] = s;
  }
}

// The parts summed in a fixed order: 32 parameters per block, its 8 warps
// take the parts w, w + 8, ... and are then added in order.
__global__ void __launch_bounds__(256)
    mlp_grad_sum(int np, int nparts, Parts in, float* __restrict__ grad,
                 float* __restrict__ loss, float inv_BK) {
  __shared__ float red[8][33];
  cudaGridDependencySynchronize();
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int p = blockIdx.x * 32 + lane;
  float g = 0.0f;
  if (p < np) {
#pragma unroll 8
    for (int b = w; b < nparts; b += 8) g += in.grad[(int64_t)b * np + p];
  }
  red[w][lane] = g;
  if (blockIdx.x == 0 && w == 0 && loss) {
    float l = 0.0f;
    for (int i = lane; i < nparts; i += 32) l += in.loss[i];
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) l += __shfl_xor_sync(0xffffffffu, l, s);
    if (lane == 0) *loss = l * inv_BK;
  }
  __syncthreads();
  if (w == 0 && p < np) {
    float s = red[0][lane];
#pragma unroll
    for (int i = 1; i < 8; ++i) s += red[i][lane];
    grad[p] = s;
  }
}

__global__ void __launch_bounds__(256)
    mlp_adam(float* __restrict__ P, const float* __restrict__ g, float* __restrict__ m,
             float* __restrict__ v, int64_t n, float lr, float b1, float b2, float eps,
             float bc1, float bc2) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float mi = fmaf(b1, m[i], (1.0f - b1) * gi);
    const float vi = fmaf(b2, v[i], (1.0f - b2) * gi * gi);
    m[i] = mi;
    v[i] = vi;
    P[i] -= lr * (mi / bc1) / (sqrtf(vi / bc2) + eps);
  }
}

// One thread per sample.  The loop over hidden units o is kept rolled: each iteration is a dot
// product over the register array h1 and an update of y, fully unrolled, so
// that the arrays stay in registers at a modest code size.
template <int KP, bool Q>
__global__ void __launch_bounds__(kThreads)
    mlp_forward(const float* __restrict__ P, int K, const float* __restrict__ x, int B,
                float* __restrict__ y_out) {
  __shared__ Net<KP> n;
  stage<KP, Q>(P, K, n);
  __syncthreads();
  const int b = blockIdx.x * kThreads + threadIdx.x;
  if (b >= B) return;
  const float xb = x[b];
  float h1[H];
#pragma unroll
  for (int i = 0; i < H; ++i) {
    const float h = gelu<Q>(fmaf(n.W1[i], xb, n.b1[i]));
    h1[i] = Q ? split_round(h) : h;
  }
  float y[KP];
#pragma unroll
  for (int k = 0; k < KP; ++k) y[k] = n.b3[k];
#pragma unroll 1
  for (int o = 0; o < H; ++o) {
    float z = n.b2[o];
#pragma unroll
    for (int i = 0; i < H; ++i) z = fmaf(n.W2[o * H + i], h1[i], z);
    float h = gelu<Q>(z);
    h = Q ? split_round(h) : h;
#pragma unroll
    for (int k = 0; k < KP; ++k) y[k] = fmaf(n.W3[k * H + o], h, y[k]);
  }
#pragma unroll
  for (int k = 0; k < KP; ++k)
    if (k < K) y_out[(int64_t)b * K + k] = y[k];
}

template <int KP, bool Q>
cudaError_t launch_train(const float* P, int K, const float* x, const float* t, int B,
                         float two_over_BK, const Parts& a, int* nparts, cudaStream_t s) {
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(mlp_train_kernel<KP, Q>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)sizeof(Train<KP>));
  if (e != cudaSuccess) return e;
  // one block per SM (the shared memory's limit), each with an equal share
  const int64_t tiles = train_tiles(B), cap = std::min(sms, kMaxParts);
  const int64_t each = (tiles + cap - 1) / cap;
  *nparts = (int)((tiles + each - 1) / each);
  mlp_train_kernel<KP, Q><<<*nparts, kTrainThreads, sizeof(Train<KP>), s>>>(P, K, x, t, B,
                                                                            two_over_BK, a);
  return cudaGetLastError();
}

template <int KP>
cudaError_t launch_train(bool q, const float* P, int K, const float* x, const float* t, int B,
                         float two_over_BK, const Parts& a, int* nparts, cudaStream_t s) {
  return q ? launch_train<KP, true>(P, K, x, t, B, two_over_BK, a, nparts, s)
           : launch_train<KP, false>(P, K, x, t, B, two_over_BK, a, nparts, s);
}

template <int KP>
cudaError_t launch_forward(bool q, const float* P, int K, const float* x, int B, float* y,
                           cudaStream_t s) {
  const int g = fwd_blocks(B);
  if (q)
    mlp_forward<KP, true><<<g, kThreads, 0, s>>>(P, K, x, B, y);
  else
    mlp_forward<KP, false><<<g, kThreads, 0, s>>>(P, K, x, B, y);
  return cudaGetLastError();
}

constexpr int64_t kMaxBatch = int64_t(1) << 24;

int check_common(const char* who, const float* P, int K, const float* x, int64_t B, int flags) {
  if (K < 1 || K > kMaxOut)
    return set_error(ION_EINVAL, "%s: K=%d outside [1, %d]", who, K, kMaxOut);
  if (B < 1 || B > kMaxBatch)
    return set_error(ION_EINVAL, "%s: B=%lld outside [1, 2^24]", who, (long long)B);
  if (!P || !x) return set_error(ION_EINVAL, "%s: NULL pointer", who);
  if (flags & ~ION_MLP_BF16) return set_error(ION_EINVAL, "%s: unknown flags 0x%x", who, flags);
  if ((reinterpret_cast<uintptr_t>(P) | reinterpret_cast<uintptr_t>(x)) % 4)
    return set_error(ION_EINVAL, "%s: arrays must be 4-byte aligned", who);
  return ION_OK;
}

// ---- training data ---------------------------------------------------------
// x = clamp(2 (log2|E| - l2lo) / (l2hi - l2lo) - 1, -1, 1) in FP64, scale =
// 2 / (l2hi - l2lo); the clamp after the rounding to float (rounding keeps
// the order).  Bound by issue and the FP64 pipe; 1,048,576
// fields: 94 us with log2() and a division, 11 us now.
__global__ void mlp_inputs_kernel(const float* __restrict__ E, int64_t n, double l2lo,
                                  double scale, float* __restrict__ x) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float e = fabsf(E[i]);
  // zero, denormal, infinite and NaN fields take the library's log2
  const double l2 = e >= 1.17549435e-38f && e <= 3.40282347e38f ? log2_f64(f64_of_f32(e))
                                                                : log2((double)e);
  x[i] = fminf(fmaxf((float)fma(l2 - l2lo, scale, -1.0), -1.0f), 1.0f);  // NaN: -1
}

// ---- standardization -------------------------------------------------------
// Y (n rows of K) is read once for both moments and once to be scaled.
// Moments: a block holds a slice of rows in registers, kHold values per
// thread, every thread on one column (threads = a multiple of K), and takes
// the slice's column sums and then its squared deviations from the slice's
// own means; mlp_moments_combine adds the slices up,
//   M2 = sum_s M2_s + sum_s n_s (mean_s - mean)^2
// (T. F. Chan, G. H. Golub, R. J. LeVeque, "Algorithms for computing the
// sample variance", Am. Stat. 37, 1983), in a fixed order.  The slices'
// means and M2 wait in T, which the last kernel then overwrites.
// A thread sums in 64-bit integers: its values in units of 2^-57 of the slice's largest
// power of 2 in the column (finer than the ulps that FP64 sums of them round by), the
// squared deviations in units of 2^-58 of the thread's largest; some 40 integer
// instructions a value in the issue time of less than one of the three FP64 ones.  Columns
// of slices with infinities or NaN, or of sizes beyond 2^400, take FP64.
// 1,048,576 x 18 values: two passes of 18 blocks took 2 x 918 us, scaling by an FP64
// division 335 us; moments by slices in FP64 140 us (107 us of FP64 issue), now 67 us
// (23 us of traffic); 15 us to combine the slices, and 40 us to scale (34 us of
// traffic; 124 us with an FP64 product instead of the pairs).
constexpr int kStdThreads = 256;
constexpr int kHold = 32;

int std_columns(int K) { return kStdThreads / K * K; }             // threads at work
int64_t std_rows(int K) { return (int64_t)(kStdThreads / K) * kHold; }  // rows of a slice

// The block's column sums of v, in a fixed order: groups of 16 rows by their
// first thread, then the groups by the threads of row 0, which alone receive
// them (the others' FP64 additions would be issued for nothing).
__device__ __forceinline__ double column_sum(double v, double* part, int K, int rows) {
  const int row = threadIdx.x / K;
  __syncthreads();
  part[threadIdx.x] = v;
  __syncthreads();
  const bool lead = row < rows && (row & 15) == 0;
  double s = v;
  if (lead)
    for (int r = 1; r < 16 && row + r < rows; ++r) s += part[threadIdx.x + r * K];
  __syncthreads();
  if (lead) part[threadIdx.x] = s;
  __syncthreads();
  if (row == 0)
    for (int r = 16; r < rows; r += 16) s += part[threadIdx.x + r * K];
  return s;
}

// An FP64 value kept in two floats' place (T is only 4-byte aligned).
__device__ __forceinline__ void put_f64(float* p, double v) {
  p[0] = __int_as_float(__double2loint(v));
  p[1] = __int_as_float(__double2hiint(v));
}
__device__ __forceinline__ double get_f64(const float* p) {
  return __hiloint2double(__float_as_int(p[1]), __float_as_int(p[0]));
}

// x 2^(57 - E), towards 0, of a double x of at most 2^(E+1) in size, E + 1023 = e.
__device__ __forceinline__ long long fixed_bits(long long x, int e) {
  const uint32_t h = (uint32_t)(x >> 32), l = (uint32_t)x;
  const uint64_t m = ((uint64_t)((h & 0xfffffu) | 0x100000u) << 32 | l) << 6;
  const uint32_t s = (uint32_t)(e + 1) - ((h >> 20) & 0x7ffu);
  const long long f = s < 64u ? (long long)(m >> s) : 0;
  return (int)h < 0 ? -f : f;
}
__device__ __forceinline__ double power_of_2(int n) {
  return __hiloint2double((1023 + n) << 20, 0);
}

// Slice blockIdx.x of the rows: its column means and M2 into
// part_out[(2 slice + which) K + k].
__global__ void __launch_bounds__(kStdThreads)
    mlp_moments_kernel(const double* __restrict__ Y, int64_t n, int K, float* part_out) {
  __shared__ double part[kStdThreads], means[kMaxOut];
  __shared__ int top[kMaxOut];
  const int rows = kStdThreads / K;
  const int64_t r0 = blockIdx.x * (int64_t)rows * kHold;
  const int ns = (int)min((int64_t)rows * kHold, n - r0);  // rows of this slice
  const int row = threadIdx.x / K, k = threadIdx.x % K;
  const bool on = row < rows;
  const double* y = Y + r0 * K + threadIdx.x;
  long long v[kHold];  // the values' bits, then the fixed-point values
  if (threadIdx.x < K) top[threadIdx.x] = 0;
  int e = 0;  // the largest exponent field
#pragma unroll
  for (int i = 0; i < kHold; ++i) {
    v[i] = on && row + i * rows < ns ? __double_as_longlong(__ldcs(y + (int64_t)i * rows * K)) : 0;
    e = max(e, (int)(v[i] >> 32) & 0x7ff00000);
  }
  __syncthreads();
  if (on) atomicMax(&top[k], e >> 20);
  __syncthreads();
  e = top[k];
  const bool fixed = e > 1023 - 400 && e < 1023 + 400;
  double s = 0.0;
  if (fixed) {
    long long sum = 0;
#pragma unroll
    for (int i = 0; i < kHold; ++i) {
      v[i] = fixed_bits(v[i], e);
      sum += v[i];
    }
    s = (double)sum * power_of_2(e - 1023 - 57);
  } else {
#pragma unroll
    for (int i = 0; i < kHold; ++i) s += __longlong_as_double(v[i]);
  }
  const double sum = column_sum(s, part, K, rows);
  if (row == 0) means[k] = sum / (double)ns;
  __syncthreads();
  const double mean = means[k];
  double q = 0.0;
  if (fixed) {
    const long long m = fixed_bits(__double_as_longlong(mean), e);
    unsigned long long all = 1, acc = 0;
#pragma unroll
    for (int i = 0; i < kHold; ++i) {
      const long long d = v[i] - m;
      v[i] = on && row + i * rows < ns ? (d < 0 ? -d : d) : 0;
      all |= (unsigned long long)v[i];
    }
    const int sh = __clzll((long long)all) - 3;  // |d| < 2^59: the largest to below 2^61
#pragma unroll
    for (int i = 0; i < kHold; ++i) {
      const uint64_t d = (uint64_t)v[i] << sh;
      acc += mul_hi64(d, d);
    }
    q = (double)(long long)acc * power_of_2(64 - 2 * sh + 2 * (e - 1023 - 57));
  } else {
#pragma unroll
    for (int i = 0; i < kHold; ++i) {
      if (on && row + i * rows < ns) {
        const double d = __longlong_as_double(v[i]) - mean;
        q = fma(d, d, q);
      }
    }
  }
  const double m2 = column_sum(q, part, K, rows);
  if (row == 0) {
    float* o = part_out + 4 * (int64_t)blockIdx.x * K;
    put_f64(o + 2 * k, mean);
    put_f64(o + 2 * (K + k), m2);
  }
}

// Block k: the mean and scale of column k from the slices' means and M2.  (What a dependent
// kernel reads of the one before is not declared __restrict__: a read-only load may be taken
// ahead of the wait.)
__global__ void __launch_bounds__(kStdThreads)
    mlp_moments_combine(const float* part_in, int64_t n, int K, int64_t slices,
                        double min_scale, double* mean_out, double* scale_out) {
  __shared__ double part[kStdThreads];
  cudaGridDependencySynchronize();
  const int k = blockIdx.x;
  const int64_t per = (int64_t)(kStdThreads / K) * kHold;
  auto total = [&](double v) {
    __syncthreads();
    part[threadIdx.x] = v;
    __syncthreads();
    for (int w = kStdThreads / 2; w > 0; w >>= 1) {
      if ((int)threadIdx.x < w) part[threadIdx.x] += part[threadIdx.x + w];
      __syncthreads();
    }
    return part[0];
  };
  double s = 0.0;
  for (int64_t i = threadIdx.x; i < slices; i += kStdThreads)
    s = fma(get_f64(part_in + 4 * i * K + 2 * k), (double)min(per, n - i * per), s);
  const double mean = total(s) / (double)n;
  double q = 0.0;
  for (int64_t i = threadIdx.x; i < slices; i += kStdThreads) {
    const double d = get_f64(part_in + 4 * i * K + 2 * k) - mean;
    q += fma(d * d, (double)min(per, n - i * per), get_f64(part_in + 4 * i * K + 2 * (K + k)));
  }
  const double m2 = total(q);
  if (threadIdx.x == 0) {
    mean_out[k] = mean;
    scale_out[k] = fmax(sqrt(m2 / (double)(n - 1)), min_scale);
  }
}

// A double as hi + lo (2^-48 relative), hi its leading 24 bits, by integer
// instructions and one int-to-float conversion; ok is false outside
// 2^-60..2^60 (and for 0).
__device__ __forceinline__ void split_bits(double x, float& hi, float& lo, bool& ok) {
  const uint32_t h = (uint32_t)__double2hiint(x), l = (uint32_t)__double2loint(x);
  const uint32_t ex = (h >> 20) & 0x7ffu, sign = h & 0x80000000u;
  ok = ex - (1023u - 60u) < 120u;
  hi = __uint_as_float(sign | (((h & 0x7fffffffu) - 0x38000000u) << 3) | (l >> 29));
  // the 29 bits below, in units of 2^(exponent - 52)
  lo = (float)(l & 0x1fffffffu) *
       __uint_as_float(sign | ((ex - (1023u + 52u - 127u)) << 23));
}

// T = (Y - mean) / scale rounded to float.  Taken in FP32 pairs (2^-44
// relative to |Y| + |mean|, about 40 FP32 and integer instructions where the
// FP64 subtraction, product and conversion cost the time of 190); where that
// error could change the rounded result (A. Ziv, "Fast evaluation of
// elementary mathematical functions with correctly rounded last bit", ACM
// TOMS 17, 1991), about one value in 10^5, or a value leaves the pairs'
// range, in FP64.  Every thread stays on one column.
__global__ void __launch_bounds__(kStdThreads)
    mlp_normalize_kernel(const double* __restrict__ Y, int64_t n, int K,
                         const double* mean, const double* scale, float* __restrict__ T) {
  constexpr int kUnroll = 8;
  cudaGridDependencySynchronize();
  const int rows = kStdThreads / K;
  if ((int)threadIdx.x >= rows * K) return;
  const int64_t step = (int64_t)rows * K;
  const int k = threadIdx.x % K;
  const double m = mean[k], sc = scale[k], inv = 1.0 / sc;
  float mh, ml, ih, il;
  bool pairs, iok;
  split_bits(m, mh, ml, pairs);
  if (m == 0.0) {
    mh = ml = 0.0f;
    pairs = true;
  }
  split_bits(inv, ih, il, iok);
  pairs = pairs && iok;
  auto one = [&](double y) -> float {
    float yh, yl;
    bool ok;
    split_bits(y, yh, yl, ok);
    // d = y - mean, q = d / scale as hi + lo
    const float s = yh - mh, z = s - yh;
    const float dl = ((yh - (s - z)) - (mh + z)) + (yl - ml);
    const float p = s * ih;
    const float e = fmaf(s, ih, -p) + fmaf(s, il, dl * ih);
    const float err = (fabsf(yh) + fabsf(mh)) * ih * 0x1p-43f;
    const float up = p + (e + err), down = p + (e - err);
    if (pairs && ok && up == down && fabsf(p) >= 0x1p-60f) return up;
    if (__double_as_longlong(y) == __double_as_longlong(m) && m - m == 0.0) return 0.0f;
    return (float)((y - m) / sc);
  };
  const int64_t all = n * K, stride = gridDim.x * step * kUnroll;
  for (int64_t i = blockIdx.x * step * kUnroll + threadIdx.x; i < all; i += stride) {
    double y[kUnroll];
    if (i + (kUnroll - 1) * step < all) {
#pragma unroll
      for (int j = 0; j < kUnroll; ++j) y[j] = __ldcs(Y + i + j * step);
#pragma unroll
      for (int j = 0; j < kUnroll; ++j) T[i + j * step] = one(y[j]);
    } else {
      for (int64_t c = i; c < all; c += step) T[c] = one(Y[c]);
    }
  }
}

// Fewer rows than hold the slices' means and M2 in T: one block per column,
// mean and then scale.
__global__ void __launch_bounds__(kStdThreads)
    mlp_moments_small(const double* __restrict__ Y, int64_t n, int K, double min_scale,
                      double* mean_out, double* scale_out) {
  __shared__ double part[kStdThreads];
  const int k = blockIdx.x;
  double mean = 0.0;
  for (int pass = 0; pass < 2; ++pass) {
    double acc = 0.0;
    for (int64_t r = threadIdx.x; r < n; r += kStdThreads) {
      const double d = Y[r * K + k] - mean;
      acc += pass ? d * d : d;
    }
    __syncthreads();
    part[threadIdx.x] = acc;
    __syncthreads();
    for (int w = kStdThreads / 2; w > 0; w >>= 1) {
      if ((int)threadIdx.x < w) part[threadIdx.x] += part[threadIdx.x + w];
      __syncthreads();
    }
    if (!pass) mean = part[0] / (double)n;
  }
  if (threadIdx.x == 0) {
    mean_out[k] = mean;
    scale_out[k] = fmax(sqrt(part[0] / (double)(n - 1)), min_scale);
  }
}

}  // namespace
}  // namespace mlp
}  // namespace ion

using namespace ion::mlp;

extern "C" {

int64_t ion_mlp_nparams(int K) {
  return (K < 1 || K > kMaxOut) ? (int64_t)ION_EINVAL : (int64_t)nparams(K);
}

size_t ion_mlp_workspace_bytes(int K, int64_t B) {
  if (K < 1 || K > kMaxOut || B < 1 || B > kMaxBatch) return 0;
  return ws_bytes(K, B);
}

int ion_mlp_loss_grad(const float* P, int K, const float* x, const float* t, int64_t B,
                      int flags, float* grad, float* loss, void* workspace,
                      size_t workspace_bytes, void* stream) {
  int rc = check_common("ion_mlp_loss_grad", P, K, x, B, flags);
  if (rc) return rc;
  if (!t || !grad) return ion::set_error(ION_EINVAL, "ion_mlp_loss_grad: NULL pointer");
  if (!workspace || workspace_bytes < ws_bytes(K, B) ||
      reinterpret_cast<uintptr_t>(workspace) % 256)
    return ion::set_error(ION_EINVAL,
                          "ion_mlp_loss_grad: workspace must be 256-byte aligned and hold "
                          "%zu bytes",
                          ws_bytes(K, B));
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const Parts a = bind(workspace, K, B);
  const bool q = (flags & ION_MLP_BF16) != 0;
  const float two_over_BK = (float)(2.0 / ((double)B * K));
  int nparts = 0;
  cudaError_t e;
  switch (padded_out(K)) {
    case 16:
      e = launch_train<16>(q, P, K, x, t, (int)B, two_over_BK, a, &nparts, s);
      break;
    case 32:
      e = launch_train<32>(q, P, K, x, t, (int)B, two_over_BK, a, &nparts, s);
      break;
    case 48:
      e = launch_train<48>(q, P, K, x, t, (int)B, two_over_BK, a, &nparts, s);
      break;
    default:
      e = launch_train<64>(q, P, K, x, t, (int)B, two_over_BK, a, &nparts, s);
      break;
  }
  if (e == cudaSuccess) {
    const int np = nparams(K);
    e = ion::launch_after(true, mlp_grad_sum, (np + 31) / 32, 256, 0, s, np, nparts, a, grad, loss,
                          (float)(1.0 / ((double)B * K)));
  }
  if (e != cudaSuccess)
    return ion::set_error(ION_ECUDA, "ion_mlp_loss_grad launch: %s", cudaGetErrorString(e));
  return ion::set_error(ION_OK, "%s", "");
}

int ion_mlp_adam(float* P, const float* grad, float* m, float* v, int64_t n, float lr,
                 float beta1, float beta2, float eps, int t, void* stream) {
  if (!P || !grad || !m || !v || n < 1)
    return ion::set_error(ION_EINVAL, "ion_mlp_adam: NULL pointer or n < 1");
  if (t < 1) return ion::set_error(ION_EINVAL, "ion_mlp_adam: step t=%d < 1", t);
  if (!(beta1 >= 0.0f && beta1 < 1.0f && beta2 >= 0.0f && beta2 < 1.0f && eps > 0.0f &&
        std::isfinite(lr)))
    return ion::set_error(ION_EINVAL, "ion_mlp_adam: bad hyper-parameters");
  const float bc1 = (float)(1.0 - std::pow((double)beta1, (double)t));
  const float bc2 = (float)(1.0 - std::pow((double)beta2, (double)t));
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const int64_t blocks = (n + 255) / 256;
  mlp_adam<<<(int)(blocks < 1024 ? blocks : 1024), 256, 0, s>>>(P, grad, m, v, n, lr, beta1,
                                                               beta2, eps, bc1, bc2);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess)
    return ion::set_error(ION_ECUDA, "ion_mlp_adam launch: %s", cudaGetErrorString(e));
  return ion::set_error(ION_OK, "%s", "");
}

int ion_mlp_forward(const float* P, int K, const float* x, int64_t B, int flags, float* y,
                    void* stream) {
  int rc = check_common("ion_mlp_forward", P, K, x, B, flags);
  if (rc) return rc;
  if (!y) return ion::set_error(ION_EINVAL, "ion_mlp_forward: y is NULL");
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const bool q = (flags & ION_MLP_BF16) != 0;
  cudaError_t e;
  switch (padded_out(K)) {
    case 16:
      e = launch_forward<16>(q, P, K, x, (int)B, y, s);
      break;
    case 32:
      e = launch_forward<32>(q, P, K, x, (int)B, y, s);
      break;
    case 48:
      e = launch_forward<48>(q, P, K, x, (int)B, y, s);
      break;
    default:
      e = launch_forward<64>(q, P, K, x, (int)B, y, s);
      break;
  }
  if (e != cudaSuccess)
    return ion::set_error(ION_ECUDA, "ion_mlp_forward launch: %s", cudaGetErrorString(e));
  return ion::set_error(ION_OK, "%s", "");
}

int ion_mlp_inputs(const float* E, int64_t n, double l2lo, double l2hi, float* x,
                   void* stream) {
  if (n < 0 || n >= (int64_t(1) << 40))
    return ion::set_error(ION_EINVAL, "ion_mlp_inputs: n=%lld outside [0, 2^40)",
                          (long long)n);
  if (!(l2lo < l2hi) || !std::isfinite(l2lo) || !std::isfinite(l2hi))
    return ion::set_error(ION_EINVAL, "ion_mlp_inputs: need finite l2lo < l2hi");
  if (n == 0) return ion::set_error(ION_OK, "%s", "");
  if (!E || !x || (reinterpret_cast<uintptr_t>(E) & 3u) || (reinterpret_cast<uintptr_t>(x) & 3u))
    return ion::set_error(ION_EINVAL, "ion_mlp_inputs: E and x must be non-NULL, 4-byte aligned");
  const int64_t blocks = (n + 255) / 256;
  mlp_inputs_kernel<<<(unsigned)blocks, 256, 0, static_cast<cudaStream_t>(stream)>>>(
      E, n, l2lo, 2.0 / (l2hi - l2lo), x);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess)
    return ion::set_error(ION_ECUDA, "ion_mlp_inputs launch: %s", cudaGetErrorString(e));
  return ion::set_error(ION_OK, "%s", "");
}

int ion_mlp_standardize(const double* Y, int64_t n, int K, double min_scale, double* mean_out,
                        double* scale_out, float* T, void* stream) {
  if (n < 2 || n >= (int64_t(1) << 32))
    return ion::set_error(ION_EINVAL, "ion_mlp_standardize: n=%lld outside [2, 2^32)",
                          (long long)n);
  if (K < 1 || K > ION_MAX_Z)
    return ion::set_error(ION_EINVAL, "ion_mlp_standardize: K=%d outside [1, %d]", K,
                          ION_MAX_Z);
  if (!(min_scale > 0.0) || !std::isfinite(min_scale))
    return ion::set_error(ION_EINVAL, "ion_mlp_standardize: min_scale must be finite and > 0");
  auto al = [](const void* p, uintptr_t a) { return (reinterpret_cast<uintptr_t>(p) & (a - 1)) == 0; };
  if (!Y || !mean_out || !scale_out || !T || !al(Y, 8) || !al(mean_out, 8) ||
      !al(scale_out, 8) || !al(T, 4))
    return ion::set_error(ION_EINVAL,
                          "ion_mlp_standardize: Y, mean_out, scale_out (8-byte aligned) and T "
                          "(4-byte aligned) must be non-NULL");
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  cudaError_t e;
  const int64_t slices = (n + std_rows(K) - 1) / std_rows(K);
  // a slice's means and M2 take four floats per column of T: four rows
  if (n >= 4 * slices) {
    mlp_moments_kernel<<<(unsigned)slices, kStdThreads, 0, s>>>(Y, n, K, T);
    e = cudaGetLastError();
    if (e == cudaSuccess)
      e = ion::launch_after(true, mlp_moments_combine, K, kStdThreads, 0, s, T, n, K, slices, min_scale,
                            mean_out, scale_out);
  } else {
    mlp_moments_small<<<K, kStdThreads, 0, s>>>(Y, n, K, min_scale, mean_out, scale_out);
    e = cudaGetLastError();
  }
  const int64_t per = (int64_t)std_columns(K) * 8;
  const int64_t need = (n * K + per - 1) / per;
  if (e == cudaSuccess)
    e = ion::launch_after(true, mlp_normalize_kernel, (unsigned)std::min<int64_t>(need, 4096),
                          kStdThreads, 0, s, Y, n, K, mean_out, scale_out, T);
  if (e != cudaSuccess)
    return ion::set_error(ION_ECUDA, "ion_mlp_standardize launch: %s", cudaGetErrorString(e));
  return ion::set_error(ION_OK, "%s", "");
}

}  // extern "C"
