// The surrogate network's own kernels: forward, loss + gradient by
// backpropagation over a batch, Adam, and the per-bin inference used inside
// the clip kernel. Network: 20 -> 64 -> GELU -> 64 -> GELU -> 2, GELU exact
// (x Phi(x)); weights are read as BF16, every product and sum is FP32.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "sep_mlp.cuh"

namespace sep {
namespace {

// Weights (BF16 -> FP32) into shared memory.
__device__ __forceinline__ void load_weights(const __nv_bfloat16* wbf, float* w) {
  for (int i = threadIdx.x; i < kNParams; i += blockDim.x) w[i] = __bfloat162float(wbf[i]);
}

constexpr int kTile = 64;        // samples per tile of the gradient kernel
constexpr int kGradThreads = 256;
constexpr int kGradCtas = 152 * 2;   // CTAs that are resident at once (two a multiprocessor: shared memory)

// Shared memory of the gradient kernel (floats). The 64 x 64 matrices keep
// block c of 4 columns of row r at block c ^ (r / 4): a thread's 4 x 4 block
// is then stored by rows and by columns without bank conflicts.
struct GradShared {
  float w1t[kIn * kH];        // W1 by input [i][j]
  float w2[kH * kH];          // W2 [j][k]
  float w2t[kH * kH];         // W2 by input [k][j]
  float w3[kOut * kH];
  float b1[kH], b2[kH], b3[4];
  float xt[kIn * kTile];      // the tile's inputs by feature [i][s]
  float x[kTile * kIn];       // and by sample
  float h1[kTile * kH];       // hidden units by sample [s][k]
  float t[kH * kTile];        // hidden units by unit [k][s]; then dL/da2 by unit [j][s]; then dL/da1 [s][k]
  float da2[kTile * kH];      // dL/da2 by sample [s][j]
  float gb1[kH], gb2[kH], gw3[kOut * kH], gb3[4];
  float loss;
};
static_assert(kTile == 64 && kH == 64, "4 x 4 blocks of 16 x 16 threads");

__device__ __forceinline__ int swz(int r, int c4) { return r * 64 + 4 * (c4 ^ ((r >> 2) & 15)); }

// acc[i][j] += sum over k < n of a[k][4 ra + i] b[k][4 cb + j] (rows of 64,
// swizzled when SA / SB).
template <bool SA, bool SB>
__device__ __forceinline__ void product(const float* a, const float* b, int n, int ra, int cb, float (&acc)[4][4]) {
#pragma unroll 4
  for (int k = 0; k < n; ++k) {
    const float4 u = *reinterpret_cast<const float4*>(a + (SA ? swz(k, ra) : k * 64 + 4 * ra));
    const float4 v = *reinterpret_cast<const float4*>(b + (SB ? swz(k, cb) : k * 64 + 4 * cb));
    const float us[4] = {u.x, u.y, u.z, u.w}, vs[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(us[i], vs[j], acc[i][j]);
  }
}

// A 4 x 4 block (rows 4 r.., columns 4 c..) into a swizzled matrix, and its transpose.
__device__ __forceinline__ void put_rows(float* m, int r, int c, const float (&v)[4][4]) {
#pragma unroll
  for (int i = 0; i < 4; ++i)
    *reinterpret_cast<float4*>(m + swz(4 * r + i, c)) = make_float4(v[i][0], v[i][1], v[i][2], v[i][3]);
}
__device__ __forceinline__ void put_columns(float* m, int r, int c, const float (&v)[4][4]) {
#pragma unroll
  for (int j = 0; j < 4; ++j)
    *reinterpret_cast<float4*>(m + swz(4 * c + j, r)) = make_float4(v[0][j], v[1][j], v[2][j], v[3][j]);
}

// Gradient of the mean squared error over n samples (x [n][20], t [n][2]),
// accumulated into grad [kNParams] and loss (sum over samples / n).
// Sample s of tile b is row idx(b * kTile + s) = (start + (b*kTile+s) * stride) mod n.
//
// Every product of the network is a 64 x 64 (64 x 20) matrix product over a
// tile of 64 samples; a thread owns a 4 x 4 block of each and reads its two
// operands as 16-byte vectors (16 multiply-adds for two reads; one product at
// a time with both operands in shared memory was bound by those reads, by
// their bank conflicts and by one set of atomics a tile). A CTA keeps its
// share of the gradient in registers over all its tiles and adds it once.
// FP32 throughout: 16,384 rows with their clearing 131 -> 45 us.
__global__ void __launch_bounds__(kGradThreads, 2) k_mlp_grad(const __nv_bfloat16* wbf, const float* x, const float* t,
                                                              int64_t n, int64_t n_used, int64_t start,
                                                              int64_t stride, float* grad, float* loss) {
  extern __shared__ __align__(16) unsigned char grad_smem[];
  GradShared& S = *reinterpret_cast<GradShared*>(grad_smem);
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  for (int i = tid; i < kNParams; i += kGradThreads) {
    const float w = __bfloat162float(wbf[i]);
    if (i < kB1) S.w1t[(i % kIn) * kH + i / kIn] = w;
    else if (i < kW2) S.b1[i - kB1] = w;
    else if (i < kB2) {
      const int j = (i - kW2) / kH, k = (i - kW2) % kH;
      S.w2[swz(j, k >> 2) + (k & 3)] = w;
      S.w2t[swz(k, j >> 2) + (j & 3)] = w;
    } else if (i < kW3) S.b2[i - kB2] = w;
    else if (i < kB3) S.w3[i - kW3] = w;
    else S.b3[i - kB3] = w;
  }
  if (tid < kH) S.gb1[tid] = S.gb2[tid] = 0.0f;
  if (tid < kOut * kH) S.gw3[tid] = 0.0f;
  if (tid < 4) S.gb3[tid] = 0.0f;
  if (tid == 0) S.loss = 0.0f;
  // this thread's share of the gradient
  float gw2[4][4] = {}, gw1[4][5] = {}, gw3[kOut][4] = {}, gb1[4] = {}, gb2[4] = {}, gb3[kOut] = {}, lsum = 0.0f;
  const int sg = tid >> 6, ig = (tid >> 4) & 3;   // W1: 16 samples and 5 inputs of the 4 units of tx
  const int64_t tiles = (n_used + kTile - 1) / kTile;
  for (int64_t b = blockIdx.x; b < tiles; b += gridDim.x) {
    const int64_t s0 = b * kTile;
    const int ns = (int)(n_used - s0 < kTile ? n_used - s0 : kTile);
    __syncthreads();   // the last tile's inputs and derivatives have been read
    for (int i = tid; i < kTile * kIn; i += kGradThreads) {
      const int s = i / kIn, k = i - s * kIn;
      float v = 0.0f;
      if (s < ns) v = x[((start + (s0 + s) * stride) % n) * kIn + k];
      S.x[i] = v;
      S.xt[k * kTile + s] = v;
    }
    __syncthreads();
    // layer 1: rows are the samples 4 ty.., columns the units 4 tx..
    float a1[4][4], h[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) a1[i][j] = S.b1[4 * tx + j];
    product<false, false>(S.xt, S.w1t, kIn, ty, tx, a1);
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) h[i][j] = gelu_f(a1[i][j]);
    put_rows(S.h1, ty, tx, h);
    put_columns(S.t, ty, tx, h);
    __syncthreads();
    // layer 2
    float a2[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) a2[i][j] = S.b2[4 * tx + j];
    product<true, true>(S.t, S.w2t, kH, ty, tx, a2);
    // layer 3: two sums over the units, by the 16 threads of a row
    float dy[4][kOut];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      float y[kOut] = {};
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        h[i][j] = gelu_f(a2[i][j]);
#pragma unroll
        for (int o = 0; o < kOut; ++o) y[o] = fmaf(S.w3[o * kH + 4 * tx + j], h[i][j], y[o]);
      }
      const int s = 4 * ty + i;
#pragma unroll
      for (int o = 0; o < kOut; ++o) {
#pragma unroll
        for (int m = 8; m > 0; m >>= 1) y[o] += __shfl_xor_sync(0xffffffffu, y[o], m);
        dy[i][o] = 0.0f;
        if (s < ns) {
          const float e = y[o] + S.b3[o] - t[((start + (s0 + s) * stride) % n) * kOut + o];
          dy[i][o] = 2.0f * e / (float)n_used;       // dL/dy
          if (tx == 0) lsum = fmaf(e, e, lsum);
        }
        gb3[o] += dy[i][o];
#pragma unroll
        for (int j = 0; j < 4; ++j) gw3[o][j] = fmaf(dy[i][o], h[i][j], gw3[o][j]);
      }
    }
    // dL/da2, by sample and by unit
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        float d = 0.0f;
#pragma unroll
        for (int o = 0; o < kOut; ++o) d = fmaf(dy[i][o], S.w3[o * kH + 4 * tx + j], d);
        h[i][j] = d * gelu_grad_f(a2[i][j]);
        gb2[j] += h[i][j];
      }
    __syncthreads();   // every thread has read the hidden units by unit
    put_rows(S.da2, ty, tx, h);
    put_columns(S.t, ty, tx, h);
    __syncthreads();
    product<true, true>(S.da2, S.h1, kTile, ty, tx, gw2);   // rows: units j, columns: inputs k
    // dL/da1
    float d1[4][4] = {};
    product<true, true>(S.t, S.w2, kH, ty, tx, d1);
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        d1[i][j] *= gelu_grad_f(a1[i][j]);
        gb1[j] += d1[i][j];
      }
    __syncthreads();   // every thread has read dL/da2 by unit
    put_rows(S.t, ty, tx, d1);
    __syncthreads();
#pragma unroll 4
    for (int s = 16 * sg; s < 16 * sg + 16; ++s) {
      const float4 u = *reinterpret_cast<const float4*>(S.t + swz(s, tx));
      const float us[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
      for (int i = 0; i < 5; ++i) {
        const float v = S.x[s * kIn + 5 * ig + i];
#pragma unroll
        for (int j = 0; j < 4; ++j) gw1[j][i] = fmaf(us[j], v, gw1[j][i]);
      }
    }
  }
  // the CTA's sums: W1 over its four sample groups, the rest over its rows
  __syncthreads();
  float* part = S.h1;   // [4][kH * kIn] floats, over h1 and the matrices behind it
#pragma unroll
  for (int j = 0; j < 4; ++j)
#pragma unroll
    for (int i = 0; i < 5; ++i) part[sg * kH * kIn + (4 * tx + j) * kIn + 5 * ig + i] = gw1[j][i];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    atomicAdd(&S.gb1[4 * tx + j], gb1[j]);
    atomicAdd(&S.gb2[4 * tx + j], gb2[j]);
#pragma unroll
    for (int o = 0; o < kOut; ++o) atomicAdd(&S.gw3[o * kH + 4 * tx + j], gw3[o][j]);
  }
  if (tx == 0) {
    atomicAdd(&S.loss, lsum);
#pragma unroll
    for (int o = 0; o < kOut; ++o) atomicAdd(&S.gb3[o], gb3[o]);
  }
  __syncthreads();
  const bool vec = ((uintptr_t)grad & 15) == 0;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    float* g = grad + kW2 + (4 * ty + i) * kH + 4 * tx;
    if (vec) {
      atomicAdd(reinterpret_cast<float4*>(g), make_float4(gw2[i][0], gw2[i][1], gw2[i][2], gw2[i][3]));
    } else {
#pragma unroll
      for (int j = 0; j < 4; ++j) atomicAdd(g + j, gw2[i][j]);
    }
  }
  for (int i = tid; i < kH * kIn; i += kGradThreads)
    atomicAdd(grad + kW1 + i, (part[i] + part[kH * kIn + i]) + (part[2 * kH * kIn + i] + part[3 * kH * kIn + i]));
  if (tid < kH) {
    atomicAdd(grad + kB1 + tid, S.gb1[tid]);
    atomicAdd(grad + kB2 + tid, S.gb2[tid]);
  }
  if (tid < kOut * kH) atomicAdd(grad + kW3 + tid, S.gw3[tid]);
  if (tid < kOut) atomicAdd(grad + kB3 + tid, S.gb3[tid]);
  if (tid == 0) atomicAdd(loss, S.loss / (float)n_used);
}
static_assert(4 * kH * kIn <= 2 * kTile * kH, "the partial sums of W1 fit h1 and the matrix behind it");

// Adam step on the FP32 master parameters; refreshes the BF16 copies (the
// training layout and the clip kernel's input-major one) and clears the
// gradient for the next batch.
__global__ void k_adam(float* theta, __nv_bfloat16* wbf, __nv_bfloat16* wbt, float* m, float* v, float* grad, float lr,
                       float b1, float b2, float eps, float c1, float c2) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= kNParams) return;
  const float g = grad[i];
  const float mi = b1 * m[i] + (1.0f - b1) * g;
  const float vi = b2 * v[i] + (1.0f - b2) * g * g;
  m[i] = mi;
  v[i] = vi;
  const float th = theta[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
  theta[i] = th;
  wbf[i] = __float2bfloat16_rn(th);
  wbt[mlp_transposed_index(i)] = __float2bfloat16_rn(th);
  grad[i] = 0.0f;
}

__global__ void k_mlp_forward(const __nv_bfloat16* wbf, const float* x, int64_t n, float* y) {
  __shared__ float W[kNParams];
  load_weights(wbf, W);
  __syncthreads();
  const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= n) return;
  float in[kIn], out[kOut];
#pragma unroll
  for (int k = 0; k < kIn; ++k) in[k] = x[s * kIn + k];
  mlp_eval(W, in, out);
  y[s * kOut] = out[0];
  y[s * kOut + 1] = out[1];
}

// p[0 .. n) and, with q, *q = 0.
__global__ void k_zero(float* p, int64_t n, float* q) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) p[i] = 0.0f;
  if (i == 0 && q) *q = 0.0f;
}

// ---- training-set preparation: keep finite rows, normalise, compact ----
constexpr int kPrepThreads = 256;
constexpr int kPrepRows = 1024;   // rows per CTA

__device__ __forceinline__ bool row_valid(const float* f, const float* t, int64_t r) {
  bool ok = isfinite(t[2 * r]) && isfinite(t[2 * r + 1]);
#pragma unroll
  for (int k = 0; k < kIn; ++k) ok = ok && isfinite(f[r * kIn + k]);
  return ok;
}

// Per CTA: number of valid rows, and FP64 sums and sums of squares of the
// 22 columns over them (partials [blocks][2][22]).
__global__ void __launch_bounds__(kPrepThreads) k_prep_stats(const float* f, const float* t, int64_t n,
                                                             int32_t* cnt, double* part) {
  __shared__ double red[2 * (kIn + kOut)][kPrepThreads / 32];
  __shared__ int rc[kPrepThreads / 32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t r0 = (int64_t)blockIdx.x * kPrepRows;
  double sum[kIn + kOut], sq[kIn + kOut];
#pragma unroll
  for (int c = 0; c < kIn + kOut; ++c) sum[c] = sq[c] = 0.0;
  int valid = 0;
  for (int i = tid; i < kPrepRows; i += kPrepThreads) {
    const int64_t r = r0 + i;
    if (r >= n || !row_valid(f, t, r)) continue;
    ++valid;
#pragma unroll
    for (int c = 0; c < kIn + kOut; ++c) {
      const double v = c < kIn ? (double)f[r * kIn + c] : (double)t[2 * r + c - kIn];
      sum[c] += v;
      sq[c] += v * v;
    }
  }
#pragma unroll
  for (int c = 0; c < kIn + kOut; ++c) {
    for (int o = 16; o > 0; o >>= 1) {
      sum[c] += __shfl_xor_sync(0xffffffffu, sum[c], o);
      sq[c] += __shfl_xor_sync(0xffffffffu, sq[c], o);
    }
  }
  valid = __reduce_add_sync(0xffffffffu, valid);
  if (lane == 0) {
#pragma unroll
    for (int c = 0; c < kIn + kOut; ++c) {
      red[c][warp] = sum[c];
      red[kIn + kOut + c][warp] = sq[c];
    }
    rc[warp] = valid;
  }
  __syncthreads();
  if (tid < 2 * (kIn + kOut)) {
    double x = 0.0;
    for (int w = 0; w < kPrepThreads / 32; ++w) x += red[tid][w];
    part[(int64_t)blockIdx.x * 2 * (kIn + kOut) + tid] = x;
  }
  if (tid == 0) {
    int x = 0;
    for (int w = 0; w < kPrepThreads / 32; ++w) x += rc[w];
    cnt[blockIdx.x] = x;
  }
}

// Valid rows of CTA b go, in order, to rows base[b] ... of (x, t), normalised.
__global__ void __launch_bounds__(kPrepThreads) k_prep_scatter(const float* f, const float* t, int64_t n,
                                                               const int64_t* base, const float* norm, float* x,
                                                               float* y) {
  __shared__ int wsum[kPrepThreads / 32];
  __shared__ int64_t off;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t r0 = (int64_t)blockIdx.x * kPrepRows;
  if (tid == 0) off = base[blockIdx.x];
  __syncthreads();
  for (int i0 = 0; i0 < kPrepRows; i0 += kPrepThreads) {
    const int64_t r = r0 + i0 + tid;
    const bool ok = r < n && row_valid(f, t, r);
    const unsigned m = __ballot_sync(0xffffffffu, ok);
    if (lane == 0) wsum[warp] = __popc(m);
    __syncthreads();
    int before = __popc(m & ((1u << lane) - 1u)), total = 0;
    for (int w = 0; w < kPrepThreads / 32; ++w) {
      if (w < warp) before += wsum[w];
      total += wsum[w];
    }
    if (ok) {
      const int64_t o = off + before;
#pragma unroll
      for (int k = 0; k < kIn; ++k) x[o * kIn + k] = (f[r * kIn + k] - norm[k]) / norm[kIn + k];
#pragma unroll
      for (int k = 0; k < kOut; ++k) y[o * kOut + k] = (t[r * kOut + k] - norm[2 * kIn + k]) / norm[2 * kIn + kOut + k];
    }
    __syncthreads();
    if (tid == 0) off += total;
    __syncthreads();
  }
}

}  // namespace

int64_t prep_blocks(int64_t n) { return (n + kPrepRows - 1) / kPrepRows; }

cudaError_t launch_prep_stats(const float* f, const float* t, int64_t n, int32_t* cnt, double* part, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  k_prep_stats<<<(unsigned)prep_blocks(n), kPrepThreads, 0, s>>>(f, t, n, cnt, part);
  return cudaGetLastError();
}

cudaError_t launch_prep_scatter(const float* f, const float* t, int64_t n, const int64_t* base, const float* norm,
                                float* x, float* y, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  k_prep_scatter<<<(unsigned)prep_blocks(n), kPrepThreads, 0, s>>>(f, t, n, base, norm, x, y);
  return cudaGetLastError();
}

size_t mlp_grad_smem() { return sizeof(GradShared); }

cudaError_t launch_mlp_grad(const __nv_bfloat16* wbf, const float* x, const float* t, int64_t n, int64_t n_used,
                            int64_t start, int64_t stride, float* grad, float* loss, cudaStream_t s) {
  if (n_used <= 0) return cudaSuccess;
  const size_t smem = mlp_grad_smem();
  cudaError_t e = cudaFuncSetAttribute(k_mlp_grad, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const int64_t tiles = (n_used + kTile - 1) / kTile;
  const int64_t blocks = tiles < kGradCtas ? tiles : kGradCtas;
  k_mlp_grad<<<(unsigned)blocks, kGradThreads, smem, s>>>(wbf, x, t, n, n_used, start, stride, grad, loss);
  return cudaGetLastError();
}

cudaError_t launch_adam(float* theta, __nv_bfloat16* wbf, __nv_bfloat16* wbt, float* m, float* v, float* grad, float lr,
                        int64_t step, cudaStream_t s) {
  const float b1 = 0.9f, b2 = 0.999f;
  const float c1 = 1.0f - powf(b1, (float)step), c2 = 1.0f - powf(b2, (float)step);
  k_adam<<<(kNParams + 255) / 256, 256, 0, s>>>(theta, wbf, wbt, m, v, grad, lr, b1, b2, 1e-8f, c1, c2);
  return cudaGetLastError();
}

cudaError_t launch_mlp_forward(const __nv_bfloat16* wbf, const float* x, int64_t n, float* y, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  k_mlp_forward<<<(unsigned)((n + 127) / 128), 128, 0, s>>>(wbf, x, n, y);
  return cudaGetLastError();
}

cudaError_t launch_zero(float* p, int64_t n, cudaStream_t s, float* q) {
  if (n <= 0) return cudaSuccess;
  k_zero<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(p, n, q);
  return cudaGetLastError();
}

}  // namespace sep
