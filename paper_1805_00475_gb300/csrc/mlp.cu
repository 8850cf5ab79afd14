// The learned edge scorer: a 3-layer perceptron F -> H -> H -> 1 (ReLU),
// fp32 training (forward, backward with the squared-error loss, Adam) and
// bf16 inference, as hand-written CUDA kernels.
//
// Parameter layout (fp32, flat): W1[F][H], b1[H], W2[H][H], b2[H], w3[H], b3.
// Activations saved for the backward pass are the post-ReLU values h1, h2
// ([rows][H] each).
//
// The H x H products (the layer, its transpose in the backward pass and the
// weight gradient) are fp32 FMAs on register tiles fed from shared memory: a
// thread owns 4 x 4 (or 2 x 4) results, so each step of the inner loop reads
// two 16-byte vectors for 16 FMAs.  They are small (34 MFMA at 2048 rows,
// about 1 us of the GPU's FMA rate); what bounds them is getting all SMs to
// work on them and the latency of staging W2 (64 KiB) once per CTA, so tiles
// are narrow (16 rows) and a CTA keeps W2 for every tile that it takes.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <string>

#include "tnc_internal.h"

namespace tnc_mlp {

constexpr int F = TNC_MLP_FEATURES;
constexpr int H = TNC_MLP_HIDDEN;
constexpr int kRows = 16;      // rows of a tile: 128 tiles at 2048 rows
constexpr int kPitch = H + 4;  // row pitch of W2 in shared memory: 16-byte aligned, transposed writes spread over banks
constexpr int OFF_W1 = 0, OFF_B1 = F * H, OFF_W2 = OFF_B1 + H, OFF_B2 = OFF_W2 + H * H, OFF_W3 = OFF_B2 + H,
              OFF_B3 = OFF_W3 + H, N_PARAMS = OFF_B3 + 1;
static_assert(N_PARAMS == TNC_MLP_PARAMS, "parameter count");

template <typename WT>
__device__ __forceinline__ float ld(const WT* p, int i);
template <>
__device__ __forceinline__ float ld<float>(const float* p, int i) {
  return p[i];
}
template <>
__device__ __forceinline__ float ld<__nv_bfloat16>(const __nv_bfloat16* p, int i) {
  return __bfloat162float(p[i]);
}

// Four consecutive weights from shared memory, from a position aligned to their size.
__device__ __forceinline__ float4 ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ float4 ld4(const __nv_bfloat16* p) {  // (a bf16 is the upper half of a float)
  const uint2 w = *reinterpret_cast<const uint2*>(p);
  return make_float4(__uint_as_float(w.x << 16), __uint_as_float(w.x & 0xFFFF0000u), __uint_as_float(w.y << 16),
                     __uint_as_float(w.y & 0xFFFF0000u));
}

// W2 in shared memory as it is, S[j * kPitch + t] = W2[j][t].  vec: P is
// 16-byte aligned (the caller's pointer may be any element's).
template <typename WT>
__device__ __forceinline__ void stage_w2(const WT* __restrict__ P, WT* S, bool vec) {
  constexpr int N = 16 / sizeof(WT);  // weights of a 16-byte copy
  if (vec) {
#pragma unroll 8
    for (int i = threadIdx.x * N; i < H * H; i += H * N) {
      const uint4 v = *reinterpret_cast<const uint4*>(P + OFF_W2 + i);
      WT* d = S + (i / H) * kPitch + i % H;
      if constexpr (sizeof(WT) == 4) {
        *reinterpret_cast<uint4*>(d) = v;
      } else {  // (rows of kPitch bf16 are 8-byte aligned)
        reinterpret_cast<uint2*>(d)[0] = make_uint2(v.x, v.y);
        reinterpret_cast<uint2*>(d)[1] = make_uint2(v.z, v.w);
      }
    }
  } else {
#pragma unroll 8
    for (int i = threadIdx.x; i < H * H; i += H) S[(i / H) * kPitch + i % H] = P[OFF_W2 + i];
  }
}

// W2, a tile of activations, its inputs: 75.0 KiB, or 42.0 KiB with bf16
// weights (below the 48 KiB that need no opt-in, which costs 1 us per call)
template <typename WT>
constexpr size_t kSmemBytes = H * kPitch * sizeof(WT) + (H * kRows + kRows * F) * sizeof(float);

// y[r] = w3 . relu(W2^T relu(W1^T x_r + b1) + b2) + b3; optionally saves h1, h2.
// H threads; in the H x H layer a warp owns 4 rows of the tile and a lane 4
// consecutive hidden units.  The sums run over the units in ascending order.
// 2048 rows: 23.6 us -> 8.0 us (fp32 weights): the latency of one tile (staging
// W2, 128 steps of the inner loop); 70000 rows 96 -> 84 us, bound by the
// shared-memory reads of the inner loop.  bf16 weights: 22.6 -> 8.3 us a call
// among others (its launch), 70000 rows 98 -> 75 us.
template <typename WT>
__global__ void __launch_bounds__(H) mlp_forward_kernel(const WT* __restrict__ P, const float* __restrict__ X,
                                                        int64_t rows, float* __restrict__ Y, float* __restrict__ h1s,
                                                        float* __restrict__ h2s, int vec) {
  extern __shared__ __align__(16) float sm[];
  WT* w2 = reinterpret_cast<WT*>(sm);
  float* h1 = reinterpret_cast<float*>(w2 + H * kPitch);  // h1[j * kRows + r]
  float* xs = h1 + H * kRows;   // xs[r * F + f]
  const int t = threadIdx.x, lane = t & 31, r4 = 4 * (t >> 5), c4 = 4 * lane;
  stage_w2(P, w2, vec != 0);
  float w1[F];
#pragma unroll
  for (int f = 0; f < F; f++) w1[f] = ld(P, OFF_W1 + f * H + t);
  const float b1 = ld(P, OFF_B1 + t), b3 = ld(P, OFF_B3);
  float b2[4], w3[4];
#pragma unroll
  for (int c = 0; c < 4; c++) {
    b2[c] = ld(P, OFF_B2 + c4 + c);
    w3[c] = ld(P, OFF_W3 + c4 + c);
  }
  for (int64_t r0 = (int64_t)blockIdx.x * kRows; r0 < rows; r0 += (int64_t)gridDim.x * kRows) {
    for (int i = t; i < kRows * F; i += H) {
      const int64_t r = r0 + i / F;
      xs[i] = r < rows ? X[r * F + i % F] : 0.f;
    }
    __syncthreads();
    float a[kRows];
#pragma unroll
    for (int r = 0; r < kRows; r++) {
      a[r] = b1;
#pragma unroll
      for (int f = 0; f < F; f++) a[r] = fmaf(xs[r * F + f], w1[f], a[r]);
      a[r] = fmaxf(a[r], 0.f);
    }
#pragma unroll
    for (int r = 0; r < kRows; r += 4)
      *reinterpret_cast<float4*>(h1 + t * kRows + r) = make_float4(a[r], a[r + 1], a[r + 2], a[r + 3]);
    if (h1s) {
#pragma unroll
      for (int r = 0; r < kRows; r++)
        if (r0 + r < rows) h1s[(r0 + r) * H + t] = a[r];
    }
    __syncthreads();
    float acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; i++)
#pragma unroll
      for (int c = 0; c < 4; c++) acc[i][c] = b2[c];
#pragma unroll 8
    for (int j = 0; j < H; j++) {
      const float4 h = *reinterpret_cast<const float4*>(h1 + j * kRows + r4);
      const float4 w = ld4(w2 + j * kPitch + c4);
      const float hv[4] = {h.x, h.y, h.z, h.w}, wv[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
      for (int i = 0; i < 4; i++)
#pragma unroll
        for (int c = 0; c < 4; c++) acc[i][c] = fmaf(hv[i], wv[c], acc[i][c]);
    }
#pragma unroll
    for (int i = 0; i < 4; i++) {
      const int64_t r = r0 + r4 + i;
      float v = 0.f, h2[4];
#pragma unroll
      for (int c = 0; c < 4; c++) {
        h2[c] = fmaxf(acc[i][c], 0.f);
        v = fmaf(h2[c], w3[c], v);
      }
      if (h2s && r < rows) {
        float* d = h2s + r * H + c4;
        if (vec) {
          *reinterpret_cast<float4*>(d) = make_float4(h2[0], h2[1], h2[2], h2[3]);
        } else {
#pragma unroll
          for (int c = 0; c < 4; c++) d[c] = h2[c];
        }
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      if (lane == 0 && r < rows) Y[r] = v + b3;
    }
    // (the next tile's first barrier separates these reads of h1 from its writes)
  }
}

// Backward pass of L = (1/n) sum_r (y_r - t_r)^2 over the n = `rows` rows of
// this call.  Pass 1 (per row): dy, dh2 = dy w3 [h2 > 0], dh1 = W2 dh2 [h1 > 0].
// The same tiling as the forward pass, W2 staged transposed (S[u][t] =
// W2[t][u]); the 128 products of a dh1 are summed 32 at a time.
// 2048 rows: 28.1 us -> 11.8 us.
__global__ void __launch_bounds__(H) mlp_backward_rows_kernel(const float* __restrict__ P,
                                                              const float* __restrict__ h1s,
                                                              const float* __restrict__ h2s,
                                                              const float* __restrict__ Y, const float* __restrict__ T,
                                                              int64_t rows, float* __restrict__ dy_out,
                                                              float* __restrict__ dh1s, float* __restrict__ dh2s) {
  extern __shared__ __align__(16) float sm[];
  float* w2t = sm;
  float* dh2 = w2t + H * kPitch;  // dh2[u * kRows + r]
  float* dy = dh2 + H * kRows;
  const int t = threadIdx.x, lane = t & 31, r4 = 4 * (t >> 5), c4 = 4 * lane;
  // a warp moves 8 u x 4 t: whole 32-byte sectors in, 32 distinct banks out (4 u + t)
#pragma unroll 8
  for (int i = t; i < H * H; i += H) {
    const int q = i >> 5, u = 8 * (q & (H / 8 - 1)) + (lane & 7), c = 4 * (q / (H / 8)) + (lane >> 3);
    w2t[u * kPitch + c] = P[OFF_W2 + c * H + u];
  }
  const float w3 = P[OFF_W3 + t];
  for (int64_t r0 = (int64_t)blockIdx.x * kRows; r0 < rows; r0 += (int64_t)gridDim.x * kRows) {
    if (t < kRows) {
      const float d = r0 + t < rows ? 2.f * (Y[r0 + t] - T[r0 + t]) / (float)rows : 0.f;
      dy[t] = d;
      if (r0 + t < rows) dy_out[r0 + t] = d;
    }
    float h2[kRows];
#pragma unroll
    for (int r = 0; r < kRows; r++) h2[r] = r0 + r < rows ? h2s[(r0 + r) * H + t] : 0.f;
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kRows; r++) {
      h2[r] = h2[r] > 0.f ? dy[r] * w3 : 0.f;
      if (r0 + r < rows) dh2s[(r0 + r) * H + t] = h2[r];
    }
#pragma unroll
    for (int r = 0; r < kRows; r += 4)
      *reinterpret_cast<float4*>(dh2 + t * kRows + r) = make_float4(h2[r], h2[r + 1], h2[r + 2], h2[r + 3]);
    __syncthreads();
    float d1[4][4];
#pragma unroll
    for (int i = 0; i < 4; i++)
#pragma unroll
      for (int c = 0; c < 4; c++) d1[i][c] = 0.f;
#pragma unroll 1
    for (int pass = 0; pass < 4; pass++) {
      float s[4][4];
#pragma unroll
      for (int i = 0; i < 4; i++)
#pragma unroll
        for (int c = 0; c < 4; c++) s[i][c] = 0.f;
#pragma unroll 8
      for (int u = pass * (H / 4); u < (pass + 1) * (H / 4); u++) {
        const float4 h = *reinterpret_cast<const float4*>(dh2 + u * kRows + r4);
        const float4 w = *reinterpret_cast<const float4*>(w2t + u * kPitch + c4);
        const float hv[4] = {h.x, h.y, h.z, h.w}, wv[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
        for (int i = 0; i < 4; i++)
#pragma unroll
          for (int c = 0; c < 4; c++) s[i][c] = fmaf(hv[i], wv[c], s[i][c]);
      }
#pragma unroll
      for (int i = 0; i < 4; i++)
#pragma unroll
        for (int c = 0; c < 4; c++) d1[i][c] += s[i][c];
    }
#pragma unroll
    for (int i = 0; i < 4; i++) {
      const int64_t r = r0 + r4 + i;
      if (r < rows) {
#pragma unroll
        for (int c = 0; c < 4; c++) dh1s[r * H + c4 + c] = h1s[r * H + c4 + c] > 0.f ? d1[i][c] : 0.f;
      }
    }
    __syncthreads();  // dh2 and dy are free for the next tile
  }
}

// Pass 2: the parameter gradients, sums over the rows.  The rows are cut into
// slices so that the whole chip shares them (a CTA per 128 gradients walking
// every row took 163.7 us at 2048 rows, a serial chain of 2048 loads);
// slice s writes its partial gradients to part + s N_PARAMS and
// a second kernel adds the slices in order (no atomics: the result does not
// depend on the schedule).  32 slices: 64 rows each at 2048 rows, 192 CTAs;
// 8.5 us, and 3.0 us to add them.
//   blockIdx.x 0..3: dW2[j][t] = sum_r h1[r][j] dh2[r][t], a 64 x 64 quarter
//   blockIdx.x 4:    dW1[f][t] = sum_r x[r][f] dh1[r][t], db1[t]
//   blockIdx.x 5:    db2[t], dw3[t] = sum_r h2[r][t] dy[r], db3
constexpr int kMaxSplits = 32;
constexpr int kSliceRows = 64;  // rows staged at a time, and the fewest that make a slice
constexpr int kParamThreads = 256;

int splits_for(int64_t rows) { return (int)std::min<int64_t>(kMaxSplits, (rows + kSliceRows - 1) / kSliceRows); }

__global__ void __launch_bounds__(kParamThreads) mlp_backward_params_kernel(
    const float* __restrict__ X, const float* __restrict__ h1s, const float* __restrict__ h2s,
    const float* __restrict__ dys, const float* __restrict__ dh1s, const float* __restrict__ dh2s, int64_t rows,
    int64_t slice, float* __restrict__ part) {
  __shared__ __align__(16) float sa[kSliceRows][64];
  __shared__ __align__(16) float sb[kSliceRows][64];
  const int t = threadIdx.x, b = blockIdx.x;
  const int64_t lo = (int64_t)blockIdx.y * slice, hi = lo + slice < rows ? lo + slice : rows;
  float* G = part + (size_t)blockIdx.y * N_PARAMS;
  if (b < 4) {
    const int j0 = (b & 1) * 64, t0 = (b >> 1) * 64;
    const int jr = 4 * (t >> 4), tc = 4 * (t & 15);
    float g[4][4];
#pragma unroll
    for (int i = 0; i < 4; i++)
#pragma unroll
      for (int c = 0; c < 4; c++) g[i][c] = 0.f;
    for (int64_t r0 = lo; r0 < hi; r0 += kSliceRows) {
      __syncthreads();
#pragma unroll 8
      for (int i = t; i < kSliceRows * 64; i += kParamThreads) {
        const int64_t r = r0 + i / 64;
        sa[i / 64][i % 64] = r < hi ? h1s[r * H + j0 + i % 64] : 0.f;
        sb[i / 64][i % 64] = r < hi ? dh2s[r * H + t0 + i % 64] : 0.f;
      }
      __syncthreads();
      const int nr = (int)(hi - r0 < kSliceRows ? hi - r0 : kSliceRows);  // (rows beyond are zero)
#pragma unroll 8
      for (int r = 0; r < nr; r++) {
        const float4 x = *reinterpret_cast<const float4*>(&sa[r][jr]);
        const float4 y = *reinterpret_cast<const float4*>(&sb[r][tc]);
        const float xv[4] = {x.x, x.y, x.z, x.w}, yv[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
        for (int i = 0; i < 4; i++)
#pragma unroll
          for (int c = 0; c < 4; c++) g[i][c] = fmaf(xv[i], yv[c], g[i][c]);
      }
    }
#pragma unroll
    for (int i = 0; i < 4; i++)
#pragma unroll
      for (int c = 0; c < 4; c++) G[OFF_W2 + (j0 + jr + i) * H + t0 + tc + c] = g[i][c];
    return;
  }
  // two halves of the threads take alternate rows of the slice
  const int col = t & (H - 1), half = t >> 7;
  float* red = &sa[0][0];
  if (b == 4) {
    float g[F], g1 = 0.f;
#pragma unroll
    for (int f = 0; f < F; f++) g[f] = 0.f;
#pragma unroll 4
    for (int64_t r = lo + half; r < hi; r += 2) {
      const float d = dh1s[r * H + col];
      g1 += d;
#pragma unroll
      for (int f = 0; f < F; f++) g[f] = fmaf(X[r * F + f], d, g[f]);
    }
    if (half) {
#pragma unroll
      for (int f = 0; f < F; f++) red[f * H + col] = g[f];
      red[F * H + col] = g1;
    }
    __syncthreads();
    if (!half) {
#pragma unroll
      for (int f = 0; f < F; f++) G[OFF_W1 + f * H + col] = g[f] + red[f * H + col];
      G[OFF_B1 + col] = g1 + red[F * H + col];
    }
    return;
  }
  float g2 = 0.f, g3 = 0.f, gb3 = 0.f;
#pragma unroll 4
  for (int64_t r = lo + half; r < hi; r += 2) {
    const float d = dys[r];
    g2 += dh2s[r * H + col];
    g3 = fmaf(h2s[r * H + col], d, g3);
    gb3 += d;
  }
  if (half) {
    red[col] = g2;
    red[H + col] = g3;
    if (col == 0) red[2 * H] = gb3;
  }
  __syncthreads();
  if (!half) {
    G[OFF_B2 + col] = g2 + red[col];
    G[OFF_W3 + col] = g3 + red[H + col];
    if (col == 0) G[OFF_B3] = gb3 + red[2 * H];
  }
}

// Gradients = the slices' partial gradients, added in slice order.
__global__ void __launch_bounds__(128) mlp_add_slices_kernel(const float* __restrict__ part, int n,
                                                             float* __restrict__ G) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N_PARAMS) return;
  float g = 0.f;
#pragma unroll 8
  for (int s = 0; s < n; s++) g += part[(size_t)s * N_PARAMS + i];
  G[i] = g;
}

__global__ void adam_kernel(float* __restrict__ P, const float* __restrict__ G, float* __restrict__ M,
                            float* __restrict__ V, int n, float lr, float b1, float b2, float eps, float c1, float c2) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const float g = G[i];
    const float m = b1 * M[i] + (1.f - b1) * g;
    const float v = b2 * V[i] + (1.f - b2) * g * g;
    M[i] = m;
    V[i] = v;
    P[i] -= lr * (m / c1) / (sqrtf(v / c2) + eps);
  }
}

__global__ void to_bf16_kernel(const float* __restrict__ P, __nv_bfloat16* __restrict__ Q, int n) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) Q[i] = __float2bfloat16(P[i]);
}

// Squared error of a batch, accumulated into loss[0] (sum over rows).
__global__ void sqerr_kernel(const float* __restrict__ Y, const float* __restrict__ T, int64_t rows, float* loss) {
  float s = 0.f;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < rows; i += (int64_t)gridDim.x * blockDim.x) {
    const float d = Y[i] - T[i];
    s += d * d;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) atomicAdd(loss, s);
}

}  // namespace tnc_mlp

using namespace tnc;

namespace {
#define MLP_TRY(call)                                                                               \
  do {                                                                                              \
    cudaError_t e_ = (call);                                                                        \
    if (e_ != cudaSuccess) return set_error(TNC_ERR_CUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
  } while (0)

// CTAs for the tiles of `rows` rows: one per tile, at most three per SM (the
// shared memory they need), each keeping W2 for all its tiles.
unsigned blocks_for(int64_t rows) {
  return (unsigned)std::min<int64_t>((rows + tnc_mlp::kRows - 1) / tnc_mlp::kRows, 3 * 152);
}

bool aligned16(const void* p) { return ((uintptr_t)p & 15u) == 0; }

// The fp32 kernels' dynamic shared memory limit (a property of the kernel on
// the current device; setting it again is harmless).
template <typename K>
int allow_smem(K kernel) {
  MLP_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)tnc_mlp::kSmemBytes<float>));
  return TNC_OK;
}
}  // namespace

namespace tnc {

// Synchronous copy for host code compiled without CUDA headers: dir 0 = host
// to device, 1 = device to host (the stream is synchronised).
void copy_device(void* dst, const void* src, size_t bytes, int dir, void* stream, int* rc) {
  cudaStream_t st = (cudaStream_t)stream;
  cudaError_t e = cudaMemcpyAsync(dst, src, bytes, dir == 0 ? cudaMemcpyHostToDevice : cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) *rc = set_error(TNC_ERR_CUDA, std::string("copy: ") + cudaGetErrorString(e));
}

int mlp_forward_dev(const float* P, const float* X, int64_t rows, float* Y, float* h1, float* h2, void* stream) {
  if (rows <= 0) return TNC_OK;
  if (int rc = allow_smem(tnc_mlp::mlp_forward_kernel<float>)) return rc;
  const int vec = aligned16(P) && aligned16(h2);
  tnc_mlp::mlp_forward_kernel<float><<<blocks_for(rows), tnc_mlp::H, tnc_mlp::kSmemBytes<float>, (cudaStream_t)stream>>>(
      P, X, rows, Y, h1, h2, vec);
  MLP_TRY(cudaGetLastError());
  return TNC_OK;
}

int mlp_forward_bf16_dev(const void* Pb, const float* X, int64_t rows, float* Y, void* stream) {
  if (rows <= 0) return TNC_OK;
  tnc_mlp::mlp_forward_kernel<__nv_bfloat16>
      <<<blocks_for(rows), tnc_mlp::H, tnc_mlp::kSmemBytes<__nv_bfloat16>, (cudaStream_t)stream>>>(
          (const __nv_bfloat16*)Pb, X, rows, Y, nullptr, nullptr, aligned16(Pb));
  MLP_TRY(cudaGetLastError());
  return TNC_OK;
}

}  // namespace tnc

extern "C" {

int tnc_mlp_forward(const float* d_params, const float* d_x, int64_t rows, float* d_y, float* d_h1, float* d_h2,
                    void* cuda_stream) {
  clear_error();
  if (!d_params || !d_x || !d_y || rows < 0) return set_error(TNC_ERR_INVALID, "bad mlp_forward arguments");
  return mlp_forward_dev(d_params, d_x, rows, d_y, d_h1, d_h2, cuda_stream);
}

int tnc_mlp_backward(const float* d_params, const float* d_x, const float* d_h1, const float* d_h2, const float* d_y,
                     const float* d_t, int64_t rows, float* d_scratch, float* d_grads, void* cuda_stream) {
  clear_error();
  if (!d_params || !d_x || !d_h1 || !d_h2 || !d_y || !d_t || !d_scratch || !d_grads || rows < 0)
    return set_error(TNC_ERR_INVALID, "bad mlp_backward arguments");
  cudaStream_t st = (cudaStream_t)cuda_stream;
  if (rows == 0) {
    MLP_TRY(cudaMemsetAsync(d_grads, 0, (size_t)TNC_MLP_PARAMS * sizeof(float), st));
    return TNC_OK;
  }
  float* dy = d_scratch;
  float* dh1 = dy + rows;
  float* dh2 = dh1 + rows * TNC_MLP_HIDDEN;
  float* part = dh2 + rows * TNC_MLP_HIDDEN;
  if (int rc = allow_smem(tnc_mlp::mlp_backward_rows_kernel)) return rc;
  tnc_mlp::mlp_backward_rows_kernel<<<blocks_for(rows), tnc_mlp::H, tnc_mlp::kSmemBytes<float>, st>>>(
      d_params, d_h1, d_h2, d_y, d_t, rows, dy, dh1, dh2);
  const int64_t slice = (rows + tnc_mlp::splits_for(rows) - 1) / tnc_mlp::splits_for(rows);
  const int n = (int)((rows + slice - 1) / slice);
  tnc_mlp::mlp_backward_params_kernel<<<dim3(6, (unsigned)n), tnc_mlp::kParamThreads, 0, st>>>(
      d_x, d_h1, d_h2, dy, dh1, dh2, rows, slice, n > 1 ? part : d_grads);
  if (n > 1)
    tnc_mlp::mlp_add_slices_kernel<<<(TNC_MLP_PARAMS + 127) / 128, 128, 0, st>>>(part, n, d_grads);
  MLP_TRY(cudaGetLastError());
  return TNC_OK;
}

int tnc_mlp_adam(float* d_params, const float* d_grads, float* d_m, float* d_v, int32_t step, float lr,
                 void* cuda_stream) {
  clear_error();
  if (!d_params || !d_grads || !d_m || !d_v || step < 1) return set_error(TNC_ERR_INVALID, "bad mlp_adam arguments");
  const float b1 = 0.9f, b2 = 0.999f;
  const float c1 = 1.f - std::pow(b1, (float)step), c2 = 1.f - std::pow(b2, (float)step);
  tnc_mlp::adam_kernel<<<72, 256, 0, (cudaStream_t)cuda_stream>>>(d_params, d_grads, d_m, d_v, TNC_MLP_PARAMS, lr, b1,
                                                                   b2, 1e-8f, c1, c2);
  MLP_TRY(cudaGetLastError());
  return TNC_OK;
}

int tnc_mlp_to_bf16(const float* d_params, void* d_params_bf16, void* cuda_stream) {
  clear_error();
  if (!d_params || !d_params_bf16) return set_error(TNC_ERR_INVALID, "NULL argument");
  tnc_mlp::to_bf16_kernel<<<72, 256, 0, (cudaStream_t)cuda_stream>>>(d_params, (__nv_bfloat16*)d_params_bf16,
                                                                      TNC_MLP_PARAMS);
  MLP_TRY(cudaGetLastError());
  return TNC_OK;
}

int tnc_mlp_forward_bf16(const void* d_params_bf16, const float* d_x, int64_t rows, float* d_y, void* cuda_stream) {
  clear_error();
  if (!d_params_bf16 || !d_x || !d_y || rows < 0) return set_error(TNC_ERR_INVALID, "bad mlp_forward_bf16 arguments");
  return mlp_forward_bf16_dev(d_params_bf16, d_x, rows, d_y, cuda_stream);
}

// dy, dh1 and dh2 of every row, and the row slices' partial gradients
size_t tnc_mlp_backward_scratch_floats(int64_t rows) {
  if (rows <= 0) return 0;
  const int n = tnc_mlp::splits_for(rows);
  return (size_t)rows * (1 + 2 * TNC_MLP_HIDDEN) + (n > 1 ? (size_t)n * TNC_MLP_PARAMS : 0);
}

size_t tnc_mlp_train_workspace_bytes(int32_t batch) {
  if (batch <= 0) return 0;
  const size_t b = (size_t)batch;
  // y, h1, h2 and backward scratch (dy, dh1, dh2) for a batch; grads, Adam m and v; loss
  return (b + 2 * b * TNC_MLP_HIDDEN + tnc_mlp_backward_scratch_floats(batch) + 3 * (size_t)TNC_MLP_PARAMS + 64) *
         sizeof(float);
}

// Mini-batch Adam on the squared error.  Epochs walk the rows in the order
// given (the caller shuffles them once); every epoch's mean loss is reported.
int tnc_mlp_train(float* d_params, const float* d_x, const float* d_t, int64_t rows, int32_t epochs, int32_t batch,
                  float lr, void* d_ws, size_t ws_bytes, void* cuda_stream, float* loss_out) {
  clear_error();
  if (!d_params || !d_x || !d_t || rows <= 0 || epochs <= 0 || batch <= 0 || !d_ws)
    return set_error(TNC_ERR_INVALID, "bad mlp_train arguments");
  if (ws_bytes < tnc_mlp_train_workspace_bytes(batch)) return set_error(TNC_ERR_BUFFER, "workspace too small");
  cudaStream_t st = (cudaStream_t)cuda_stream;
  float* y = (float*)d_ws;
  float* h1 = y + batch;
  float* h2 = h1 + (size_t)batch * TNC_MLP_HIDDEN;
  float* scratch = h2 + (size_t)batch * TNC_MLP_HIDDEN;
  float* g = scratch + tnc_mlp_backward_scratch_floats(batch);
  float* m = g + TNC_MLP_PARAMS;
  float* v = m + TNC_MLP_PARAMS;
  float* loss = v + TNC_MLP_PARAMS;
  MLP_TRY(cudaMemsetAsync(m, 0, 2 * (size_t)TNC_MLP_PARAMS * sizeof(float), st));
  int32_t step = 0;
  for (int32_t e = 0; e < epochs; e++) {
    MLP_TRY(cudaMemsetAsync(loss, 0, sizeof(float), st));
    for (int64_t r0 = 0; r0 < rows; r0 += batch) {
      const int64_t nb = std::min<int64_t>(batch, rows - r0);
      const float* xb = d_x + r0 * TNC_MLP_FEATURES;
      const float* tb = d_t + r0;
      int rc = mlp_forward_dev(d_params, xb, nb, y, h1, h2, st);
      if (rc) return rc;
      tnc_mlp::sqerr_kernel<<<std::max<unsigned>(1, (unsigned)std::min<int64_t>((nb + 255) / 256, 64)), 256, 0, st>>>(
          y, tb, nb, loss);
      rc = tnc_mlp_backward(d_params, xb, h1, h2, y, tb, nb, scratch, g, st);
      if (rc) return rc;
      rc = tnc_mlp_adam(d_params, g, m, v, ++step, lr, st);
      if (rc) return rc;
    }
    if (loss_out) {
      float l = 0;
      MLP_TRY(cudaMemcpyAsync(&l, loss, sizeof(float), cudaMemcpyDeviceToHost, st));
      MLP_TRY(cudaStreamSynchronize(st));
      loss_out[e] = l / (float)rows;
    }
  }
  MLP_TRY(cudaStreamSynchronize(st));
  return TNC_OK;
}

}  // extern "C"
