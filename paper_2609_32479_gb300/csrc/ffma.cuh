// fp32 matrix products on the CUDA cores, one tile per CTA of 256 threads with the
// activations in shared memory and the weights staged through it, and the fp32
// element-wise functions that go with them.
#pragma once

#include <stdint.h>

namespace tf_ffma {

constexpr int NTHREADS = 256;
constexpr int KC = 16;   // k per staged weight chunk (every K of the encoder and the head is a multiple of 16)

// sigma(x) = 1 / (1 + e^-x): the library exponential and the IEEE division (e^-x = inf
// gives 0)
__device__ __forceinline__ float sigm(float x) { return 1.0f / (1.0f + expf(-x)); }
__device__ __forceinline__ float silu(float x) { return x * sigm(x); }

// floats of the two staging buffers for CN columns a thread
__host__ __device__ constexpr int stage_floats(int cn) { return 2 * KC * (16 * cn + 4); }

// The thread's place in a tile of 16 RM rows x 16 CN columns: rows row() + 16 r, r <
// RM; columns col(c), c < CN.  A warp covers 4 rows x 8 column groups, so its reads
// of both operands fall in different banks (rows of the activations are padded to
// 4 mod 32 floats where the width is a multiple of 32).
__device__ __forceinline__ int row0() { return ((threadIdx.x >> 6) << 2) + ((threadIdx.x & 31) >> 3); }
__device__ __forceinline__ int colg() { return (((threadIdx.x >> 5) & 1) << 3) + (threadIdx.x & 7); }
template <int CN>
__device__ __forceinline__ int col(int c) {
  if (CN == 8) return (c >> 2) * 64 + 4 * colg() + (c & 3);
  return CN * colg() + c;
}

// acc[r][c] += sum_k A[row0() + 16 r][k] W[wrow(col(c))][k], k in order.  A: shared
// memory, row stride lda (a multiple of 4); W: global, row stride ldw, 16-byte
// aligned rows; wrow(n) is the weight row of the tile's column n, negative for none
// (read as zeros).  A must be complete only when the first barrier inside is
// passed; the caller synchronises before it changes A.  par: the staging buffer in
// turn, carried from call to call (one barrier a chunk suffices then).
//
// A chunk's global loads are in flight while the chunk before it is computed.  Per
// 4 k a thread loads RM + CN 16-byte pieces for 4 RM CN multiply-adds.
template <int RM, int CN, class WRow>
__device__ __forceinline__ void block_gemm(float (&acc)[RM][CN], const float* __restrict__ A, int lda,
                                           const float* __restrict__ W, int ldw, WRow&& wrow, int K, float* ws,
                                           int& par) {
  constexpr int N = 16 * CN, LDS = N + 4, PER = (N * 4 + NTHREADS - 1) / NTHREADS;
  const int tid = threadIdx.x;
  const float* src[PER];
  float4 v[PER];
#pragma unroll
  for (int i = 0; i < PER; ++i) {
    const int idx = tid + i * NTHREADS, n = idx >> 2, j = idx & 3;
    const int wr = idx < N * 4 ? wrow(n) : -1;
    src[i] = wr >= 0 ? W + (size_t)wr * ldw + 4 * j : nullptr;
    v[i] = src[i] ? __ldg(reinterpret_cast<const float4*>(src[i])) : make_float4(0.f, 0.f, 0.f, 0.f);
  }
  const float* a0 = A + row0() * lda;
  for (int k0 = 0; k0 < K; k0 += KC) {
    float* w = ws + par * (KC * LDS);
    par ^= 1;
#pragma unroll
    for (int i = 0; i < PER; ++i) {
      const int idx = tid + i * NTHREADS, n = idx >> 2, j = idx & 3;
      if (N * 4 % NTHREADS == 0 || idx < N * 4) {
        float* d = w + 4 * j * LDS + n;
        d[0] = v[i].x;
        d[LDS] = v[i].y;
        d[2 * LDS] = v[i].z;
        d[3 * LDS] = v[i].w;
      }
    }
    __syncthreads();
    if (k0 + KC < K) {
#pragma unroll
      for (int i = 0; i < PER; ++i)
        if (src[i]) v[i] = __ldg(reinterpret_cast<const float4*>(src[i] + k0 + KC));
    }
#pragma unroll
    for (int k = 0; k < KC; k += 4) {
      float4 a[RM];
#pragma unroll
      for (int r = 0; r < RM; ++r) a[r] = *reinterpret_cast<const float4*>(a0 + 16 * r * lda + k0 + k);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        float b[CN];
        const float* wk = w + (k + j) * LDS;
        if constexpr (CN == 2) {
          const float2 t = *reinterpret_cast<const float2*>(wk + 2 * colg());
          b[0] = t.x;
          b[1] = t.y;
        } else {
#pragma unroll
          for (int c = 0; c < CN; c += 4) {
            const float4 t = *reinterpret_cast<const float4*>(wk + (c >> 2) * 64 + 4 * colg());
            b[c] = t.x;
            b[c + 1] = t.y;
            b[c + 2] = t.z;
            b[c + 3] = t.w;
          }
        }
#pragma unroll
        for (int r = 0; r < RM; ++r) {
          const float x = j == 0 ? a[r].x : j == 1 ? a[r].y : j == 2 ? a[r].z : a[r].w;
#pragma unroll
          for (int c = 0; c < CN; ++c) acc[r][c] = fmaf(x, b[c], acc[r][c]);
        }
      }
    }
  }
}

template <int RM, int CN>
__device__ __forceinline__ void zero(float (&acc)[RM][CN]) {
#pragma unroll
  for (int r = 0; r < RM; ++r)
#pragma unroll
    for (int c = 0; c < CN; ++c) acc[r][c] = 0.0f;
}

// RMSNorm with gain of rows of D values (D a multiple of 4), one warp a row:
// y = x / sqrt(mean(x^2) + eps) * g.  x and y may be the same row.
__device__ __forceinline__ void norm_row(const float* x, float* y, const float* __restrict__ g, int D, float eps,
                                         int lane) {
  float ss = 0.0f;
  for (int c = lane; c < D; c += 32) ss = fmaf(x[c], x[c], ss);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
  const float inv = 1.0f / sqrtf(ss / (float)D + eps);
  for (int c = lane; c < D; c += 32) y[c] = x[c] * inv * __ldg(g + c);
}

// The head (Sec. 3.2-3.3) on 16 RM pooled vectors in shared memory pv (row stride
// ldp, already normalised): hid = SiLU(W_1 pv + b_1) (128 wide, row stride 132), the
// quantiles W_2 hid + b_2 handed to emit(row, output, value).  hid may not overlap
// pv or ws (stage_floats(8) floats).
template <int RM, class Emit>
__device__ __forceinline__ void head_rows(const float* pv, int ldp, int P, const float* __restrict__ w1,
                                          const float* __restrict__ b1, const float* __restrict__ w2,
                                          const float* __restrict__ b2, int Q, float* hid, float* ws, int& par,
                                          Emit&& emit) {
  {
    float acc[RM][8];
    zero<RM, 8>(acc);
    block_gemm<RM, 8>(acc, pv, ldp, w1, P, [](int n) { return n; }, P, ws, par);
#pragma unroll
    for (int r = 0; r < RM; ++r)
#pragma unroll
      for (int c = 0; c < 8; ++c) hid[(row0() + 16 * r) * 132 + col<8>(c)] = silu(acc[r][c] + __ldg(b1 + col<8>(c)));
  }
  for (int n0 = 0; n0 < Q; n0 += 64) {
    __syncthreads();   // hid complete; the staging buffers at rest
    float acc[RM][4];
    zero<RM, 4>(acc);
    par = 0;
    block_gemm<RM, 4>(acc, hid, 132, w2, 128, [&](int n) { return n0 + n < Q ? n0 + n : -1; }, 128, ws, par);
#pragma unroll
    for (int r = 0; r < RM; ++r)
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const int n = n0 + col<4>(c);
        if (n < Q) emit(row0() + 16 * r, n, acc[r][c] + __ldg(b2 + n));
      }
  }
}

}  // namespace tf_ffma
