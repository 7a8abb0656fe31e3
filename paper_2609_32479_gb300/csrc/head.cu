// The regression head (Sec. 3.2-3.3) on given pooled vectors: RMSNorm, W_h1 with
// SiLU, W_h2, medians, for the kernel paths that leave the pooled vectors in global
// memory.  fp32 on the CUDA cores.
#include <cuda_runtime.h>
#include <math.h>

#include "ffma.cuh"
#include "trackfit_internal.h"

namespace {

struct HeadArgs {
  const float* pooled;   // [B][P]
  const int32_t* n_hits;
  int64_t B;
  int T, P, Q, NQ;
  float rms_eps;
  const float *g, *w1, *b1, *w2, *b2;
  float *out, *out_q, *out_pool;   // [B][5], [B][Q] or null, [B][P] or null (may be pooled itself)
  unsigned long long* err;
};

size_t head_smem(int RM, int P) {
  return (size_t)(16 * RM * (P + 4) + 16 * RM * 132 + tf_ffma::stage_floats(8)) * 4;
}

// One CTA takes 16 RM tracks: the pooled vectors normed into shared memory (a warp a
// track), then the two products.  Tracks with an invalid hit count take part as
// zero vectors and leave NaN rows.
template <int RM>
__global__ void __launch_bounds__(tf_ffma::NTHREADS) head_kernel(const __grid_constant__ HeadArgs h) {
  using namespace tf_ffma;
  extern __shared__ float4 sm4[];
  const int ldp = h.P + 4, rows = 16 * RM;
  float* pv = reinterpret_cast<float*>(sm4);   // [rows][ldp]
  float* hid = pv + rows * ldp;                // [rows][132]
  float* ws = hid + rows * 132;
  __shared__ int bad_s[16 * RM];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t t0 = (int64_t)blockIdx.x * rows;
  const int nt = (int)(h.B - t0 < rows ? h.B - t0 : rows);
  const float qnan = __int_as_float(0x7fc00000);
  for (int i = warp; i < rows; i += NTHREADS / 32) {
    bool bad = true;
    if (i < nt) {
      const int n = h.n_hits[t0 + i];
      bad = n < 1 || n > h.T;
    }
    float* row = pv + i * ldp;
    if (bad) {
      for (int c = lane; c < h.P; c += 32) row[c] = 0.0f;
      if (i < nt && h.out_pool)
        for (int c = lane; c < h.P; c += 32) h.out_pool[(t0 + i) * h.P + c] = qnan;
    } else {
      const float* src = h.pooled + (t0 + i) * h.P;
      for (int c = lane; c < h.P; c += 32) {
        const float v = src[c];
        row[c] = v;
        if (h.out_pool && h.out_pool != h.pooled) h.out_pool[(t0 + i) * h.P + c] = v;
      }
      __syncwarp();
      norm_row(row, row, h.g, h.P, h.rms_eps, lane);
    }
    if (lane == 0) {
      bad_s[i] = bad;
      if (bad && i < nt) atomicAdd(h.err, 1ull);
    }
  }
  int par = 0;
  head_rows<RM>(pv, ldp, h.P, h.w1, h.b1, h.w2, h.b2, h.Q, hid, ws, par, [&](int r, int o, float v) {
    if (r >= nt) return;
    if (bad_s[r]) v = qnan;
    if (h.out_q) h.out_q[(t0 + r) * h.Q + o] = v;
    if (o % h.NQ == h.NQ / 2) h.out[(t0 + r) * 5 + o / h.NQ] = v;
  });
}

}  // namespace

cudaError_t tf_head_prepare() {
  const cudaError_t e = tf_allow_smem(head_kernel<1>);
  return e != cudaSuccess ? e : tf_allow_smem(head_kernel<2>);
}

// 32 tracks a CTA; 16 while that leaves SMs without a CTA (a small batch is bound by
// the latency of one CTA's chain of weight chunks, which does not grow with them).
cudaError_t tf_head(const tf_shape& s, const tf_blob_off& o, const float* W, const float* pooled,
                    const int32_t* n_hits, int64_t B, int nsm, float* out, float* out_q, float* out_pool,
                    unsigned long long* err, cudaStream_t st) {
  HeadArgs h{pooled, n_hits, B, s.T, s.P, s.Q, s.NQ, s.rms_eps, W + o.head_g, W + o.head_w1, W + o.head_b1,
             W + o.head_w2, W + o.head_b2, out, out_q, out_pool, err};
  if (B > (int64_t)32 * nsm)
    head_kernel<2><<<(unsigned)((B + 31) / 32), tf_ffma::NTHREADS, head_smem(2, s.P), st>>>(h);
  else
    head_kernel<1><<<(unsigned)((B + 15) / 16), tf_ffma::NTHREADS, head_smem(1, s.P), st>>>(h);
  return cudaPeekAtLastError();
}
