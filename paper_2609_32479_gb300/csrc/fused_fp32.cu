// The whole fp32 encoder (gated-merge topology, d_model up to 128) in one kernel: a
// CTA takes whole tracks of up to 64 hits through the embedding, every layer, the
// pooling and the head, with every activation in shared memory.
//
// Layer by layer the same work was one launch a step with the activations in
// global memory: 16 launches for two layers (152 us at 256 tracks, all latency), and
// at 16,384 tracks of 8.5 hits in 12 rows 5.36 ms, of which the products ran on padded rows.
// Here only valid hits take part and a batch is one launch (two with the
// packing).  What bounds it is the multiply-add pipe at large batches, and at small ones
// the chain of weight chunks from L2.
#include <cuda_runtime.h>
#include <math.h>

#include "ffma.cuh"
#include "trackfit_internal.h"

namespace {

using namespace tf_ffma;

struct FusedArgs {
  tf_shape s;
  tf_blob_off o;
  const float* W;
  const float* hits;       // padded [B][T][F], or packed rows with offs
  const int64_t* offs;
  const int32_t* n_hits;
  int64_t B;
  int group;               // > 0: item i is the tracks i group ..; 0: slab i of the packing
  const int32_t* order;
  const int2* slab;
  const int32_t* n_slabs;
  int ldx, ldy, ldr;       // row strides of x, of the states, of the projections (floats)
  float *out, *out_q, *out_pool;
  unsigned long long* err;
};

struct Meta {
  int trk[TF_SLAB_TRACKS], n[TF_SLAB_TRACKS], r0[TF_SLAB_TRACKS + 1];
  uint8_t slot[TF_SLAB], t[TF_SLAB];
  int cnt;
};

// RM: 16 RM rows of hits; CP, CD: columns a thread of the projection chunks (16 CP =
// 4 x the chunk's channels) and of the d_model wide products.
template <int RM, int CP, int CD>
__global__ void __launch_bounds__(NTHREADS, CP == 8 ? 1 : 2) encoder_fp32_kernel(const __grid_constant__ FusedArgs p) {
  extern __shared__ float4 sm4[];
  __shared__ Meta m;
  constexpr int ROWS = 16 * RM, CH = 4 * CP;
  const tf_shape& s = p.s;
  const int D = s.D, H = s.H, F = s.F, ldx = p.ldx, ldy = p.ldy, ldr = p.ldr;
  float* X = reinterpret_cast<float*>(sm4);   // [ROWS][ldx] residual stream
  float* XH = X + ROWS * ldx;                 // [ROWS][ldx] normed stream
  float* Y = XH + ROWS * ldx;                 // [ROWS][ldy] Fourier vector, then the states
  float* PR = Y + ROWS * ldy;                 // [ROWS][ldr] projections of a chunk, hidden values
  float* ws = PR + ROWS * ldr;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int items = p.group ? (int)((p.B + p.group - 1) / p.group) : *p.n_slabs;
  for (int item = blockIdx.x; item < items; item += gridDim.x) {
  __syncthreads();   // the previous item's shared memory is no longer read
  if (warp == 0) {   // the tracks of this item and their rows
    int b0, cnt;
    if (p.group) {
      b0 = item * p.group;
      cnt = (int)(p.B - b0 < p.group ? p.B - b0 : p.group);
    } else {
      const int2 sl = p.slab[item];
      b0 = sl.x;
      cnt = sl.y;
    }
    int trk = 0, n = 0, full = 0;
    if (lane < cnt) {
      trk = p.group ? b0 + lane : p.order[b0 + lane];
      full = p.n_hits[trk];
      n = full < 1 || full > s.T ? 0 : full;
    }
    int e = n;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int u = __shfl_up_sync(0xffffffffu, e, o);
      if (lane >= o) e += u;
    }
    if (lane < cnt) {
      m.trk[lane] = trk;
      m.n[lane] = n;
      m.r0[lane] = e - n;
      for (int t = 0; t < n; ++t) {
        m.slot[e - n + t] = (uint8_t)lane;
        m.t[e - n + t] = (uint8_t)t;
      }
      if (!n) atomicAdd(p.err, 1ull);
    }
    if (lane == 31) m.r0[TF_SLAB_TRACKS] = e;   // all rows
    if (lane == 0) m.cnt = cnt;
  }
  __syncthreads();
  const int cnt = m.cnt, R = m.r0[TF_SLAB_TRACKS];
  int par = 0;
  // Fourier features (Sec. 3.2): u = (v - min) / (max - min) and the argument s_k u as
  // unevaluated sums of two floats, reduced modulo 2 exactly, so the sine and cosine
  // carry only the final rounding of the argument (before it the sum is 1.7e-13 off at
  // most, features in their range: an fp64 evaluation rounded to the same argument in each
  // of 12,000 draws, features up to 100 times their range among them)
  for (int i = tid; i < R * F * TRACKFIT_MAX_FOURIER; i += NTHREADS) {
    const int k = i % TRACKFIT_MAX_FOURIER, rf = i / TRACKFIT_MAX_FOURIER, r = rf / F, f = rf - r * F;
    const int64_t b = m.trk[m.slot[r]];
    const int64_t row = (p.offs ? p.offs[b] : b * s.T) + m.t[r];
    const float v = p.hits[row * F + f];
    const float mn = -s.feat_min[f], ih = s.feat_inv_range[f];
    const float dh = v + mn, bv = dh - v, dl = (v - (dh - bv)) + (mn - bv);
    const float uh = dh * ih;
    const float ul = fmaf(dh, ih, -uh) + fmaf(dh, s.feat_inv_lo[f], dl * ih);
    const float sk = s.scale[k], xh = uh * sk, xl = fmaf(uh, sk, -xh) + ul * sk;
    const float a = (xh - 2.0f * rintf(0.5f * xh)) + xl;
    float sn, cs;
    sincospif(a, &sn, &cs);
    float* e = Y + r * ldy + f * 2 * TRACKFIT_MAX_FOURIER + k;
    e[0] = sn;
    e[TRACKFIT_MAX_FOURIER] = cs;
  }
  // one d_model wide product, column tile by column tile: f(row, column, sum)
  auto dense = [&](const float* A, int lda, size_t w, int K, auto&& f) {
    for (int n0 = 0; n0 < D; n0 += 16 * CD) {
      float acc[RM][CD];
      zero<RM, CD>(acc);
      block_gemm<RM, CD>(acc, A, lda, p.W + w, K, [&](int n) { return n0 + n < D ? n0 + n : -1; }, K, ws, par);
#pragma unroll
      for (int r = 0; r < RM; ++r)
#pragma unroll
        for (int c = 0; c < CD; ++c) {
          const int n = n0 + col<CD>(c);
          if (n < D) f(row0() + 16 * r, n, acc[r][c]);
        }
    }
  };
  const float* W = p.W;
  __syncthreads();
  dense(Y, ldy, p.o.emb_w1, s.E, [&](int r, int n, float v) { PR[r * ldr + n] = silu(v + __ldg(W + p.o.emb_b1 + n)); });
  __syncthreads();
  dense(PR, ldr, p.o.emb_w2, D, [&](int r, int n, float v) { X[r * ldx + n] = v + __ldg(W + p.o.emb_b2 + n); });
  const bool endpoints = s.pool == TRACKFIT_POOL_ENDPOINTS;
  for (int l = 0; l < s.L; ++l) {
    const tf_layer_off& lo = p.o.layer[l];
    __syncthreads();
    for (int r = warp; r < R; r += NTHREADS / 32) norm_row(X + r * ldx, XH + r * ldx, W + lo.g, D, s.rms_eps, lane);
    for (int c0 = 0; c0 < H; c0 += CH) {   // z and n of CH channels, both directions, then their scans
      __syncthreads();
      par = 0;
      float acc[RM][CP];
      zero<RM, CP>(acc);
      block_gemm<RM, CP>(acc, XH, ldx, W + lo.w_in, D, [&](int n) { return (n / CH) * H + c0 + n % CH; }, D, ws, par);
#pragma unroll
      for (int r = 0; r < RM; ++r)
#pragma unroll
        for (int c = 0; c < CP; ++c) {
          const int n = col<CP>(c), q = n / CH;   // q: z_f, n_f, z_b, n_b
          const float v = acc[r][c] + __ldg(W + lo.b_in + q * H + c0 + n % CH);
          PR[(row0() + 16 * r) * ldr + n] = (q & 1) ? v : sigm(v);
        }
      __syncthreads();
      for (int i = tid; i < cnt * 2 * CH; i += NTHREADS) {   // Eq. 2, one (track, direction, channel) a thread
        const int c = i % CH, d = (i / CH) & 1, k = i / (2 * CH), n = m.n[k];
        const int step = d ? -1 : 1;
        const float* z = PR + (m.r0[k] + (d ? n - 1 : 0)) * ldr + 2 * d * CH + c;
        float* y = Y + (m.r0[k] + (d ? n - 1 : 0)) * ldy + d * H + c0 + c;
        float h = 0.0f;
        for (int t = 0; t < n; ++t) {
          h = fmaf(z[0], z[CH] - h, h);
          *y = h;
          z += step * ldr;
          y += step * ldy;
        }
      }
    }
    if (endpoints && l == s.L - 1) break;
    __syncthreads();
    par = 0;
    // x' = x + (W_m [h_f; h_b] + b_m) sigma(p_g), in place
    for (int n0 = 0; n0 < D; n0 += 16 * CD) {
      float gt[RM][CD], acc[RM][CD];
      zero<RM, CD>(gt);
      zero<RM, CD>(acc);
      auto wr = [&](int n) { return n0 + n < D ? n0 + n : -1; };
      block_gemm<RM, CD>(gt, XH, ldx, W + lo.w_in + (size_t)4 * H * D, D, wr, D, ws, par);
      block_gemm<RM, CD>(acc, Y, ldy, W + lo.w_m, 2 * H, wr, 2 * H, ws, par);
#pragma unroll
      for (int r = 0; r < RM; ++r)
#pragma unroll
        for (int c = 0; c < CD; ++c) {
          const int n = n0 + col<CD>(c);
          if (n >= D) continue;
          float* x = X + (row0() + 16 * r) * ldx + n;
          *x += (acc[r][c] + __ldg(W + lo.b_m + n)) * sigm(gt[r][c] + __ldg(W + lo.b_in + 4 * H + n));
        }
    }
    __syncthreads();
    dense(X, ldx, lo.w1, D, [&](int r, int n, float v) { PR[r * ldr + n] = silu(v + __ldg(W + lo.b1 + n)); });
    __syncthreads();
    dense(PR, ldr, lo.w2, D, [&](int r, int n, float v) { X[r * ldx + n] += v + __ldg(W + lo.b2 + n); });
  }
  __syncthreads();
  // pooling, hits in order, into the normed stream's place; then the head
  const int P = s.P, ldp = P + 4;
  float* pv = XH;
  float* hid = PR;
  if (!endpoints) {
    for (int i = tid; i < cnt * P; i += NTHREADS) {
      const int k = i / P, c = i - k * P, n = m.n[k];
      float a = 0.0f;
      for (int t = 0; t < n; ++t) a += X[(m.r0[k] + t) * ldx + c];
      pv[k * ldp + c] = n ? a / (float)n : 0.0f;
    }
  } else {
    for (int i = tid; i < cnt * P; i += NTHREADS) {
      const int k = i / P, c = i - k * P, n = m.n[k];
      pv[k * ldp + c] = n ? Y[(m.r0[k] + (c < H ? n - 1 : 0)) * ldy + c] : 0.0f;
    }
  }
  __syncthreads();
  for (int k = warp; k < cnt; k += NTHREADS / 32) {
    if (p.out_pool)
      for (int c = lane; c < P; c += 32) p.out_pool[(size_t)m.trk[k] * P + c] = m.n[k] ? pv[k * ldp + c] : NAN;
    __syncwarp();
    norm_row(pv + k * ldp, pv + k * ldp, W + p.o.head_g, P, s.rms_eps, lane);
  }
  __syncthreads();
  par = 0;
  float* ws_head = Y;   // the states have been read
  head_rows<1>(pv, ldp, P, W + p.o.head_w1, W + p.o.head_b1, W + p.o.head_w2, W + p.o.head_b2, s.Q, hid, ws_head, par,
               [&](int r, int o, float v) {
                 if (r >= cnt) return;
                 const size_t b = m.trk[r];
                 if (!m.n[r]) v = NAN;
                 if (p.out_q) p.out_q[b * s.Q + o] = v;
                 if (o % s.NQ == s.NQ / 2) p.out[b * 5 + o / s.NQ] = v;
               });
  }
}

struct Plan {
  int RM, CP, CD, ldx, ldy, ldr;
  size_t smem;
};

int imax(int a, int b) { return a > b ? a : b; }

Plan shape_plan(const tf_shape& s, int RM) {
  Plan q;
  q.RM = RM;
  q.CP = s.D == 128 ? 8 : s.H % 16 == 0 ? 4 : 2;
  q.CD = s.D == 128 ? 8 : s.D % 64 == 0 ? 4 : 2;
  const int rows = 16 * RM;
  q.ldx = s.D + 4;
  q.ldy = imax(2 * s.H, s.E) + 4;
  q.ldr = imax(16 * q.CP, s.D) + 4;
  // the head's 16 pooled vectors, hidden values and staging lie in the places of the
  // normed stream, the projections and the states
  const int xh = imax(rows * q.ldx, 16 * (s.P + 4)), pr = imax(rows * q.ldr, 16 * 132);
  q.ldx = imax(q.ldx, (xh + rows - 1) / rows);
  q.ldx = (q.ldx + 3) / 4 * 4;
  q.ldr = imax(q.ldr, (pr + rows - 1) / rows);
  q.ldr = (q.ldr + 3) / 4 * 4;
  q.ldy = imax(q.ldy, (stage_floats(8) + rows - 1) / rows);
  q.ldy = (q.ldy + 3) / 4 * 4;
  q.smem = ((size_t)rows * (2 * q.ldx + q.ldy + q.ldr) + stage_floats(q.CP > q.CD ? q.CP : q.CD)) * 4;
  return q;
}

using Kernel = void (*)(const FusedArgs);
Kernel pick(const Plan& q) {
  if (q.RM == 4) return q.CP == 8 ? encoder_fp32_kernel<4, 8, 8> : q.CP == 4 ? (q.CD == 4 ? encoder_fp32_kernel<4, 4, 4> : encoder_fp32_kernel<4, 4, 2>) : (q.CD == 4 ? encoder_fp32_kernel<4, 2, 4> : encoder_fp32_kernel<4, 2, 2>);
  return q.CP == 8 ? encoder_fp32_kernel<1, 8, 8> : q.CP == 4 ? (q.CD == 4 ? encoder_fp32_kernel<1, 4, 4> : encoder_fp32_kernel<1, 4, 2>) : (q.CD == 4 ? encoder_fp32_kernel<1, 2, 4> : encoder_fp32_kernel<1, 2, 2>);
}

}  // namespace

// fp32, gated-merge topology, d_model up to 128 (wider does not fit: the states of 64
// hits alone take 3 d_model x 256 bytes of an SM's 227 KB).
bool tf_fused_fp32_supported(const tf_shape& s) {
  return s.precision == TRACKFIT_FP32 && s.topology == TRACKFIT_TOPOLOGY_MERGE && s.D <= 128 &&
         shape_plan(s, 4).smem + sizeof(Meta) <= 226 * 1024;
}

cudaError_t tf_fused_fp32_prepare(const tf_shape& s) {
  for (int RM : {1, 4}) {
    const cudaError_t e = tf_allow_smem(pick(shape_plan(s, RM)));
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// One launch over B tracks (packed with two more).  While every CTA slot of the chip
// can take its tracks whole at once (and in 16 rows if they fit), the batch goes out
// as runs of consecutive tracks, without packing: its time is one CTA's chain of
// steps then, which neither packing nor fuller CTAs would shorten.  Above that the
// slabs of the packing keep 97 % of the rows busy.  An SM has two slots, or one at d_model
// 128 (by registers) and where shared memory holds only one CTA of 64 rows (d_model 80 up,
// any with 15 features): with two assumed there, 304 tracks of 20 hits at d_model 96 ran
// unpacked in two waves, more than 1.5 times the 226 us of one.
int tf_fused_fp32_forward(const tf_shape& s, const tf_blob_off& o, const float* W, const tf_pack& pk,
                          unsigned long long* err, const float* hits, const int32_t* n_hits, const int64_t* offs,
                          int64_t B, float* out, float* out_q, float* out_pool, cudaStream_t st, trackfit_ctx* prof) {
  int dev = 0, nsm = 0, sm_smem = 0, reserved = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sm_smem, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev) != cudaSuccess)
    return TRACKFIT_ERR_CUDA;
  const Plan q1 = shape_plan(s, 1), q4 = shape_plan(s, 4);
  auto slots_of = [&](const Plan& q) -> int64_t {
    const bool two = q.CP != 8 && 2 * (q.smem + sizeof(Meta) + reserved) <= (size_t)sm_smem;
    return (int64_t)nsm * (two ? 2 : 1);
  };
  const int64_t slots1 = slots_of(q1), slots4 = slots_of(q4);
  for (int64_t c0 = 0; c0 < B; c0 += pk.cap) {
    const int64_t nb = B - c0 < pk.cap ? B - c0 : pk.cap;
    const int64_t each1 = (nb + slots1 - 1) / slots1, each4 = (nb + slots4 - 1) / slots4;
    const bool small = each1 * s.T <= 16, flat = small || (each4 * s.T <= TF_SLAB && each4 <= TF_SLAB_TRACKS);
    const Plan& q = small ? q1 : q4;
    const int64_t slots = small ? slots1 : slots4, each = small ? each1 : each4;
    FusedArgs p{s, o, W, offs ? hits : hits + c0 * s.T * s.F, offs ? offs + c0 : nullptr, n_hits + c0, nb,
                flat ? (int)each : 0, pk.order, pk.slab, pk.n_slabs, q.ldx, q.ldy, q.ldr,
                out + c0 * 5, out_q ? out_q + c0 * s.Q : nullptr, out_pool ? out_pool + c0 * s.P : nullptr, err};
    if (!flat) {
      const cudaError_t e = tf_plan(p.n_hits, nb, s.T, nsm, pk.order, pk.slab, pk.n_slabs, st);
      if (e != cudaSuccess) {
        tf_note_cuda(e, "plan launch");
        return TRACKFIT_ERR_CUDA;
      }
    }
    const int64_t items = flat ? (nb + each - 1) / each : nb;
    if (prof) tf_prof_begin(prof, st);
    pick(q)<<<(unsigned)(items < slots ? items : slots), NTHREADS, q.smem, st>>>(p);
    if (prof) tf_prof_end(prof, st);
    const cudaError_t e = cudaPeekAtLastError();
    if (e != cudaSuccess) {
      tf_note_cuda(e, "encoder_fp32_kernel launch");
      return TRACKFIT_ERR_CUDA;
    }
  }
  return TRACKFIT_OK;
}
