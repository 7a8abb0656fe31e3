// The Transformer encoder (App. A.3: pre-norm attention within each track and a SiLU MLP,
// mean readout, 16-bit operands) for d_model 128 and 4 or 8 heads, in one tensor-core
// kernel behind the Fourier rows.
//
// As separate launches (rows.cu) every intermediate of a hit went through HBM, 7.8 KB a hit
// and layer: at 131,072 tracks of 12.5 hits and three layers the products took 7.3 ms
// and the attention 3.3 ms.  Here a tile of 128 packed hits (two slabs of whole tracks)
// stays on its SM from the Fourier vector to the pooled mean:
//   D[hit][channel] = Act[hit][k] W[channel][k],
// accumulators in TMEM with one hit a lane: norms are sums along a thread's columns, and
// attention needs only the other hits of the track.
//
// Warp roles (608 threads): 0 TMA producer, 1 MMA issuer and TMEM owner, 2-17 epilogue
// (TMEM lane quadrant = warp % 4, 32-column group = (warp - 2) / 4, with four heads the
// head), 18 loader of the tile's metadata.  The steps of a tile follow one another: a
// product group, then its epilogue (one hand-over each way).
// TMEM: columns 0-127 the fp32 residual stream, 128-511 the group's results (q, k, v; the
// MLP's hidden values; or 128 columns to be added to the stream).
// Shared memory: SA, the 16-bit operand of the d_model wide products (K-major, two 64-k
// blocks); KV, one head-interleaved fp32 matrix of the tile's keys, then its values,
// then (16-bit) the MLP's hidden operand, at the end the last stream for the pooling; the
// ring of 16 KB weight blocks (and Fourier blocks).
#include <cstring>
#include <new>
#include <vector>

#include "tiles.cuh"

namespace {

constexpr int TR_MAX_H = 320;                        // MLP width: its operand takes KV's place
constexpr int TR_LD = 132;                           // floats of a row of KV (4 mod 32: rows in different banks)
constexpr int TR_SA = 0, TR_KV = 32768, TR_RING = 32768 + 5 * 16384;   // KV: 128 rows (67.6 KB), or 5 operand blocks
static_assert(TILE * TR_LD * 4 <= TR_RING - TR_KV && TR_MAX_H / 64 * 16384 <= TR_RING - TR_KV, "KV too small");
constexpr int TR_MAX_STAGES = 6;
constexpr uint64_t TR_DRAIN_NS = 200000000ull;
constexpr size_t TR_WS_BUDGET = (size_t)4 << 30;     // bytes of the Fourier rows

enum { TM_F = 0, TM_E1, TM_E2, TM_QKV, TM_O, TM_1, TM_2, TM_MAPS };

struct TrParams {
  CUtensorMap tm[TM_MAPS];
  TileSrc src;
  float* pool;                  // [B][128]
  int L, H, KE, last_nk, nst;
  int n1, n1_tiles;             // columns of one MLP1 product, products
  uint32_t idesc, idesc1;       // N = 128, N = n1
  float rms_eps;
  const float* vec;             // b_e1, b_e2, then per layer g1, b_qkv, b_o, g2, b_1, b_2
  unsigned long long* err;
  uint64_t wait_ns;
  int hold_tile;                // test hook: CTA 0's loader holds this tile's metadata hand-over (-1: none)
};

struct TrMisc {
  uint64_t full[TR_MAX_STAGES], empty[TR_MAX_STAGES];
  uint64_t acc_bar, op_bar, drain_bar;
  uint64_t meta_full[2], meta_free[2];
  uint32_t tmem_base;
  int abort_flag;
  TileMeta meta[2];
  uint8_t tpos[2][TILE];
  alignas(16) float part[2][4][TILE];   // sums of squares of the four column groups, two norms in turn
};
constexpr size_t TR_SMEM_REST = sizeof(TrMisc) + 1024;

__device__ __forceinline__ void tr_abort(TrMisc* m, unsigned long long* err) {
  if (atomicExch(&m->abort_flag, 1) == 0) atomicAdd(err + 1, 1ull);
}
__device__ __forceinline__ void named_sync(int id, int n) { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory"); }

// 8 values of operand row r (a hit), k columns 8 c8 .. 8 c8 + 7, into a K-major operand of 64-k
// blocks with 128-byte swizzle.
template <bool FP16>
__device__ __forceinline__ void put8(uint32_t buf, int r, int c8, const float* v) {
  st_shared_v4(buf + (uint32_t)((c8 >> 3) * 16384 + r * 128 + (((c8 & 7) ^ (r & 7)) << 4)), pack2<FP16>(v[0], v[1]),
               pack2<FP16>(v[2], v[3]), pack2<FP16>(v[4], v[5]), pack2<FP16>(v[6], v[7]));
}
// v + b for N consecutive columns (the same for every lane)
template <int N>
__device__ __forceinline__ void add_bias(float (&v)[N], const float* __restrict__ b) {
#pragma unroll
  for (int i = 0; i < N; i += 4) {
    const float4 w = __ldg(reinterpret_cast<const float4*>(b + i));
    v[i] += w.x;
    v[i + 1] += w.y;
    v[i + 2] += w.z;
    v[i + 3] += w.w;
  }
}
// SiLU on a pair of values (sigmoid2 of tc_epilogue.cuh)
template <int N>
__device__ __forceinline__ void silu_all(float (&v)[N]) {
#pragma unroll
  for (int i = 0; i < N; i += 2) {
    const f2 x(v[i], v[i + 1]);
    f2 e(0.0f), sg(0.0f);
    sigmoid2(mul2(x, f2(-LOG2E_F)), e, sg);
    mul2(x, sg).get(v[i], v[i + 1]);
  }
}

// Attention of one head of width DH for the thread's hit: the keys, then the values, of its
// slab's hits go through KV (the two warps of a slab's lane quadrants and this column
// group exchange theirs: named barrier bar, 64 threads).  Two passes over the track's
// keys, four at a time: the scores into the TMEM columns that the head's own k and then
// q have left (2 DH keys) and their maximum, then the exponentials, their sum and the
// weighted values.  Every sum runs in a fixed order.  Bound by the reads of keys and values
// from shared memory; eight at a time read a track's last key more often to no end (131,072
// tracks of 12.5 hits, 6.52 -> 6.25 ms with four).
template <int DH>
__device__ __forceinline__ void attend(float (&o)[DH], float* kv, int row, int ch, uint32_t tq, uint32_t tk, uint32_t tv,
                                       const float* bq, const float* bk, const float* bv, int start, int n, int steps,
                                       int bar) {
  float* own = kv + row * TR_LD + ch;
  {
    float k[DH];
#pragma unroll
    for (int i = 0; i < DH; i += 16) {
      float t[16];
      tmem_ld16(tk + i, t);
      tmem_ld_wait();
#pragma unroll
      for (int c = 0; c < 16; ++c) k[i + c] = t[c];
    }
    add_bias<DH>(k, bk);
#pragma unroll
    for (int i = 0; i < DH; i += 4) *reinterpret_cast<float4*>(own + i) = make_float4(k[i], k[i + 1], k[i + 2], k[i + 3]);
  }
  const float scale = rsqrtf((float)DH);
  float q[DH], m = -INFINITY;
#pragma unroll
  for (int i = 0; i < DH; i += 16) {
    float t[16];
    tmem_ld16(tq + i, t);
    tmem_ld_wait();
#pragma unroll
    for (int c = 0; c < 16; ++c) q[i + c] = t[c];
  }
  add_bias<DH>(q, bq);
  tc_fence_before();
  named_sync(bar, 64);   // the slab's keys of this column group are in KV
  const int last = start + (n > 0 ? n - 1 : 0);
#pragma unroll 1
  for (int s = 0; s < steps; ++s) {
    float sc[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float* kr = kv + min(start + 4 * s + j, last) * TR_LD + ch;
      float a = 0.0f;
#pragma unroll
      for (int i = 0; i < DH; i += 4) {
        const float4 k4 = *reinterpret_cast<const float4*>(kr + i);
        a = fmaf(q[i], k4.x, a);
        a = fmaf(q[i + 1], k4.y, a);
        a = fmaf(q[i + 2], k4.z, a);
        a = fmaf(q[i + 3], k4.w, a);
      }
      sc[j] = 4 * s + j < n ? a * scale : -INFINITY;
      m = fmaxf(m, sc[j]);
    }
    tmem_st4(s < DH / 4 ? tk + 4 * s : tq + 4 * s - DH, sc);
  }
  tmem_st_wait();
  {
    float v[DH];
#pragma unroll
    for (int i = 0; i < DH; i += 16) {
      float t[16];
      tmem_ld16(tv + i, t);
      tmem_ld_wait();
#pragma unroll
      for (int c = 0; c < 16; ++c) v[i + c] = t[c];
    }
    add_bias<DH>(v, bv);
    named_sync(bar, 64);   // both warps are done with the keys
#pragma unroll
    for (int i = 0; i < DH; i += 4) *reinterpret_cast<float4*>(own + i) = make_float4(v[i], v[i + 1], v[i + 2], v[i + 3]);
  }
  named_sync(bar, 64);   // the values are in KV
#pragma unroll
  for (int i = 0; i < DH; ++i) o[i] = 0.0f;
  float l = 0.0f;
#pragma unroll 1
  for (int s = 0; s < steps; ++s) {
    float sc[4];
    tmem_ld4(s < DH / 4 ? tk + 4 * s : tq + 4 * s - DH, sc);
    tmem_ld_wait();
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float p = 4 * s + j < n ? expf(sc[j] - m) : 0.0f;
      l += p;
      const float* vr = kv + min(start + 4 * s + j, last) * TR_LD + ch;
#pragma unroll
      for (int i = 0; i < DH; i += 4) {
        const float4 v4 = *reinterpret_cast<const float4*>(vr + i);
        o[i] = fmaf(p, v4.x, o[i]);
        o[i + 1] = fmaf(p, v4.y, o[i + 1]);
        o[i + 2] = fmaf(p, v4.z, o[i + 2]);
        o[i + 3] = fmaf(p, v4.w, o[i + 3]);
      }
    }
  }
  const float inv = n > 0 ? 1.0f / l : 0.0f;
#pragma unroll
  for (int i = 0; i < DH; ++i) o[i] *= inv;
}

template <bool FP16, int DH>
__global__ void __launch_bounds__(NT, 1) transformer_kernel(const __grid_constant__ TrParams p) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t* gbase = smem_raw + (base - raw);
  TrMisc* m = reinterpret_cast<TrMisc*>(gbase + TR_RING + p.nst * A_BLOCK);
  const uint32_t ring = base + TR_RING, sa = base + TR_SA, su = base + TR_KV;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t full0 = smem_u32(&m->full[0]), empty0 = smem_u32(&m->empty[0]);
  const uint32_t acc_bar = smem_u32(&m->acc_bar), op_bar = smem_u32(&m->op_bar), drain_bar = smem_u32(&m->drain_bar);
  if (threadIdx.x == 0) {
    for (int s = 0; s < p.nst; ++s) {
      mbar_init(full0 + 8 * s, 1);
      mbar_init(empty0 + 8 * s, 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(smem_u32(&m->meta_full[b]), 1);
      mbar_init(smem_u32(&m->meta_free[b]), NE / 32);
    }
    mbar_init(acc_bar, 1);
    mbar_init(op_bar, NE / 32);
    mbar_init(drain_bar, 1);
    m->abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == 1) {
    tmem_alloc(smem_u32(&m->tmem_base), 512);
    tmem_relinquish();
  }
  if (warp == 0 && lane == 0)
    for (int i = 0; i < TM_MAPS; ++i) prefetch_tmap(&p.tm[i]);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = m->tmem_base;
  const int n_slabs = *p.src.n_slabs, n_tiles = (n_slabs + 1) >> 1;
  volatile int* abort = &m->abort_flag;
  const int kh = (p.H + 63) / 64;   // 64-k blocks of the hidden operand

  if (warp == 0) {
    // TMA producer: one lane, blocks in the issuer's order
    if (elect_one()) {
      uint32_t stage = 0, phase = 0;
      int issued = 0;
      bool ok = true;
      auto load = [&](int map, int c0, int c1, uint32_t bytes) {
        if (!ok) return;
        const uint32_t full = full0 + 8 * stage;
        if (!mbar_wait(empty0 + 8 * stage, phase ^ 1u, abort, p.wait_ns)) {
          tr_abort(m, p.err);
          ok = false;
          return;
        }
        mbar_arrive_expect_tx(full, bytes);
        tma_load_2d(ring + stage * A_BLOCK, &p.tm[map], full, c0, c1);
        ++issued;
        if (++stage == (uint32_t)p.nst) {
          stage = 0;
          phase ^= 1u;
        }
      };
      for (int t = blockIdx.x; t < n_tiles && ok; t += gridDim.x) {
        for (int kc = 0; kc < p.KE; ++kc) {
          load(TM_F, kc * 64, t * TILE, A_BLOCK);
          load(TM_E1, kc * 64, 0, A_BLOCK);
        }
        for (int kc = 0; kc < 2; ++kc) load(TM_E2, kc * 64, 0, A_BLOCK);
        for (int l = 0; l < p.L; ++l) {
          for (int r = 0; r < 3; ++r)
            for (int kc = 0; kc < 2; ++kc) load(TM_QKV, kc * 64, (3 * l + r) * 128, A_BLOCK);
          for (int kc = 0; kc < 2; ++kc) load(TM_O, kc * 64, l * 128, A_BLOCK);
          for (int r = 0; r < p.n1_tiles; ++r)
            for (int kc = 0; kc < 2; ++kc) load(TM_1, kc * 64, l * p.H + r * p.n1, (uint32_t)p.n1 * 128u);
          for (int kc = 0; kc < kh; ++kc) load(TM_2, kc * 64, l * 128, A_BLOCK);
        }
      }
      if (*abort) {   // let the copies already issued land before the CTA can exit
        volatile int never = 0;
        for (int k = 0; k < p.nst && k < issued; ++k) {
          const int i = issued - 1 - k;
          mbar_wait(full0 + 8 * (i % p.nst), (uint32_t)((i / p.nst) & 1), &never, TR_DRAIN_NS);
        }
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    // MMA issuer: one lane for the whole loop.  Activations are the A operand, weights B,
    // both K-major.
    if (elect_one()) {
      uint32_t stage = 0, phase = 0, op_k = 0;
      bool ok = true;
      auto wait_bar = [&](uint32_t bar, uint32_t parity) {
        if (ok && !mbar_wait(bar, parity, abort, p.wait_ns)) {
          tr_abort(m, p.err);
          ok = false;
        }
      };
      const uint64_t desc = sdesc_sw128(base, 16, 1024);
      const uint32_t lo0 = desc_lo(desc), hi = desc_hi(desc), ring_lo = lo0 + (TR_RING >> 4);
      auto stage_lo = [&]() { return ring_lo + stage * (A_BLOCK >> 4); };
      auto next_stage = [&]() {
        if (++stage == (uint32_t)p.nst) {
          stage = 0;
          phase ^= 1u;
        }
      };
      auto operand = [&]() { wait_bar(op_bar, op_k++ & 1u); };   // the epilogue's next hand-over
      auto commit = [&]() { if (ok) umma_commit(acc_bar); };
      // K columns of the operand at byte offset off, against the next blocks of the ring
      auto product = [&](uint32_t d, uint32_t off, int K, uint32_t idesc) {
        uint32_t a_lo = lo0 + (off >> 4);
        for (int k = 0; k < K; k += 64, a_lo += A_BLOCK >> 4) {
          wait_bar(full0 + 8 * stage, phase);
          if (!ok) return;
          tc_fence_after();
          if (K - k >= 64) {
            umma4_f16<2>(d, a_lo, hi, stage_lo(), hi, idesc, k);
          } else {
            for (int j = 0; j < (K - k) / 16; ++j)
              umma_f16(d, ((uint64_t)hi << 32) | (a_lo + 2 * j), ((uint64_t)hi << 32) | (stage_lo() + 2 * j), idesc,
                          (k | j) ? 1u : 0u);
          }
          umma_commit(empty0 + 8 * stage);
          next_stage();
        }
      };
      for (int t = blockIdx.x; t < n_tiles && ok; t += gridDim.x) {
        if (t != (int)blockIdx.x) operand();   // the tile before has left the accumulators
        for (int kc = 0; kc < p.KE; ++kc) {    // embedding product 1: Fourier rows and weights alternate in the ring
          wait_bar(full0 + 8 * stage, phase);
          const uint32_t a0 = stage_lo(), e0 = empty0 + 8 * stage;
          next_stage();
          wait_bar(full0 + 8 * stage, phase);
          if (!ok) break;
          tc_fence_after();
          if (kc + 1 < p.KE || p.last_nk == 4)
            umma4_f16<2>(tmem + 128, a0, hi, stage_lo(), hi, p.idesc, kc);
          else
            umma2_f16<2>(tmem + 128, a0, hi, stage_lo(), hi, p.idesc, kc);
          umma_commit(e0);
          umma_commit(empty0 + 8 * stage);
          next_stage();
        }
        commit();
        operand();
        product(tmem + 128, TR_SA, 128, p.idesc);
        commit();
        for (int l = 0; l < p.L && ok; ++l) {
          operand();
          for (int r = 0; r < 3; ++r) product(tmem + 128 + 128 * r, TR_SA, 128, p.idesc);
          commit();
          operand();
          product(tmem + 128, TR_SA, 128, p.idesc);
          commit();
          operand();
          for (int r = 0; r < p.n1_tiles; ++r) product(tmem + 128 + (uint32_t)(r * p.n1), TR_SA, 128, p.idesc1);
          commit();
          operand();
          product(tmem + 128, TR_KV, p.H, p.idesc);
          commit();
        }
      }
      // no MMA may still run when TMEM is released
      umma_commit(drain_bar);
      volatile int never = 0;
      mbar_wait(drain_bar, 0, &never, TR_DRAIN_NS);
    }
    __syncwarp();
  } else if (warp < 2 + NE / 32) {
    // Epilogue.  A failed wait sets the abort flag and every later wait fails fast, but no
    // warp leaves the loop early: all of them meet at the named barriers.  `alive` (the same
    // for a warp's lanes): every wait of this warp has succeeded; only then is the metadata of
    // its tile complete and kept until the warp releases it, and may an address be formed from
    // it.
    bool alive = true;
    const int q = warp & 3, cg = (warp - 2) >> 2, row = 32 * q + lane, c0 = 32 * cg;
    const int pair_bar = 1 + (q >> 1) * 4 + cg;   // 1-8: a slab's two quadrants, one column group
    const uint32_t tl = tmem + ((uint32_t)(32 * q) << 16);
    const uint32_t tx = tl + c0, ta = tl + 128 + c0;
    float* kv = reinterpret_cast<float*>(gbase + TR_KV);
    uint32_t acc_k = 0, norms = 0;
    auto wait_on = [&](uint32_t bar, uint32_t parity) {
      const bool got = mbar_wait(bar, parity, abort, p.wait_ns);
      if (!__all_sync(0xffffffffu, got)) {
        if (lane == 0) tr_abort(m, p.err);
        alive = false;
      }
      tc_fence_after();
    };
    auto wait_acc = [&]() { wait_on(acc_bar, acc_k++ & 1u); };
    auto signal = [&]() {
      fence_proxy_async_smem();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(op_bar);
    };
    // x = res + (acc + b), kept in TMEM; its norm times the gain into SA
    auto stream = [&](bool first, const float* b, const float* gain) {
      float v[32];
      tmem_ld32(ta, v);
      tmem_ld_wait();
      add_bias<32>(v, b + c0);
      if (!first) {
        float x[32];
        tmem_ld32(tx, x);
        tmem_ld_wait();
#pragma unroll
        for (int i = 0; i < 32; ++i) v[i] = x[i] + v[i];
      }
      if (!gain) {   // the last layer: the stream goes to KV for the pooling
#pragma unroll
        for (int i = 0; i < 32; i += 4)
          *reinterpret_cast<float4*>(kv + row * TR_LD + c0 + i) = make_float4(v[i], v[i + 1], v[i + 2], v[i + 3]);
        return;
      }
      tmem_st32(tx, v);
      float ss = 0.0f;
#pragma unroll
      for (int i = 0; i < 32; ++i) ss = fmaf(v[i], v[i], ss);
      float(*part)[TILE] = m->part[norms++ & 1u];
      part[cg][row] = ss;
      named_sync(9 + q, 128);   // the quadrant's four column groups
      const float tot = (part[0][row] + part[1][row]) + (part[2][row] + part[3][row]);
      const float inv = 1.0f / sqrtf(tot / 128.0f + p.rms_eps);
#pragma unroll
      for (int i = 0; i < 32; i += 4) {
        const float4 w = __ldg(reinterpret_cast<const float4*>(gain + c0 + i));
        v[i] = v[i] * inv * w.x;
        v[i + 1] = v[i + 1] * inv * w.y;
        v[i + 2] = v[i + 2] * inv * w.z;
        v[i + 3] = v[i + 3] * inv * w.w;
      }
#pragma unroll
      for (int i = 0; i < 32; i += 8) put8<FP16>(sa, row, (c0 + i) >> 3, v + i);
      tmem_st_wait();
    };
    const int per_layer = 128 + 384 + 128 + 128 + p.H + 128;
    int i = 0;
    for (int t = blockIdx.x; t < n_tiles; t += gridDim.x, ++i) {
      wait_acc();
      {
        float v[32];
        tmem_ld32(ta, v);
        tmem_ld_wait();
        add_bias<32>(v, p.vec + c0);
        silu_all<32>(v);
#pragma unroll
        for (int k = 0; k < 32; k += 8) put8<FP16>(sa, row, (c0 + k) >> 3, v + k);
      }
      signal();
      const float* vec = p.vec + 256;   // the layer's g1, b_qkv, b_o, g2, b_1, b_2
      wait_acc();
      stream(true, p.vec + 128, vec);
      signal();
      wait_on(smem_u32(&m->meta_full[i & 1]), (uint32_t)(i >> 1) & 1u);
      const TileMeta* md = &m->meta[i & 1];
      int n = 0, start = row;
      if (alive && (md->col_flags[row] & F_VALID)) {
        n = md->slot_n[md->col_slot[row]];
        start = row - m->tpos[i & 1][row];
      }
      const int steps = (__reduce_max_sync(0xffffffffu, n) + 3) >> 2;
#pragma unroll 1
      for (int l = 0; l < p.L; ++l, vec += per_layer) {
        wait_acc();   // q, k, v
#pragma unroll 1
        for (int h = 0; h < 32 / DH; ++h) {   // the column group's heads
          const int ch = c0 + h * DH;
          float o[DH];
          const uint32_t tq = tl + 128 + ch;
          attend<DH>(o, kv, row, ch, tq, tq + 128, tq + 256, vec + 128 + ch, vec + 256 + ch, vec + 384 + ch, start, n,
                     steps, pair_bar);
#pragma unroll
          for (int k = 0; k < DH; k += 8) put8<FP16>(sa, row, (ch + k) >> 3, o + k);
        }
        signal();
        wait_acc();
        stream(false, vec + 512, vec + 640);
        signal();
        wait_acc();
        for (int u = cg; u < p.H / 16; u += 4) {   // the MLP's hidden values, 16 columns at a time
          float v[16];
          tmem_ld16(tl + 128 + 16 * u, v);
          tmem_ld_wait();
          add_bias<16>(v, vec + 768 + 16 * u);
          silu_all<16>(v);
          put8<FP16>(su, row, 2 * u, v);
          put8<FP16>(su, row, 2 * u + 1, v + 8);
        }
        signal();
        wait_acc();
        const bool last = l + 1 == p.L;
        stream(false, vec + 768 + p.H, last ? nullptr : vec + per_layer);
        if (!last || t + (int)gridDim.x < n_tiles) signal();
      }
      // mean pooling, each track's hits in order: thread (track of the tile, channel)
      named_sync(13, NE);
      if (alive) {
        const int te = threadIdx.x - 64, c = te & 127;
        for (int w = 0; w < 4; ++w)   // tracks by their first row, in turn over the four thread groups
          for (uint32_t f = md->m_first[w >> 1][w & 1]; f; f &= f - 1) {
            const int r0 = 32 * w + __ffs(f) - 1, slot = md->col_slot[r0], cnt = md->slot_n[slot];
            if ((slot & 3) != (te >> 7)) continue;
            float a = 0.0f;
            for (int k = 0; k < cnt; ++k) a += kv[(r0 + k) * TR_LD + c];
            p.pool[(size_t)md->slot_track[slot] * 128 + c] = a / (float)cnt;
          }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&m->meta_free[i & 1]));
    }
  } else {
    // loader warp: the metadata of a tile, one tile ahead
    int i = 0;
    for (int t = blockIdx.x; t < n_tiles; t += gridDim.x, ++i) {
      const int b = i & 1;
      if (i >= 2) {
        const bool got = mbar_wait(smem_u32(&m->meta_free[b]), (uint32_t)((i >> 1) - 1) & 1u, abort, p.wait_ns);
        if (!__all_sync(0xffffffffu, got) && lane == 0) tr_abort(m, p.err);
        // after a failure anywhere a release may have come from a warp that gave up: stop, so
        // that the metadata others still read stays as it is
        if (!__all_sync(0xffffffffu, got && !*abort)) break;
      }
      load_meta(p.src, m->tpos[b], &m->meta[b], 2 * t, n_slabs, lane);
      __threadfence_block();
      __syncwarp();
      if (i == p.hold_tile && blockIdx.x == 0) hold_hand_over(abort, p.wait_ns);
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&m->meta_full[b]));
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
}

}  // namespace

struct tf_tr_state {
  int nsm;
  int64_t chunk;      // tracks at a time
  size_t smem;
  void *dev, *pack;
  uint16_t* four;     // Fourier rows
  float* pool;        // [chunk][128]
  TrParams p;
};

namespace {

// Columns of one MLP1 product: an equal split of the width into multiples of 16 up to 128
// (0 if there is none).
int mlp_split(int H) {
  for (int parts = (H + 127) / 128; parts <= H / 16; ++parts)
    if (H % parts == 0 && (H / parts) % 16 == 0) return H / parts;
  return 0;
}

using TrKernel = void (*)(const TrParams);
TrKernel tr_kernel(const tf_shape& s) {
  if (s.precision == TRACKFIT_FP16_PROJ) return s.NH == 4 ? transformer_kernel<true, 32> : transformer_kernel<true, 16>;
  return s.NH == 4 ? transformer_kernel<false, 32> : transformer_kernel<false, 16>;
}

}  // namespace

// d_model 128, four heads (or eight, with tracks of up to 32 hits: a head's scores lie in
// the 2 x 128 / heads columns its query and key leave), MLP width up to 320 (its operand
// takes the keys' place in shared memory).  Others run as separate launches (rows.cu).
bool tf_tr_supported(const tf_shape& s) {
  return (s.precision == TRACKFIT_BF16_PROJ || s.precision == TRACKFIT_FP16_PROJ) &&
         s.topology == TRACKFIT_TOPOLOGY_ATTENTION && s.D == 128 && (s.NH == 4 || (s.NH == 8 && s.T <= 32)) &&
         s.H <= TR_MAX_H && mlp_split(s.H) != 0 && s.K == TRACKFIT_MAX_FOURIER;
}

void tf_tr_destroy(tf_tr_state* c) {
  if (!c) return;
  tf_free(c->dev);
  tf_free(c->pack);
  tf_free(c->four);
  tf_free(c->pool);
  delete c;
}

int tf_tr_create(trackfit_ctx* h, const float* W, tf_tr_state** out) {
  const tf_shape& s = h->s;
  const tf_blob_off& o = h->off;
  tf_tr_state* c = new (std::nothrow) tf_tr_state();
  if (!c) return TRACKFIT_ERR_OOM;
  *out = c;   // freed by the caller's tf_tr_destroy on any failure below
  const bool fp16 = s.precision == TRACKFIT_FP16_PROJ;
  int dev = 0, optin = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&c->nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess)
    return TRACKFIT_ERR_CUDA;
  TrParams& p = c->p;
  p.L = s.L;
  p.H = s.H;
  p.KE = (s.E + 63) / 64;
  p.last_nk = (s.E - 64 * (p.KE - 1)) / 16;
  p.n1 = mlp_split(s.H);
  p.n1_tiles = s.H / p.n1;
  p.rms_eps = s.rms_eps;
  p.nst = (optin - (int)TR_SMEM_REST - TR_RING) / A_BLOCK;
  if (p.nst > TR_MAX_STAGES) p.nst = TR_MAX_STAGES;
  if (p.nst < 3) return TRACKFIT_ERR_UNSUPPORTED;
  c->smem = TR_RING + (size_t)p.nst * A_BLOCK + TR_SMEM_REST;
  p.idesc = idesc_f16(128, 128, fp16 ? 0u : 1u, false, false);
  p.idesc1 = idesc_f16(128, p.n1, fp16 ? 0u : 1u, false, false);
  // 16-bit weights, each product's matrices of all layers stacked, [N][K]
  const size_t D = s.D, H = s.H, E = s.E, L = s.L;
  std::vector<uint16_t> w;
  w.reserve(D * E + D * D + L * (4 * D * D + 2 * D * H));
  auto mat = [&](size_t off, size_t n) {
    for (size_t i = 0; i < n; ++i) w.push_back(to_16(W[off + i], fp16));
  };
  mat(o.emb_w1, D * E);
  mat(o.emb_w2, D * D);
  const size_t at_qkv = w.size();
  for (size_t l = 0; l < L; ++l) mat(o.layer[l].w_in, 3 * D * D);
  const size_t at_o = w.size();
  for (size_t l = 0; l < L; ++l) mat(o.layer[l].w_m, D * D);
  const size_t at_1 = w.size();
  for (size_t l = 0; l < L; ++l) mat(o.layer[l].w1, H * D);
  const size_t at_2 = w.size();
  for (size_t l = 0; l < L; ++l) mat(o.layer[l].w2, D * H);
  std::vector<float> v;
  auto vec = [&](size_t off, size_t n) { v.insert(v.end(), W + off, W + off + n); };
  vec(o.emb_b1, D);
  vec(o.emb_b2, D);
  for (size_t l = 0; l < L; ++l) {
    const tf_layer_off& lo = o.layer[l];
    vec(lo.g, D);
    vec(lo.b_in, 3 * D);
    vec(lo.b_m, D);
    vec(lo.g2, D);
    vec(lo.b1, H);
    vec(lo.b2, D);
  }
  const size_t wbytes = (w.size() * 2 + 255) / 256 * 256;
  int st = tf_status_from_cuda(tf_malloc(&c->dev, wbytes + v.size() * 4));
  if (st != TRACKFIT_OK) return st;
  const uint16_t* dw = static_cast<uint16_t*>(c->dev);
  float* dv = reinterpret_cast<float*>(static_cast<char*>(c->dev) + wbytes);
  st = tf_status_from_cuda(cudaMemcpy(c->dev, w.data(), w.size() * 2, cudaMemcpyHostToDevice));
  if (st == TRACKFIT_OK) st = tf_status_from_cuda(cudaMemcpy(dv, v.data(), v.size() * 4, cudaMemcpyHostToDevice));
  if (st != TRACKFIT_OK) return st;
  p.vec = dv;
  int64_t chunk = 1 << 20;
  while (chunk > 1024 && (size_t)tf_slab_bound(chunk, s.T) * SLAB * E * 2 + (size_t)chunk * D * 4 > TR_WS_BUDGET) chunk -= 1024;
  c->chunk = chunk;
  const int64_t cap = (tf_slab_bound(chunk, s.T) + 1) / 2 * TILE;
  st = tf_status_from_cuda(tf_malloc(&c->pack, tf_pack_bytes(chunk)));
  if (st == TRACKFIT_OK) st = tf_status_from_cuda(tf_malloc((void**)&c->four, (size_t)cap * E * 2));
  if (st == TRACKFIT_OK) st = tf_status_from_cuda(tf_malloc((void**)&c->pool, (size_t)chunk * D * 4));
  // a last tile of one slab reads the rows of a slab that is not there: zeros, or an
  // earlier batch's, in rows of their own
  if (st == TRACKFIT_OK) st = tf_status_from_cuda(cudaMemset(c->four, 0, (size_t)cap * E * 2));
  if (st != TRACKFIT_OK) return st;
  if (!tile_map(&p.tm[TM_F], c->four, (uint64_t)cap, E, fp16) || !tile_map(&p.tm[TM_E1], dw, D, E, fp16) ||
      !tile_map(&p.tm[TM_E2], dw + D * E, D, D, fp16) || !tile_map(&p.tm[TM_QKV], dw + at_qkv, L * 3 * D, D, fp16) ||
      !tile_map(&p.tm[TM_O], dw + at_o, L * D, D, fp16) ||
      !tile_map(&p.tm[TM_1], dw + at_1, L * H, D, fp16, (uint32_t)p.n1) ||
      !tile_map(&p.tm[TM_2], dw + at_2, L * D, H, fp16))
    return TRACKFIT_ERR_CUDA;
  if (tf_allow_smem(tr_kernel(s)) != cudaSuccess) return TRACKFIT_ERR_CUDA;
  if (tf_head_prepare() != cudaSuccess) return TRACKFIT_ERR_CUDA;
  return TRACKFIT_OK;
}

int tf_tr_forward(trackfit_ctx* h, tf_tr_state* c, uint64_t wait_ns, int hold_tile, const float* hits,
                  const int32_t* n_hits, int64_t B, float* out, float* out_q, float* out_pool, cudaStream_t st, const int64_t* offs) {
  const tf_shape& s = h->s;
  TrParams p = c->p;
  p.err = h->d_err;
  p.wait_ns = wait_ns;
  p.hold_tile = hold_tile;
  const tf_pack pk = tf_pack_in(c->pack, c->chunk);
  p.src.T = s.T;
  p.src.slab = pk.slab;
  p.src.order = pk.order;
  p.src.n_slabs = pk.n_slabs;
  for (int64_t c0 = 0; c0 < B; c0 += c->chunk) {
    const int64_t nb = B - c0 < c->chunk ? B - c0 : c->chunk;
    p.src.hits = offs ? hits : hits + c0 * s.T * s.F;
    p.src.offs = offs ? offs + c0 : nullptr;
    p.src.n_hits = n_hits + c0;
    p.pool = out_pool ? out_pool + c0 * s.P : c->pool;
    cudaError_t e = tf_plan(p.src.n_hits, nb, s.T, c->nsm, pk.order, pk.slab, pk.n_slabs, st);
    if (e == cudaSuccess) e = fourier_slabs(p.src, s, nb, c->nsm, c->four, st);
    if (e == cudaSuccess) {
      tf_prof_begin(h, st);
      tr_kernel(s)<<<c->nsm, NT, c->smem, st>>>(p);
      tf_prof_end(h, st);
      e = tf_head(s, h->off, h->d_w, p.pool, p.src.n_hits, nb, c->nsm, out + c0 * 5, out_q ? out_q + c0 * s.Q : nullptr,
                  out_pool ? p.pool : nullptr, h->d_err, st);
    }
    if (e == cudaSuccess) e = cudaPeekAtLastError();
    if (e != cudaSuccess) {
      tf_note_cuda(e, "transformer_kernel launch");
      return TRACKFIT_ERR_CUDA;
    }
  }
  return TRACKFIT_OK;
}
