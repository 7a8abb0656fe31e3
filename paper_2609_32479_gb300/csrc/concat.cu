// The paper's own model (Sec. 3.2: concatenated directions into the next layer, endpoint
// readout, 16-bit operands) for d_model 128 and up to two layers, in one tensor-core kernel
// behind the Fourier rows.
//
// As separate launches (rows.cu) each layer's fp32 projections went through HBM, 6 KB a
// hit and layer: at 131,072 tracks of 12.5 hits the products took 2.7 ms and the scans
// 1.8 ms.  Here a tile of 128 packed hits (two slabs of whole tracks, as in
// tc_forward.cu) stays on its SM from the Fourier vector to the readout:
//   D[channel][hit] = W[channel][k] Act[k][hit],
// accumulators in TMEM with one channel a lane, so that an epilogue thread owns a channel
// and walks the hits of its tracks; the scans run in registers on the accumulators.
//
// Warp roles (608 threads): 0 TMA producer, 1 MMA issuer and TMEM owner, 2-17 epilogue,
// 18 loader of the tile's column metadata.  The Fourier vector (480 rows for 15
// features, 120 KB a tile) is not kept: its 64-row chunks stream through the same ring of
// 16 KB blocks as the weights, K-major from global memory.  Shared memory: X (the embedding
// output, 128 k-rows) and Y (the states of layer 0, 384 k-rows; the embedding's hidden
// values lie in its first 128 rows before).  TMEM: two buffers of 256 columns, filled by
// turns: every product group (the embedding's two, then z and n of 64 channels of both
// directions) waits only until the epilogue has copied the group before last to registers.
#include <cstring>
#include <new>
#include <vector>

#include "tiles.cuh"

namespace {

constexpr int CT_H = 192, CT_NDC = 3;                // hidden width, chunks of 64 channels
constexpr int CT_Y = 0, CT_X = 98304, CT_RING = 131072;
constexpr int CT_MAX_STAGES = 6;
constexpr uint64_t CT_DRAIN_NS = 200000000ull;
constexpr size_t CT_WS_BUDGET = (size_t)4 << 30;     // bytes of the Fourier rows

enum { CM_F = 0, CM_E1, CM_E2, CM_IN0, CM_IN1, CM_MAPS };

struct CatParams {
  CUtensorMap tm[CM_MAPS];
  TileSrc src;
  float* pool;          // [B][2 H] endpoint states
  int L, KE, nst;       // layers, 64-row chunks of the Fourier vector, ring stages
  int last_nk;          // 16-row steps of its last chunk: 2 or 4 (E is a multiple of 32)
  uint32_t idesc_mn, idesc_k;   // activations MN-major (shared memory) or K-major (Fourier rows)
  const float *b_e1, *b_e2;     // [128]
  const float* b_in;            // [L][NDC * 256], chunk order
  unsigned long long* err;
  uint64_t wait_ns;
  int hold_tile;        // test hook: CTA 0's loader holds this tile's metadata hand-over (-1: none)
};

struct CatMisc {
  uint64_t full[CT_MAX_STAGES], empty[CT_MAX_STAGES];
  uint64_t acc_full[2], acc_free[2], op_bar, drain_bar;
  uint64_t meta_full[2], meta_free[2];
  uint32_t tmem_base;
  int abort_flag;
  TileMeta meta[2];
  float carry[2][2][128];   // by chunk parity: a slab's second segment may read one while its first writes the next
};
constexpr size_t CT_SMEM_REST = sizeof(CatMisc) + 1024;

__device__ __forceinline__ void cat_abort(CatMisc* m, unsigned long long* err) {
  if (atomicExch(&m->abort_flag, 1) == 0) atomicAdd(err + 1, 1ull);
}

// The endpoint states of the tracks that end (forward) or start (reverse) in the
// thread's 32 columns: states h of channel ch of [h_f; h_b].
__device__ __forceinline__ void put_endpoints(const ECtx& x, const float (&h)[32], int ch) {
  const uint32_t ends = x.q < 2 ? x.md->m_last[x.half][x.sub] : x.md->m_first[x.half][x.sub];
#pragma unroll
  for (int j = 0; j < 32; ++j)
    if (ends & (1u << j)) x.pool[(size_t)x.md->slot_track[x.md->col_slot[x.col0 + j]] * (2 * CT_H) + ch] = h[j];
}

template <bool FP16>
__global__ void __launch_bounds__(NT, 1) concat_kernel(const __grid_constant__ CatParams p) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  CatMisc* m = reinterpret_cast<CatMisc*>(smem_raw + (base - raw) + CT_RING + p.nst * A_BLOCK);
  const uint32_t ring = base + CT_RING;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t full0 = smem_u32(&m->full[0]), empty0 = smem_u32(&m->empty[0]);
  const uint32_t acc_full = smem_u32(&m->acc_full[0]), acc_free = smem_u32(&m->acc_free[0]);
  const uint32_t op_bar = smem_u32(&m->op_bar), drain_bar = smem_u32(&m->drain_bar);
  if (threadIdx.x == 0) {
    for (int s = 0; s < p.nst; ++s) {
      mbar_init(full0 + 8 * s, 1);
      mbar_init(empty0 + 8 * s, 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(acc_full + 8 * b, 1);
      mbar_init(acc_free + 8 * b, NE / 32);
      mbar_init(smem_u32(&m->meta_full[b]), 1);
      mbar_init(smem_u32(&m->meta_free[b]), NE / 32);
    }
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
    for (int i = 0; i < CM_MAPS; ++i) prefetch_tmap(&p.tm[i]);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = m->tmem_base;
  const int n_slabs = *p.src.n_slabs, n_tiles = (n_slabs + 1) >> 1;
  volatile int* abort = &m->abort_flag;

  if (warp == 0) {
    // TMA producer: one lane
    if (elect_one()) {
      uint32_t stage = 0, phase = 0;
      int issued = 0;
      bool ok = true;
      auto load = [&](int map, int c0, int c1) {
        if (!ok) return;
        const uint32_t full = full0 + 8 * stage;
        if (!mbar_wait(empty0 + 8 * stage, phase ^ 1u, abort, p.wait_ns)) {
          cat_abort(m, p.err);
          ok = false;
          return;
        }
        mbar_arrive_expect_tx(full, A_BLOCK);
        tma_load_2d(ring + stage * A_BLOCK, &p.tm[map], full, c0, c1);
        ++issued;
        if (++stage == (uint32_t)p.nst) {
          stage = 0;
          phase ^= 1u;
        }
      };
      for (int t = blockIdx.x; t < n_tiles && ok; t += gridDim.x) {
        for (int kc = 0; kc < p.KE; ++kc) {
          load(CM_E1, kc * 64, 0);
          load(CM_F, kc * 64, t * TILE);
        }
        for (int kc = 0; kc < 2; ++kc) load(CM_E2, kc * 64, 0);
        for (int l = 0; l < p.L; ++l)
          for (int r = 0; r < 2 * CT_NDC; ++r)   // z, then n, of each chunk
            for (int kc = 0; kc < (l ? 6 : 2); ++kc) load(l ? CM_IN1 : CM_IN0, kc * 64, r * 128);
      }
      if (*abort) {   // let the copies already issued land before the CTA can exit
        volatile int never = 0;
        for (int k = 0; k < p.nst && k < issued; ++k) {
          const int i = issued - 1 - k;
          mbar_wait(full0 + 8 * (i % p.nst), (uint32_t)((i / p.nst) & 1), &never, CT_DRAIN_NS);
        }
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    // MMA issuer: one lane for the whole loop (an elected branch and a vote at each wait
    // cost twice the time of the products; the whole warp in step, as in tc_forward.cu, was
    // 1 % slower here)
    if (elect_one()) {
      uint32_t stage = 0, phase = 0, g = 0, op_k = 0;
      bool ok = true;
      auto wait_bar = [&](uint32_t bar, uint32_t parity) {
        if (ok && !mbar_wait(bar, parity, abort, p.wait_ns)) {
          cat_abort(m, p.err);
          ok = false;
        }
      };
      const uint64_t a_desc = sdesc_sw128(ring, 16, 1024), b_desc = sdesc_sw128(base, B_LBO, B_SBO);
      const uint32_t a_lo0 = desc_lo(a_desc), a_hi = desc_hi(a_desc), b_lo0 = desc_lo(b_desc), b_hi = desc_hi(b_desc);
      constexpr uint32_t BSTEP = (2 * B_SBO) >> 4;
      auto stage_lo = [&]() { return a_lo0 + stage * (A_BLOCK >> 4); };
      auto next_stage = [&]() {
        if (++stage == (uint32_t)p.nst) {
          stage = 0;
          phase ^= 1u;
        }
      };
      // the group's accumulator buffer, free once the epilogue has read group g - 2
      auto begin = [&]() -> uint32_t {
        if (g >= 2) wait_bar(acc_free + 8 * (g & 1u), ((g >> 1) - 1u) & 1u);
        return tmem + (g & 1u) * 256u;
      };
      auto end = [&]() {
        if (ok) umma_commit(acc_full + 8 * (g & 1u));
        ++g;
      };
      auto operand = [&]() { wait_bar(op_bar, op_k++ & 1u); };   // the epilogue's next operand hand-over
      // kb (even) weight blocks against the activations at byte offset off of shared memory
      auto product = [&](uint32_t d, uint32_t off, int kb) {
        uint32_t b_lo = b_lo0 + (off >> 4);
        for (int kc = 0; kc < kb; kc += 2, b_lo += 8 * BSTEP) {
          wait_bar(full0 + 8 * stage, phase);
          const uint32_t a0 = stage_lo(), e0 = empty0 + 8 * stage;
          next_stage();
          wait_bar(full0 + 8 * stage, phase);
          if (!ok) return;
          tc_fence_after();
          umma4_f16<BSTEP>(d, a0, a_hi, b_lo, b_hi, p.idesc_mn, kc);
          umma_commit(e0);
          umma4_f16<BSTEP>(d, stage_lo(), a_hi, b_lo + 4 * BSTEP, b_hi, p.idesc_mn, 1u);
          umma_commit(empty0 + 8 * stage);
          next_stage();
        }
      };
      for (int t = blockIdx.x; t < n_tiles && ok; t += gridDim.x) {
        {   // embedding product 1: weights and Fourier rows alternate in the ring
          const uint32_t d = begin();
          for (int kc = 0; kc < p.KE; ++kc) {
            wait_bar(full0 + 8 * stage, phase);
            const uint32_t a0 = stage_lo(), e0 = empty0 + 8 * stage;
            next_stage();
            wait_bar(full0 + 8 * stage, phase);
            if (!ok) break;
            tc_fence_after();
            if (kc + 1 < p.KE || p.last_nk == 4)
              umma4_f16<2>(d, a0, a_hi, stage_lo(), a_hi, p.idesc_k, kc);
            else
              umma2_f16<2>(d, a0, a_hi, stage_lo(), a_hi, p.idesc_k, kc);
            umma_commit(e0);
            umma_commit(empty0 + 8 * stage);
            next_stage();
          }
          end();
        }
        {   // embedding product 2 from the hidden values (Y's first rows)
          const uint32_t d = begin();
          operand();
          product(d, CT_Y, 2);
          end();
        }
        for (int l = 0; l < p.L && ok; ++l)
          for (int dc = 0; dc < CT_NDC; ++dc) {
            const uint32_t d = begin();
            if (dc == 0) operand();
            product(d, l ? CT_Y : CT_X, l ? 6 : 2);
            product(d + 128, l ? CT_Y : CT_X, l ? 6 : 2);
            end();
          }
      }
      // no MMA may still run when TMEM is released
      umma_commit(drain_bar);
      volatile int never = 0;
      mbar_wait(drain_bar, 0, &never, CT_DRAIN_NS);
    }
    __syncwarp();
  } else if (warp < 2 + NE / 32) {
    // Epilogue.  The warps run decoupled: each arrives on the hand-over barriers itself
    // (16 arrivals).  One operand barrier is enough: between two operand hand-overs every
    // warp waits for a product that the issuer starts only after the first of them.  A
    // failed wait sets the abort flag and every later wait fails fast, but no warp leaves
    // the loop early (the segments of a slab meet at named barriers).  `alive` (the same for
    // a warp's lanes): every wait of this warp has succeeded; only then is the metadata of its
    // tile complete and kept until the warp releases it, and may an address be formed from it.
    bool alive = true;
    ECtx x;
    x.q = warp & 3;
    x.seg = (warp - 2) >> 2;
    x.half = x.seg >> 1;
    x.sub = x.seg & 1;
    x.lane = lane;
    x.c = 32 * x.q + lane;
    x.col0 = SEGW * x.seg;
    x.te = threadIdx.x - 64;
    x.pool = p.pool;
    const uint32_t tq = tmem + ((uint32_t)(32 * x.q) << 16);
    uint32_t g = 0;
    auto wait_on = [&](uint32_t bar, uint32_t parity) {
      const bool got = mbar_wait(bar, parity, abort, p.wait_ns);
      if (!__all_sync(0xffffffffu, got)) {
        if (lane == 0) cat_abort(m, p.err);
        alive = false;
      }
      tc_fence_after();
    };
    auto arrive = [&](uint32_t bar, bool wrote_operands) {
      if (wrote_operands) fence_proxy_async_smem();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar);
    };
    auto wait_group = [&]() {
      wait_on(acc_full + 8 * (g & 1u), (g >> 1) & 1u);
      x.zn = tq + (g & 1u) * 256u;
    };
    auto free_group = [&]() {
      arrive(acc_free + 8 * (g & 1u), false);
      ++g;
    };
    // a 128-channel product group: f of every value (with its bias) to k-row c of buf
    auto operand_rows = [&](float bias, uint32_t buf, auto&& f) {
      wait_group();
      float v[32];
      tmem_ld32(x.zn + x.col0, v);
      tmem_ld_wait();
      free_group();
#pragma unroll
      for (int i = 0; i < 32; ++i) v[i] = f(v[i] + bias);
      store_row32<FP16>(buf, x.c, x.col0, v);
      arrive(op_bar, true);
    };
    int i = 0;
    for (int t = blockIdx.x; t < n_tiles; t += gridDim.x, ++i) {
      operand_rows(p.b_e1[x.c], base + CT_Y, [](float v) { return silu(v); });
      operand_rows(p.b_e2[x.c], base + CT_X, [](float v) { return v; });
      wait_on(smem_u32(&m->meta_full[i & 1]), (uint32_t)(i >> 1) & 1u);
      x.md = &m->meta[i & 1];
      for (int l = 0; l < p.L; ++l) {
        const bool last = l + 1 == p.L;
#pragma unroll 1
        for (int dc = 0; dc < CT_NDC; ++dc) {
          const float* b = p.b_in + (l * CT_NDC + dc) * 256 + x.c;
          const float bz = b[0], bn = b[128];
          wait_group();
          float z[32], n[32];
          scan_load(x, z, n);
          free_group();
          scan_gates(x, z, n, bz, bn);
          x.carry = m->carry[g & 1u];
          scan_chain<true>(x, z, n);
          if (!last) {
            store_row32<FP16>(base + CT_Y + dc * 32768, x.c, x.col0, z);
          } else if (alive) {
            put_endpoints(x, z, (x.c >> 6) * CT_H + dc * 64 + (x.c & 63));
          }
        }
        if (!last) arrive(op_bar, true);
      }
      arrive(smem_u32(&m->meta_free[i & 1]), false);
    }
  } else {
    // loader warp: the column metadata of a tile, one tile ahead
    int i = 0;
    for (int t = blockIdx.x; t < n_tiles; t += gridDim.x, ++i) {
      const int b = i & 1;
      if (i >= 2) {
        const bool got = mbar_wait(smem_u32(&m->meta_free[b]), (uint32_t)((i >> 1) - 1) & 1u, abort, p.wait_ns);
        if (!__all_sync(0xffffffffu, got) && lane == 0) cat_abort(m, p.err);
        // after a failure anywhere a release may have come from a warp that gave up: stop, so
        // that the metadata others still read stays as it is
        if (!__all_sync(0xffffffffu, got && !*abort)) break;
      }
      load_meta(p.src, nullptr, &m->meta[b], 2 * t, n_slabs, lane);
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

struct tf_cat_state {
  int nsm;
  int64_t chunk;      // tracks at a time
  size_t smem;
  void *dev, *pack;   // weights and biases; packing
  uint16_t* four;     // Fourier rows
  float* pool;        // [chunk][2 H]
  CatParams p;
};

// d_model 128 (the hidden width is then 192), endpoint readout, one or two layers: the
// states of one layer and the embedding output are what shared memory holds.  Others
// run as separate launches (rows.cu).
bool tf_cat_supported(const tf_shape& s) {
  return (s.precision == TRACKFIT_BF16_PROJ || s.precision == TRACKFIT_FP16_PROJ) &&
         s.topology == TRACKFIT_TOPOLOGY_CONCAT && s.pool == TRACKFIT_POOL_ENDPOINTS && s.D == 128 && s.H == CT_H &&
         s.L <= 2 && s.K == TRACKFIT_MAX_FOURIER;
}

void tf_cat_destroy(tf_cat_state* c) {
  if (!c) return;
  tf_free(c->dev);
  tf_free(c->pack);
  tf_free(c->four);
  tf_free(c->pool);
  delete c;
}

int tf_cat_create(trackfit_ctx* h, const float* W, tf_cat_state** out) {
  const tf_shape& s = h->s;
  const tf_blob_off& o = h->off;
  tf_cat_state* c = new (std::nothrow) tf_cat_state();
  if (!c) return TRACKFIT_ERR_OOM;
  *out = c;   // freed by the caller's tf_cat_destroy on any failure below
  const bool fp16 = s.precision == TRACKFIT_FP16_PROJ;
  int dev = 0, optin = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&c->nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess)
    return TRACKFIT_ERR_CUDA;
  CatParams& p = c->p;
  p.L = s.L;
  p.KE = (s.E + 63) / 64;
  p.last_nk = (s.E - 64 * (p.KE - 1)) / 16;
  p.nst = (optin - (int)CT_SMEM_REST - CT_RING) / A_BLOCK;
  if (p.nst > CT_MAX_STAGES) p.nst = CT_MAX_STAGES;
  if (p.nst < 4) return TRACKFIT_ERR_UNSUPPORTED;
  c->smem = CT_RING + (size_t)p.nst * A_BLOCK + CT_SMEM_REST;
  p.idesc_mn = idesc_f16(128, 128, fp16 ? 0u : 1u, false, true);
  p.idesc_k = idesc_f16(128, 128, fp16 ? 0u : 1u, false, false);
  // weights: W_e1 [128][E], W_e2 [128][128], then per layer the rows in chunk order (64
  // forward z, 64 reverse z, the same of n, for each 64 channels) and, after layer 0,
  // the columns too (Y holds chunk by chunk 64 forward and 64 reverse states)
  const size_t D = s.D, H = s.H, E = s.E, rows = CT_NDC * 256;
  std::vector<uint16_t> w(D * E + D * D + rows * D + rows * 2 * H);
  std::vector<float> b(2 * D + 2 * rows, 0.0f);
  size_t at = 0;
  for (size_t i = 0; i < D * E; ++i) w[at++] = to_16(W[o.emb_w1 + i], fp16);
  for (size_t i = 0; i < D * D; ++i) w[at++] = to_16(W[o.emb_w2 + i], fp16);
  for (size_t i = 0; i < D; ++i) {
    b[i] = W[o.emb_b1 + i];
    b[D + i] = W[o.emb_b2 + i];
  }
  for (int l = 0; l < s.L; ++l) {
    const tf_layer_off& lo = o.layer[l];
    const size_t I = l ? 2 * H : D;
    for (size_t r = 0; r < rows; ++r) {
      const size_t dc = r / 256, n = (r / 128) & 1, dir = (r / 64) & 1, ch = dc * 64 + (r & 63);
      const size_t src = (2 * dir + n) * H + ch;
      for (size_t k = 0; k < I; ++k) {
        const size_t kk = l ? ((k / 64) & 1) * H + (k / 128) * 64 + (k & 63) : k;
        w[at++] = to_16(W[lo.w_in + src * I + kk], fp16);
      }
      b[2 * D + l * rows + r] = W[lo.b_in + src];
    }
  }
  const size_t wbytes = (w.size() * 2 + 255) / 256 * 256;
  int st = tf_status_from_cuda(tf_malloc(&c->dev, wbytes + b.size() * 4));
  if (st != TRACKFIT_OK) return st;
  uint16_t* dw = static_cast<uint16_t*>(c->dev);
  float* db = reinterpret_cast<float*>(static_cast<char*>(c->dev) + wbytes);
  st = tf_status_from_cuda(cudaMemcpy(dw, w.data(), w.size() * 2, cudaMemcpyHostToDevice));
  if (st == TRACKFIT_OK) st = tf_status_from_cuda(cudaMemcpy(db, b.data(), b.size() * 4, cudaMemcpyHostToDevice));
  if (st != TRACKFIT_OK) return st;
  p.b_e1 = db;
  p.b_e2 = db + D;
  p.b_in = db + 2 * D;
  int64_t chunk = 1 << 20;
  while (chunk > 1024 && (size_t)tf_slab_bound(chunk, s.T) * SLAB * E * 2 + (size_t)chunk * 2 * H * 4 > CT_WS_BUDGET) chunk -= 1024;
  c->chunk = chunk;
  const int64_t cap = (tf_slab_bound(chunk, s.T) + 1) / 2 * TILE;
  if (st == TRACKFIT_OK) st = tf_status_from_cuda(tf_malloc(&c->pack, tf_pack_bytes(chunk)));
  if (st == TRACKFIT_OK) st = tf_status_from_cuda(tf_malloc((void**)&c->four, (size_t)cap * E * 2));
  if (st == TRACKFIT_OK) st = tf_status_from_cuda(tf_malloc((void**)&c->pool, (size_t)chunk * 2 * H * 4));
  // a last tile of one slab reads the rows of a slab that is not there: zeros, or an
  // earlier batch's, in columns of their own
  if (st == TRACKFIT_OK) st = tf_status_from_cuda(cudaMemset(c->four, 0, (size_t)cap * E * 2));
  if (st != TRACKFIT_OK) return st;
  const uint16_t *we2 = dw + D * E, *w0 = we2 + D * D, *w1 = w0 + rows * D;
  if (!tile_map(&p.tm[CM_F], c->four, (uint64_t)cap, E, fp16) || !tile_map(&p.tm[CM_E1], dw, D, E, fp16) ||
      !tile_map(&p.tm[CM_E2], we2, D, D, fp16) || !tile_map(&p.tm[CM_IN0], w0, rows, D, fp16) ||
      !tile_map(&p.tm[CM_IN1], w1, rows, 2 * H, fp16))
    return TRACKFIT_ERR_CUDA;
  if (tf_allow_smem(concat_kernel<false>) != cudaSuccess || tf_allow_smem(concat_kernel<true>) != cudaSuccess)
    return TRACKFIT_ERR_CUDA;
  if (tf_head_prepare() != cudaSuccess) return TRACKFIT_ERR_CUDA;
  return TRACKFIT_OK;
}

int tf_cat_forward(trackfit_ctx* h, tf_cat_state* c, uint64_t wait_ns, int hold_tile, const float* hits,
                   const int32_t* n_hits, int64_t B, float* out, float* out_q, float* out_pool, cudaStream_t st, const int64_t* offs) {
  const tf_shape& s = h->s;
  CatParams p = c->p;
  const bool fp16 = s.precision == TRACKFIT_FP16_PROJ;
  p.err = h->d_err;
  p.wait_ns = wait_ns;
  p.hold_tile = hold_tile;
  p.src.T = s.T;
  const tf_pack pk = tf_pack_in(c->pack, c->chunk);
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
      if (fp16)
        concat_kernel<true><<<c->nsm, NT, c->smem, st>>>(p);
      else
        concat_kernel<false><<<c->nsm, NT, c->smem, st>>>(p);
      tf_prof_end(h, st);
      e = tf_head(s, h->off, h->d_w, p.pool, p.src.n_hits, nb, c->nsm, out + c0 * 5, out_q ? out_q + c0 * s.Q : nullptr,
                  out_pool ? p.pool : nullptr, h->d_err, st);
    }
    if (e == cudaSuccess) e = cudaPeekAtLastError();
    if (e != cudaSuccess) {
      tf_note_cuda(e, "concat_kernel launch");
      return TRACKFIT_ERR_CUDA;
    }
  }
  return TRACKFIT_OK;
}
