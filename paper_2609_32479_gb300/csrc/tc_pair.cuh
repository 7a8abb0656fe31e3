// The fused encoder for d_model 128: two tiles of 128 hits in turn.
//
// At this width the epilogue's work on a product takes about as long as the product,
// and with one tile in flight each waited for the other: the MMA issuer stood still for
// 52 % of the time (14.6 ms at 262,144 tracks of six layers, 0.287 of the tensor peak).
// Here the epilogue warps do every step for tile 0 and then for tile 1, so that the
// products of one run while the other is in the epilogue.
//
// TMEM: the merge accumulators, then x', of tile u in columns 128 u; one pair of z and n
// columns (256, 384) that the two tiles use by turns (a tile's columns are free as soon
// as the epilogue has copied them to registers); the output gate and MLP1 of tile u in
// 256 + 128 u.  Shared memory: per tile XB (128 k-rows) and HB (128 k-rows); the Fourier
// operand's 160 rows take HB and the first 32 rows of XB, both free at that time.
// Weights are streamed for each tile by itself (a z/n block would have to stay until the
// other tile's columns are free).  A CTA's last tile runs alone if it has no partner.
//
// Each tile has its own set of barriers, and each set sees the same hand-overs in the
// same order as a tile by itself; the issuer waits for the release of the z/n columns by
// the other tile as well (S_W_X), in place of the tile's own.
#pragma once

enum { W_X = 4 };
constexpr int P_XB = 0, P_HB = 32768, P_TILE = 65536, P_A = 2 * P_TILE;   // shared memory: per tile XB and HB, then the weight ring

// The sequence of weight blocks of nt tiles (1 or 2) through the encoder.
// f(u, map, row, col, nk, tmem_col, bsel, bk, acc, wait, commit) as for walk_tile; u:
// the tile; wait: a sum of W_E, W_H and W_X.
template <class F>
inline void walk_pair(int L, int NDC, int ROWS_IN, int nt, F&& f) {
  // the embedding's first product goes to the gate columns, so it can run while the
  // epilogue still pools the tiles before
  for (int u = 0; u < nt; ++u)
    for (int kc = 0; kc < 3; ++kc)
      f(u, MAP_E1, 0, kc * 64, kc == 2 ? 2 : 4, 256 + 128 * u, kc == 2 ? BSEL_XB : BSEL_HB, kc == 2 ? 0 : kc * 64,
        kc > 0, kc == 0 ? W_E : W_NONE, kc == 2 ? C_ACC : C_NONE);
  // a 128 x 128 product from XB
  auto dense = [&](int u, int map, int r0, int tcol, bool onto, int wait, int commit) {
    for (int kc = 0; kc < 2; ++kc)
      f(u, map, r0, kc * 64, 4, tcol, BSEL_XB, kc * 64, onto || kc > 0, kc == 0 ? wait : W_NONE,
        kc == 1 ? commit : C_NONE);
  };
  for (int u = 0; u < nt; ++u) dense(u, MAP_E2, 0, 128 * u, false, W_E, C_ACC);
  for (int l = 0; l < L; ++l) {
    const int rb = l * ROWS_IN;
    auto merge = [&](int u, int k, int commit) {
      for (int kc = 0; kc < 2; ++kc)
        f(u, MAP_M, l * 128, k * 128 + kc * 64, 4, 128 * u, BSEL_HB, kc * 64, k > 0 || kc > 0, kc == 0 ? W_H : W_NONE,
          kc == 1 ? commit : C_NONE);
    };
    for (int k = 0; k < NDC; ++k)
      for (int u = 0; u < nt; ++u) {
        // x_hat of the tile, and the z/n columns released by whichever tile had them
        int wait = k == 0 ? W_E : W_NONE;
        if (nt == 1)
          wait = W_E;
        else if (u == 1 || k > 0)
          wait |= W_X;
        dense(u, MAP_IN, rb + k * 256, 256, false, wait, C_NONE);
        dense(u, MAP_IN, rb + k * 256 + 128, 384, false, W_NONE, C_ACC);
        if (k > 0) merge(u, k - 1, C_HB);
      }
    for (int u = 0; u < nt; ++u) {
      dense(u, MAP_IN, rb + NDC * 256, 256 + 128 * u, false, nt == 1 ? (int)W_E : u == 0 ? (int)W_X : 0, C_NONE);
      merge(u, NDC - 1, C_ACC);
    }
    for (int u = 0; u < nt; ++u) dense(u, MAP_1, l * 128, 256 + 128 * u, false, W_E, C_ACC);
    for (int u = 0; u < nt; ++u) dense(u, MAP_2, l * 128, 128 * u, true, W_E, C_ACC);   // onto x'
  }
}

struct PairMisc {
  uint64_t full[MAX_STAGES], empty[MAX_STAGES];
  uint64_t acc_bar[2][2], e_bar[2][2], hb_bar[2], eh_bar[2], drain_bar;   // [tile]([alternating])
  uint64_t meta_full[4], meta_free[4];   // [2 x (pair mod 2) + tile]
  uint32_t tmem_base;
  int abort_flag;
  TileMeta meta[4];
  LoaderScratch ls;
  alignas(16) float part[2][4][TILE];
  float carry[2][2][128];
  alignas(16) float rinv[NE / 32][32];
};

// THIN: a tile is one slab, with half the columns and half the epilogue warps, and a CTA
// has at most one.  While every slab can have a CTA of its own the batch's time is one
// tile's chain of steps, and that is shorter then (101 tracks: 145 -> 120 us a call).
template <bool THIN>
constexpr int PAIR_EPI = THIN ? NE / 64 : NE / 32;   // epilogue warps
template <bool THIN>
constexpr int PAIR_NT = 32 * (PAIR_EPI<THIN> + 3);

template <bool FP16, bool THIN>
__global__ void __launch_bounds__(PAIR_NT<THIN>, 1) tc_pair_kernel(const __grid_constant__ TcParams p) {
  constexpr int EW = PAIR_EPI<THIN>;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t* gbase = smem_raw + (base - raw);
  PairMisc* m = reinterpret_cast<PairMisc*>(gbase + p.off_misc);
  const uint32_t ab = base + P_A;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t full0 = smem_u32(&m->full[0]), empty0 = smem_u32(&m->empty[0]);
  const uint32_t acc_bar = smem_u32(&m->acc_bar[0][0]), e_bar = smem_u32(&m->e_bar[0][0]);
  const uint32_t hb_bar = smem_u32(&m->hb_bar[0]), eh_bar = smem_u32(&m->eh_bar[0]);
  const uint32_t drain_bar = smem_u32(&m->drain_bar);

  if (threadIdx.x == 0) {
    for (int s = 0; s < p.nst; ++s) {
      mbar_init(full0 + 8 * s, 1);
      mbar_init(empty0 + 8 * s, 1);
    }
    for (int i = 0; i < 4; ++i) {
      mbar_init(acc_bar + 8 * i, 1);
      mbar_init(e_bar + 8 * i, EW);   // one arrival per epilogue warp
      mbar_init(smem_u32(&m->meta_full[i]), 1);
      mbar_init(smem_u32(&m->meta_free[i]), EW);
    }
    for (int u = 0; u < 2; ++u) {
      mbar_init(hb_bar + 8 * u, 1);
      mbar_init(eh_bar + 8 * u, EW);
    }
    mbar_init(drain_bar, 1);
    m->abort_flag = 0;
    fence_mbar_init();
  }
  // the steps of one tile, then those of two
  Step* tab = reinterpret_cast<Step*>(gbase + p.off_misc + sizeof(PairMisc));
  const int n1 = p.n_sched, n2 = p.n_sched2;
  for (int i = threadIdx.x; i < n1 + n2; i += blockDim.x) tab[i] = p.sched[i];
  if (warp == 1) {
    tmem_alloc(smem_u32(&m->tmem_base), 512);
    tmem_relinquish();
  }
  if (warp == 0 && lane == 0)
    for (int i = 0; i < NMAPS; ++i) prefetch_tmap(&p.tm[i]);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = m->tmem_base;
  const int n_slabs = *p.src.n_slabs;
  const int n_tiles = THIN ? n_slabs : (n_slabs + 1) >> 1;
  int mine = 0;   // this CTA's tiles: blockIdx.x + j gridDim.x
  if ((int)blockIdx.x < n_tiles) mine = (n_tiles - 1 - (int)blockIdx.x) / (int)gridDim.x + 1;
  volatile int* abort = &m->abort_flag;

  // the loader's scratch for the CTA's first tiles, in the part of their XB that the Fourier
  // operand leaves free
  auto first_hits = [&](int u) { return reinterpret_cast<LoaderScratch*>(gbase + P_XB + u * P_TILE + 16384); };

  if (warp == 0) {
    // TMA producer: the 16 KB weight blocks in schedule order, one ring stage each; as in
    // the one-tile kernel, one lane's copies are let through by a predicate
    uint32_t stage = 0, phase = 0;
    const uint32_t me = elect_one() ? 1u : 0u;
    bool ok = true;
    int issued = 0;
    for (int j = 0; j < mine && ok; j += 2) {
      const bool two = j + 1 < mine;
      const Step* t = two ? tab + n1 : tab;
      const int n = two ? n2 : n1;
      for (int i = 0; i < n && ok; ++i) {
        const Step e = t[i];
        const CUtensorMap* map = &p.tm[e.prod & 15u];
        int c0 = (int)((e.prod >> 4) & 15u) * 64;
        const int c1 = (int)(e.prod >> 8), nb = (e.mma & S_TAIL) ? 1 : 2;
        for (int b = 0; b < nb; ++b, c0 += 64) {
          const uint32_t full = full0 + 8 * stage;
          if (!mbar_wait(empty0 + 8 * stage, phase ^ 1u, abort, p.wait_ns)) {
            set_abort(&m->abort_flag, p.err);
            ok = false;
          }
          ok = __all_sync(0xffffffffu, ok);
          if (!ok) break;
          mbar_arrive_expect_tx_if(full, A_BLOCK, me);
          tma_load_2d_if(ab + stage * A_BLOCK, map, full, c0, c1, me);
          ++issued;
          if (++stage == (uint32_t)p.nst) {
            stage = 0;
            phase ^= 1u;
          }
        }
      }
    }
    __syncwarp();
    if (*abort) {   // let the copies already issued land before the CTA can exit
      volatile int never = 0;
      for (int k = 0; k < p.nst && k < issued; ++k) {
        const int i = issued - 1 - k;
        mbar_wait(full0 + 8 * (i % p.nst), (uint32_t)((i / p.nst) & 1), &never, DRAIN_NS);
      }
    }
  } else if (warp == 1) {
    // MMA issuer: one straight line and one vote a step, as in the one-tile kernel
    uint32_t stage = 0, phase = 0;
    uint32_t e_k0 = 0, e_k1 = 0, h_k0 = 0, h_k1 = 0, a_k0 = 0, a_k1 = 0;   // hand-overs and commits so far, by tile
    const uint32_t me = elect_one() ? 1u : 0u;
    bool ok = true;
    const uint64_t a_desc = sdesc_sw128(ab, 16, 1024), b_desc = sdesc_sw128(base, B_LBO, B_SBO);
    const uint32_t a_lo0 = desc_lo(a_desc), a_hi = desc_hi(a_desc), b_lo0 = desc_lo(b_desc), b_hi = desc_hi(b_desc);
    constexpr uint32_t BSTEP = (2 * B_SBO) >> 4;
    const uint32_t idesc = THIN ? p.idesc_thin : p.idesc;   // N = 64, 128
    auto wait_bar = [&](uint32_t bar, uint32_t parity) {
      if (!mbar_wait(bar, parity, abort, p.wait_ns)) {
        set_abort(&m->abort_flag, p.err);
        ok = false;
      }
    };
    auto wait_e = [&](uint32_t u) {   // tile u's k-th operand hand-over arrives on e_bar[u][k % 2]
      const uint32_t k = u ? e_k1 : e_k0;
      e_k0 += u ^ 1u;
      e_k1 += u;
      wait_bar(e_bar + 16 * u + 8 * (k & 1u), (k >> 1) & 1u);
    };
    for (int j = 0; j < mine && ok; j += 2) {
      const bool two = j + 1 < mine;
      const int n = two ? n2 : n1;
      const Step* t = two ? tab + n1 : tab;
      uint32_t e = t[0].mma;
      for (int i = 0; i < n; ++i) {
        const uint32_t en = t[i + 1 < n ? i + 1 : 0].mma, u = (e & S_TILE) ? 1u : 0u;
        if (e & S_W_E) wait_e(u);
        if (e & S_W_X) wait_e(u ^ 1u);
        if (e & S_W_H) {
          const uint32_t k = u ? h_k1 : h_k0;
          h_k0 += u ^ 1u;
          h_k1 += u;
          wait_bar(eh_bar + 8 * u, k & 1u);
        }
        wait_bar(full0 + 8 * stage, phase);
        const uint32_t a_lo = a_lo0 + stage * (A_BLOCK >> 4), b_lo = b_lo0 + (e & 0xFFFFu);
        const uint32_t d = tmem + ((e & S_COL) >> 16) * 128u;
        if (e & S_TAIL) {
          ok = __all_sync(0xffffffffu, ok);
          if (!ok) break;
          tc_fence_after();
          umma2_f16_if<BSTEP>(d, a_lo, a_hi, b_lo, b_hi, idesc, 1u, me);
          umma_commit_if(empty0 + 8 * stage, me);
        } else {
          const uint32_t s0 = stage;
          if (++stage == (uint32_t)p.nst) {
            stage = 0;
            phase ^= 1u;
          }
          wait_bar(full0 + 8 * stage, phase);
          ok = __all_sync(0xffffffffu, ok);
          if (!ok) break;
          tc_fence_after();
          umma4_f16_if<BSTEP>(d, a_lo, a_hi, b_lo, b_hi, idesc, e & S_ACC, me);
          umma_commit_if(empty0 + 8 * s0, me);
          umma4_f16_if<BSTEP>(d, a_lo0 + stage * (A_BLOCK >> 4), a_hi, b_lo + 4 * BSTEP, b_hi, idesc, 1u, me);
          umma_commit_if(empty0 + 8 * stage, me);
        }
        if (e & S_C_ACC) {   // tile u's k-th accumulator commit goes to acc_bar[u][k % 2]
          const uint32_t k = u ? a_k1 : a_k0;
          a_k0 += u ^ 1u;
          a_k1 += u;
          umma_commit_if(acc_bar + 16 * u + 8 * (k & 1u), me);
        } else if (e & S_C_HB) {
          umma_commit_if(hb_bar + 8 * u, me);
        }
        e = en;
        if (++stage == (uint32_t)p.nst) {
          stage = 0;
          phase ^= 1u;
        }
      }
    }
    __syncwarp();
    // no MMA may still run when TMEM is released (by the lane that issued them)
    umma_commit_if(drain_bar, me);
    volatile int never = 0;
    mbar_wait(drain_bar, 0, &never, DRAIN_NS);
    __syncwarp();
  } else if (warp < 2 + EW) {
    // Epilogue: every step for tile 0, then for tile 1.  The warps run decoupled, as in
    // the one-tile kernel; its argument that no warp is two hand-overs ahead or two
    // commits behind holds for each tile's own barriers.  A failed wait sets the abort
    // flag and every later wait fails fast, but no warp leaves the loop early; `alive` as in
    // the one-tile kernel.
    bool alive = true;
    const int q = warp & 3, seg = (warp - 2) >> 2;
    ECtx x;
    x.q = q;
    x.seg = seg;
    x.half = seg >> 1;
    x.sub = seg & 1;
    x.lane = lane;
    x.c = 32 * q + lane;
    x.col0 = SEGW * seg;
    x.te = threadIdx.x - 64;
    x.zn = tmem + ((uint32_t)(32 * q) << 16) + 256;
    x.rinv = m->rinv[warp - 2];
    x.pool = p.pool;
    x.rms_eps = p.rms_eps;
    int pair = 0;
    auto tile = [&](int u) {   // the context of tile u
      x.xb = base + P_XB + u * P_TILE;
      x.hb = base + P_HB + u * P_TILE;
      x.acc = x.zn - 256 + 128 * u;
      x.gt = x.zn + 128 * u;
      x.xs = p.xs + ((size_t)blockIdx.x * 2 + u) * TILE * 128;
      x.part = m->part[u];
      x.carry = m->carry[u];
      x.md = &m->meta[2 * (pair & 1) + u];
    };
    uint32_t e_k0 = 0, e_k1 = 0, a_k0 = 0, a_k1 = 0, hb_k0 = 0, hb_k1 = 0;
    auto arrive = [&](uint32_t bar, bool wrote_operands) {
      if (wrote_operands) fence_proxy_async_smem();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar);
    };
    auto signal_e = [&](int u, bool wrote_operands) {
      const uint32_t k = u ? e_k1 : e_k0;
      if (u) ++e_k1; else ++e_k0;
      arrive(e_bar + 16 * u + 8 * (k & 1u), wrote_operands);
    };
    auto wait_on = [&](uint32_t bar, uint32_t parity) {
      const bool got = mbar_wait(bar, parity, abort, p.wait_ns);
      if (!__all_sync(0xffffffffu, got)) {
        if (lane == 0) set_abort(&m->abort_flag, p.err);
        alive = false;
      }
      tc_fence_after();
    };
    auto wait_acc = [&](int u) {
      const uint32_t k = u ? a_k1 : a_k0;
      if (u) ++a_k1; else ++a_k0;
      wait_on(acc_bar + 16 * u + 8 * (k & 1u), (k >> 1) & 1u);
    };
    auto wait_hb = [&](int u) {
      const uint32_t k = u ? hb_k1 : hb_k0;
      if (u) ++hb_k1; else ++hb_k0;
      wait_on(hb_bar + 8 * u, k & 1u);
    };
    // the Fourier operand of tile u of a pair: the loads need the loader's hand-over,
    // the stores need the tile's HB and XB free.
    const uint8_t* fbuf = p.fbuf + (size_t)blockIdx.x * 4 * EB_BYTES;
    // a thread's r-th 16-byte chunk of the operand
    auto chunk = [&](int r) -> uint32_t { return (uint32_t)(r * EW * 32 + x.te) * 16u; };
    auto fetch = [&](int pr, int u, uint4 (&v)[5]) {
      const int b = 2 * (pr & 1) + u;
      wait_on(smem_u32(&m->meta_full[b]), (uint32_t)(pr >> 1) & 1u);
#pragma unroll
      for (int r = 0; r < 5; ++r) v[r] = __ldcg(reinterpret_cast<const uint4*>(fbuf + b * EB_BYTES + chunk(r)));
    };
    auto put = [&](int u, const uint4 (&v)[5]) {
      const uint32_t hb = base + P_HB + u * P_TILE, xb = base + P_XB + u * P_TILE;
#pragma unroll
      for (int r = 0; r < 4; ++r) st_shared_v4(hb + chunk(r), v[r].x, v[r].y, v[r].z, v[r].w);
      st_shared_v4(xb + chunk(4) - 128 * 256, v[4].x, v[4].y, v[4].z, v[4].w);   // k-rows 128-159
      signal_e(u, true);
    };
    // The CTA's first tiles: nothing runs yet that could hide their operand, so the epilogue
    // warps form it themselves instead of the loader warp alone (a call of 101 tracks
    // 115 -> 93 us, 4,096 tracks of 64 hits 1,129 -> 1,077 us)
    for (int u = 0; u < 2 && u < mine; ++u) {
      wait_on(smem_u32(&m->meta_full[u]), 0);
      const uint32_t hb = base + P_HB + u * P_TILE, xb = base + P_XB + u * P_TILE;
      fourier_operand<FP16>(p.src, first_hits(u), &m->meta[u], (THIN ? SLAB : TILE) / 8, x.te, EW * 32,
                            [&](int row, int g, uint4 v) {
                              st_shared_v4(row < 128 ? hb + bchunk(row, g) : xb + bchunk(row - 128, g), v.x, v.y, v.z, v.w);
                            });
      signal_e(u, true);
    }
    for (int j = 0; j < mine; j += 2, ++pair) {
      const int nt = j + 1 < mine ? 2 : 1;
#pragma unroll 1
      for (int u = 0; u < nt; ++u) {
        tile(u);
        ep_silu<FP16, 1>(x, p.b_e1, [&]() { wait_acc(u); });
        signal_e(u, true);
      }
#pragma unroll 1
      for (int l = -1; l < p.L; ++l) {
        // l = -1: the embedding output; the residual stream and x_hat of layer l + 1
        // are formed at the end of layer l
        if (l >= 0) {
#pragma unroll 1
          for (int dc = 0; dc < p.NDC; ++dc) {
            const size_t rb = (size_t)l * p.ROWS_IN + dc * 256;
            const float bz = p.b_in[rb + x.c], bn = p.b_in[rb + 128 + x.c];
#pragma unroll 1
            for (int u = 0; u < nt; ++u) {
              tile(u);
              wait_acc(u);
              float z[32], n[32];
              scan_load(x, z, n);
              signal_e(u, false);   // the z/n columns are free
              scan_gates(x, z, n, bz, bn);
              // HB still feeds the merge of the previous chunk (the gate hand-over
              // covers the last merge of the previous layer)
              if (dc > 0) wait_hb(u);
              scan_chain_store<FP16>(x, z, n);
              arrive(eh_bar + 8 * u, true);
            }
          }
          const float bm = p.b_m[(size_t)l * 128 + x.c], bg = p.b_in[(size_t)l * p.ROWS_IN + p.NDC * 256 + x.c],
                      b1 = p.b_1[(size_t)l * 128 + x.c];
#pragma unroll 1
          for (int u = 0; u < nt; ++u) {
            tile(u);
            float xg[32];
            gate_x_load<1>(x, 0, xg);
            wait_acc(u);
            ep_gate<FP16>(x, 0, xg, bm, bg);
            signal_e(u, true);
          }
#pragma unroll 1
          for (int u = 0; u < nt; ++u) {
            tile(u);
            wait_acc(u);
            ep_silu_mt<FP16>(x, b1, 0, x.xb, 0);
            signal_e(u, true);
          }
        }
        if (l + 1 < p.L) {
          const float* bias = l < 0 ? p.b_e2 : p.b_2 + (size_t)l * 128;
#pragma unroll 1
          for (int u = 0; u < nt; ++u) {
            tile(u);
            ep_residual<FP16, 1>(x, bias, p.g + (size_t)(l + 1) * 128, [&]() { wait_acc(u); },
                                 [&]() { signal_e(u, true); });
          }
        } else {
          // once a tile's last MLP2 has completed, its HB and XB are free: the next
          // pair's Fourier operand goes in and its first product runs while this pair is
          // pooled, tile 0 by the warps of each slab's first segment, tile 1 by the others
#pragma unroll 1
          for (int u = 0; u < nt; ++u) {
            const bool more = !THIN && j + 2 + u < mine;
            uint4 fv[5];
            if (more) fetch(pair + 1, u, fv);
            wait_acc(u);
            if (more) put(u, fv);
          }
          if (alive && x.sub < nt) {
            tile(x.sub);
            ep_pool<1>(x, 0, p.b_2 + (size_t)l * 128);
          }
          for (int u = 0; u < nt; ++u) arrive(smem_u32(&m->meta_free[2 * (pair & 1) + u]), false);
        }
      }
    }
  } else {
    // loader warp: tile set-up one pair ahead of the epilogue
    uint8_t* fbuf = p.fbuf + (size_t)blockIdx.x * 4 * EB_BYTES;
    for (int j = 0; j < mine; ++j) {
      const int pr = j >> 1, b = 2 * (pr & 1) + (j & 1);
      if (pr >= 2) {   // the buffer last held a tile of pair pr - 2
        const bool got = mbar_wait(smem_u32(&m->meta_free[b]), (uint32_t)((pr >> 1) - 1) & 1u, abort, p.wait_ns);
        if (!__all_sync(0xffffffffu, got) && lane == 0) set_abort(&m->abort_flag, p.err);
        if (!__all_sync(0xffffffffu, got && !*abort)) break;   // as in the one-tile kernel
      }
      const int t = (int)blockIdx.x + j * (int)gridDim.x;
      const int s0 = THIN ? t : 2 * t, end = THIN ? t + 1 : n_slabs;
      if (j < 2) {
        load_meta(p.src, first_hits(j)->col_tpos, &m->meta[b], s0, end, lane);
        load_hits(p.src, first_hits(j), &m->meta[b], lane);
      } else {
        load_tile<FP16>(p.src, &m->ls, &m->meta[b], fbuf + b * EB_BYTES, s0, end, lane);
      }
      __threadfence_block();
      __syncwarp();
      if (j == p.hold_tile && blockIdx.x == 0) hold_hand_over(abort, p.wait_ns);
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
