// Device code that the fused tensor-core kernels share (tc_forward.cu: d_model 256, one
// tile of 128 hits at a time; tc_pair.cuh: d_model 128, two tiles in turn): the operand
// layout, the epilogue steps of one tile and the loader's tile set-up.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <math.h>

#include "sm100_ptx.cuh"
#include "trackfit_internal.h"

namespace {

using namespace sm100;

constexpr int NT = 608;                   // warp 0 TMA, warp 1 MMA issuer, warps 2..17 epilogue, warp 18 loader
constexpr int NE = 512;                   // epilogue threads
constexpr int SEGW = 32;                  // hit columns per epilogue thread (half a slab)
constexpr int TILE = 128;
constexpr int SLAB = TF_SLAB;
constexpr int MAX_TRK_TILE = 2 * TF_SLAB_TRACKS;
constexpr int A_BLOCK = 128 * 64 * 2;     // one 128-row x 64-k 16-bit weight block
constexpr int EB_BYTES = 160 * 256;       // Fourier operand: 160 k-rows x 128 hits bf16
constexpr int B_SBO = 2048;               // k-group stride of the MN-major activation operand
constexpr int B_LBO = 1024;               // 64-hit atom stride
enum { F_FIRST = 1, F_LAST = 2, F_VALID = 4 };

// Where a tile's hits come from, for the loader warp.
struct TileSrc {
  const float* hits;
  const int64_t* offs;   // packed input: track b's hits are rows offs[b] .. of hits (null: padded [B][T][5])
  const int32_t* n_hits;
  const int2* slab;      // the packing (tf_pack): slab s = tracks order[slab[s].x ..], slab[s].y of them
  const int32_t* order;
  const int32_t* n_slabs;
  int T;
  int scale_doubling;    // scale[k + 3] == 2 scale[k] for every k: Fourier by angle doubling
  float feat_min[5], feat_inv_hi[5], feat_inv_lo[5], scale[16];
};
struct LoaderScratch {
  uint8_t col_tpos[TILE];
  float hs[TILE][5];
};

// Column metadata of one tile, written by the loader warp one tile ahead (two
// buffers, alternating by tile).
struct TileMeta {
  int slot_track[MAX_TRK_TILE], slot_n[MAX_TRK_TILE];
  uint8_t col_flags[TILE], col_slot[TILE];
  // per column half h, 32-column word w: bit j = column 64h + 32w + j starts a
  // track (first), ends one (last), holds a hit (valid)
  uint32_t m_first[2][2], m_last[2][2], m_valid[2][2];
};
__device__ __forceinline__ float sigm(float x) { return __fdividef(1.0f, 1.0f + __expf(-x)); }
__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float rcp_approx(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
constexpr float LOG2E_F = 1.4426950408889634f;
__device__ __forceinline__ float silu(float x) { return x * sigm(x); }
// The MLP's SiLU inside the fused kernel uses one MUFU operation per value
// instead of two (ex2 and rcp), from SiLU(x) = (x / 2)(1 + tanh(x / 2)):
// tanh.approx has a relative error of about 2^-11, and the result is rounded
// to a 16-bit operand right away (measured: no change in the error against the
// oracle).  The output gate does not: its value scales the merge into the fp32
// residual stream, where that error showed up on every track, so it takes the
// two-operation sigmoid, as do the scan gates (a = 1 - sigma there also needs
// relative accuracy as sigma -> 1).
__device__ __forceinline__ float tanh_approx(float x) {
  float y;
  asm("tanh.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
// Two floats in one 64-bit register: the packed fp32 operations are the IEEE ones on each
// half and take one issue slot for two values.
struct f2 {
  uint64_t v;
  __device__ __forceinline__ f2(float a, float b) { asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(a), "f"(b)); }
  __device__ __forceinline__ explicit f2(float a) : f2(a, a) {}
  __device__ __forceinline__ void get(float& a, float& b) const { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }
};
__device__ __forceinline__ f2 add2(f2 a, f2 b) {
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(a.v) : "l"(a.v), "l"(b.v));
  return a;
}
__device__ __forceinline__ f2 mul2(f2 a, f2 b) {
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(a.v) : "l"(a.v), "l"(b.v));
  return a;
}
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) {
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(a.v) : "l"(a.v), "l"(b.v), "l"(c.v));
  return a;
}
// For two arguments t = -x log2 e: e = 2^t and sigma(x) = 1 / (1 + e), by the hardware's
// exponential and reciprocal (e = inf gives sigma = 0, a NaN passes).  Issued instructions
// bound the gates more than the special-function unit does: with the reciprocal formed by
// Newton steps on the multiply-add pipe, two at a time, d_model 128 took 12.65 ms instead
// of 12.00 at 262,144 tracks of six layers.
__device__ __forceinline__ void sigmoid2(f2 t, f2& e, f2& sg) {
  float t0, t1, d0, d1;
  t.get(t0, t1);
  e = f2(ex2_approx(t0), ex2_approx(t1));
  add2(e, f2(1.0f)).get(d0, d1);
  sg = f2(rcp_approx(d0), rcp_approx(d1));
}
// The smaller of x and y; NaN if x is NaN (fminf would drop it).
__device__ __forceinline__ float min_nan(float x, float y) {
  float m;
  asm("min.NaN.f32 %0, %1, %2;" : "=f"(m) : "f"(x), "f"(y));
  return m;
}

// Operand conversion (round to nearest even): bf16, or fp16 when FP16 is set.
template <bool FP16>
__device__ __forceinline__ uint32_t pack2(float a, float b) {   // a -> low half (lower column)
  if constexpr (FP16) {
    __half2 v = __floats2half2_rn(a, b);
    return *reinterpret_cast<uint32_t*>(&v);
  } else {
    __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<uint32_t*>(&v);
  }
}

// Byte offset, inside an MN-major 128-byte-swizzled operand with 128 columns, of
// the 16-byte chunk that holds columns [8*n8, 8*n8+8) of k-row k.  Atoms are 8
// k-rows x 64 columns (1 KB); the two column atoms of a k-group are adjacent.
__device__ __forceinline__ uint32_t bchunk(int k, int n8) {
  return (uint32_t)((k >> 3) * B_SBO + (n8 >> 3) * B_LBO + (k & 7) * 128 + (((n8 & 7) ^ (k & 7)) << 4));
}

__device__ __forceinline__ void st_shared_v4(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
  asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}

// Write 32 consecutive columns [n0, n0+32) of k-row k (n0 % 32 == 0) as 16-bit operands.
template <bool FP16>
__device__ __forceinline__ void store_row32(uint32_t buf, int k, int n0, const float (&v)[32]) {
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    st_shared_v4(buf + bchunk(k, (n0 >> 3) + c), pack2<FP16>(v[8 * c + 0], v[8 * c + 1]),
                 pack2<FP16>(v[8 * c + 2], v[8 * c + 3]), pack2<FP16>(v[8 * c + 4], v[8 * c + 5]),
                 pack2<FP16>(v[8 * c + 6], v[8 * c + 7]));
  }
}

template <bool FP16>
__device__ __forceinline__ void store_row16(uint32_t buf, int k, int n0, const float (&v)[16]) {
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    st_shared_v4(buf + bchunk(k, (n0 >> 3) + c), pack2<FP16>(v[8 * c + 0], v[8 * c + 1]),
                 pack2<FP16>(v[8 * c + 2], v[8 * c + 3]), pack2<FP16>(v[8 * c + 4], v[8 * c + 5]),
                 pack2<FP16>(v[8 * c + 6], v[8 * c + 7]));
  }
}

// The four epilogue warps of one 32-column segment (one per TMEM quadrant):
// barrier 10 + seg, 128 threads.
__device__ __forceinline__ void seg_sync(int seg) { asm volatile("bar.sync %0, 128;" ::"r"(10 + seg) : "memory"); }

// ------------------------------------------------------------------ epilogue
struct ECtx {
  const TileMeta* md;   // metadata of the tile being processed
  uint32_t xb, hb;      // its activation operands in shared memory
  uint32_t acc, zn, gt; // TMEM columns (with the warp's lane offset): accumulators, z/n, gate and MLP1
  float* xs;            // its residual scratch
  float (*part)[TILE];  // partial column sums of the four quadrants
  float (*carry)[128];  // [slab][channel]: scan states between a slab's column segments
  float* rinv;          // the warp's 32 inverse RMS values
  float* pool;
  float rms_eps;
  // quadrant q (TMEM lanes / channels 32q..), column segment seg = 32-column
  // quarter of the tile (slab half = seg / 2, position in the slab sub = seg % 2)
  int q, lane, seg, half, sub, c, col0, te;
};

// The two epilogue warps that share a quadrant and a slab hand a recurrence state
// from the slab's first 32 columns to the second, or back in the reverse
// direction: barrier 2 + 2q + half, 64 threads, both warps synchronising once
// per hand-over.  (The leading warp must not merely arrive: a warp that could
// arrive twice before its partner synchronises would complete a barrier
// instance on its own and leave the partner's last one unmatched.  In normal
// operation the state-buffer wait keeps the leader within one hand-over, but
// after an expired wait every wait fails fast and that bound is gone; with a
// synchronisation on both sides the two warps pair up whatever the waits do.
// The partner reaches its side before its own scan, so the leader, which
// scans first, seldom waits.)
__device__ __forceinline__ void carry_pass(const ECtx& x) {
  asm volatile("bar.sync %0, 64;" ::"r"(2 + 2 * x.q + x.half) : "memory");
}
__device__ __forceinline__ void carry_wait(const ECtx& x) {
  asm volatile("bar.sync %0, 64;" ::"r"(2 + 2 * x.q + x.half) : "memory");
}

// silu(acc + b) of the 128-channel tile mt, with the half argument from one FMA (the
// rounded sum halved: exact) -> k-rows row0 + c of buf (b: the
// thread's channel's bias, loaded before the wait for the product)
template <bool FP16>
__device__ __forceinline__ void ep_silu_mt(const ECtx& x, float b, int mt, uint32_t buf, int row0) {
  float v[32];
  tmem_ld32(x.gt + mt * 128 + x.col0, v);
  tmem_ld_wait();
  const f2 hb(0.5f * b);
#pragma unroll
  for (int i = 0; i < 32; i += 2) {
    const f2 h = fma2(f2(v[i], v[i + 1]), f2(0.5f), hb);
    float h0, h1;
    h.get(h0, h1);
    fma2(h, f2(tanh_approx(h0), tanh_approx(h1)), h).get(v[i], v[i + 1]);
  }
  store_row32<FP16>(buf, row0 + x.c, x.col0, v);
}
// silu(acc + bias) of the embedding's first product (in the gate columns) -> XB rows [mt*128 + c], all tiles read under one TMEM wait;
// the biases are loaded before the wait for the product (wait_first)
template <bool FP16, int MT, class W>
__device__ __forceinline__ void ep_silu(const ECtx& x, const float* bias, W&& wait_first) {
  float bv[MT];
#pragma unroll
  for (int mt = 0; mt < MT; ++mt) bv[mt] = bias[mt * 128 + x.c];
  wait_first();
  float v[MT][32];
#pragma unroll
  for (int mt = 0; mt < MT; ++mt) tmem_ld32(x.gt + mt * 128 + x.col0, v[mt]);
  tmem_ld_wait();
#pragma unroll
  for (int mt = 0; mt < MT; ++mt) {
    const float b = bv[mt];
#pragma unroll
    for (int i = 0; i < 32; ++i) v[mt][i] = silu(v[mt][i] + b);
    store_row32<FP16>(x.xb, mt * 128 + x.c, x.col0, v[mt]);
  }
}
// X = acc + bias (a layer's accumulator already holds x' plus the MLP2 product).
// X goes to the per-CTA scratch (read back once, by the next layer's gate
// epilogue) and the RMS-normalised x_hat to XB (recomputing X from TMEM); the
// last layer's X is mean-pooled instead (ep_pool).
// Sum of v over the 32 lanes for 16 columns at once: afterwards lane L holds the
// total of column L & 15 (both halves of the warp hold the same 16 totals).
__device__ __forceinline__ float reduce_scatter16(float (&v)[16], int lane) {
#pragma unroll
  for (int off = 8; off >= 1; off >>= 1) {
    const bool upper = (lane & off) != 0;
#pragma unroll
    for (int i = 0; i < off; ++i) {
      const float send = upper ? v[i] : v[i + off];
      const float keep = upper ? v[i + off] : v[i];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, send, off);
    }
  }
  return v[0] + __shfl_xor_sync(0xffffffffu, v[0], 16);
}

template <bool FP16, int MT, class W, class S>
__device__ __forceinline__ void ep_residual(const ECtx& x, const float* bias, const float* gain, W&& wait_tile,
                                              S&& signal_tile) {
  // bias and gain of the thread's channels, loaded before the wait for the
  // first tile's product so that their latency hides behind it
  constexpr int D = 128 * MT;   // d_model
  const uint32_t vm = x.md->m_valid[x.half][x.sub];   // bit i: column col0 + i holds a hit
  // X = acc + bias (the accumulator already holds x' + MLP for a layer, the
  // embedding product for the embedding).  Pad columns are not cleared in X:
  // their x_hat is 0 (their inverse RMS is set to 0), so every product gives
  // them its bias, and their values stay finite and in their own columns (the
  // products and norms are per column, the scans restart at each track's ends,
  // pooling skips them).  The products complete one 128-channel tile at a time,
  // each waited for in turn (wait_tile): tile 0 is summed while tile 1 is still
  // being computed, and x_hat is handed over per tile (signal_tile) so the next
  // products can start on its K rows.  Only the sums of squares stand between
  // the last product and the first hand-over: X goes to the scratch after both
  // hand-overs (each thread later reads back only its own values, and the
  // accumulator columns still hold X until the next layer's first merge, which
  // waits for this thread's scan hand-over).
  float bias_v[MT], gain_v[MT];
#pragma unroll
  for (int mt = 0; mt < MT; ++mt) {
    bias_v[mt] = bias[mt * 128 + x.c];
    gain_v[mt] = gain[mt * 128 + x.c];
  }
  float sq[32];
#pragma unroll
  for (int i = 0; i < 32; ++i) sq[i] = 0.0f;
#pragma unroll
  for (int mt = 0; mt < MT; ++mt) {
    wait_tile();
#pragma unroll
    for (int hh = 0; hh < 2; ++hh) {
      float v[16];
      tmem_ld16(x.acc + mt * 128 + x.col0 + 16 * hh, v);
      tmem_ld_wait();
#pragma unroll
      for (int i = 0; i < 16; i += 2) {
        const f2 val = add2(f2(v[i], v[i + 1]), f2(bias_v[mt]));
        fma2(val, val, f2(sq[16 * hh + i], sq[16 * hh + i + 1])).get(sq[16 * hh + i], sq[16 * hh + i + 1]);
      }
    }
  }
#pragma unroll
  for (int hh = 0; hh < 2; ++hh) {
    float h16[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) h16[i] = sq[16 * hh + i];
    const float t = reduce_scatter16(h16, x.lane);
    if (x.lane < 16) x.part[x.q][x.col0 + 16 * hh + x.lane] = t;
  }
  // the column sums over all channels: the four quadrants' partial sums of this
  // segment's columns; every warp then forms the 32 inverse RMS values itself
  // (the same sum in the same order, so the four copies are identical) in a
  // slice of its own
  seg_sync(x.seg);
  float* rw = x.rinv;
  uint32_t bad;   // columns whose sum is no number: x_hat 0 (see scan_chain_store)
  {
    const int c = x.col0 + x.lane;
    const float t = x.part[0][c] + x.part[1][c] + x.part[2][c] + x.part[3][c];
    rw[x.lane] = ((vm >> x.lane) & 1u) ? 1.0f / sqrtf(t / (float)D + x.rms_eps) : 0.0f;
    bad = __ballot_sync(0xffffffffu, !(t < INFINITY));
  }
  __syncwarp();
#pragma unroll
  for (int mt = 0; mt < MT; ++mt) {
    const float g = gain_v[mt];
#pragma unroll
    for (int hh = 0; hh < 2; ++hh) {
      const int c0 = x.col0 + 16 * hh;
      float v[16], rv[16];
      tmem_ld16(x.acc + mt * 128 + c0, v);
      const float4* rp = reinterpret_cast<const float4*>(rw + 16 * hh);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float4 r4 = rp[i];
        rv[4 * i] = r4.x;
        rv[4 * i + 1] = r4.y;
        rv[4 * i + 2] = r4.z;
        rv[4 * i + 3] = r4.w;
      }
      tmem_ld_wait();
#pragma unroll
      for (int i = 0; i < 16; i += 2)
        mul2(mul2(add2(f2(v[i], v[i + 1]), f2(bias_v[mt])), f2(g)), f2(rv[i], rv[i + 1])).get(v[i], v[i + 1]);
      if (bad) {
#pragma unroll
        for (int i = 0; i < 16; ++i)
          if ((bad >> (16 * hh + i)) & 1u) v[i] = 0.0f;
      }
      store_row16<FP16>(x.xb, mt * 128 + x.c, c0, v);
    }
    signal_tile();   // x_hat of this tile is in XB
  }
  // the residual stream to the scratch (a warp's store: one 128-byte line)
#pragma unroll
  for (int mt = 0; mt < MT; ++mt) {
#pragma unroll
    for (int hh = 0; hh < 2; ++hh) {
      const int c0 = x.col0 + 16 * hh;
      float v[16];
      tmem_ld16(x.acc + mt * 128 + c0, v);
      tmem_ld_wait();
      float* xp = x.xs + (size_t)c0 * D + mt * 128 + x.c;
#pragma unroll
      for (int i = 0; i < 16; ++i) xp[(size_t)i * D] = v[i] + bias_v[mt];
    }
  }
}

// Masked mean pooling of the last layer's output X = acc + bias, only with the tile's
// metadata at hand (its stores are indexed by it).  The warp of
// quadrant q and slab half pools channel tile mt (channels 128 mt + 32 q + lane)
// over all 64 columns of the slab, each track's hits summed in order from its
// first: the two warps of a slab's segments take different channel tiles, or
// different hit tiles.  The column loops stay rolled: this runs once per tile, and its code is cold.
template <int MT>
__device__ __forceinline__ void ep_pool(const ECtx& x, int mt, const float* bias) {
  constexpr int D = 128 * MT;
  const int ch = mt * 128 + x.c;
  const float bv = bias[ch];
  const uint8_t* flags = x.md->col_flags;
  float run = 0.0f;
#pragma unroll 1
  for (int k = 0; k < 4; ++k) {   // 16-column groups of the slab
    const int c0 = SLAB * x.half + 16 * k;
    const uint32_t vm = x.md->m_valid[x.half][k >> 1] >> (16 * (k & 1));
    float v[16];
    tmem_ld16(x.acc + mt * 128 + c0, v);
    tmem_ld_wait();
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const float val = ((vm >> i) & 1u) ? v[i] + bv : 0.0f;
      const int fl = flags[c0 + i];
      run = (fl & F_FIRST) ? val : run + val;
      if (fl & F_LAST) {
        const int s = x.md->col_slot[c0 + i];
        x.pool[(size_t)x.md->slot_track[s] * D + ch] = run / (float)x.md->slot_n[s];
      }
    }
  }
}

// X of the thread's channel in tile mt and its 32 columns, read back from the
// scratch; issued before the wait for the gate's inputs so the loads' latency
// hides behind it.
template <int MT>
__device__ __forceinline__ void gate_x_load(const ECtx& x, int mt, float (&xv)[32]) {
  constexpr int D = 128 * MT;
  const float* xp = x.xs + (size_t)x.col0 * D + mt * 128 + x.c;
#pragma unroll
  for (int i = 0; i < 32; ++i) xv[i] = xp[(size_t)i * D];
}
// x' = X + (M + b_m) * sigma(p_g + b_g) for the 128-channel tile mt -> TMEM columns
// 128 mt.. (in place of the merge accumulator; MLP2 accumulates onto it) and XB
// rows 128 mt + c.
template <bool FP16>
__device__ __forceinline__ void ep_gate(const ECtx& x, int mt, const float (&xv)[32], float bm, float bg) {
  const int ch_g = mt * 128 + x.c;
  const float cg = -bg * LOG2E_F;
#pragma unroll
  for (int hh = 0; hh < 2; ++hh) {
    const int c0 = x.col0 + 16 * hh;
    float mv[16], gv[16];
    tmem_ld16(x.acc + mt * 128 + c0, mv);
    tmem_ld16(x.gt + mt * 128 + c0, gv);
    tmem_ld_wait();
#pragma unroll
    for (int i = 0; i < 16; i += 2) {
      f2 e(0.0f), sg(0.0f);
      sigmoid2(fma2(f2(gv[i], gv[i + 1]), f2(-LOG2E_F), f2(cg)), e, sg);
      fma2(add2(f2(mv[i], mv[i + 1]), f2(bm)), sg, f2(xv[16 * hh + i], xv[16 * hh + i + 1])).get(mv[i], mv[i + 1]);
    }
    tmem_st16(x.acc + mt * 128 + c0, mv);   // x' where MLP2 will accumulate
    store_row16<FP16>(x.xb, ch_g, c0, mv);
  }
  tmem_st_wait();
}

// Scan chunk of one layer.  The chunk holds 64 channels of both directions:
// TMEM lanes 0-63 (quadrants 0, 1) run the forward recurrence over the hits in
// time order, lanes 64-127 (quadrants 2, 3) the reverse one.  Each thread owns a
// 32-column segment; the two segments of a slab run one after the other, the
// leading one handing its final state to the other (carry_pass / carry_wait).  The
// z/n accumulators are first copied to registers (scan_load) so the issuer can
// reuse their TMEM columns for the next chunk while the gates and the recurrence
// run; the states then go to HB.
__device__ __forceinline__ void scan_load(const ECtx& x, float (&z)[32], float (&n)[32]) {
  tmem_ld32(x.zn + x.col0, z);
  tmem_ld32(x.zn + 128 + x.col0, n);
  tmem_ld_wait();
}
// The gates, independent across hits, in the form h_t = a_t h_{t-1} + b_t of the
// linear scan: with s = sigma(z + b_z) = 1 / (1 + e), e = 2^(-(z + b_z) log2 e),
// a = 1 - s = e s (no cancellation as s -> 1) and b = s (n + b_n).  The argument of e is
// held at 126: beyond it the reciprocal would be flushed to zero and a with it, where a
// is 1 (s is 1.2e-38 there instead of less).  Where the recurrence restarts (a track's
// first hit forward, its last in reverse) a = 0.  a replaces z, b replaces n.
__device__ __forceinline__ void scan_gates(const ECtx& x, float (&z)[32], float (&n)[32], float bz, float bn) {
  const uint32_t rm = x.q < 2 ? x.md->m_first[x.half][x.sub] : x.md->m_last[x.half][x.sub];
  const float cz = -bz * LOG2E_F;
#pragma unroll
  for (int j = 0; j < 32; j += 2) {
    f2 e(0.0f), sg(0.0f);
    float t0, t1;
    fma2(f2(z[j], z[j + 1]), f2(-LOG2E_F), f2(cz)).get(t0, t1);
    sigmoid2(f2(min_nan(t0, 126.0f), min_nan(t1, 126.0f)), e, sg);
    mul2(e, sg).get(z[j], z[j + 1]);
    if (rm & (1u << j)) z[j] = 0.0f;
    if (rm & (2u << j)) z[j + 1] = 0.0f;
    mul2(sg, add2(f2(n[j], n[j + 1]), f2(bn))).get(n[j], n[j + 1]);
  }
}
// Eq. 2 per channel over this thread's 32 columns (one FMA per hit on the serial
// path), the states replacing z.  Tracks fill a slab from its first column, so
// padding only trails the last track: the forward state is never read after it,
// and in reverse the last track's end restarts the state (a = 0 there: the
// finite state coming from the padding is multiplied away).  Values left in
// padding columns stay in padding columns (every product and norm is per
// column) and stay finite (their x_hat is 0), so they need no clearing here.
// SELECT: the state after a restart is b itself, so that an infinity or NaN of one
// track stays out of the next (a second, predicated instruction on the serial path).
template <bool SELECT>
__device__ __forceinline__ void scan_chain(const ECtx& x, float (&a)[32], const float (&b)[32]) {
  const bool fwd = x.q < 2;
  const bool leads = fwd ? x.sub == 0 : x.sub == 1;
  float h = 0.0f;
  if (!leads) {
    carry_wait(x);
    h = x.carry[x.half][x.c];
  }
  const uint32_t rm = fwd ? x.md->m_first[x.half][x.sub] : x.md->m_last[x.half][x.sub];
  auto step = [&](int j) {
    if constexpr (SELECT) {
      asm("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %3, 0;\n\t"
          "@!p fma.rn.f32 %0, %1, %0, %2;\n\t@p mov.f32 %0, %2;\n\t}"
          : "+f"(h)
          : "f"(a[j]), "f"(b[j]), "r"(rm & (1u << j)));
    } else {
      h = fmaf(a[j], h, b[j]);
    }
    a[j] = h;
  };
  if (fwd) {
#pragma unroll
    for (int j = 0; j < 32; ++j) step(j);
  } else {
#pragma unroll
    for (int j = 31; j >= 0; --j) step(j);
  }
  if (leads) {
    x.carry[x.half][x.c] = h;
    carry_pass(x);
  }
}
// The gated-merge kernels: a restart is a = 0, one FMA a hit on the serial path.  That
// needs a finite state before it, or an infinity or NaN of one track would reach the next
// in its slab.  So a column whose residual stream is not finite has x_hat 0 (ep_residual) and
// with it finite gates and candidates; the stream itself keeps the column's value, adds to
// it and is pooled, so the track's own result is no number either way.  (x_hat itself is at
// most sqrt(d_model) times the gain, within 16 bits for any gain below 4,000.)  Selecting at
// every restart instead cost 12 % (262,144 tracks of six layers, 12.1 to 13.5 ms).
template <bool FP16>
__device__ __forceinline__ void scan_chain_store(const ECtx& x, float (&a)[32], const float (&b)[32]) {
  scan_chain<false>(x, a, b);
  store_row32<FP16>(x.hb, x.c, x.col0, a);
}

// Test hook: hold a loader's hand-over past the waiters' limit (at most twice the limit, and
// no longer once a wait has given up), so that the epilogue's wait for it expires; the
// metadata itself is complete.
__device__ __forceinline__ void hold_hand_over(volatile int* abort, uint64_t wait_ns) {
  const uint64_t t0 = globaltimer();
  while (!*abort && globaltimer() - t0 < 2 * wait_ns) {
  }
}

// Tile set-up, run one tile ahead by the loader warp while the epilogue warps
// work on the current tile: the column metadata of the tile's two slabs (into
// the metadata buffer md), the features of its hits, and the Fourier operand
// (the B operand of the embedding's first product) as the byte image of HB in
// the CTA's global buffer fb, from which the epilogue copies it at tile start.
// The tile's slabs are s0 and, if there is one before end, s0 + 1.
__device__ __forceinline__ void load_meta(const TileSrc& p, uint8_t* col_tpos, TileMeta* md, int s0, int end, int lane) {
  for (int c = lane; c < TILE; c += 32) md->col_flags[c] = 0;
  __syncwarp();
  int ns = 0;
  for (int hf = 0; hf < 2; ++hf) {
    const int s = s0 + hf;
    if (s >= end) break;
    const int2 sl = p.slab[s];
    const int b0 = sl.x, cnt = sl.y;
    int n = 0, trk = 0;
    if (lane < cnt) {
      trk = p.order[b0 + lane];
      n = p.n_hits[trk];
      if (n < 1 || n > p.T) n = 0;   // rejected by the packer's validity check: no columns
    }
    int incl = n;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    if (lane < cnt) {
      const int slot = ns + lane;
      const int c0 = SLAB * hf + incl - n;
      md->slot_track[slot] = trk;
      md->slot_n[slot] = n;
      for (int t = 0; t < n; ++t) {
        const int col = c0 + t;
        md->col_flags[col] = (uint8_t)(F_VALID | (t == 0 ? F_FIRST : 0) | (t == n - 1 ? F_LAST : 0));
        md->col_slot[col] = (uint8_t)slot;
        if (col_tpos) col_tpos[col] = (uint8_t)t;
      }
    }
    ns += cnt;
  }
  __syncwarp();
  if (lane < 4) {   // column bitmasks
    const int hf = lane >> 1, w = lane & 1;
    uint32_t fm = 0, lm = 0, vm = 0;
    for (int j = 0; j < 32; ++j) {
      const int f = md->col_flags[SLAB * hf + 32 * w + j];
      fm |= (uint32_t)((f & F_FIRST) != 0) << j;
      lm |= (uint32_t)((f & F_LAST) != 0) << j;
      vm |= (uint32_t)((f & F_VALID) != 0) << j;
    }
    md->m_first[hf][w] = fm;
    md->m_last[hf][w] = lm;
    md->m_valid[hf][w] = vm;
  }
  __syncwarp();
}

// The features of the tile's hits.
__device__ __forceinline__ void load_hits(const TileSrc& p, LoaderScratch* m, const TileMeta* md, int lane) {
  for (int idx = lane; idx < TILE * 5; idx += 32) {
    const int col = idx / 5, f = idx - col * 5;
    float v = 0.0f;
    if (md->col_flags[col] & F_VALID) {
      const size_t trk = (size_t)md->slot_track[md->col_slot[col]];
      const size_t row = p.offs ? (size_t)p.offs[trk] + m->col_tpos[col] : trk * p.T + m->col_tpos[col];
      v = p.hits[row * 5 + f];
    }
    m->hs[col][f] = v;
  }
  __syncwarp();
}

// The Fourier operand of the tile's first 8 groups columns, the work items first, first +
// stride, ..: store(k-row, group of 8 columns, 16-byte chunk).
template <bool FP16, class Store>
__device__ __forceinline__ void fourier_operand(const TileSrc& p, const LoaderScratch* m, const TileMeta* md, int groups,
                                                int first, int stride, Store&& store) {
  // u = (v - min) / (max - min) and the argument s_k * u as unevaluated sums of
  // two floats (error-free TwoSum / TwoProduct with fma), reduced modulo 2
  // exactly, so sin(pi s_k u) carries only the final fp32 rounding.
  auto arg = [&](int col, int f, float sk) -> float {
    const float v = m->hs[col][f], mn = -p.feat_min[f];
    const float dh = v + mn;
    const float bv = dh - v;
    const float dl = (v - (dh - bv)) + (mn - bv);
    const float uh = dh * p.feat_inv_hi[f];
    const float ul = fmaf(dh, p.feat_inv_hi[f], -uh) + fmaf(dh, p.feat_inv_lo[f], dl * p.feat_inv_hi[f]);
    const float xh = uh * sk;
    const float xl = fmaf(uh, sk, -xh) + ul * sk;
    return (xh - 2.0f * rintf(0.5f * xh)) + xl;
  };
  auto put = [&](int row, int g, const float (&v)[8]) {
    store(row, g, make_uint4(pack2<FP16>(v[0], v[1]), pack2<FP16>(v[2], v[3]), pack2<FP16>(v[4], v[5]), pack2<FP16>(v[6], v[7])));
  };
  // one work item = 8 columns of one feature and one evaluated scale, stored as
  // 16-byte chunks of the operand.  With s_{k+3} = 2 s_k, sin/cos are evaluated
  // for the scales k = 0-2, 6-8, 12-14 only and the others follow by one step of
  // the double angle identities (2 s c, (c - s)(c + s)), so no value is more than
  // one doubling (a few ulp) from an evaluated one.
  const int n_eval = p.scale_doubling ? 9 : 16;
  for (int it = first; it < groups * 5 * n_eval; it += stride) {
    const int g = it % groups, fk = it / groups, f = fk % 5, bi = fk / 5;
    const int kb = p.scale_doubling ? (bi / 3) * 6 + bi % 3 : bi;
    float sn[8], cs[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int col = 8 * g + j;
      sn[j] = 0.0f;
      cs[j] = 0.0f;
      if (md->col_flags[col] & F_VALID) {
        const float r = arg(col, f, p.scale[kb]);
        sn[j] = sinpif(r);
        cs[j] = cospif(r);
      }
    }
    put(f * 32 + kb, g, sn);
    put(f * 32 + 16 + kb, g, cs);
    if (p.scale_doubling && kb + 3 < 16) {
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const float s2 = 2.0f * sn[j] * cs[j], c2 = (cs[j] - sn[j]) * (cs[j] + sn[j]);
        sn[j] = s2;
        cs[j] = c2;
      }
      put(f * 32 + kb + 3, g, sn);
      put(f * 32 + 16 + kb + 3, g, cs);
    }
  }
}

template <bool FP16>
__device__ __forceinline__ void load_tile(const TileSrc& p, LoaderScratch* m, TileMeta* md, uint8_t* fb, int s0,
                                          int end, int lane) {
  load_meta(p, m->col_tpos, md, s0, end, lane);
  load_hits(p, m, md, lane);
  fourier_operand<FP16>(p, m, md, TILE / 8, lane, 32,
                        [&](int row, int g, uint4 v) { *reinterpret_cast<uint4*>(fb + bchunk(row, g)) = v; });
}

}  // namespace
