// tcgen05 path: one persistent, warp-specialised kernel runs the whole encoder
// forward (embedding, every minGRU layer, pooling) for the 16-bit-operand
// configs; the head (head.cu) then runs on the pooled vectors.
//
// Orientation: every per-hit matrix product is computed transposed,
//   D[channel][hit] = W[channel][k] * Act[k][hit],
// with the weights as the M=128 operand (K-major, TMA-staged from L2/HBM with
// 128-byte swizzle) and the activations of one tile of 128 packed hits as the
// N=128 operand (MN-major, written by the epilogue warps straight into shared
// memory).  The fp32 accumulator lives in tensor memory with lane = channel and
// column = hit, so each epilogue thread owns one channel and walks the hits of
// its tracks in order: the gated scans of Eq. 2 run in registers without any
// cross-thread exchange.
//
// Tile: 128 hit columns = two 64-column slabs; each slab holds whole tracks
// (packed by best fit, unpadded).  Warp roles (608 threads):
//   warp 0       TMA producer of weight blocks (warp-wide loop, one elected lane issues)
//   warp 1       tcgen05.mma issuer (warp-wide loop, one elected lane issues), TMEM owner
//   warps 2..17  epilogue: TMEM lane quadrant = warp % 4, 32-column segment = (warp-2)/4
//   warp 18      loader: column metadata and Fourier operand of the next tile
// TMEM (512 columns): R0,R1 = merge accumulators, then x' with the MLP2 product
// accumulated onto it (d_model rows); R2,R3 = z and n of one scan chunk, then the
// output-gate projection, then MLP1 (and the embedding's first product).
// The fp32 residual stream of the tile lives in a per-CTA global scratch slab
// (L2-resident), never in HBM-sized intermediates.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cudaTypedefs.h>
#include <math.h>

#include <cstring>
#include <new>
#include <vector>

#include "tc_epilogue.cuh"

namespace {

constexpr int A_STAGE = 2 * A_BLOCK;      // a pipeline stage holds two consecutive blocks
constexpr int MAX_SCHED = 1024;           // schedule steps per tile
constexpr int MISC_BYTES = 10240;
constexpr int MAX_STAGES = 8;
constexpr int64_t MAXB = TF_PACK_TRACKS;  // tracks per launch chunk
constexpr int64_t POOL_TRACKS = 1048576;  // tracks per launch chunk when the pooled means go to the internal buffer
constexpr uint64_t WAIT_NS = 2000000000ull;   // bounded-wait limit (a handle's test hook may lower it)
constexpr uint64_t DRAIN_NS = 200000000ull;

enum { MAP_E1 = 0, MAP_E2, MAP_IN, MAP_M, MAP_1, MAP_2, NMAPS };
enum { BSEL_XB = 0, BSEL_HB = 1 };
// Hand-overs around a schedule block: before its first MMA the issuer waits for
// the epilogue's next hand-over on e_bar (W_E; two barriers used alternately) or
// eh_bar (W_H); after its last MMA it commits to acc_bar (C_ACC; two barriers
// used alternately) or hb_bar (C_HB).
enum { W_NONE = 0, W_E = 1, W_H = 2 };
enum { C_NONE = 0, C_ACC = 1, C_HB = 2 };
// A schedule step: two consecutive 64-k blocks of one product (a weight row block and
// K columns col, col + 64), one ring stage at d_model 256.  TAIL: the last 32 k-rows of the
// Fourier operand, a half block each of the step's one (d_model 128) or two 128-channel
// tiles.  prod: map | col/64 << 4 | row << 8; mma: the B operand's offset / 16 in the
// activation buffers | flags << 16, with the accumulator columns / 128 in flags' low bits.
struct Step {
  uint32_t prod, mma;
};
constexpr uint32_t S_COL = 3u << 16, S_ACC = 1u << 18, S_TAIL = 1u << 19, S_W_E = 1u << 20, S_W_H = 1u << 21,
                   S_W_X = 1u << 22, S_C_ACC = 1u << 23, S_C_HB = 1u << 24, S_TILE = 1u << 25;

constexpr int SCHED_BYTES = MAX_SCHED * (int)sizeof(Step);   // the schedule, copied to shared memory

struct TcParams {
  CUtensorMap tm[NMAPS];
  TileSrc src;
  float* pool;   // [B][D] pooled means (the caller's buffer or an internal one)
  float* xs;
  const Step* sched;   // the steps of a tile (d_model 128: then those of two tiles)
  int n_sched, n_sched2;
  const float* b_e1;
  const float* b_e2;
  const float* g;
  const float* b_in;
  const float* b_m;
  const float* b_1;
  const float* b_2;
  unsigned long long* err;
  uint64_t wait_ns;     // limit of every bounded wait
  int hold_tile;        // test hook: CTA 0's loader holds this tile's metadata hand-over (-1: none)
  int D, L, NDC, ROWS_IN, nst;
  uint32_t idesc, idesc_thin;   // N = 128, 64
  int off_xb, off_hb, off_a, off_misc;
  int fp16;
  float rms_eps;
  uint8_t* fbuf;        // per CTA Fourier operands (byte images) written by the loader warp: two for each tile in flight
};

struct Misc {
  uint64_t full[MAX_STAGES], empty[MAX_STAGES];
  uint64_t acc_bar[2], e_bar[2], hb_bar, eh_bar, drain_bar;
  uint64_t meta_full[2], meta_free[2];   // loader -> epilogue, epilogue -> loader
  uint32_t tmem_base;
  int abort_flag;
  TileMeta meta[2];
  LoaderScratch ls;
  alignas(16) float part[4][TILE];
  float carry[2][128];   // [slab][channel]: scan states between a slab's column segments
  alignas(16) float rinv[NE / 32][32];   // per epilogue warp: 1 / RMS of its 32 columns
};
static_assert(sizeof(Misc) <= MISC_BYTES, "misc region too small");

// The static sequence of 128x64 weight blocks of one tile, in the order the MMA
// issuer consumes them, two blocks a step (waits fall on the first of a step, commits on
// the second).  f(map, row, col, nk, tmem_col, bsel, bk, acc, wait, commit):
// nk MMAs of K=16 read the block, accumulate into TMEM columns tmem_col, with
// the activation operand bsel starting at k-row bk; acc = accumulate onto the
// existing accumulator; wait / commit = hand-overs (W_*, C_*).
//
// Within a layer the scan chunks are software-pipelined: as soon as the
// epilogue has copied the z/n accumulators of chunk k into registers, the
// issuer computes z/n of chunk k+1 into the same TMEM columns, and the merge
// product of chunk k follows once its states h(k) are in shared memory.
template <class F>
inline void walk_tile(const TcParams& p, F&& f) {   // d_model 256
  // the embedding's first product goes to the z/n columns, so it can run while
  // the epilogue still pools the previous tile from columns 0..
  for (int mt = 0; mt < 2; ++mt)
    for (int kc = 0; kc < 2; ++kc)
      f(MAP_E1, mt * 128, kc * 64, 4, 256 + mt * 128, BSEL_HB, kc * 64, kc > 0, (mt == 0 && kc == 0) ? W_E : W_NONE,
        C_NONE);
  for (int mt = 0; mt < 2; ++mt)   // its last 32 k-rows
    f(MAP_E1, mt * 128, 128, 2, 256 + mt * 128, BSEL_HB, 128, true, W_NONE, mt == 1 ? C_ACC : C_NONE);
  for (int mt = 0; mt < 2; ++mt)   // committed per 128-channel tile, like MLP2
    for (int kc = 0; kc < 4; ++kc)
      f(MAP_E2, mt * 128, kc * 64, 4, mt * 128, BSEL_XB, kc * 64, kc > 0, (mt == 0 && kc == 0) ? W_E : W_NONE,
        kc == 3 ? C_ACC : C_NONE);
  for (int l = 0; l < p.L; ++l) {
    const int rb = l * p.ROWS_IN;
    auto zn = [&](int k) {   // z and n of scan chunk k -> TMEM columns 256.. and 384..
      for (int kc = 0; kc < 4; ++kc)
        f(MAP_IN, rb + k * 256, kc * 64, 4, 256, BSEL_XB, kc * 64, kc > 0, kc == 0 ? W_E : W_NONE, C_NONE);
      for (int kc = 0; kc < 4; ++kc)
        f(MAP_IN, rb + k * 256 + 128, kc * 64, 4, 384, BSEL_XB, kc * 64, kc > 0, W_NONE, kc == 3 ? C_ACC : C_NONE);
    };
    // x_hat arrives one 128-channel tile at a time (K rows 0-127, then 128-255)
    for (int kh = 0; kh < 2; ++kh) {
      for (int kc = 2 * kh; kc < 2 * kh + 2; ++kc)
        f(MAP_IN, rb, kc * 64, 4, 256, BSEL_XB, kc * 64, kc > 0, kc == 2 * kh ? W_E : W_NONE, C_NONE);
      for (int kc = 2 * kh; kc < 2 * kh + 2; ++kc)
        f(MAP_IN, rb + 128, kc * 64, 4, 384, BSEL_XB, kc * 64, kc > 0, W_NONE, kc == 3 ? C_ACC : C_NONE);
    }
    for (int k = 0; k < p.NDC; ++k) {
      if (k + 1 < p.NDC) {
        zn(k + 1);
      } else {   // output-gate projection into the z/n columns once the last chunk is out
        for (int mt = 0; mt < 2; ++mt)
          for (int kc = 0; kc < 4; ++kc)
            f(MAP_IN, rb + p.NDC * 256 + mt * 128, kc * 64, 4, 256 + mt * 128, BSEL_XB, kc * 64, kc > 0,
              (mt == 0 && kc == 0) ? W_E : W_NONE, C_NONE);
      }
      // merge of chunk k: M[D] += W_m[:, chunk] * h(k).  The last one completes
      // the gate epilogue's inputs one 128-channel tile at a time.
      const bool last = k + 1 == p.NDC;
      for (int mt = 0; mt < 2; ++mt)
        for (int kc = 0; kc < 2; ++kc)
          f(MAP_M, l * p.D + mt * 128, k * 128 + kc * 64, 4, mt * 128, BSEL_HB, kc * 64, k > 0 || kc > 0,
            (mt == 0 && kc == 0) ? W_H : W_NONE, kc == 1 && (last || mt == 1) ? (last ? C_ACC : C_HB) : C_NONE);
    }
    // pipelined by 128-channel tile: MLP1's first K half (x' of tile 0, XB rows
    // 0-127) starts once the gate epilogue of tile 0 is out, the rest once tile 1
    // is; MLP2's K rows 0-127 (SiLU of tile 0) come from HB, rows 128-255 (SiLU of
    // tile 1) from XB.
    const int r1 = l * p.D;
    // MLP1 goes to the z/n columns (free once the gate epilogue of the tile has
    // read them); MLP2 accumulates onto x', which the gate epilogue left in the
    // merge columns
    for (int kc = 0; kc < 4; ++kc)
      f(MAP_1, r1, kc * 64, 4, 256, BSEL_XB, kc * 64, kc > 0, (kc & 1) ? W_NONE : W_E, kc == 3 ? C_ACC : C_NONE);
    for (int kc = 0; kc < 4; ++kc)
      f(MAP_1, r1 + 128, kc * 64, 4, 384, BSEL_XB, kc * 64, kc > 0, W_NONE, kc == 3 ? C_ACC : C_NONE);
    // MLP2: K rows 0-127 (HB) of both output tiles once the SiLU of tile 0 is
    // in, then rows 128-255 (XB), tile 0 first (the residual starts on it)
    for (int kh = 0; kh < 2; ++kh)
      for (int mt = 0; mt < 2; ++mt)
        for (int kc = 2 * kh; kc < 2 * kh + 2; ++kc)
          f(MAP_2, r1 + mt * 128, kc * 64, 4, mt * 128, kh == 0 ? BSEL_HB : BSEL_XB, kc * 64, true,
            (mt == 0 && kc == 2 * kh) ? W_E : W_NONE, kc == 3 ? C_ACC : C_NONE);
  }
}

__device__ __forceinline__ void set_abort(int* flag, unsigned long long* err) {
  if (atomicExch(flag, 1) == 0) atomicAdd(err + 1, 1ull);
}

// Tile start on the epilogue side: the Fourier operand from the CTA's global
// buffer into HB (five 16-byte chunks per thread, all loads in flight at once).
// The loads bypass L1 (ld.global.cg): the buffer is rewritten by the loader warp
// every other tile, and a line of an earlier tile's operand must not be served
// from L1.  The loads (fourier_fetch) can be issued before HB is free; the
// stores (fourier_put) only after.
static_assert(EB_BYTES == 5 * 16 * NE, "one chunk per thread per round");
__device__ __forceinline__ void fourier_fetch(const ECtx& x, const uint8_t* fb, uint4 (&v)[5]) {
#pragma unroll
  for (int r = 0; r < 5; ++r) v[r] = __ldcg(reinterpret_cast<const uint4*>(fb) + r * NE + x.te);
}
__device__ __forceinline__ void fourier_put(const ECtx& x, const uint4 (&v)[5]) {
#pragma unroll
  for (int r = 0; r < 5; ++r) st_shared_v4(x.hb + 16 * (r * NE + x.te), v[r].x, v[r].y, v[r].z, v[r].w);
}

template <bool FP16>
__global__ void __launch_bounds__(NT, 1) tc_forward_kernel(const __grid_constant__ TcParams p) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t* gbase = smem_raw + (base - raw);
  const uint32_t xb = base + p.off_xb, hb = base + p.off_hb, ab = base + p.off_a;
  Misc* m = reinterpret_cast<Misc*>(gbase + p.off_misc);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t full0 = smem_u32(&m->full[0]), empty0 = smem_u32(&m->empty[0]);
  const uint32_t acc_bar0 = smem_u32(&m->acc_bar[0]), acc_bar1 = smem_u32(&m->acc_bar[1]);
  const uint32_t e_bar0 = smem_u32(&m->e_bar[0]), e_bar1 = smem_u32(&m->e_bar[1]);
  const uint32_t hb_bar = smem_u32(&m->hb_bar), eh_bar = smem_u32(&m->eh_bar);
  const uint32_t drain_bar = smem_u32(&m->drain_bar);

  if (threadIdx.x == 0) {
    for (int s = 0; s < p.nst; ++s) {
      mbar_init(full0 + 8 * s, 1);
      mbar_init(empty0 + 8 * s, 1);
    }
    mbar_init(acc_bar0, 1);
    mbar_init(acc_bar1, 1);
    mbar_init(e_bar0, NE / 32);   // one arrival per epilogue warp
    mbar_init(e_bar1, NE / 32);
    mbar_init(hb_bar, 1);
    mbar_init(eh_bar, NE / 32);
    mbar_init(drain_bar, 1);
    for (int b = 0; b < 2; ++b) {
      mbar_init(smem_u32(&m->meta_full[b]), 1);
      mbar_init(smem_u32(&m->meta_free[b]), NE / 32);
    }
    m->abort_flag = 0;
    fence_mbar_init();
  }
  Step* sched_s = reinterpret_cast<Step*>(gbase + p.off_misc + MISC_BYTES);
  for (int i = threadIdx.x; i < p.n_sched; i += blockDim.x) sched_s[i] = p.sched[i];
  if (warp == 1) {
    tmem_alloc(smem_u32(&m->tmem_base), 512);
    tmem_relinquish();
  }
  if (warp == 0 && lane == 0)
    for (int i = 0; i < NMAPS; ++i) prefetch_tmap(&p.tm[i]);
  static_assert(NT == 608 && NE == 512 && SEGW == 32, "warp roles assume 19 warps");
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = m->tmem_base;
  const int n_slabs = *p.src.n_slabs;
  const int n_tiles = (n_slabs + 1) >> 1;
  volatile int* abort = &m->abort_flag;

  // the loader's scratch for the CTA's first tile: XB is free until that tile's embedding
  LoaderScratch* first_hits = reinterpret_cast<LoaderScratch*>(gbase + p.off_xb);

  if (warp == 0) {
    // TMA producer: a step's two 16 KB weight blocks per stage, in schedule order.  The
    // whole warp walks the schedule and waits; one lane's copies are let through by a
    // predicate (see the issuer).
    uint32_t stage = 0, phase = 0;
    const uint32_t me = elect_one() ? 1u : 0u;
    bool ok = true;
    int issued = 0;
    for (int t = blockIdx.x; t < n_tiles && ok; t += gridDim.x) {
      for (int i = 0; i < p.n_sched; ++i) {
        const Step e = sched_s[i];
        const CUtensorMap* map = &p.tm[e.prod & 15u];
        const int c0 = (int)((e.prod >> 4) & 15u) * 64, c1 = (int)(e.prod >> 8);
        const bool tail = e.mma & S_TAIL;
        const uint32_t full = full0 + 8 * stage, dst = ab + stage * A_STAGE;
        if (!mbar_wait(empty0 + 8 * stage, phase ^ 1u, abort, p.wait_ns)) {
          set_abort(&m->abort_flag, p.err);
          ok = false;
        }
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        mbar_arrive_expect_tx_if(full, A_STAGE, me);
        tma_load_2d_if(dst, map, full, c0, c1, me);
        tma_load_2d_if(dst + A_BLOCK, map, full, tail ? c0 : c0 + 64, tail ? c1 + 128 : c1, me);
        ++issued;
        if (++stage == (uint32_t)p.nst) {
          stage = 0;
          phase ^= 1u;
        }
      }
    }
    __syncwarp();
    if (*abort) {
      // let the copies already issued land before the CTA can exit
      volatile int never = 0;
      for (int k = 0; k < p.nst && k < issued; ++k) {
        const int i = issued - 1 - k;
        mbar_wait(full0 + 8 * (i % p.nst), (uint32_t)((i / p.nst) & 1), &never, DRAIN_NS);
      }
    }
  } else if (warp == 1) {
    // MMA issuer.  It must hand the tensor pipe 8 products every 512 cycles while five
    // warps share its scheduler, so its own instructions count: with a branch around an
    // elected lane, a vote after each wait and a block a time it took 755 cycles for 4
    // products beside busy warps (N = 64 products took as long as N = 128).  So the whole
    // warp runs one straight line a step, the instructions of all lanes but one are
    // switched off by a predicate, and the next step's entry is loaded ahead: 314
    // cycles for 4.  Every lane waits for itself, so the lanes vote once a step: one left
    // behind by the length of the ring would test a parity two phases old (the vote takes
    // 0.5 to 1 %; one lane alone for the whole loop took 3.47 ms instead of 3.26 for 20,011
    // tracks).
    uint32_t stage = 0, phase = 0, e_k = 0, h_k = 0, a_k = 0;
    const uint32_t me = elect_one() ? 1u : 0u;
    bool ok = true;
    const uint64_t a_desc = sdesc_sw128(ab, 16, 1024), b_desc = sdesc_sw128(base, B_LBO, B_SBO);
    const uint32_t a_lo0 = desc_lo(a_desc), a_hi = desc_hi(a_desc), b_lo0 = desc_lo(b_desc), b_hi = desc_hi(b_desc);
    constexpr uint32_t BSTEP = (2 * B_SBO) >> 4;
    const uint32_t idesc = p.idesc;
    auto wait_bar = [&](uint32_t bar, uint32_t parity) {
      if (!mbar_wait(bar, parity, abort, p.wait_ns)) {
        set_abort(&m->abort_flag, p.err);
        ok = false;
      }
    };
    for (int t = blockIdx.x; t < n_tiles && ok; t += gridDim.x) {
      uint32_t e = sched_s[0].mma;
      for (int i = 0; i < p.n_sched; ++i) {
        const uint32_t en = sched_s[i + 1 < p.n_sched ? i + 1 : 0].mma;
        if (e & S_W_E) {   // the k-th W_E hand-over arrives on e_bar[k % 2]
          wait_bar(e_bar0 + 8 * (e_k & 1u), (e_k >> 1) & 1u);
          ++e_k;
        } else if (e & S_W_H) {
          wait_bar(eh_bar, h_k & 1u);
          ++h_k;
        }
        wait_bar(full0 + 8 * stage, phase);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        tc_fence_after();
        const uint32_t a_lo = a_lo0 + stage * (A_STAGE >> 4), b_lo = b_lo0 + (e & 0xFFFFu);
        const uint32_t d = tmem + ((e & S_COL) >> 16) * 128u;
        if (!(e & S_TAIL)) {
          umma4_f16_if<BSTEP>(d, a_lo, a_hi, b_lo, b_hi, idesc, e & S_ACC, me);
          umma4_f16_if<BSTEP>(d, a_lo + (A_BLOCK >> 4), a_hi, b_lo + 4 * BSTEP, b_hi, idesc, 1u, me);
        } else {
          umma2_f16_if<BSTEP>(d, a_lo, a_hi, b_lo, b_hi, idesc, 1u, me);
          umma2_f16_if<BSTEP>(d + 128u, a_lo + (A_BLOCK >> 4), a_hi, b_lo, b_hi, idesc, 1u, me);
        }
        umma_commit_if(empty0 + 8 * stage, me);
        // The k-th accumulator commit goes to acc_bar[k % 2] (some commits come in
        // pairs with no epilogue hand-over between them; see the epilogue).
        if (e & S_C_ACC) {
          umma_commit_if(acc_bar0 + 8 * (a_k & 1u), me);
          ++a_k;
        } else if (e & S_C_HB) {
          umma_commit_if(hb_bar, me);
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
  } else if (warp < 2 + NE / 32) {
    ECtx x;
    x.xb = xb;
    x.hb = hb;
    x.q = warp & 3;
    x.seg = (warp - 2) >> 2;
    x.half = x.seg >> 1;
    x.sub = x.seg & 1;
    x.lane = lane;
    x.c = 32 * x.q + lane;
    x.col0 = SEGW * x.seg;
    x.te = threadIdx.x - 64;
    x.acc = tmem + ((uint32_t)(32 * x.q) << 16);
    x.zn = x.gt = x.acc + 256;
    x.xs = p.xs + (size_t)blockIdx.x * TILE * p.D;
    x.part = m->part;
    x.carry = m->carry;
    x.rinv = m->rinv[warp - 2];
    x.pool = p.pool;
    x.rms_eps = p.rms_eps;
    uint32_t acc_ph0 = 0, acc_ph1 = 0, hb_phase = 0;
    // The epilogue warps run decoupled: each makes its shared-memory operand
    // writes visible to the async proxy, orders its TMEM reads and arrives on the
    // hand-over barrier itself (e_bar and eh_bar count one arrival per warp), and
    // each polls the MMA commits itself.  Some consecutive hand-overs do not wait
    // for the issuer in between (gate tile 0 then 1, SiLU 0 then 1, x_hat 0 then
    // 1), so a warp can arrive for the next one before a slower warp has arrived
    // for the current one; on a single counting barrier that arrival would
    // complete the current phase early.  The W_E hand-overs therefore alternate
    // between two barriers: a warp is never more than one hand-over ahead of
    // another (the one after a pair waits for a product that needs both).  The
    // accumulator commits come in such pairs too (the last merge's two channel
    // tiles, MLP1's, MLP2's, the embedding's second product): a warp that starts
    // its wait for the first of a pair after the second has landed would see the
    // phase parity flipped twice, so they alternate between two barriers as
    // well (a warp is never two commits behind: the issuer makes commit k + 2
    // only after a hand-over that every warp gives after its wait for commit k).
    // A failed wait sets the abort flag and every later wait fails fast, but no
    // warp leaves the loop early: all warps keep taking the same sequence of named
    // barriers (the column-norm exchanges, the segment hand-overs), so none of
    // them can be left waiting.  `alive` (the same for a warp's lanes): every wait of
    // this warp has succeeded.  Only then is the metadata of its tile complete and kept
    // until the warp releases it (the loader stops at the first failure), so only then may
    // an address be formed from it.
    bool alive = true;
    auto signal_to = [&](uint32_t bar, bool wrote_operands) {
      if (wrote_operands) fence_proxy_async_smem();   // costly: only after operand writes
      tc_fence_before();
      __syncwarp();
      if (x.lane == 0) mbar_arrive(bar);
    };
    uint32_t e_k = 0;   // W_E hand-overs so far: the next goes to e_bar[e_k % 2]
    auto signal_e = [&](bool wrote_operands) {
      signal_to((e_k & 1u) ? e_bar1 : e_bar0, wrote_operands);
      ++e_k;
    };
    auto signal = [&]() { signal_e(true); };
    auto wait_on = [&](uint32_t bar, uint32_t& ph) {
      const bool got = mbar_wait(bar, ph, abort, p.wait_ns);   // try_wait: suspends instead of polling
      if (!__all_sync(0xffffffffu, got)) {
        if (x.lane == 0) set_abort(&m->abort_flag, p.err);
        alive = false;
      }
      ph ^= 1u;
      tc_fence_after();
    };
    uint32_t acc_k = 0;   // accumulator commits waited for so far: the next is on acc_bar[acc_k % 2]
    auto wait_acc = [&]() {
      if (acc_k & 1u)
        wait_on(acc_bar1, acc_ph1);
      else
        wait_on(acc_bar0, acc_ph0);
      ++acc_k;
    };
    const uint8_t* fbuf = p.fbuf + (size_t)blockIdx.x * 2 * EB_BYTES;
    uint32_t meta_ph[2] = {0u, 0u};
    // tile start: the loader's metadata and Fourier operand of the CTA's i-th tile
    // the loads wait for the loader's hand-over of tile i; the stores, after
    // which the operand is handed to the issuer, need HB free
    auto tile_fetch = [&](int i, uint4 (&v)[5]) {
      const int b = i & 1;
      wait_on(smem_u32(&m->meta_full[b]), meta_ph[b]);
      fourier_fetch(x, fbuf + b * EB_BYTES, v);
    };
    auto tile_put = [&](const uint4 (&v)[5]) {
      fourier_put(x, v);
      signal();
    };
    // The CTA's first tile: nothing runs yet that could hide its operand, so the epilogue
    // warps form it themselves instead of the loader warp alone (20,011 tracks 3.29 -> 3.26 ms)
    if ((int)blockIdx.x < n_tiles) {
      wait_on(smem_u32(&m->meta_full[0]), meta_ph[0]);
      fourier_operand<FP16>(p.src, first_hits, &m->meta[0], TILE / 8, x.te, NE, [&](int row, int g, uint4 v) {
        st_shared_v4(hb + bchunk(row, g), v.x, v.y, v.z, v.w);
      });
      signal();
    }
    int i = 0;
    for (int t = blockIdx.x; t < n_tiles; t += gridDim.x, ++i) {
      x.md = &m->meta[i & 1];
      ep_silu<FP16, 2>(x, p.b_e1, wait_acc);
      signal();
      ep_residual<FP16, 2>(x, p.b_e2, p.g, wait_acc, signal);   // embedding output X0
      for (int l = 0; l < p.L; ++l) {
        for (int dc = 0; dc < p.NDC; ++dc) {
          // biases are loaded before the wait so their latency hides behind it
          const size_t rb = (size_t)l * p.ROWS_IN + dc * 256;
          const float bz = p.b_in[rb + x.c], bn = p.b_in[rb + 128 + x.c];
          wait_acc();
          float z[32], n[32];
          scan_load(x, z, n);
          signal_e(false);   // the z/n columns are free for the next chunk
          scan_gates(x, z, n, bz, bn);
          // HB still feeds the merge of the previous chunk (the gate hand-over
          // covers the last merge of the previous layer)
          if (dc > 0) wait_on(hb_bar, hb_phase);
          scan_chain_store<FP16>(x, z, n);
          signal_to(eh_bar, true);
        }
        // gate and MLP1 epilogues one 128-channel tile at a time (the issuer
        // pipelines the next tile's products behind each); the
        // SiLU of tile 0 goes to HB (MLP1 still reads XB rows 0-127 then)
        // the biases of the thread's channels are loaded ahead of the waits
        const float* b1 = p.b_1 + (size_t)l * p.D;
        const float* bmp = p.b_m + (size_t)l * p.D;
        const float* bgp = p.b_in + (size_t)l * p.ROWS_IN + p.NDC * 256;
        const float bm0 = bmp[x.c], bg0 = bgp[x.c], b10 = b1[x.c];
        float xg[32];
        gate_x_load<2>(x, 0, xg);
        wait_acc();
        ep_gate<FP16>(x, 0, xg, bm0, bg0);
        signal();
        const float bm1 = bmp[128 + x.c], bg1 = bgp[128 + x.c], b11 = b1[128 + x.c];
        gate_x_load<2>(x, 1, xg);
        wait_acc();
        ep_gate<FP16>(x, 1, xg, bm1, bg1);
        signal();
        wait_acc();
        ep_silu_mt<FP16>(x, b10, 0, x.hb, 0);
        signal();
        wait_acc();
        ep_silu_mt<FP16>(x, b11, 1, x.xb, 128);
        signal();
        if (l + 1 < p.L) {
          ep_residual<FP16, 2>(x, p.b_2 + (size_t)l * p.D, p.g + (size_t)(l + 1) * p.D, wait_acc, signal);
        } else {
          // once both output tiles of the last MLP2 have completed, HB and XB
          // are free: the next tile's Fourier operand (fetched before the
          // waits) goes in and its first product (into the z/n columns) runs
          // while this tile is pooled
          const bool more = t + (int)gridDim.x < n_tiles;
          uint4 fv[5];
          if (more) tile_fetch(i + 1, fv);
          wait_acc();
          wait_acc();
          if (more) tile_put(fv);
          if (alive) ep_pool<2>(x, x.sub, p.b_2 + (size_t)l * p.D);
          signal_to(smem_u32(&m->meta_free[i & 1]), false);   // this tile's metadata is no longer read
        }
      }
    }
  } else {
    // loader warp: tile set-up one tile ahead of the epilogue
    uint8_t* fbuf = p.fbuf + (size_t)blockIdx.x * 2 * EB_BYTES;
    uint32_t free_ph[2] = {0u, 0u};
    int i = 0;
    for (int t = blockIdx.x; t < n_tiles; t += gridDim.x, ++i) {
      const int b = i & 1;
      if (i >= 2) {   // buffer b last held the metadata of tile i - 2
        const bool got = mbar_wait(smem_u32(&m->meta_free[b]), free_ph[b], abort, p.wait_ns);
        if (!__all_sync(0xffffffffu, got) && lane == 0) set_abort(&m->abort_flag, p.err);
        // after a failure anywhere a release may have come from a warp that gave up: stop, so
        // that the metadata others still read stays as it is
        if (!__all_sync(0xffffffffu, got && !*abort)) break;
        free_ph[b] ^= 1u;
      }
      if (i == 0) {
        load_meta(p.src, first_hits->col_tpos, &m->meta[b], 2 * t, n_slabs, lane);
        load_hits(p.src, first_hits, &m->meta[b], lane);
      } else {
        load_tile<FP16>(p.src, &m->ls, &m->meta[b], fbuf + b * EB_BYTES, 2 * t, n_slabs, lane);
      }
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

#include "tc_pair.cuh"

// ------------------------------------------------------------------ UMMA probe
// D[128][128] = A[128][K] * B[K][128] through the same TMA / descriptor / TMEM
// path as the fused kernel (test hook for the operand layouts).
__global__ void __launch_bounds__(128, 1) umma_probe_kernel(const __grid_constant__ CUtensorMap tmA,
                                                            const uint16_t* __restrict__ Bkn, int K,
                                                            float* __restrict__ Dout, uint32_t idesc,
                                                            unsigned long long* err) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t* gbase = smem_raw + (base - raw);
  const uint32_t a_s = base;                 // K/64 blocks of 16 KB
  const uint32_t b_s = base + (K / 64) * A_BLOCK;
  uint64_t* bars = reinterpret_cast<uint64_t*>(gbase + (K / 64) * A_BLOCK + K * 256);
  uint32_t* tbase = reinterpret_cast<uint32_t*>(bars + 2);
  int* abortp = reinterpret_cast<int*>(bars + 3);
  const uint32_t tma_bar = smem_u32(&bars[0]), mma_bar = smem_u32(&bars[1]);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    mbar_init(tma_bar, 1);
    mbar_init(mma_bar, 1);
    *abortp = 0;
    fence_mbar_init();
  }
  if (warp == 0) {
    tmem_alloc(smem_u32(tbase), 128);
    tmem_relinquish();
  }
  // B operand written by the threads, exactly as the epilogue does
  for (int idx = threadIdx.x; idx < K * 16; idx += 128) {
    const int k = idx >> 4, n8 = idx & 15;
    const uint16_t* src = Bkn + (size_t)k * 128 + n8 * 8;
    uint32_t w[4];
    for (int i = 0; i < 4; ++i) w[i] = (uint32_t)src[2 * i] | ((uint32_t)src[2 * i + 1] << 16);
    st_shared_v4(b_s + bchunk(k, n8), w[0], w[1], w[2], w[3]);
  }
  fence_proxy_async_smem();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tbase;
  volatile int* abort = abortp;
  bool ok = true;
  if (threadIdx.x == 0) {
    mbar_arrive_expect_tx(tma_bar, (K / 64) * A_BLOCK);
    for (int kc = 0; kc < K / 64; ++kc) tma_load_2d(a_s + kc * A_BLOCK, &tmA, tma_bar, kc * 64, 0);
    ok = mbar_wait(tma_bar, 0, abort, WAIT_NS);
    if (ok) {
      tc_fence_after();
      for (int kc = 0; kc < K / 64; ++kc)
        for (int k = 0; k < 4; ++k) {
          const uint64_t ad = sdesc_sw128(a_s + kc * A_BLOCK + 32 * k, 16, 1024);
          const uint64_t bd = sdesc_sw128(b_s + ((kc * 64 + 16 * k) >> 3) * B_SBO, B_LBO, B_SBO);
          umma_f16(tmem, ad, bd, idesc, (kc || k) ? 1u : 0u);
        }
      umma_commit(mma_bar);
    } else {
      atomicAdd(err + 1, 1ull);
      *abortp = 1;
    }
  }
  __syncthreads();
  if (!*abort) {
    if (mbar_wait(mma_bar, 0, abort, WAIT_NS)) {
      tc_fence_after();
      const uint32_t tq = tmem + ((uint32_t)(32 * warp) << 16);
      for (int ch = 0; ch < 4; ++ch) {
        float v[32];
        tmem_ld32(tq + 32 * ch, v);
        tmem_ld_wait();
        for (int i = 0; i < 32; ++i) Dout[(size_t)(32 * warp + lane) * 128 + 32 * ch + i] = v[i];
      }
    } else if (lane == 0) {
      atomicAdd(err + 1, 1ull);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc(tmem, 128);
  }
}

// ------------------------------------------------------------------ host side
uint16_t fp16_bits(float f) {
  const __half v = __float2half_rn(f);
  return *reinterpret_cast<const uint16_t*>(&v);
}
uint16_t bf16_bits(float f) {
  uint32_t u;
  std::memcpy(&u, &f, 4);
  if ((u & 0x7f800000u) == 0x7f800000u && (u & 0x007fffffu)) return 0x7fc0;
  u += 0x7fffu + ((u >> 16) & 1u);
  return (uint16_t)(u >> 16);
}

PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  }
  return fn;
}

// bf16 matrix [rows][cols] row-major -> tensor map with 64 x 128 boxes, 128 B swizzle.
bool make_map(CUtensorMap* m, const void* ptr, uint64_t rows, uint64_t cols, bool fp16 = false) {
  auto fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[2] = {cols, rows};
  cuuint64_t strides[1] = {cols * 2};
  cuuint32_t box[2] = {64, 128};
  cuuint32_t es[2] = {1, 1};
  return fn(m, fp16 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(ptr), dims, strides, box, es,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

struct tf_tc_state {
  int nsm = 0, nst = 0, NDC = 0, ROWS_IN = 0, KM = 0;
  size_t smem = 0;
  int off_xb = 0, off_hb = 0, off_a = 0, off_misc = 0;
  uint32_t idesc = 0, idesc_thin = 0;
  void* dev = nullptr;  // one allocation for all weights
  uint16_t *w_e1 = nullptr, *w_e2 = nullptr, *w_in = nullptr, *w_m = nullptr, *w_1 = nullptr, *w_2 = nullptr;
  float *b_e1 = nullptr, *b_e2 = nullptr, *g = nullptr, *b_in = nullptr, *b_m = nullptr, *b_1 = nullptr,
        *b_2 = nullptr;
  void* pack = nullptr;   // packing buffers for MAXB tracks
  Step* sched = nullptr;   // steps of one tile, then (d_model 128) of two
  int n_sched = 0, n_sched2 = 0;
  float* xs = nullptr;
  uint8_t* fbuf = nullptr;
  float* pool = nullptr;   // pooled means when the caller passes no buffer [POOL_TRACKS][D]
  uint64_t wait_ns = WAIT_NS;   // test hook (trackfit_debug_wait_limit)
  int hold_tile = -1;
  CUtensorMap tm[NMAPS];
};

// Steps of a tile at d_model 128: the embedding's 2 + 1, a layer's products.
static int pair_steps(int L, int NDC) { return 3 + L * (3 * NDC + 3); }

// The steps of one tile (nt = 1) or of two in turn (d_model 128, nt = 2): walk_tile's or
// walk_pair's blocks, two at a time.
static std::vector<Step> build_schedule(int D, int L, int NDC, int ROWS_IN, int nt) {
  std::vector<Step> out;
  bool second = false;
  auto put = [&](int u, int map, int row, int col, int nk, int tcol, int bsel, int bk, int acc, int wait, int commit) {
    const uint32_t commits = (commit == C_ACC ? S_C_ACC : 0u) | (commit == C_HB ? S_C_HB : 0u);
    if (!second) {
      const int off = D == 128 ? u * P_TILE + (bsel == BSEL_HB ? P_HB : P_XB) : (bsel == BSEL_HB ? D * 256 : 0);
      out.push_back({(uint32_t)map | ((uint32_t)(col >> 6) << 4) | ((uint32_t)row << 8),
                     (uint32_t)((off + (bk >> 3) * B_SBO) >> 4) | ((uint32_t)(tcol >> 7) << 16) | (acc ? S_ACC : 0u) |
                         (nk == 2 ? S_TAIL : 0u) | ((wait & W_E) ? S_W_E : 0u) | ((wait & W_H) ? S_W_H : 0u) |
                         ((wait & W_X) ? S_W_X : 0u) | (u ? S_TILE : 0u)});
    }
    out.back().mma |= commits;
    second = !second && !(D == 128 && nk == 2);   // d_model 128: the tail is a step of one block
  };
  if (D == 128) {
    walk_pair(L, NDC, ROWS_IN, nt, put);
  } else {
    TcParams q;
    std::memset(&q, 0, sizeof(q));
    q.D = D;
    q.L = L;
    q.NDC = NDC;
    q.ROWS_IN = ROWS_IN;
    walk_tile(q, [&](int map, int row, int col, int nk, int tcol, int bsel, int bk, int acc, int wait, int commit) {
      put(0, map, row, col, nk, tcol, bsel, bk, acc, wait, commit);
    });
  }
  return out;
}

struct ScheduleCounter {   // a callable for walk_tile and walk_pair on either side
  int64_t c[6] = {0, 0, 0, 0, 0, 0};
  uint8_t* codes = nullptr;   // optional: per block wait | commit << 2, in order
  int64_t cap = 0;
  bool two = false;           // two tiles in turn: wait | commit << 3 | tile << 5
  void operator()(int u, int, int, int, int nk, int, int, int, int, int wait, int commit) {
    if (c[0] < cap) codes[c[0]] = (uint8_t)(two ? wait | (commit << 3) | (u << 5) : wait | (commit << 2));
    ++c[0];
    c[1] += nk;
    c[2] += ((wait & W_E) != 0) + ((wait & W_X) != 0);
    c[3] += (wait & W_H) != 0;
    c[4] += commit == C_ACC;
    c[5] += commit == C_HB;
  }
  void operator()(int map, int row, int col, int nk, int tcol, int bsel, int bk, int acc, int wait, int commit) {
    (*this)(0, map, row, col, nk, tcol, bsel, bk, acc, wait, commit);
  }
};

// Totals of the fused kernel's block schedules, from the walks the kernel's steps are made
// from (host only, no device needed): counts[0] blocks, [1] MMA instructions (128 x 128 x 16
// each), [2] W_E and [3] W_H hand-over waits, [4] C_ACC and [5] C_HB commits of a tile by
// itself; with n >= 12, [6..11] the same of two tiles in turn (d_model 128, else 0).  With
// codes, also each block's waits and commit in issue order (at most cap blocks): the lone
// tile's, then, with n >= 12, the two tiles'.
int tf_tc_schedule_counts(const tf_shape& s, int64_t* counts, int n, uint8_t* codes, int64_t cap) {
  if (n < 6 || (cap > 0 && !codes)) return TRACKFIT_ERR_INVALID_ARG;
  TcParams q;
  memset(&q, 0, sizeof(q));
  q.D = s.D;
  q.L = s.L;
  q.NDC = s.H / 64;
  q.ROWS_IN = q.NDC * 256 + s.D;
  ScheduleCounter c, c2;
  c.codes = codes;
  c.cap = cap;
  if (s.D == 128)
    walk_pair(q.L, q.NDC, q.ROWS_IN, 1, c);
  else
    walk_tile(q, c);
  for (int i = 0; i < 6; ++i) counts[i] = c.c[i];
  if (n < 12) return TRACKFIT_OK;
  c2.two = true;
  if (cap > c.c[0]) {
    c2.codes = codes + c.c[0];
    c2.cap = cap - c.c[0];
  }
  if (s.D == 128) walk_pair(q.L, q.NDC, q.ROWS_IN, 2, c2);
  for (int i = 0; i < 6; ++i) counts[6 + i] = c2.c[i];
  return TRACKFIT_OK;
}

int tf_tc_wait_limit(trackfit_ctx* h, int64_t limit_ns, int hold_tile) {
  if (!h->tc) return TRACKFIT_ERR_UNSUPPORTED;
  if (limit_ns < 0 || hold_tile < -1) return TRACKFIT_ERR_INVALID_ARG;
  h->tc->wait_ns = limit_ns > 0 ? (uint64_t)limit_ns : WAIT_NS;
  h->tc->hold_tile = hold_tile;
  return TRACKFIT_OK;
}

bool tf_tc_supported(const tf_shape& s) {
  return (s.precision == TRACKFIT_BF16_PROJ || s.precision == TRACKFIT_FP16_PROJ) && s.pool == TRACKFIT_POOL_MEAN &&
         s.topology == TRACKFIT_TOPOLOGY_MERGE && (s.D == 128 || s.D == 256) &&
         s.H % 64 == 0 && s.T <= 64 && s.Hh == 128 && s.Q <= 75 && s.F == 5 && s.K == 16;
}

void tf_tc_destroy(trackfit_ctx* h) {
  if (!h || !h->tc) return;
  tf_tc_state* t = h->tc;
  tf_free(t->dev);
  tf_free(t->pack);
  tf_free(t->xs);
  tf_free(t->fbuf);
  tf_free(t->pool);
  tf_free(t->sched);
  delete t;
  h->tc = nullptr;
}

int tf_tc_create(trackfit_ctx* h, const float* W) {
  const tf_shape& s = h->s;
  const tf_blob_off& o = h->off;
  tf_tc_state* t = new (std::nothrow) tf_tc_state();
  if (!t) return TRACKFIT_ERR_OOM;
  h->tc = t;
  const int D = s.D, H = s.H, L = s.L, E = s.E;
  t->NDC = H / 64;
  t->ROWS_IN = t->NDC * 256 + D;
  t->KM = t->NDC * 128;
  const bool fp16 = s.precision == TRACKFIT_FP16_PROJ;
  t->idesc = idesc_f16(128, 128, fp16 ? 0u : 1u, false, true);
  t->idesc_thin = idesc_f16(128, 64, fp16 ? 0u : 1u, false, true);
  int dev = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&t->nsm, cudaDevAttrMultiProcessorCount, dev);
  int smem_optin = 0;
  cudaDeviceGetAttribute(&smem_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (D == 128) {   // two tiles in turn (tc_pair.cuh)
    const int rest = (int)sizeof(PairMisc) + 3 * pair_steps(L, t->NDC) * (int)sizeof(Step);   // one tile's and two tiles'
    t->nst = (smem_optin - 1024 - rest - P_A) / A_BLOCK;
    if (t->nst > MAX_STAGES) t->nst = MAX_STAGES;
    if (t->nst < 3) return TRACKFIT_ERR_UNSUPPORTED;
    t->off_misc = P_A + t->nst * A_BLOCK;
    t->smem = (size_t)t->off_misc + rest + 1024;
  } else {
    t->off_xb = 0;
    t->off_hb = D * 256;
    t->off_a = t->off_hb + EB_BYTES;
    const int avail = smem_optin - 1024 - MISC_BYTES - SCHED_BYTES - t->off_a;
    t->nst = avail / A_STAGE;
    if (t->nst > MAX_STAGES) t->nst = MAX_STAGES;
    if (t->nst < 2) return TRACKFIT_ERR_UNSUPPORTED;
    t->off_misc = t->off_a + t->nst * A_STAGE;
    t->smem = (size_t)t->off_misc + MISC_BYTES + SCHED_BYTES + 1024;
  }
  // ---- repack weights (bf16 GEMM operands, fp32 biases/head)
  const size_t n_e1 = (size_t)D * E, n_e2 = (size_t)D * D, n_in = (size_t)L * t->ROWS_IN * D,
               n_m = (size_t)L * D * t->KM, n_11 = (size_t)L * D * D;
  std::vector<uint16_t> we1(n_e1), we2(n_e2), win(n_in, 0), wm(n_m, 0), w1(n_11), w2(n_11);
  std::vector<float> bin((size_t)L * t->ROWS_IN, 0.0f), gg((size_t)L * D), bm((size_t)L * D), b1((size_t)L * D),
      b2((size_t)L * D);
  uint16_t (*cv)(float) = fp16 ? fp16_bits : bf16_bits;
  for (size_t i = 0; i < n_e1; ++i) we1[i] = cv(W[o.emb_w1 + i]);
  for (size_t i = 0; i < n_e2; ++i) we2[i] = cv(W[o.emb_w2 + i]);
  for (int l = 0; l < L; ++l) {
    const tf_layer_off& lo = o.layer[l];
    const size_t rb = (size_t)l * t->ROWS_IN;
    // scan chunk dc = 64 channels of both directions: rows 0-63 forward,
    // rows 64-127 reverse (z block, then n block); the merge columns follow
    for (int dc = 0; dc < t->NDC; ++dc) {
      for (int c = 0; c < 128; ++c) {
        const int dir = c >> 6, ch = dc * 64 + (c & 63);
        const int src_z = (dir == 0 ? 0 : 2 * H) + ch, src_n = (dir == 0 ? H : 3 * H) + ch;
        for (int k = 0; k < D; ++k) {
          win[(rb + dc * 256 + c) * D + k] = cv(W[lo.w_in + (size_t)src_z * D + k]);
          win[(rb + dc * 256 + 128 + c) * D + k] = cv(W[lo.w_in + (size_t)src_n * D + k]);
        }
        bin[rb + dc * 256 + c] = W[lo.b_in + src_z];
        bin[rb + dc * 256 + 128 + c] = W[lo.b_in + src_n];
        for (int r = 0; r < D; ++r)
          wm[((size_t)l * D + r) * t->KM + dc * 128 + c] = cv(W[lo.w_m + (size_t)r * 2 * H + dir * H + ch]);
      }
    }
    for (int c = 0; c < D; ++c) {
      for (int k = 0; k < D; ++k)
        win[(rb + t->NDC * 256 + c) * D + k] = cv(W[lo.w_in + (size_t)(4 * H + c) * D + k]);
      bin[rb + t->NDC * 256 + c] = W[lo.b_in + 4 * H + c];
    }
    for (size_t i = 0; i < (size_t)D * D; ++i) {
      w1[(size_t)l * D * D + i] = cv(W[lo.w1 + i]);
      w2[(size_t)l * D * D + i] = cv(W[lo.w2 + i]);
    }
    for (int c = 0; c < D; ++c) {
      gg[(size_t)l * D + c] = W[lo.g + c];
      bm[(size_t)l * D + c] = W[lo.b_m + c];
      b1[(size_t)l * D + c] = W[lo.b1 + c];
      b2[(size_t)l * D + c] = W[lo.b2 + c];
    }
  }

  // ---- one device allocation for everything the kernel reads
  struct Part {
    const void* src;
    size_t bytes;
    void** dst;
  };
  std::vector<Part> parts = {
      {we1.data(), n_e1 * 2, (void**)&t->w_e1},
      {we2.data(), n_e2 * 2, (void**)&t->w_e2},
      {win.data(), n_in * 2, (void**)&t->w_in},
      {wm.data(), n_m * 2, (void**)&t->w_m},
      {w1.data(), n_11 * 2, (void**)&t->w_1},
      {w2.data(), n_11 * 2, (void**)&t->w_2},
      {W + o.emb_b1, (size_t)D * 4, (void**)&t->b_e1},
      {W + o.emb_b2, (size_t)D * 4, (void**)&t->b_e2},
      {gg.data(), gg.size() * 4, (void**)&t->g},
      {bin.data(), bin.size() * 4, (void**)&t->b_in},
      {bm.data(), bm.size() * 4, (void**)&t->b_m},
      {b1.data(), b1.size() * 4, (void**)&t->b_1},
      {b2.data(), b2.size() * 4, (void**)&t->b_2},
  };
  size_t total = 0;
  for (auto& pt : parts) total += (pt.bytes + 255) & ~(size_t)255;
  if (tf_malloc((void**)&t->dev, total) != cudaSuccess) return TRACKFIT_ERR_OOM;
  size_t off = 0;
  for (auto& pt : parts) {
    *pt.dst = static_cast<char*>(t->dev) + off;
    if (cudaMemcpy(*pt.dst, pt.src, pt.bytes, cudaMemcpyHostToDevice) != cudaSuccess) return TRACKFIT_ERR_CUDA;
    off += (pt.bytes + 255) & ~(size_t)255;
  }
  // ---- packing buffers and the per-CTA residual scratch
  if (tf_malloc(&t->pack, tf_pack_bytes(MAXB)) != cudaSuccess) return TRACKFIT_ERR_OOM;
  if (tf_malloc((void**)&t->xs, (size_t)t->nsm * TILE * 256 * sizeof(float)) != cudaSuccess) return TRACKFIT_ERR_OOM;
  if (tf_malloc((void**)&t->fbuf, (size_t)t->nsm * (D == 128 ? 4 : 2) * EB_BYTES) != cudaSuccess) return TRACKFIT_ERR_OOM;
  if (tf_malloc((void**)&t->pool, (size_t)POOL_TRACKS * D * sizeof(float)) != cudaSuccess) return TRACKFIT_ERR_OOM;
  // ---- tensor maps
  bool ok = make_map(&t->tm[MAP_E1], t->w_e1, D, E, fp16) && make_map(&t->tm[MAP_E2], t->w_e2, D, D, fp16) &&
            make_map(&t->tm[MAP_IN], t->w_in, (uint64_t)L * t->ROWS_IN, D, fp16) &&
            make_map(&t->tm[MAP_M], t->w_m, (uint64_t)L * D, t->KM, fp16) &&
            make_map(&t->tm[MAP_1], t->w_1, (uint64_t)L * D, D, fp16) &&
            make_map(&t->tm[MAP_2], t->w_2, (uint64_t)L * D, D, fp16);
  if (!ok) return TRACKFIT_ERR_CUDA;
  // ---- the schedules
  {
    std::vector<Step> steps = build_schedule(D, L, t->NDC, t->ROWS_IN, 1);
    t->n_sched = (int)steps.size();
    if (D == 128) {
      const std::vector<Step> two = build_schedule(D, L, t->NDC, t->ROWS_IN, 2);
      t->n_sched2 = (int)two.size();
      steps.insert(steps.end(), two.begin(), two.end());
    }
    if (t->n_sched > MAX_SCHED || (D == 128 && (int)steps.size() > 3 * pair_steps(L, t->NDC))) return TRACKFIT_ERR_UNSUPPORTED;
    if (tf_malloc((void**)&t->sched, steps.size() * sizeof(Step)) != cudaSuccess) return TRACKFIT_ERR_OOM;
    if (cudaMemcpy(t->sched, steps.data(), steps.size() * sizeof(Step), cudaMemcpyHostToDevice) != cudaSuccess)
      return TRACKFIT_ERR_CUDA;
  }
  if (tf_allow_smem(tc_forward_kernel<false>) != cudaSuccess || tf_allow_smem(tc_forward_kernel<true>) != cudaSuccess ||
      tf_allow_smem(tc_pair_kernel<false, false>) != cudaSuccess ||
      tf_allow_smem(tc_pair_kernel<true, false>) != cudaSuccess ||
      tf_allow_smem(tc_pair_kernel<false, true>) != cudaSuccess ||
      tf_allow_smem(tc_pair_kernel<true, true>) != cudaSuccess)
    return TRACKFIT_ERR_CUDA;
  if (tf_head_prepare() != cudaSuccess)
    return TRACKFIT_ERR_CUDA;
  return TRACKFIT_OK;
}

int tf_tc_forward(trackfit_ctx* h, const float* hits, const int32_t* n_hits, int64_t B, float* out, float* out_q,
                  float* out_pool, cudaStream_t st, const int64_t* offs) {
  tf_tc_state* t = h->tc;
  const tf_shape& s = h->s;
  TcParams p;
  std::memset(&p, 0, sizeof(p));
  for (int i = 0; i < NMAPS; ++i) p.tm[i] = t->tm[i];
  p.xs = t->xs;
  p.fbuf = t->fbuf;
  const tf_pack pk = tf_pack_in(t->pack, MAXB);
  p.src.slab = pk.slab;
  p.src.order = pk.order;
  p.src.n_slabs = pk.n_slabs;
  p.sched = t->sched;
  p.n_sched = t->n_sched;
  p.n_sched2 = t->n_sched2;
  p.b_e1 = t->b_e1;
  p.b_e2 = t->b_e2;
  p.g = t->g;
  p.b_in = t->b_in;
  p.b_m = t->b_m;
  p.b_1 = t->b_1;
  p.b_2 = t->b_2;
  p.err = h->d_err;
  p.wait_ns = t->wait_ns;
  p.hold_tile = t->hold_tile;
  p.src.T = s.T;
  p.D = s.D;
  p.L = s.L;
  p.NDC = t->NDC;
  p.ROWS_IN = t->ROWS_IN;
  p.nst = t->nst;
  p.idesc = t->idesc;
  p.idesc_thin = t->idesc_thin;
  p.off_xb = t->off_xb;
  p.off_hb = t->off_hb;
  p.off_a = t->off_a;
  p.off_misc = t->off_misc;
  p.rms_eps = s.rms_eps;
  p.fp16 = s.precision == TRACKFIT_FP16_PROJ;
  for (int f = 0; f < 5; ++f) {
    const double inv = 1.0 / s.feat_range_d[f];
    p.src.feat_min[f] = s.feat_min[f];
    p.src.feat_inv_hi[f] = (float)inv;
    p.src.feat_inv_lo[f] = (float)(inv - (double)p.src.feat_inv_hi[f]);
  }
  for (int k = 0; k < 16; ++k) p.src.scale[k] = s.scale[k];
  p.src.scale_doubling = 1;
  for (int k = 0; k + 3 < 16; ++k)
    if (s.scale[k + 3] != 2.0f * s.scale[k]) p.src.scale_doubling = 0;
  // without a caller buffer the pooled means go to the internal one, which
  // bounds the launch chunk
  const int64_t chunk = out_pool ? MAXB : POOL_TRACKS;
  for (int64_t c0 = 0; c0 < B; c0 += chunk) {
    const int64_t nb = (B - c0 < chunk) ? B - c0 : chunk;
    if (tf_plan(n_hits + c0, nb, s.T, t->nsm, pk.order, pk.slab, pk.n_slabs, st) != cudaSuccess) return TRACKFIT_ERR_CUDA;
    p.src.hits = offs ? hits : hits + c0 * s.T * 5;
    p.src.offs = offs ? offs + c0 : nullptr;
    p.src.n_hits = n_hits + c0;
    p.pool = out_pool ? out_pool + c0 * s.P : t->pool;
    tf_prof_begin(h, st);
    // a CTA for every slab there can be: one-slab tiles (d_model 128)
    const bool thin = s.D == 128 && tf_slab_bound(nb, s.T) <= t->nsm;
    const auto kernel = s.D == 128 ? (p.fp16 ? (thin ? tc_pair_kernel<true, true> : tc_pair_kernel<true, false>)
                                             : (thin ? tc_pair_kernel<false, true> : tc_pair_kernel<false, false>))
                                   : (p.fp16 ? tc_forward_kernel<true> : tc_forward_kernel<false>);
    kernel<<<t->nsm, thin ? PAIR_NT<true> : NT, t->smem, st>>>(p);
    tf_prof_end(h, st);
    if (tf_head(s, h->off, h->d_w, p.pool, p.src.n_hits, nb, t->nsm, out + c0 * 5, out_q ? out_q + c0 * s.Q : nullptr,
                out_pool ? p.pool : nullptr, h->d_err, st) != cudaSuccess)
      return TRACKFIT_ERR_CUDA;
    if (cudaPeekAtLastError() != cudaSuccess) return TRACKFIT_ERR_CUDA;
  }
  return TRACKFIT_OK;
}

// UMMA layout probe: A device bf16 [128][K] (K-major), Bkn device bf16 [K][128],
// D device fp32 [128][128]; K in {64, 128, 192, 256}.  Synchronous.
int tf_tc_probe(trackfit_ctx* h, const uint16_t* A, const uint16_t* Bkn, int K, float* D, cudaStream_t st) {
  if (K < 64 || K > 256 || (K % 64) != 0) return TRACKFIT_ERR_INVALID_ARG;
  CUtensorMap m;
  if (!make_map(&m, A, 128, (uint64_t)K)) return TRACKFIT_ERR_CUDA;
  const size_t smem = (size_t)(K / 64) * A_BLOCK + (size_t)K * 256 + 64 + 1024;
  if (cudaFuncSetAttribute(umma_probe_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
    return TRACKFIT_ERR_CUDA;
  umma_probe_kernel<<<1, 128, smem, st>>>(m, Bkn, K, D, idesc_f16(128, 128, 1u, false, true), h->d_err);
  if (cudaPeekAtLastError() != cudaSuccess) return TRACKFIT_ERR_CUDA;
  return TRACKFIT_OK;
}
