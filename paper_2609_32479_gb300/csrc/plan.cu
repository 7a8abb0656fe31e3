// Packing of whole tracks into slabs: at most TF_SLAB hits and TF_SLAB_TRACKS
// tracks each, the unit that the fused kernels work on.
#include "trackfit_internal.h"

namespace {

// One CTA packs a segment of blockDim.x tracks, one thread a track: a counting
// sort by hit count, then best fit by the first warp: each slab takes the longest
// remaining tracks that still fit until none does.  Lengths are at most 64, so the
// lengths that are left are one 64-bit mask, the longest that fits is a count of
// its leading zeros, and as many tracks of a length as fit are taken at once.
// Tracks with an invalid hit count take a slot but no columns, at the end.  The
// packing of a segment depends on its hit counts alone; where its slabs lie among
// those of the other segments does not, and neither matters to a track's results.
//
// It is bound by the latency of the first warp's steps (about three a slab), so their
// state is in registers: with the counts in shared memory and an integer division a step
// took 400 cycles (98 us for 256 tracks of 64 hits, 31 us for 997 of 12.5), and one lane
// walking a table of counts took 57 us for 101 tracks, 531 us for segments of 1,024.
template <int SEG>
__global__ void __launch_bounds__(SEG) plan_kernel(const int32_t* __restrict__ n_hits, int64_t B, int T,
                                                   int32_t* __restrict__ order, int2* __restrict__ slab,
                                                   int32_t* __restrict__ n_slabs) {
  constexpr int NW = SEG / 32, NL = TF_SLAB + 1;
  __shared__ int16_t hist[NW][NL + 1], items[SEG], first[SEG + 1];
  __shared__ int16_t cnt[NL], pos[NL];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int64_t b0 = (int64_t)blockIdx.x * SEG;
  const int nt = (int)(B - b0 < SEG ? B - b0 : SEG);
  for (int i = tid; i < NW * (NL + 1); i += SEG) (&hist[0][0])[i] = 0;
  int len = -1;   // past the batch: in no bucket
  if (tid < nt) {
    len = n_hits[b0 + tid];
    if (len < 1 || len > T) len = 0;
  }
  __syncthreads();
  const uint32_t same = __match_any_sync(0xffffffffu, len);
  const int rank = __popc(same & ((1u << lane) - 1u));
  if (len >= 0 && rank == 0) hist[warp][len] = (int16_t)__popc(same);
  __syncthreads();
  for (int l = tid; l < NL; l += SEG) {   // exclusive sums over the warps
    int s = 0;
    for (int w = 0; w < NW; ++w) {
      const int v = hist[w][l];
      hist[w][l] = (int16_t)s;
      s += v;
    }
    cnt[l] = (int16_t)s;
  }
  __syncthreads();
  if (warp == 0) {   // exclusive sums over the lengths 0 .. 64
    int carry = 0;
    for (int l0 = 0; l0 < NL; l0 += 32) {
      const int l = l0 + lane, v = l < NL ? cnt[l] : 0;
      int s = v;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, s, o);
        if (lane >= o) s += u;
      }
      if (l < NL) pos[l] = (int16_t)(carry + s - v);
      carry += __shfl_sync(0xffffffffu, s, 31);
    }
  }
  __syncthreads();
  if (len >= 0) items[pos[len] + hist[warp][len] + rank] = (int16_t)tid;
  __syncthreads();
  if (warp != 0) return;
  // Lane i keeps, for the lengths i + 1 and i + 33: tracks left and where the next of them
  // is in items (packed), and 1 / length in 16 fractional bits.  A step's chain of
  // dependent operations is then a few integer instructions and two shuffles.
  uint32_t lo = (uint32_t)cnt[lane + 1] | ((uint32_t)pos[lane + 1] << 16);
  uint32_t hi = (uint32_t)cnt[lane + 33] | ((uint32_t)pos[lane + 33] << 16);
  const uint32_t inv_lo = 65536u / (lane + 1) + 1u, inv_hi = 65536u / (lane + 33) + 1u;   // exact up to 64
  uint64_t left = (uint64_t)__ballot_sync(0xffffffffu, (lo & 0xffffu) != 0) |
                  (uint64_t)__ballot_sync(0xffffffffu, (hi & 0xffffu) != 0) << 32;   // bit l - 1: tracks of l hits remain
  int o = 0, ns = 0, cap = TF_SLAB, ntr = 0;
  if (lane == 0) first[0] = 0;
  while (left) {
    uint64_t fits = cap == TF_SLAB ? left : left & ((1ull << cap) - 1ull);
    if (fits == 0 || ntr == TF_SLAB_TRACKS) {   // the slab is full
      ++ns;
      if (lane == 0) first[ns] = (int16_t)o;
      cap = TF_SLAB;
      ntr = 0;
      fits = left;
    }
    const int b = 63 - __clzll((long long)fits), l = b + 1;
    const uint32_t cp = __shfl_sync(0xffffffffu, b < 32 ? lo : hi, b & 31);
    const uint32_t inv = __shfl_sync(0xffffffffu, b < 32 ? inv_lo : inv_hi, b & 31);
    const int c = (int)(cp & 0xffffu), at = (int)(cp >> 16);
    const int k = min(min(c, (int)(((uint32_t)cap * inv) >> 16)), TF_SLAB_TRACKS - ntr);
    if (k == c) left &= ~(1ull << b);
    if (lane == (b & 31)) {   // k tracks fewer, the next one k further
      const uint32_t d = ((uint32_t)k << 16) - (uint32_t)k;
      if (b < 32)
        lo += d;
      else
        hi += d;
    }
    if (lane < k) order[b0 + o + lane] = (int32_t)(b0 + items[at + lane]);
    o += k;
    ntr += k;
    cap -= k * l;
  }
  for (int bad = cnt[0], at = 0; bad > 0;) {   // tracks with an invalid hit count
    if (ntr == TF_SLAB_TRACKS) {
      ++ns;
      if (lane == 0) first[ns] = (int16_t)o;
      ntr = 0;
    }
    const int k = min(bad, TF_SLAB_TRACKS - ntr);
    if (lane < k) order[b0 + o + lane] = (int32_t)(b0 + items[at + lane]);
    at += k;
    o += k;
    ntr += k;
    bad -= k;
  }
  ++ns;   // the last slab (a segment has at least one track)
  if (lane == 0) first[ns] = (int16_t)o;
  int base = 0;
  if (lane == 0) base = atomicAdd(n_slabs, ns);
  base = __shfl_sync(0xffffffffu, base, 0);
  __syncwarp();
  for (int i = lane; i < ns; i += 32)
    slab[base + i] = make_int2((int)b0 + first[i], first[i + 1] - first[i]);
}

}  // namespace

// Segments of 1,024 tracks leave one slab in 200 part-filled; below one such
// segment for each SM the plan's own latency counts for more than the fill, and
// segments of 256 take a quarter of the steps.  Up to 2,048 tracks the tiles hardly fill
// the chip once, so the fill counts for nothing: segments of 64.  With the state in
// registers, a whole call of 101 tracks 121 -> 115 us (d_model 128) and 106 -> 84 us (997
// tracks of the paper's model); 4,096 tracks of 64 hits 1,160 -> 1,129 us.
cudaError_t tf_plan(const int32_t* n_hits, int64_t B, int T, int nsm, int32_t* order, int2* slab, int32_t* n_slabs,
                    cudaStream_t st) {
  cudaError_t e = cudaMemsetAsync(n_slabs, 0, sizeof(int32_t), st);
  if (e != cudaSuccess) return e;
  if (B >= (int64_t)1024 * nsm)
    plan_kernel<1024><<<(unsigned)((B + 1023) / 1024), 1024, 0, st>>>(n_hits, B, T, order, slab, n_slabs);
  else if (B <= 2048)
    plan_kernel<64><<<(unsigned)((B + 63) / 64), 64, 0, st>>>(n_hits, B, T, order, slab, n_slabs);
  else
    plan_kernel<256><<<(unsigned)((B + 255) / 256), 256, 0, st>>>(n_hits, B, T, order, slab, n_slabs);
  return cudaPeekAtLastError();
}
