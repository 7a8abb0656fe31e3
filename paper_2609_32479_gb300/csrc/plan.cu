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
// It is bound by the latency of the first warp's steps (about three a slab).  One
// lane walking a table of counts took 57 us for 101 tracks and 531 us for segments
// of 1,024.
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
  uint64_t left = 0;   // bit l - 1: tracks of l hits remain
#pragma unroll
  for (int h = 0; h < 2; ++h)
    left |= (uint64_t)__ballot_sync(0xffffffffu, cnt[32 * h + lane + 1] > 0) << (32 * h);
  int o = 0, ns = 0, cap = TF_SLAB, ntr = 0, bad = cnt[0];
  if (lane == 0) first[0] = 0;
  while (left || bad) {
    const uint64_t fits = cap == TF_SLAB ? left : left & ((1ull << cap) - 1ull);
    int l = 0, k = 0;
    if (ntr < TF_SLAB_TRACKS) {
      if (fits) {
        l = 64 - __clzll((long long)fits);
        const int c = cnt[l];
        k = min(min(c, cap / l), TF_SLAB_TRACKS - ntr);
        if (k == c) left &= ~(1ull << (l - 1));
      } else if (!left) {
        k = min(bad, TF_SLAB_TRACKS - ntr);
        bad -= k;
      }
    }
    if (k == 0) {   // the slab is full
      ++ns;
      if (lane == 0) first[ns] = (int16_t)o;
      cap = TF_SLAB;
      ntr = 0;
      continue;
    }
    const int at = pos[l];
    if (lane < k) order[b0 + o + lane] = (int32_t)(b0 + items[at + lane]);
    __syncwarp();
    if (lane == 0) {
      pos[l] = (int16_t)(at + k);
      cnt[l] = (int16_t)(cnt[l] - k);
    }
    __syncwarp();
    o += k;
    ntr += k;
    cap -= k * l;
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
// segments of 256 take a quarter of the steps.
cudaError_t tf_plan(const int32_t* n_hits, int64_t B, int T, int nsm, int32_t* order, int2* slab, int32_t* n_slabs,
                    cudaStream_t st) {
  cudaError_t e = cudaMemsetAsync(n_slabs, 0, sizeof(int32_t), st);
  if (e != cudaSuccess) return e;
  if (B >= (int64_t)1024 * nsm)
    plan_kernel<1024><<<(unsigned)((B + 1023) / 1024), 1024, 0, st>>>(n_hits, B, T, order, slab, n_slabs);
  else
    plan_kernel<256><<<(unsigned)((B + 255) / 256), 256, 0, st>>>(n_hits, B, T, order, slab, n_slabs);
  return cudaPeekAtLastError();
}
