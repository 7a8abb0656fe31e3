// What the kernels on tiles of packed hits with materialised Fourier rows share
// (concat.cu, transformer.cu): the Fourier rows in tile order and the host's helpers.
#pragma once

#include <cuda.h>
#include <cudaTypedefs.h>

#include "tc_epilogue.cuh"

namespace {

// ------------------------------------------------------------------ Fourier rows
// Sec. 3.2, for the hits of a slab: row 64 s + column holds the hit's Fourier vector
// (per feature 16 sines, 16 cosines); columns without a hit hold zeros.  One thread per
// (column, feature), the argument as in rows.cu (an unevaluated sum of two floats,
// reduced modulo 2 exactly; with scales 2^(k/3) nine of 16 evaluated, the others by
// one double-angle step).
template <bool FP16>
__global__ void __launch_bounds__(256) fourier_slab_kernel(const TileSrc src, const __grid_constant__ tf_shape s,
                                                           uint16_t* __restrict__ e) {
  __shared__ int64_t row_s[SLAB];
  const int n_slabs = *src.n_slabs;
  for (int sl = blockIdx.x; sl < n_slabs; sl += gridDim.x) {
    __syncthreads();
    if (threadIdx.x < 32) {
      const int lane = threadIdx.x;
      const int2 d = src.slab[sl];
      int n = 0;
      int64_t r = 0;
      if (lane < d.y) {
        const int b = src.order[d.x + lane];
        n = src.n_hits[b];
        if (n < 1 || n > s.T) n = 0;
        r = src.offs ? src.offs[b] : (int64_t)b * s.T;
      }
      int end = n;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, end, o);
        if (lane >= o) end += u;
      }
      for (int t = 0; t < n; ++t) row_s[end - n + t] = r + t;
      const int all = __shfl_sync(0xffffffffu, end, 31);
      for (int c = all + lane; c < SLAB; c += 32) row_s[c] = -1;
    }
    __syncthreads();
    for (int i = threadIdx.x; i < SLAB * s.F; i += 256) {
      const int c = i / s.F, f = i - c * s.F;
      uint4* o = reinterpret_cast<uint4*>(e + ((size_t)sl * SLAB + c) * s.E + f * 2 * TRACKFIT_MAX_FOURIER);
      const int64_t row = row_s[c];
      if (row < 0) {
#pragma unroll
        for (int q = 0; q < 4; ++q) o[q] = make_uint4(0u, 0u, 0u, 0u);
        continue;
      }
      const float v = src.hits[row * s.F + f];
      const float mn = -s.feat_min[f], ih = s.feat_inv_range[f];
      const float dh = v + mn, bv = dh - v, dl = (v - (dh - bv)) + (mn - bv);
      const float uh = dh * ih;
      const float ul = fmaf(dh, ih, -uh) + fmaf(dh, s.feat_inv_lo[f], dl * ih);
      float sv[TRACKFIT_MAX_FOURIER], cv[TRACKFIT_MAX_FOURIER];
#pragma unroll
      for (int k = 0; k < TRACKFIT_MAX_FOURIER; ++k) {
        if (src.scale_doubling && (k % 6) >= 3) {   // s_k = 2 s_{k-3}
          sv[k] = 2.0f * sv[k - 3] * cv[k - 3];
          cv[k] = (cv[k - 3] - sv[k - 3]) * (cv[k - 3] + sv[k - 3]);
          continue;
        }
        const float sk = s.scale[k], xh = uh * sk, xl = fmaf(uh, sk, -xh) + ul * sk;
        sincospif((xh - 2.0f * rintf(0.5f * xh)) + xl, &sv[k], &cv[k]);
      }
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        o[q] = make_uint4(pack2<FP16>(sv[8 * q], sv[8 * q + 1]), pack2<FP16>(sv[8 * q + 2], sv[8 * q + 3]),
                          pack2<FP16>(sv[8 * q + 4], sv[8 * q + 5]), pack2<FP16>(sv[8 * q + 6], sv[8 * q + 7]));
        o[2 + q] = make_uint4(pack2<FP16>(cv[8 * q], cv[8 * q + 1]), pack2<FP16>(cv[8 * q + 2], cv[8 * q + 3]),
                              pack2<FP16>(cv[8 * q + 4], cv[8 * q + 5]), pack2<FP16>(cv[8 * q + 6], cv[8 * q + 7]));
      }
    }
  }
}

inline cudaError_t fourier_slabs(TileSrc src, const tf_shape& s, int64_t tracks, int nsm, uint16_t* e, cudaStream_t st) {
  src.scale_doubling = 1;
  for (int k = 0; k + 3 < TRACKFIT_MAX_FOURIER; ++k)
    if (s.scale[k + 3] != 2.0f * s.scale[k]) src.scale_doubling = 0;
  const unsigned grid = (unsigned)(tracks < 8 * nsm ? tracks : 8 * nsm);   // slabs are at most the tracks
  if (s.precision == TRACKFIT_FP16_PROJ)
    fourier_slab_kernel<true><<<grid, 256, 0, st>>>(src, s, e);
  else
    fourier_slab_kernel<false><<<grid, 256, 0, st>>>(src, s, e);
  return cudaPeekAtLastError();
}

// 16-bit matrix [rows][cols] row-major -> tensor map of 64-column x box_rows boxes with
// 128-byte swizzle (out-of-range elements read as zero).
inline bool tile_map(CUtensorMap* m, const void* ptr, uint64_t rows, uint64_t cols, bool fp16,
                     uint32_t box_rows = 128) {
  void* f = nullptr;
  cudaDriverEntryPointQueryResult q;
  if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) != cudaSuccess ||
      q != cudaDriverEntryPointSuccess)
    return false;
  cuuint64_t dims[2] = {cols, rows}, strides[1] = {cols * 2};
  cuuint32_t box[2] = {64, box_rows}, es[2] = {1, 1};
  return reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(f)(
             m, fp16 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(ptr),
             dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
             CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

inline uint16_t to_16(float f, bool fp16) {
  if (fp16) {
    const __half v = __float2half_rn(f);
    return *reinterpret_cast<const uint16_t*>(&v);
  }
  const __nv_bfloat16 v = __float2bfloat16_rn(f);
  return *reinterpret_cast<const uint16_t*>(&v);
}

}  // namespace
