// Shared by the tensor-core softmax kernels: tensor maps, the pre-pass and the
// merge of split prefixes.
#pragma once

#include <cuda.h>

#include "common.cuh"
#include "kernels.h"

namespace flare {

constexpr int kRowsM = 128;  // query rows per row tile (tensor-memory lanes)

// bf16 tensor map of `rank` dimensions with the 128-byte swizzle.
bool encode_map(CUtensorMap* m, const void* ptr, int rank, const uint64_t* dims,
                const uint64_t* strides, const uint32_t* box);
// Validates the requests and orders the work units (one CTA).
cudaError_t launch_softmax_order(const SoftmaxParams& p, cudaStream_t stream);

// Merge of the split partials of one row tile (rows mtile*128 ..) of one
// (request, kv head): out = sum_s w_s o_s with w_s = exp(lse_s - lse) and
// lse = log sum_s exp(lse_s) (the splits' partial outputs are already
// normalised by their own row sums).  The weights go to shared memory first
// (one thread per row); then every thread combines 8 (row, 4-column) pieces at
// a time with all their loads in flight.  All threads of the CTA call this;
// `wts` holds 128 * n_split floats.
template <int D>
__device__ void merge_splits(const SoftmaxParams& p, int item, int r, int kvh, int mtile,
                             float* wts) {
  const int M = p.B * p.G;
  const int ns = p.n_split;
  const int m0 = mtile * kRowsM;
  const int rows = min(kRowsM, M - m0);
  const size_t base = (size_t)item * ns * M + m0;  // row i of split s at base + s * M + i
  for (int i = threadIdx.x; i < rows; i += blockDim.x) {
    float mx = -INFINITY;
    for (int s = 0; s < ns; ++s) mx = fmaxf(mx, p.ws_lse[base + (size_t)s * M + i]);
    float den = 0.f;
    for (int s = 0; s < ns; ++s) {
      const float l = p.ws_lse[base + (size_t)s * M + i];
      const float e = l == -INFINITY ? 0.f : expf(l - mx);
      wts[i * ns + s] = e;
      den += e;
    }
    const float inv = 1.f / den;
    for (int s = 0; s < ns; ++s) wts[i * ns + s] *= inv;
    const int m = m0 + i, t = m / p.G, g = m % p.G;
    if (p.lse) p.lse[((size_t)r * p.B + t) * p.Hq + kvh * p.G + g] = mx + logf(den);
  }
  __syncthreads();
  constexpr int kC = D / 4;  // 4-column pieces per row
  constexpr int kBatch = 8;
  const int n_items = rows * kC;
  for (int i0 = threadIdx.x; i0 < n_items; i0 += kBatch * blockDim.x) {
    float4 acc[kBatch];
#pragma unroll
    for (int k = 0; k < kBatch; ++k) acc[k] = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int s = 0; s < ns; ++s) {
      float4 o[kBatch];
#pragma unroll
      for (int k = 0; k < kBatch; ++k) {
        const int it = i0 + k * blockDim.x;
        o[k] = it < n_items ? *reinterpret_cast<const float4*>(
                                  p.ws_o + (base + (size_t)s * M + it / kC) * D + (it % kC) * 4)
                            : make_float4(0.f, 0.f, 0.f, 0.f);
      }
#pragma unroll
      for (int k = 0; k < kBatch; ++k) {
        const int it = i0 + k * blockDim.x;
        const float w = it < n_items ? wts[(it / kC) * ns + s] : 0.f;
        acc[k].x = fmaf(w, o[k].x, acc[k].x);
        acc[k].y = fmaf(w, o[k].y, acc[k].y);
        acc[k].z = fmaf(w, o[k].z, acc[k].z);
        acc[k].w = fmaf(w, o[k].w, acc[k].w);
      }
    }
#pragma unroll
    for (int k = 0; k < kBatch; ++k) {
      const int it = i0 + k * blockDim.x;
      if (it >= n_items) continue;
      const int m = m0 + it / kC, t = m / p.G, g = m % p.G;
      const size_t orow = ((size_t)r * p.B + t) * p.Hq + kvh * p.G + g;
      __nv_bfloat162 lo = __floats2bfloat162_rn(acc[k].x, acc[k].y);
      __nv_bfloat162 hi = __floats2bfloat162_rn(acc[k].z, acc[k].w);
      *reinterpret_cast<uint2*>(static_cast<__nv_bfloat16*>(p.out) + orow * D + (it % kC) * 4) =
          make_uint2(*reinterpret_cast<uint32_t*>(&lo), *reinterpret_cast<uint32_t*>(&hi));
    }
  }
}

// Publishes this CTA's split partial and, if it is the last split of its row
// tile to finish, merges them all (all threads of the CTA call this).
template <int D>
__device__ void finish_split(const SoftmaxParams& p, int item, int r, int kvh, int mtile,
                             int n_mt, int* last_flag, float* wts) {
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0)
    *last_flag = atomicAdd(&p.counters[(size_t)item * n_mt + mtile], 1) == p.n_split - 1;
  __syncthreads();
  if (*last_flag) {
    __threadfence();
    merge_splits<D>(p, item, r, kvh, mtile, wts);
  }
}

}  // namespace flare
