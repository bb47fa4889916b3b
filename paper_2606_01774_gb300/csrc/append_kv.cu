// KV append of the state-update pass: the finalized block's keys and values
// become part of the paged prefix.  Positions prefix_len[r] + t for the
// first n = append_len[r] (or B) block tokens, through the page table.
//
// The call moves little (8 MB for 64 requests, blocks of 32) and is bound by the
// latency of one thread's chain: the lengths, then the page ids and the source
// together, then the store.  A request's block is one run of 16-byte chunks in the
// source, split over CTAs of 256 threads by kChunks chunks a thread, all loaded
// before the first is stored; every CTA checks the whole request, so nothing of
// a request with a bad page id is written.  With one CTA per request each thread ran
// the chain eight times: 64 requests, blocks of 32 (2 heads, D = 256) 8.0 -> 2.7 us,
// one request 7.9 -> 2.2, 128 requests, blocks of 64 24.3 -> 6.3, 256 requests, blocks
// of 16 (4 heads, D = 128) 6.0 -> 3.6.  One or four chunks a thread: within 0.4 us.
#include "common.cuh"
#include "kernels.h"

namespace flare {

namespace {
constexpr int kAppendThreads = 256;
constexpr int kChunks = 2;
constexpr int kMaxBlock = 64;  // tokens of a block; at least one thread each
}  // namespace

__global__ void __launch_bounds__(kAppendThreads)
    append_kv_kernel(SoftmaxParams p, const int32_t* append_len, void* k_pool, void* v_pool,
                     int row_shift) {  // log2 of the 16-byte chunks of a (token, head) row
  stream_order();
  __shared__ int pages[kMaxBlock];
  const int r = blockIdx.x, tid = threadIdx.x;
  const int P = p.prefix_len[r];
  const int n = append_len ? append_len[r] : p.B;
  int bad = 0;
  if (n < 0 || n > p.B) bad = FLARE_DEV_BAD_ACCEPT_LEN;
  else if (P < 0 || (long)P + n > (long)p.max_pages * p.page_size) bad = FLARE_DEV_BAD_PREFIX_LEN;
  const size_t block = ((size_t)p.B * p.Hkv) << row_shift;  // chunks of a request
  const size_t total = bad ? 0 : ((size_t)n * p.Hkv) << row_shift;
  const uint4* kb = static_cast<const uint4*>(p.k_blk) + r * block;
  const uint4* vb = static_cast<const uint4*>(p.v_blk) + r * block;
  constexpr int kStep = kAppendThreads * kChunks;
  const size_t first = (size_t)blockIdx.y * kStep;
  if (first >= total && blockIdx.y > 0) return;
  int badpg = 0;
  if (!bad && tid < n) {
    const int pg = p.page_table[(size_t)r * p.max_pages + (P + tid) / p.page_size];
    pages[tid] = pg;
    badpg = pg < 0 || pg >= p.num_pages;
  }
  for (size_t e0 = first + tid;; e0 += (size_t)gridDim.y * kStep) {
    uint4 kv[kChunks], vv[kChunks];
#pragma unroll
    for (int u = 0; u < kChunks; ++u) {
      const size_t e = e0 + u * kAppendThreads;
      if (e < total) kv[u] = kb[e], vv[u] = vb[e];
    }
    if (e0 == first + tid) {
      if (__syncthreads_or(badpg)) bad = FLARE_DEV_BAD_PAGE;
      if (bad) {
        if (tid == 0 && blockIdx.y == 0) flag(p.dev_status, bad);
        return;
      }
    }
    if (e0 >= total) return;
#pragma unroll
    for (int u = 0; u < kChunks; ++u) {
      const size_t e = e0 + u * kAppendThreads;
      if (e >= total) break;
      const unsigned row = (unsigned)(e >> row_shift);
      const int t = (int)(row / (unsigned)p.Hkv), hk = (int)(row % (unsigned)p.Hkv);
      const size_t dst = ((((size_t)pages[t] * p.Hkv + hk) * p.page_size + (P + t) % p.page_size)
                          << row_shift) + (e & ((1u << row_shift) - 1));
      static_cast<uint4*>(k_pool)[dst] = kv[u];
      static_cast<uint4*>(v_pool)[dst] = vv[u];
    }
  }
}

cudaError_t launch_append_kv(const SoftmaxParams& p, const int32_t* append_len, void* k_pool,
                             void* v_pool, int elem_bytes, cudaStream_t stream) {
  if (p.R == 0) return cudaSuccess;
  int row_shift = 0;  // D is 64, 128 or 256
  while ((16 << row_shift) < p.D * elem_bytes) ++row_shift;
  const size_t block = ((size_t)p.B * p.Hkv) << row_shift;
  const size_t slices = (block + kAppendThreads * kChunks - 1) / (kAppendThreads * kChunks);
  const dim3 grid((unsigned)p.R, (unsigned)(slices < 65535 ? slices : 65535));
  launch_kernel(append_kv_kernel, grid, kAppendThreads, 0, stream, p, append_len, k_pool, v_pool,
                row_shift);
  note_launches(1);
  return cudaGetLastError();
}

}  // namespace flare
