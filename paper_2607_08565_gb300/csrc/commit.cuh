// Device code of a commit that the index with and without an LRU share.
#pragma once

#include "smetric_impl.cuh"
#include "table.cuh"

namespace smetric {

// Checks of a batch to commit and the queue drain, by one CTA: every request's
// instance (in [-1, N)) and local hit (in [0, L_r]); a bad value clears the
// batch flag, so that nothing is committed and the loads stay as they were.
// Otherwise, with `load`, it sums per instance the tokens each request routed
// there must prefill or fetch (L_r - local hit) and sets
// load_i <- (load_i + that sum) >> 1. Integer sums, so the order of the
// atomics does not matter. Returns whether the batch is to be committed.
__device__ __forceinline__ bool drain_batch(const int64_t* __restrict__ off, int32_t n, int N,
                                            const int32_t* __restrict__ instance,
                                            const int32_t* __restrict__ local_hit, int32_t* __restrict__ batch_ok,
                                            int64_t* __restrict__ load, int32_t* status) {
  __shared__ unsigned long long acc[SMETRIC_MAX_INSTANCES];
  __shared__ int bad;
  if (threadIdx.x == 0) bad = 0;
  for (int i = threadIdx.x; i < N; i += blockDim.x) acc[i] = 0;
  const bool offsets_ok = *batch_ok != 0;
  __syncthreads();
  if (!offsets_ok) return false;
  for (int64_t r = threadIdx.x; r < n; r += blockDim.x) {
    const int32_t i = instance[r];
    const int64_t L = off[r + 1] - off[r], h = local_hit ? local_hit[r] : 0;
    if (i < -1 || i >= N || h < 0 || h > L) { bad = 1; continue; }
    if (i >= 0 && load) atomicAdd(&acc[i], (unsigned long long)(L - h));
  }
  __syncthreads();
  if (bad) {
    if (threadIdx.x == 0) {
      *batch_ok = 0;
      latch_error(status, SMETRIC_ERR_INVALID_ARG);
    }
    return false;
  }
  if (load)
    for (int i = threadIdx.x; i < N; i += blockDim.x) load[i] = (load[i] + (int64_t)acc[i]) >> 1;
  return true;
}

// Largest r in [lo, n) with block_off[r] <= f, given block_off[lo] <= f < block_off[n].
__device__ __forceinline__ int32_t request_of(const int64_t* __restrict__ block_off, int32_t lo, int32_t n, int64_t f) {
  int32_t hi = n;
  while (hi - lo > 1) {
    const int32_t mid = (lo + hi) >> 1;
    if (__ldg(block_off + mid) <= f) lo = mid; else hi = mid;
  }
  return lo;
}

// One block of a committed request adds its hash to the local tier of the
// request's instance and, with `global`, to the global tier, in one entry
// access. A request routed to -1 (an invalid batch) adds nothing; another
// out-of-range instance latches INVALID_ARG. Returns whether it was committed.
__device__ __forceinline__ bool commit_block(uint8_t* tags, uint64_t* table, uint64_t n_buckets, int ew, int N,
                                             uint64_t key, int32_t i, bool global, int32_t* status) {
  if (i == -1) return false;
  if (i < -1 || i >= N || key < 2) {
    latch_error(status, SMETRIC_ERR_INVALID_ARG);
    return false;
  }
  if (!insert_key(tags, table, ew, n_buckets, key, global ? tier_bits(i, N) : tier_bits(i)))
    latch_error(status, SMETRIC_ERR_TABLE_FULL);
  return true;
}

}  // namespace smetric
