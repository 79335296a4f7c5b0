// Device-side LRU of capped KV$ tiers.
//
// Each serving instance's local KV$ and the global store are bounded and
// evict their least recently used blocks (Section 2: the instance that ran a
// request caches its blocks; capacity is finite). The recency order is the
// one the replay between batches uses: a block touched by request r of a
// batch at block position b has stamp (batch, r, -b), so within a request
// the deepest blocks are the least recent; after a batch's touches a tier
// over its cap evicts its smallest stamps until it is at the cap.
//
// Each capped tier keeps its keys in a record region, least recent first,
// one record per key. A commit rewrites every region from the current record
// buffer into the other one: the old records whose key the batch touched in
// that tier are dropped, the batch's touches of the tier follow in stamp
// order (a key touched several times once, at its last touch), and the
// first (count - cap) records are evicted instead of written. A commit moves
// 8 bytes per record twice and little more: whether a record's key was touched
// is asked of a bitmap first (8 bits per touch and more, so that about one key
// in nine that was not touched goes on to the exact set), and a record's
// survival is kept as a bit. Six launches per batch:
//   k_lru_plan    one CTA: the batch's checks and the queue drain; per request
//                 its first touch position in its local tier's and in the
//                 global tier's touch list (a stable prefix over the requests
//                 routed to each instance); per tier the touch count and the
//                 touch-list, set, filter and tile offsets.
//   k_lru_touch   thread per block: the block into the index (commit_block);
//                 its touch (deepest block first) into its tiers' touch lists,
//                 the batch's (tier, key) -> last touch sets (noting the
//                 touch's entry there) and their filters.
//   k_lru_flags   CTAs over tiles of 1,024 records-then-touches of one tier: a
//                 bit for whether each survives the rewrite, and the tile's
//                 count.
//   k_lru_scan    one CTA: exclusive scan of the tile counts; per tier its
//                 surviving count and the excess over its cap.
//   k_lru_write   CTAs over the tiles: each survivor's rank in its tier; the first
//                 `excess` go to the list of evicted keys, the rest to the
//                 other buffer.
//   k_lru_evict   thread per evicted key: remove_tier, which gives a slot back
//                 when its key leaves its last tier (a tier's evictions are
//                 its first records: done in place they are a few CTAs' serial
//                 work); the new lengths; the sets and filters cleared.
// Measured, 256 requests and 190k blocks a commit, 16 local tiers of 200k
// blocks (3.2M records), global tier uncapped, the batch's requests on few
// instances: 80 us of kernels (plan 13, touch 21, flags 24, scan 5, write 11,
// evict 6.5), against 159 with a set lookup per record in both passes (43 and
// 61 us), one warp's plan after the drain (8 and 11) and the touches apart from
// the inserts (16 and 13).

#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <new>

#include "smetric_impl.cuh"
#include "commit.cuh"
#include "launch.cuh"
#include "table.cuh"
#include "call_range.cuh"

using namespace smetric;

namespace {

constexpr int kLruThreads = 256;
constexpr int kLruPer = 4;                           // rounds of 32 consecutive elements that a warp owns in a tile
// 1,024 elements: a batch often goes to few instances, whose tiles then have all
// the lookups; 4,096 a tile left those to a few dozen CTAs (31 us instead of 24
// for the flags kernel at 190k touches of one tier).
constexpr int64_t kLruTile = kLruThreads * kLruPer;
// CTAs an SM of the two kernels over the tiles, at most. The caps say how many
// tiles there may be, the tiers' lengths how many there are: a CTA for each that
// may be made a commit of 3,200 blocks on 272M capped blocks take 324 us (these
// limits 75), and 95 on 48M (66). Full tiers want many CTAs, so that the tiles
// with the lookups spread: 717k blocks a commit on 48M records take 872 us with
// 192 of the flags kernel, 882 with 64, 870 with a CTA a tile.
constexpr int kFlagCtas = 192, kWriteCtas = 64;
constexpr int kLruTileWords = (int)(kLruTile / 32);  // flag words of a tile
constexpr int64_t kMaxCap = 1LL << 40;

// Rows of the per-tier plan (n_tiers + 1 entries each; the extra entry of
// kTile0 is the total tile count).
enum LruPlan {
  kRingOff = 0,  // the tier's record region in each buffer
  kCap,          // its cap (0: not capped)
  kLen,          // records in the current buffer
  kTouches,      // touches this batch
  kTouchOff,     // first touch in the touch lists
  kSetOff,       // first entry of its set
  kSetMask,      // set entries - 1 (-1: no set)
  kBitOff,       // first word of its filter
  kBitMask,      // filter bits - 1
  kTile0,        // first tile
  kExcess,       // records to evict
  kNewLen,       // records after the rewrite
  kEvictOff,     // first evicted key
  kLruPlanFields
};

__device__ __forceinline__ int64_t* row(int64_t* plan, int n_tiers, int f) { return plan + (int64_t)f * (n_tiers + 1); }
__device__ __forceinline__ const int64_t* row(const int64_t* plan, int n_tiers, int f) {
  return plan + (int64_t)f * (n_tiers + 1);
}

// Batch set of one tier: open addressing over (key, last touch + 1) pairs,
// key 0 = empty; sized >= 2 x the tier's touches, so a probe always ends.
// Returns the key's entry.
__device__ __forceinline__ uint64_t set_put(uint64_t* set, int64_t mask, uint64_t key, uint64_t v) {
  uint64_t s = key & (uint64_t)mask;
  for (int64_t t = 0; t <= mask; ++t) {
    unsigned long long* e = reinterpret_cast<unsigned long long*>(set + 2 * s);
    const unsigned long long old = atomicCAS(e, 0ull, (unsigned long long)key);
    if (old == 0ull || old == key) {
      atomicMax(e + 1, (unsigned long long)v);
      return s;
    }
    s = (s + 1) & (uint64_t)mask;
  }
  return s;
}

constexpr uint32_t kNowhere = 0xffffffffu;  // an entry past 2^32: looked up by its key

__device__ __forceinline__ ulonglong2 set_entry(const uint64_t* set, uint64_t s) {
  return __ldg(reinterpret_cast<const ulonglong2*>(set + 2 * s));
}

// The value of `key` in a set (0: absent), whose home entry is e.
__device__ __forceinline__ uint64_t set_get(const uint64_t* set, int64_t mask, uint64_t key, ulonglong2 e) {
  uint64_t s = key & (uint64_t)mask;
  for (int64_t t = 0; t <= mask; ++t) {
    if (e.x == key) return e.y;
    if (e.x == 0) return 0;
    s = (s + 1) & (uint64_t)mask;
    e = set_entry(set, s);
  }
  return 0;
}

__device__ __forceinline__ int64_t next_pow2(int64_t v) {
  int64_t p = 1;
  while (p < v) p <<= 1;
  return p;
}

// A key's bit in a filter; the sets use the low bits.
__device__ __forceinline__ uint32_t filter_bit(uint64_t key, int64_t mask) { return (uint32_t)(key >> 32) & (uint32_t)mask; }

// Its shared memory: running totals, and a round's totals per warp, of N + 1 tiers.
constexpr size_t plan_smem(int N) { return (size_t)33 * (N + 1) * sizeof(int64_t); }

// One CTA: checks and drain, then rounds of 1,024 requests, 32 to a warp.
// Within a warp, the lanes routed to the same instance (__match_any_sync) sum
// the blocks of their lower lanes; the warps' totals per instance are scanned
// over the warps in shared memory, and the running totals carry across rounds.
// So req_off[r] is the number of blocks of earlier requests routed to r's
// instance, and req_off[R + r] that of all earlier committed requests (global
// tier).
__global__ void __launch_bounds__(1024)
    k_lru_plan(const int64_t* __restrict__ off, const int64_t* __restrict__ block_off, int32_t n,
               const int32_t* __restrict__ instance, const int32_t* __restrict__ local_hit, int32_t* batch_ok, int N,
               bool local_capped, bool global_touch, int64_t* plan, int64_t* __restrict__ req_off, int64_t R,
               int64_t* __restrict__ load, int32_t* status) {
  pdl_enter();
  extern __shared__ int64_t lsm[];
  int64_t* const run = lsm;            // [N + 1]: running totals, the global tier's last
  int64_t* const cnt = lsm + (N + 1);  // [32][N + 1]: a round's totals per warp
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nt = N + 1;
  const bool ok = drain_batch(off, n, N, instance, local_hit, batch_ok, load, status);
  for (int i = threadIdx.x; i < nt; i += blockDim.x) run[i] = 0;
  __syncthreads();
  for (int32_t base = 0; ok && base < n; base += 1024) {
    const int32_t r = base + (int32_t)threadIdx.x;
    for (int i = lane; i < nt; i += 32) cnt[warp * nt + i] = 0;
    __syncwarp();
    int32_t i = -1;
    int64_t nb = 0;
    if (r < n) {
      i = instance[r];
      nb = block_off[r + 1] - block_off[r];
      if (i < 0 || i >= N) {
        i = -1;
        nb = 0;
      }
    }
    const unsigned peers = __match_any_sync(0xffffffffu, i);
    int64_t acc = 0, gacc = 0;
#pragma unroll 4
    for (int k = 0; k < 32; ++k) {
      const int64_t v = __shfl_sync(0xffffffffu, nb, k);
      if (k < lane) {
        gacc += v;
        if ((peers >> k) & 1u) acc += v;
      }
    }
    if (i >= 0 && lane == 31 - __clz(peers)) cnt[warp * nt + i] = acc + nb;
    if (lane == 31) cnt[warp * nt + N] = gacc + nb;
    __syncthreads();
    for (int t = threadIdx.x; t < nt; t += blockDim.x) {
      int64_t x = run[t];
      for (int w = 0; w < 32; ++w) {
        const int64_t v = cnt[w * nt + t];
        cnt[w * nt + t] = x;
        x += v;
      }
      run[t] = x;
    }
    __syncthreads();
    if (r < n && i >= 0) {
      req_off[r] = cnt[warp * nt + i] + acc;
      req_off[R + r] = cnt[warp * nt + N] + gacc;
    }
    __syncthreads();
  }
  if (warp != 0) return;
  // per tier: touches, then the offsets of the touch lists, sets, filters and tiles
  int64_t t_off = 0, s_off = 0, b_off = 0, tile0 = 0;
  for (int base = 0; base < nt; base += 32) {
    const int t = base + lane;
    int64_t T = 0, S = 0, F = 0, tiles = 0;  // F: filter words
    if (t < nt) {
      const bool capped = row(plan, nt, kCap)[t] > 0;
      T = !capped ? 0 : (t < N ? (local_capped ? run[t] : 0) : (global_touch ? run[N] : 0));
      S = T > 0 ? next_pow2(2 * T) : 0;
      F = T > 0 ? max((int64_t)1, min(next_pow2(8 * T), (int64_t)1 << 32) / 32) : 0;
      tiles = (row(plan, nt, kLen)[t] + T + kLruTile - 1) / kLruTile;
    }
    int64_t pt = T, ps = S, pb = F, pl = tiles;  // inclusive warp scans
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int64_t a = __shfl_up_sync(0xffffffffu, pt, d), b = __shfl_up_sync(0xffffffffu, ps, d),
                    c = __shfl_up_sync(0xffffffffu, pl, d), e = __shfl_up_sync(0xffffffffu, pb, d);
      if (lane >= d) {
        pt += a;
        ps += b;
        pl += c;
        pb += e;
      }
    }
    if (t < nt) {
      row(plan, nt, kTouches)[t] = T;
      row(plan, nt, kTouchOff)[t] = t_off + pt - T;
      row(plan, nt, kSetOff)[t] = s_off + ps - S;
      row(plan, nt, kSetMask)[t] = S - 1;
      row(plan, nt, kBitOff)[t] = b_off + pb - F;
      row(plan, nt, kBitMask)[t] = 32 * F - 1;
      row(plan, nt, kTile0)[t] = tile0 + pl - tiles;
    }
    t_off += __shfl_sync(0xffffffffu, pt, 31);
    s_off += __shfl_sync(0xffffffffu, ps, 31);
    b_off += __shfl_sync(0xffffffffu, pb, 31);
    tile0 += __shfl_sync(0xffffffffu, pl, 31);
  }
  if (lane == 0) row(plan, nt, kTile0)[nt] = tile0;  // total tiles
  if (lane == 0) row(plan, nt, kSetOff)[nt] = s_off;  // set entries in use
  if (lane == 0) row(plan, nt, kBitOff)[nt] = b_off;  // and filter words
}

// Thread per block f of the batch (request r, position b of n_r): into the
// index, and its touch, whose position in a tier's list is the tier's count of
// earlier requests' blocks plus n_r - 1 - b (deepest block first). The plan has
// counted every block of a request that goes to an instance, so a block whose
// hash is refused (below 2) has its places all the same: it leaves key 0 there,
// which k_lru_flags passes over.
__global__ void __launch_bounds__(256)
    k_lru_touch(uint8_t* tags, uint64_t* table, uint64_t n_buckets, int ew, const int64_t* __restrict__ block_off,
                int32_t n, const int32_t* __restrict__ instance, const uint64_t* __restrict__ H,
                const int32_t* __restrict__ batch_ok, int N, bool global, bool local_capped, bool global_touch,
                const int64_t* __restrict__ plan, const int64_t* __restrict__ req_off, int64_t R,
                uint64_t* __restrict__ touches, uint32_t* __restrict__ where, uint64_t* __restrict__ set,
                uint32_t* __restrict__ filter, int32_t* status) {
  pdl_enter();
  if (!*batch_ok) return;
  const int nt = N + 1;
  const int64_t total = block_off[n];
  int32_t r = 0;
  auto touch = [&](int t, int64_t q, uint64_t key) {
    touches[row(plan, nt, kTouchOff)[t] + q] = key;
    if (key == 0) return;
    const uint32_t bit = filter_bit(key, row(plan, nt, kBitMask)[t]);
    atomicOr(filter + row(plan, nt, kBitOff)[t] + (bit >> 5), 1u << (bit & 31));
    const uint64_t e = set_put(set + 2 * row(plan, nt, kSetOff)[t], row(plan, nt, kSetMask)[t], key, (uint64_t)q + 1);
    where[row(plan, nt, kTouchOff)[t] + q] = e < kNowhere ? (uint32_t)e : kNowhere;
  };
  for (int64_t f = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; f < total;
       f += (int64_t)gridDim.x * blockDim.x) {
    r = request_of(block_off, r, n, f);
    const int32_t i = instance[r];
    uint64_t key = H[f];
    if (!commit_block(tags, table, n_buckets, ew, N, key, i, global, status)) {
      if (i < 0 || i >= N) continue;  // no places
      key = 0;
    }
    const int64_t back = block_off[r + 1] - 1 - f;  // n_r - 1 - b
    if (local_capped) touch(i, req_off[r] + back, key);
    if (global_touch) touch(N, req_off[R + r] + back, key);
  }
}

// The tier of tile k: the largest t with kTile0[t] <= k (tiers without
// tiles share their successor's first tile and are skipped).
__device__ __forceinline__ int tier_of_tile(const int64_t* tile0, int nt, int64_t k) {
  int lo = 0, hi = nt;  // tile0[lo] <= k < tile0[hi]
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (tile0[mid] <= k) lo = mid; else hi = mid;
  }
  return lo;
}

// What a tile's CTA needs of its tier's plan.
struct LruTile {
  int64_t j0;          // the tile's first element of the tier's rewrite
  int64_t len, touch;  // records, then touches
  const uint64_t* ring;
  const uint64_t* touches;
  int t;
};

__device__ __forceinline__ LruTile tile_of(const int64_t* plan, int nt, int64_t k, const uint64_t* ring,
                                           const uint64_t* touches) {
  LruTile x;
  x.t = tier_of_tile(row(plan, nt, kTile0), nt, k);
  x.j0 = (k - row(plan, nt, kTile0)[x.t]) * kLruTile;
  x.len = row(plan, nt, kLen)[x.t];
  x.touch = row(plan, nt, kTouches)[x.t];
  x.ring = ring + row(plan, nt, kRingOff)[x.t];
  x.touches = touches + row(plan, nt, kTouchOff)[x.t];
  return x;
}

// Key of element j: a record (j < len) or the touch j - len; 0 past both.
__device__ __forceinline__ uint64_t element(const LruTile& x, int64_t j) {
  return j < x.len ? __ldg(x.ring + j) : j - x.len < x.touch ? __ldg(x.touches + (j - x.len)) : 0ull;
}

// One CTA: exclusive scan of the tile counts into tile_off (total at the end),
// each thread a run of consecutive tiles, then each tier's survivors, excess
// over its cap and new length, and the scan of the excesses.
__global__ void __launch_bounds__(1024)
    k_lru_scan(int64_t* __restrict__ plan, int nt, const int64_t* __restrict__ tile_cnt,
               int64_t* __restrict__ tile_off) {
  pdl_enter();
  __shared__ int64_t ws[32];
  __shared__ int64_t excess[SMETRIC_MAX_INSTANCES + 1];
  const int64_t* tile0 = row(plan, nt, kTile0);
  const int64_t total = tile0[nt];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t per = (total + 1023) / 1024;
  const int64_t a = min(total, threadIdx.x * per), e = min(total, a + per);
  int64_t v = 0;
  for (int64_t k = a; k < e; ++k) v += tile_cnt[k];
  int64_t x = v;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const int64_t y = __shfl_up_sync(0xffffffffu, x, d);
    if (lane >= d) x += y;
  }
  if (lane == 31) ws[w] = x;
  __syncthreads();
  if (w == 0) {
    int64_t y = ws[lane];
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int64_t z = __shfl_up_sync(0xffffffffu, y, d);
      if (lane >= d) y += z;
    }
    ws[lane] = y;  // inclusive over the warps
  }
  __syncthreads();
  int64_t at = (w > 0 ? ws[w - 1] : 0) + x - v;
  for (int64_t k = a; k < e; ++k) {
    tile_off[k] = at;
    at += tile_cnt[k];
  }
  if (threadIdx.x == 0) tile_off[total] = ws[31];
  __syncthreads();
  for (int t = threadIdx.x; t < nt; t += blockDim.x) {
    const int64_t kept = tile_off[tile0[t + 1]] - tile_off[tile0[t]];
    const int64_t cap = row(plan, nt, kCap)[t];
    const int64_t ex = cap > 0 && kept > cap ? kept - cap : 0;
    row(plan, nt, kExcess)[t] = ex;
    row(plan, nt, kNewLen)[t] = kept - ex;
    excess[t] = ex;
  }
  __syncthreads();
  if (w == 0) {
    int64_t off = 0;
    for (int t0 = 0; t0 < nt; t0 += 32) {
      const int t = t0 + lane;
      const int64_t ex = t < nt ? excess[t] : 0;
      int64_t y = ex;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const int64_t z = __shfl_up_sync(0xffffffffu, y, d);
        if (lane >= d) y += z;
      }
      if (t < nt) row(plan, nt, kEvictOff)[t] = off + y - ex;
      off += __shfl_sync(0xffffffffu, y, 31);
    }
    if (lane == 0) row(plan, nt, kEvictOff)[nt] = off;
  }
}

// Flags and count of tile k, by one CTA.
__device__ __forceinline__ void flag_tile(int64_t k, const int64_t* __restrict__ plan, int nt, const uint64_t* __restrict__ ring,
                                          const uint64_t* __restrict__ touches, const uint32_t* __restrict__ where,
                                          const uint64_t* __restrict__ set, const uint32_t* __restrict__ filter, uint32_t* __restrict__ keep,
                                          int64_t* __restrict__ tile_cnt) {
  const LruTile x = tile_of(plan, nt, k, ring, touches);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t j0 = x.j0 + (int64_t)w * 32 * kLruPer + lane;
  const int64_t mask = row(plan, nt, kSetMask)[x.t], bmask = row(plan, nt, kBitMask)[x.t];
  const uint64_t* const tset = set + 2 * row(plan, nt, kSetOff)[x.t];
  const uint32_t* const bits = filter + row(plan, nt, kBitOff)[x.t];
  const uint32_t* const twhere = where + row(plan, nt, kTouchOff)[x.t];
  // Records stay unless the set says otherwise, touches go unless it does: the
  // elements to look up there (the filter's answers, and every touch) are
  // gathered first, so that the CTA looks all of them up at once.
  __shared__ uint32_t words[kLruTileWords];
  __shared__ uint16_t ask[kLruTile];
  __shared__ int asks;
  if (threadIdx.x == 0) asks = 0;
  uint64_t key[kLruPer];
#pragma unroll
  for (int e = 0; e < kLruPer; ++e) key[e] = element(x, j0 + 32 * e);
  uint32_t maybe = 0;  // bit e: element e's key may have been touched
  if (mask >= 0) {
#pragma unroll
    for (int e = 0; e < kLruPer; ++e) {
      const uint32_t b = filter_bit(key[e], bmask);
      const bool hit = (__ldg(bits + (b >> 5)) >> (b & 31)) & 1u;
      maybe |= (uint32_t)(hit && key[e] != 0) << e;  // (0: past the tile's elements, or a refused touch)
    }
  }
#pragma unroll
  for (int e = 0; e < kLruPer; ++e) {
    const unsigned m = __ballot_sync(0xffffffffu, j0 + 32 * e < x.len);
    if (lane == 0) words[w * kLruPer + e] = m;
  }
  __syncthreads();
  const int mine = __popc(maybe);
  int incl = mine;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const int a = __shfl_up_sync(0xffffffffu, incl, d);
    if (lane >= d) incl += a;
  }
  int at = 0;
  if (lane == 31) at = atomicAdd(&asks, incl);
  at = __shfl_sync(0xffffffffu, at, 31) + incl - mine;
  for (uint32_t left = maybe; left; left &= left - 1)
    ask[at++] = (uint16_t)(w * 32 * kLruPer + 32 * (__ffs(left) - 1) + lane);
  __syncthreads();
  constexpr int A = 4;  // a thread's lookups in flight (all of a tile of touches)
  for (int p = threadIdx.x; p < asks; p += A * kLruThreads) {
    int el[A];
    uint64_t kv[A];
    ulonglong2 home[A];
#pragma unroll
    for (int u = 0; u < A; ++u) {
      el[u] = p + u * kLruThreads < asks ? ask[p + u * kLruThreads] : -1;
      kv[u] = el[u] >= 0 ? element(x, x.j0 + el[u]) : 0;
    }
#pragma unroll
    for (int u = 0; u < A; ++u)
      if (el[u] >= 0) {  // a touch's entry is known, a record's key is probed for
        const int64_t q = x.j0 + el[u] - x.len;
        const uint32_t at = q >= 0 ? __ldg(twhere + q) : kNowhere;
        home[u] = set_entry(tset, at != kNowhere ? at : kv[u] & (uint64_t)mask);
      }
#pragma unroll
    for (int u = 0; u < A; ++u) {
      if (el[u] < 0) continue;
      const int64_t q = x.j0 + el[u] - x.len;
      const uint64_t last = set_get(tset, mask, kv[u], home[u]);
      if (q < 0) {  // a record stays if its key was not touched,
        if (last != 0) atomicAnd(words + (el[u] >> 5), ~(1u << (el[u] & 31)));
      } else if (last == (uint64_t)q + 1) {  // a touch if it is its key's last
        atomicOr(words + (el[u] >> 5), 1u << (el[u] & 31));
      }
    }
  }
  __syncthreads();
  if (threadIdx.x < 32) {
    int c = 0;
#pragma unroll
    for (int u = 0; u < kLruTileWords / 32; ++u) {
      const uint32_t m = words[32 * u + lane];
      keep[k * kLruTileWords + 32 * u + lane] = m;
      c += __popc(m);
    }
    c = __reduce_add_sync(0xffffffffu, c);
    if (lane == 0) tile_cnt[k] = c;
  }
}

// LOOP: a CTA takes every gridDim.x-th tile, with fewer CTAs than there may be
// tiles. (Without it the loop's two registers would cost 0.3 % of a commit.)
template <bool LOOP>
__global__ void __launch_bounds__(kLruThreads)
    k_lru_flags(const int64_t* __restrict__ plan, int nt, const uint64_t* __restrict__ ring,
                const uint64_t* __restrict__ touches, const uint32_t* __restrict__ where,
                const uint64_t* __restrict__ set, const uint32_t* __restrict__ filter, uint32_t* __restrict__ keep,
                int64_t* __restrict__ tile_cnt) {
  pdl_enter();
  const int64_t total = row(plan, nt, kTile0)[nt];
  for (int64_t k = blockIdx.x; k < total; k += gridDim.x) {
    flag_tile(k, plan, nt, ring, touches, where, set, filter, keep, tile_cnt);
    if (!LOOP) return;
    __syncthreads();  // the next tile takes the shared arrays
  }
}

__global__ void __launch_bounds__(kLruThreads)
    k_lru_write(const int64_t* __restrict__ plan, int nt, const uint64_t* __restrict__ ring,
                uint64_t* __restrict__ next, const uint64_t* __restrict__ touches, const uint32_t* __restrict__ keep,
                const int64_t* __restrict__ tile_off, uint64_t* __restrict__ evicted) {
  pdl_enter();
  const int64_t* tile0 = row(plan, nt, kTile0);
  const int64_t total = tile0[nt];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int64_t k = blockIdx.x; k < total; k += gridDim.x) {
    const LruTile x = tile_of(plan, nt, k, ring, touches);
    // lane e < kLruPer has the warp's flag word e; survivors of the CTA's earlier warps
    const uint32_t* const words = keep + k * kLruTileWords;
    const uint32_t mine = lane < kLruPer ? words[w * kLruPer + lane] : 0;
    int before = 0;
    for (int u = lane; u < w * kLruPer; u += 32) before += __popc(words[u]);
    before = __reduce_add_sync(0xffffffffu, before);
    int64_t rank = tile_off[k] - tile_off[tile0[x.t]] + before;
    const int64_t ex = row(plan, nt, kExcess)[x.t];
    const int64_t j0 = x.j0 + (int64_t)w * 32 * kLruPer + lane;
    uint64_t* const out = next + row(plan, nt, kRingOff)[x.t] - ex;
    uint64_t* const gone = evicted + row(plan, nt, kEvictOff)[x.t];
    uint64_t key[kLruPer];
#pragma unroll
    for (int e = 0; e < kLruPer; ++e) key[e] = element(x, j0 + 32 * e);
#pragma unroll
    for (int e = 0; e < kLruPer; ++e) {
      const uint32_t m = __shfl_sync(0xffffffffu, mine, e);
      const int64_t at = rank + __popc(m & ((1u << lane) - 1));
      if ((m >> lane) & 1u) (at >= ex ? out : gone)[at] = key[e];
      rank += __popc(m);
    }
  }
}

__global__ void __launch_bounds__(256)
    k_lru_evict(int64_t* __restrict__ plan, int nt, const uint64_t* __restrict__ evicted, uint64_t* __restrict__ set,
                uint32_t* __restrict__ filter, uint8_t* tags, uint64_t* table, int ew, int W, uint64_t n_buckets) {
  pdl_enter();
  const int64_t* const off = row(plan, nt, kEvictOff);
  const int64_t total = off[nt];
  const int64_t i0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, step = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = i0; i < total; i += step) {
    const int t = tier_of_tile(off, nt, i);  // (the same search: tiers without evictions share an offset)
    remove_tier(tags, table, ew, W, n_buckets, evicted[i], t >> 6, 1ull << (t & 63));  // the global tier is bit N
  }
  // the sets and filters are done with: cleared for the next batch
  const int64_t used = row(plan, nt, kSetOff)[nt], words = row(plan, nt, kBitOff)[nt];
  for (int64_t i = i0; i < used; i += step) reinterpret_cast<ulonglong2*>(set)[i] = make_ulonglong2(0ull, 0ull);
  for (int64_t i = i0; i < words; i += step) filter[i] = 0;
  if (blockIdx.x == 0)
    for (int t = threadIdx.x; t < nt; t += blockDim.x) row(plan, nt, kLen)[t] = row(plan, nt, kNewLen)[t];
}

}  // namespace

namespace smetric {

void lru_free(smetric_index* idx) {
  LruState* L = idx->lru;
  if (!L) return;
  cudaFree(L->ring[0]);
  cudaFree(L->ring[1]);
  cudaFree(L->plan);
  cudaFree(L->req_off);
  cudaFree(L->touches);
  cudaFree(L->set);
  cudaFree(L->where);
  cudaFree(L->filter);
  cudaFree(L->keep);
  cudaFree(L->evicted);
  cudaFree(L->tile_cnt);
  cudaFree(L->tile_off);
  delete L;
  idx->lru = nullptr;
}

int lru_reset(smetric_index* idx, cudaStream_t s) {
  LruState* L = idx->lru;
  if (!L) return SMETRIC_OK;
  return cuda_status(
      cudaMemsetAsync(L->plan + (int64_t)kLen * (L->n_tiers + 1), 0, (L->n_tiers + 1) * sizeof(int64_t), s));
}

int lru_commit(smetric_index* idx, const int64_t* d_offsets, const int32_t* d_instance, const int32_t* d_local_hit,
               const uint64_t* d_hashes, int32_t n, bool global, int64_t* d_load, cudaStream_t s) {
  LruState* L = idx->lru;
  const int N = idx->cfg.num_instances, nt = L->n_tiers;
  const bool local_capped = L->local_cap > 0, global_touch = global && L->global_cap > 0;
  const int64_t R = idx->cfg.max_batch_requests;
  const int64_t max_blocks = idx->cfg.max_batch_tokens / idx->cfg.block_size;
  int rc;
  const size_t smem = plan_smem(N);
  const int64_t want = (max_blocks + 255) / 256;
  const unsigned grid = (unsigned)std::max<int64_t>(1, std::min<int64_t>(want, (int64_t)idx->num_sms * 8));
  const int64_t tiles = L->max_tiles;
  const unsigned fgrid = (unsigned)std::min<int64_t>(tiles, (int64_t)idx->num_sms * kFlagCtas);
  const unsigned wgrid = (unsigned)std::min<int64_t>(tiles, (int64_t)idx->num_sms * kWriteCtas);
  const uint64_t* ring = L->ring[L->cur];
  uint64_t* next = L->ring[L->cur ^ 1];
  if ((rc = launch_k(k_lru_plan, dim3(1), dim3(1024), smem, s, true, d_offsets, (const int64_t*)idx->block_off, n,
                     d_instance, d_local_hit, idx->batch_ok, N, local_capped, global_touch, L->plan, L->req_off, R,
                     d_load, idx->status)) ||
      (rc = launch_k(k_lru_touch, dim3(grid), dim3(256), 0, s, true, idx->tags, idx->table, idx->n_buckets, idx->EW,
                     (const int64_t*)idx->block_off, n, d_instance, d_hashes, (const int32_t*)idx->batch_ok, N, global,
                     local_capped, global_touch, (const int64_t*)L->plan, (const int64_t*)L->req_off, R, L->touches,
                     L->where, L->set, L->filter, idx->status)) ||
      (rc = launch_k(tiles > fgrid ? k_lru_flags<true> : k_lru_flags<false>, dim3(fgrid), dim3(kLruThreads), 0, s, true,
                     (const int64_t*)L->plan, nt, ring,
                     (const uint64_t*)L->touches, (const uint32_t*)L->where, (const uint64_t*)L->set,
                     (const uint32_t*)L->filter, L->keep, L->tile_cnt)) ||
      (rc = launch_k(k_lru_scan, dim3(1), dim3(1024), 0, s, true, L->plan, nt, (const int64_t*)L->tile_cnt,
                     L->tile_off)) ||
      (rc = launch_k(k_lru_write, dim3(wgrid), dim3(kLruThreads), 0, s, true,
                     (const int64_t*)L->plan, nt, ring, next, (const uint64_t*)L->touches, (const uint32_t*)L->keep,
                     (const int64_t*)L->tile_off, L->evicted)) ||
      (rc = launch_k(k_lru_evict, dim3(grid), dim3(256), 0, s, true, L->plan, nt, (const uint64_t*)L->evicted, L->set,
                     L->filter, idx->tags, idx->table, idx->EW, idx->W, idx->n_buckets)))
    return rc;
  idx->launches += 6;
  L->cur ^= 1;
  return SMETRIC_OK;
}

}  // namespace smetric

extern "C" {

int smetric_index_set_lru(smetric_index* idx, int64_t local_cap, int64_t global_cap) {
  CallRange range("smetric_index_set_lru");
  int rc = check_device(idx);
  if (rc) return rc;
  if (local_cap < 0 || global_cap < 0 || local_cap > kMaxCap || global_cap > kMaxCap) return SMETRIC_ERR_INVALID_ARG;
  if (cudaDeviceSynchronize() != cudaSuccess) return cuda_status(cudaErrorUnknown);
  lru_free(idx);
  if (local_cap == 0 && global_cap == 0) return SMETRIC_OK;
  // the plan kernel's limit is every index's: the most that any N takes
  if (cudaFuncSetAttribute(k_lru_plan, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)plan_smem(SMETRIC_MAX_INSTANCES)) != cudaSuccess)
    return cuda_status(cudaErrorInvalidValue);
  const int N = idx->cfg.num_instances, nt = N + 1;
  const int64_t R = idx->cfg.max_batch_requests;
  const int64_t max_blocks = idx->cfg.max_batch_tokens / idx->cfg.block_size;
  LruState* L = new (std::nothrow) LruState();
  if (!L) return SMETRIC_ERR_OOM;
  L->local_cap = local_cap;
  L->global_cap = global_cap;
  L->n_tiers = nt;
  // host copies of the static plan rows
  int64_t* h = new (std::nothrow) int64_t[(size_t)kLruPlanFields * (nt + 1)]();
  if (!h) {
    delete L;
    return SMETRIC_ERR_OOM;
  }
  int64_t ring_total = 0;
  for (int t = 0; t < nt; ++t) {
    const int64_t cap = t < N ? local_cap : global_cap;
    h[(int64_t)kRingOff * (nt + 1) + t] = ring_total;
    h[(int64_t)kCap * (nt + 1) + t] = cap;
    ring_total += cap;
  }
  // tiles: each tier's records (<= cap) and touches, rounded up to whole tiles
  L->max_tiles = (ring_total + 2 * max_blocks) / kLruTile + nt + 1;
  L->set_entries = 8 * max_blocks + 2;
  // a tier's filter has at most 16 bits a touch, or one word; touches number at most 2 * max_blocks
  L->filter_words = max_blocks + nt + 1;
  idx->lru = L;
  const bool ok =
      cudaMalloc(&L->ring[0], std::max<int64_t>(ring_total, 1) * sizeof(uint64_t)) == cudaSuccess &&
      cudaMalloc(&L->ring[1], std::max<int64_t>(ring_total, 1) * sizeof(uint64_t)) == cudaSuccess &&
      cudaMalloc(&L->plan, (size_t)kLruPlanFields * (nt + 1) * sizeof(int64_t)) == cudaSuccess &&
      cudaMalloc(&L->req_off, std::max<int64_t>(2 * R, 1) * sizeof(int64_t)) == cudaSuccess &&
      cudaMalloc(&L->touches, std::max<int64_t>(2 * max_blocks, 1) * sizeof(uint64_t)) == cudaSuccess &&
      cudaMalloc(&L->set, L->set_entries * 2 * sizeof(uint64_t)) == cudaSuccess &&
      cudaMalloc(&L->where, std::max<int64_t>(2 * max_blocks, 1) * sizeof(uint32_t)) == cudaSuccess &&
      cudaMalloc(&L->filter, L->filter_words * sizeof(uint32_t)) == cudaSuccess &&
      cudaMalloc(&L->keep, L->max_tiles * kLruTileWords * sizeof(uint32_t)) == cudaSuccess &&
      // no tier evicts more than the batch touched in it
      cudaMalloc(&L->evicted, std::max<int64_t>(2 * max_blocks, 1) * sizeof(uint64_t)) == cudaSuccess &&
      cudaMalloc(&L->tile_cnt, (L->max_tiles + 1) * sizeof(int64_t)) == cudaSuccess &&
      cudaMalloc(&L->tile_off, (L->max_tiles + 1) * sizeof(int64_t)) == cudaSuccess &&
      cudaMemcpy(L->plan, h, (size_t)kLruPlanFields * (nt + 1) * sizeof(int64_t), cudaMemcpyHostToDevice) ==
          cudaSuccess &&
      cudaMemset(L->set, 0, L->set_entries * 2 * sizeof(uint64_t)) == cudaSuccess &&
      cudaMemset(L->filter, 0, L->filter_words * sizeof(uint32_t)) == cudaSuccess;
  delete[] h;
  if (!ok) {
    (void)cudaGetLastError();
    lru_free(idx);
    return SMETRIC_ERR_OOM;
  }
  return SMETRIC_OK;
}

int smetric_index_lru_sizes(smetric_index* idx, int64_t* d_sizes, smetric_stream_t stream) {
  CallRange range("smetric_index_lru_sizes");
  int rc = check_device(idx);
  if (rc) return rc;
  if (!d_sizes) return SMETRIC_ERR_INVALID_ARG;
  const int nt = idx->cfg.num_instances + 1;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  if (!idx->lru) return cuda_status(cudaMemsetAsync(d_sizes, 0, nt * sizeof(int64_t), s));
  return cuda_status(cudaMemcpyAsync(d_sizes, idx->lru->plan + (int64_t)kLen * (nt + 1), nt * sizeof(int64_t),
                                     cudaMemcpyDeviceToDevice, s));
}

}  // extern "C"
