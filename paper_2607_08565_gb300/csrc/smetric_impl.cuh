// Internal declarations shared by the library's translation units.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <vector>

#include "smetric.h"

namespace smetric {

constexpr uint64_t kGamma = 0x9E3779B97F4A7C15ull;
constexpr uint64_t kEmpty = 0;  // key of a never-used slot

// SplitMix64 output function (Steele, Lea & Flood, OOPSLA 2014; Stafford's
// Mix13 multipliers). Two xor-shift-multiply rounds and a final xor-shift.
__host__ __device__ __forceinline__ uint64_t mix64(uint64_t z) {
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

// The table is an array of buckets of kSlots = 15 slots. A bucket's 16-byte
// tag group (in a tag array of its own) holds a one-byte tag per slot (0:
// empty; otherwise the low key byte, 1 for 0) and, in byte 15, the bucket's
// overflow count: how many keys stored past this bucket probed through it
// (saturating at 255, which then stays). Entries (key + tier-mask words) are
// in the entry array, slot sl of bucket b at b * kSlots + sl. A key's home
// bucket is the high 64 bits of key * n_buckets (Lemire's range reduction);
// an insert takes the first empty slot in bucket order from the home bucket
// (linear probing over buckets) and counts itself in the overflow byte of
// every bucket it passed; a lookup stops at the first bucket without the key
// whose overflow count is 0. A key that leaves its last tier gives its slot
// back (tag and key zeroed, the passed buckets' counts decremented), so the
// table holds live keys only and no tombstones. At load factor 0.7 about 98%
// of keys sit in their home bucket: a lookup is one tag read plus one entry
// read.
constexpr int kBucket = 16;  // bytes of a bucket's tag group
constexpr int kSlots = 15;   // slots of a bucket

__device__ __forceinline__ uint64_t home_bucket(uint64_t key, uint64_t n_buckets) {
  return __umul64hi(key, n_buckets);
}

__host__ __device__ __forceinline__ uint32_t key_tag(uint64_t key) {
  const uint32_t t = (uint32_t)key & 0xFFu;
  return t ? t : 1u;
}

// The slots of a bucket whose tag equals `tag` (0: the empty ones), as a set
// that next_slot takes apart; byte 15, the overflow count, is left out. Bit
// 8 b + w stands for byte b of tag word w, slot 4 w + b: the zero bytes of
// x ^ tag have their top bit set by an exact test per word, and the four words'
// top bits go side by side, ~24 instructions for the 16 bytes (a per-byte
// compare and gather took ~70; a probe runs this once or twice).
__device__ __forceinline__ uint32_t slot_match(uint4 t, uint32_t tag) {
  const uint32_t rep = tag * 0x01010101u;
  const uint32_t w[4] = {t.x ^ rep, t.y ^ rep, t.z ^ rep, t.w ^ rep};
  uint32_t m = 0;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const uint32_t zero = ~(((w[i] & 0x7F7F7F7Fu) + 0x7F7F7F7Fu) | w[i]) & 0x80808080u;
    m |= zero >> (7 - i);
  }
  return m & ~(1u << 27);
}

// Takes one slot out of a set that slot_match gave.
__device__ __forceinline__ int next_slot(uint32_t& set) {
  const int p = __ffs(set) - 1;
  set &= set - 1;
  return 4 * (p & 7) + (p >> 3);
}

// A bucket's overflow count (byte 15 of its tag group).
__device__ __forceinline__ uint32_t overflow_count(uint4 t) { return t.w >> 24; }

// Buckets a lookup or an insert visits at most.
__host__ __device__ __forceinline__ uint64_t max_buckets(uint64_t n_buckets) {
  const uint64_t m = SMETRIC_MAX_PROBE / kBucket;
  return n_buckets < m ? n_buckets : m;
}

// First error wins; later ones are dropped until the host reads and clears.
__device__ __forceinline__ void latch_error(int32_t* status, int32_t code) {
  atomicCAS(reinterpret_cast<int*>(status), 0, code);
}

// Entry stride in 64-bit words for W mask words: key + W words, rounded up to
// a power of two so that no entry straddles a 32-byte sector (W = 1: 16 B,
// W = 2..3: 32 B, W = 4..7: 64 B).
__host__ __device__ constexpr int entry_words(int W) { return W == 1 ? 2 : (W <= 3 ? 4 : 8); }

// Route kernels, in launch order; names returned by smetric_profile_kernel_name.
// kChainProbe is k_lead and k_chain_probe in a route (group stage, then chain
// and probe in one kernel) and the chain alone in the calls that only hash.
enum RouteKernel { kPrep = 0, kDigest = 1, kChainProbe = 2, kWalk = 3, kNumRouteKernels = 4 };

// smetric_route_batch_host: the status and the outputs of batches of up to this
// many requests come back in one copy to the index's pinned buffer and one wait.
// (Longer ones are copied to the caller's arrays: the extra pass over 20 bytes a
// request costs the host more than the copies saved.) Inputs are always copied
// from the caller's arrays, in stream order. 16 requests of 6,000 tokens: 81 us
// a call, 83 with a copy of its own for the status, 98 with four copies down
// and the status read by a synchronous one.
constexpr int64_t kHostSmall = 2048;
constexpr size_t kStatusBytes = 16;  // before the outputs, so that one copy takes both
constexpr size_t kHostPin = kStatusBytes + (size_t)kHostSmall * 20;

struct ProfileSlot {
  cudaEvent_t ev[kNumRouteKernels + 1];
};

}  // namespace smetric

namespace smetric {

// Device-side LRU of the capped tiers (smetric_index_set_lru; kernels in
// lru.cu). Each capped tier keeps its keys in recency order, least recent
// first, in a region of one of two record buffers; a commit rewrites every
// region from one buffer into the other.
struct LruState {
  int64_t local_cap = 0, global_cap = 0;  // blocks; 0 = uncapped
  int n_tiers = 0;                        // N + 1
  uint64_t* ring[2] = {nullptr, nullptr}; // records (keys), tier t's at its region offset
  int cur = 0;                            // the buffer holding the current records
  int64_t* plan = nullptr;                // kLruPlanFields rows of n_tiers + 1 int64 (lru.cu)
  int64_t* req_off = nullptr;             // 2 * max_batch_requests: a request's first touch in its tiers
  uint64_t* touches = nullptr;            // 2 * max_blocks: the batch's touches, tier after tier
  uint64_t* set = nullptr;                // set_entries (key, last touch + 1) pairs
  int64_t set_entries = 0;
  uint32_t* where = nullptr;              // 2 * max_blocks: each touch's entry in its tier's set
  uint32_t* filter = nullptr;             // filter_words: a bit per hash of a touched key, tier after tier
  int64_t filter_words = 0;
  uint32_t* keep = nullptr;               // max_tiles * kLruTile flags, one bit each
  uint64_t* evicted = nullptr;            // 2 * max_blocks: the batch's evicted keys, tier after tier
  int64_t* tile_cnt = nullptr;            // max_tiles + 1, then their exclusive scan
  int64_t* tile_off = nullptr;
  int64_t max_tiles = 0;
};

}  // namespace smetric

struct smetric_index {
  smetric_index_config cfg;
  int device;
  int num_sms;
  int W;   // tier-mask words per key
  int EW;  // entry stride in 64-bit words
  uint64_t n_buckets;  // ceil(capacity_slots / kSlots)
  uint64_t* table;     // n_buckets * kSlots entries of EW words
  uint8_t* tags;       // n_buckets tag groups of kBucket bytes
  int32_t* status;  // device: first latched error
  // route scratch
  int64_t* block_off;  // max_batch_requests + 1: first block of each request
  uint64_t* digest;    // max_batch_tokens / B: per-block digests d_b
  uint64_t* hashes;    // max_batch_tokens / B: per-block chain hashes h_b
  uint64_t* masks;     // W * max_batch_tokens / B: per-block tier masks
  uint64_t* chunk_and; // W * (max_batch_tokens / B / 32 + R + 1): AND of each request-aligned 32-block chunk's masks
  uint64_t* groups;    // 2 * group_slots: (first-block hash, INT32_MAX - leader) pairs
  uint64_t group_slots;  // power of two >= 2 * max_batch_requests
  int32_t* lead;       // max_batch_requests: the request whose masks a request shares
  int32_t* share;      // max_batch_requests: leading blocks taken from the leader
  int32_t* summ;       // max_batch_requests * (num_instances + 1): run ends c_i, then g (the sequential variant)
  uint64_t* sk_tmp;     // max_batch_requests: session keys nobody reads (session links); a route's k_lead marks
  int64_t* chunk_off;  // max_batch_requests + 1: first 32-block chunk of each request
  int32_t* batch_ok;   // device flag written by the prep kernel
  // staging for smetric_route_batch_host
  int32_t* st_tokens;
  int64_t* st_in;       // num_instances loads, then max_batch_requests + 1 offsets
  uint64_t* st_out;     // after the status word: a batch's session keys, then its 3 n int32 outputs (20 bytes a request)
  unsigned char* st_pin;  // pinned host memory: the status, and kHostSmall requests' outputs
  int digest_occ;  // resident digest CTAs per SM (0 until the first route)
  smetric::LruState* lru;  // capped tiers' recency (NULL: no tier capped)
  // observability
  int64_t launches;
  bool profiling;
  std::vector<smetric::ProfileSlot> prof_pool;  // free event sets
  std::vector<smetric::ProfileSlot> prof_used;  // recorded, not yet read
};

namespace smetric {
// Returns SMETRIC_OK if the index is usable from the current device.
int check_device(const smetric_index* idx);
// Sets the shared-memory limits of the index's kernels; false on a CUDA error.
bool kernel_limits(const smetric_index* idx);
// Maps a CUDA error to SMETRIC_ERR_CUDA (clearing the sticky-free error state).
int cuda_status(cudaError_t e);
// Inserts a routed batch's block hashes into its chosen instances' local tiers
// (and the global tier); block_off must hold the batch's block offsets.
int launch_commit(smetric_index* idx, const int32_t* d_instance, const uint64_t* d_hashes, int32_t n,
                  int64_t max_blocks, bool global, cudaStream_t s);
// The same on an index with an LRU, with the batch's checks and the queue drain
// before it (drain_batch): then the capped tiers' recency lists take the
// batch's touches and evict what exceeds each cap.
int lru_commit(smetric_index* idx, const int64_t* d_offsets, const int32_t* d_instance, const int32_t* d_local_hit,
               const uint64_t* d_hashes, int32_t n, bool global, int64_t* d_load, cudaStream_t s);
// Empties every recency list (after the table is cleared).
int lru_reset(smetric_index* idx, cudaStream_t s);
// Frees the LRU state.
void lru_free(smetric_index* idx);
}  // namespace smetric
