// Batched routing: block chain hash, session key, two-tier longest-prefix
// match, integer cost and argmin (Figure 6 and Figure 10 of the paper, with
// every request of the batch routed against one snapshot of index and load).
//
// Kernels per batch, in stream order:
//   k_prep        a CTA per 8,192 requests (up to 128): validates offsets and
//                 loads; scans the per-request full-block counts into block_off
//                 and the 32-block chunk counts into chunk_off.
//   k_digest_tma  HBM-bound block digests d_b: chunk q of request r is its
//                 blocks 32q..32q+31, one 2D TMA tile of 32 overlapping rows
//                 (each block's bytes rounded out to 16-byte boundaries); a
//                 CTA takes a contiguous range of chunks, its warps
//                 interleaved over it; lane j folds block j's B/2 words.
//                 The lane holding a request's first block also inserts the
//                 request's group key (its first-block hash) into the group
//                 table. (k_digest and k_digest_any cover block sizes the
//                 tensor maps do not.)
//   k_lead        one warp per request: its group's leader (the group's lowest
//                 request index), the shared prefix (leading blocks with the
//                 leader's digests), and whether the chain kernel takes it.
//   k_chain_probe one CTA per SM. Chain warps (one lane per request the CTA
//                 owns) run the serial chain h_b over the digests in a ring in
//                 shared memory; beside them, probe warps fill the ring, write
//                 the session keys (and the hashes, where wanted) and probe
//                 every block not shared: the tier masks of h_b from the index
//                 (15 tags of the home bucket, then the matching entry), and
//                 the AND of each 32-block chunk's masks.
//   k_walk        one warp per request walks the runs of the local tiers and
//                 the global tier (a member over its leader's probes up to
//                 its shared prefix), 32 chunks per step from the chunk ANDs
//                 and block by block where a run ends; a short tail past the
//                 shared prefix that the chain kernel left out is chained and
//                 probed here; then lanes = instances for the cost and a
//                 shuffle argmin with ties to the lowest id (or one of the
//                 policy scores).

#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <utility>
#include <atomic>
#include <cstring>

#include "smetric_impl.cuh"
#include "commit.cuh"
#include "launch.cuh"

using namespace smetric;

namespace {

constexpr unsigned kFull = 0xffffffffu;

constexpr int kChunk = 32;        // blocks per digest task (one per lane)
constexpr int kDigestWarps = 8;   // most warps per digest CTA
// Most shared memory of a digest CTA without tile copies. The limit on dynamic
// shared memory belongs to the kernel, which every index (and the call without
// one) shares: it is always set to this, never to what one block size needs.
constexpr size_t kDigestSmem = 200 * 1024;
// Warps per TMA digest CTA, one CTA an SM: 32 for B = 16 and 32, then as many
// rows as shared memory holds, 24 for B = 64 and 12 for 128. (The largest box is
// 256 elements wide, so B = 256 stays with k_digest_any.) Measured, 205M tokens
// with B = 32: 138 us; two CTAs of 24 warps 142.6, three of 16 145, one of 28
// 144.6, two stages a warp 147 and more. 98M tokens with B = 16: 88 us, 90.6
// with two CTAs of 24. Routes of 2,466 requests of 17,144 tokens with B = 128:
// 79 us, 170 with k_digest_any.
constexpr int tma_warps(int HB) { return HB <= 16 ? 32 : HB <= 32 ? 24 : 12; }
// Copy stages per TMA digest warp. The kernel is written for any number: for one
// alone, without its loops over stages, ptxas took 32 to 36 registers instead of
// 40, and routes 274 us instead of 269 (8,192 requests, B = 32) and 399 instead
// of 289 (4,099 requests, N = 256, B = 16).
constexpr int kTmaStages = 1;
constexpr int kMatchWarps = 8;    // warps per walk CTA
constexpr int kGroupAhead = 8;    // 32-block rounds of digests a group warp compares at once

// ---------------------------------------------------------------------------
// prep
// ---------------------------------------------------------------------------

__device__ __forceinline__ int64_t warp_incl_scan(int64_t v, int lane) {
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    int64_t t = __shfl_up_sync(kFull, v, d);
    if (lane >= d) v += t;
  }
  return v;
}

constexpr int kPrepThreads = 1024;
constexpr int kPrepRounds = 8;  // rounds of 32 consecutive requests per warp
constexpr int kPrepPass = kPrepThreads * kPrepRounds;  // requests a CTA scans at a time
constexpr int64_t kPrepMaxCtas = 128;  // past 128 passes a CTA takes several

// CTA j scans the j-th stretch of requests (a pass of kPrepPass while there are
// no more than kPrepMaxCtas of them), after adding up the counts of all
// requests before it by itself: reading 8 bytes a request again costs less than
// waiting for another CTA, and what it costs is mostly the latency of a load.
// The last CTA has seen every request then: it alone checks the batch, writes
// the totals and the batch's flag. 32,768 requests: 16.5 us; 30 with one CTA
// that took its passes one after another.
inline int64_t prep_passes(int64_t n) {  // of one CTA
  const int64_t passes = std::max<int64_t>(1, (n + kPrepPass - 1) / kPrepPass);
  return (passes + kPrepMaxCtas - 1) / kPrepMaxCtas;
}
inline unsigned prep_grid(int64_t n) {
  const int64_t stretch = prep_passes(n) * kPrepPass;
  return (unsigned)std::max<int64_t>(1, (n + stretch - 1) / stretch);
}

__global__ void __launch_bounds__(kPrepThreads) k_prep(int passes, const int64_t* __restrict__ off, int32_t n,
                                              int64_t n_tokens, int B, const int64_t* __restrict__ load,
                                              int n_load, int64_t* __restrict__ block_off,
                                              int64_t* __restrict__ chunk_off, int32_t* batch_ok,
                                              int32_t* status, int64_t max_load, int64_t max_len,
                                              const int64_t* __restrict__ est_hit,
                                              const int64_t* __restrict__ aux0 = nullptr, int64_t aux0_max = 0,
                                              const int64_t* __restrict__ aux1 = nullptr, int64_t aux1_max = 0) {
  constexpr int NS = 2;  // scans: full blocks, and 32-block chunks (when chunk_off is wanted)
  constexpr int R = kPrepRounds;
  __shared__ int64_t warp_tot[NS][32], warp_before[NS][32];
  __shared__ int64_t pass_tot[NS];
  __shared__ int bad_all;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
  const bool last = blockIdx.x == gridDim.x - 1;
  if (tid == 0) bad_all = 0;
  __syncthreads();
  int bad = 0;  // bit 0: invalid offsets, bit 1: out-of-range length or load
  if (last) {
    for (int i = tid; i < n_load; i += blockDim.x) {
      const int64_t v = load[i];
      if (v < 0 || v > max_load) bad |= 2;
      if (aux0 && (aux0[i] < 0 || aux0[i] > aux0_max)) bad |= 2;  // further per-instance inputs
      if (aux1 && (aux1[i] < 0 || aux1[i] > aux1_max)) bad |= 2;
    }
    if (est_hit)  // the policy's expected hits, each in [0, 2^31)
      for (int64_t r = tid; r < n; r += blockDim.x) {
        const int64_t v = est_hit[r];
        if (v < 0 || v > (int64_t)INT32_MAX) bad |= 2;
      }
  }
  // full blocks of a request from its two offsets, and their checks
  auto blocks = [&](int64_t a, int64_t b) -> uint32_t {
    if (a < 0 || b < a || b > n_tokens) { bad |= 1; return 0; }
    if (b - a > max_len) { bad |= 2; return 0; }
    return (uint32_t)(b - a) / (uint32_t)B;
  };
  // A CTA gives each warp R rounds of 32 consecutive requests (lane = request),
  // so that offsets are loaded and both outputs stored coalesced. Every offset
  // of the pass is loaded before any is used; the counts stay in registers
  // between the warp sums and the scans that write the outputs.
  const int64_t start = (int64_t)blockIdx.x * passes * kPrepPass;
  int64_t before[NS] = {0, 0};  // this thread's share of the counts before the stretch
#pragma unroll 8
  for (int64_t r = tid; r < start; r += kPrepThreads) {
    const uint32_t nb = blocks(__ldg(off + r), __ldg(off + r + 1));
    before[0] += nb;
    before[1] += (nb + 31) >> 5;
  }
  for (int64_t first = start; first < start + (int64_t)passes * kPrepPass && (first == start || first < n);
       first += kPrepPass) {
    const int64_t seg = first + (int64_t)warp * 32 * R + lane;
    int64_t a[R], b[R];
#pragma unroll
    for (int i = 0; i < R; ++i) {
      const int64_t r = seg + 32 * i;
      a[i] = r < n ? off[r] : 0;
      b[i] = r < n ? off[r + 1] : 0;
    }
    uint32_t nbv[R];
#pragma unroll
    for (int i = 0; i < R; ++i) nbv[i] = seg + 32 * i < n ? blocks(a[i], b[i]) : 0;
    auto cnt = [&](int k, int i) -> int64_t { return k == 0 ? nbv[i] : (nbv[i] + 31) >> 5; };
#pragma unroll
    for (int k = 0; k < NS; ++k) {
      int64_t t = 0;
#pragma unroll
      for (int i = 0; i < R; ++i) t += cnt(k, i);
#pragma unroll
      for (int d = 16; d > 0; d >>= 1) t += __shfl_xor_sync(kFull, t, d);
      if (start > 0 && first == start) {
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) before[k] += __shfl_xor_sync(kFull, before[k], d);
      }
      if (lane == 0) {
        warp_tot[k][warp] = t;
        warp_before[k][warp] = before[k];
      }
    }
    __syncthreads();
    if (warp < NS) {  // warp k: scan k
      const int k = warp;
      const int64_t t = lane < nw ? warp_tot[k][lane] : 0;
      int64_t carry = first > start ? pass_tot[k] : lane < nw ? warp_before[k][lane] : 0;
      if (start > 0 && first == start) {
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) carry += __shfl_xor_sync(kFull, carry, d);
      }
      __syncwarp();
      const int64_t ti = warp_incl_scan(t, lane);
      if (lane < nw) warp_tot[k][lane] = carry + ti - t;  // exclusive
      if (lane == 31) pass_tot[k] = carry + ti;
    }
    __syncthreads();
    // both scans side by side, so that their shuffle chains overlap; rounds
    // past the last request are skipped (the test is warp-uniform)
    int64_t run[NS];
#pragma unroll
    for (int k = 0; k < NS; ++k) run[k] = warp_tot[k][warp];  // this warp's exclusive start
#pragma unroll
    for (int i = 0; i < R; ++i) {
      if (seg - lane + 32 * i >= n) break;
      const int64_t r = seg + 32 * i;
      const int64_t c0 = cnt(0, i), c1 = cnt(1, i);
      const int64_t i0 = warp_incl_scan(c0, lane), i1 = warp_incl_scan(c1, lane);
      if (r < n) {
        block_off[r] = run[0] + i0 - c0;
        if (chunk_off) chunk_off[r] = run[1] + i1 - c1;
      }
      run[0] += __shfl_sync(kFull, i0, 31);
      run[1] += __shfl_sync(kFull, i1, 31);
    }
    __syncthreads();  // warp_tot is rewritten by the next pass
  }
  if (bad) atomicOr(&bad_all, bad);
  __syncthreads();
  if (last && tid == 0) {
    block_off[n] = pass_tot[0];
    if (chunk_off) chunk_off[n] = pass_tot[1];
    const int ba = bad_all;
    *batch_ok = ba == 0;
    if (ba & 1) latch_error(status, SMETRIC_ERR_INVALID_ARG);
    else if (ba & 2) latch_error(status, SMETRIC_ERR_OVERFLOW);
  }
}

// ---------------------------------------------------------------------------
// digest
// ---------------------------------------------------------------------------

// The group stage works from the digests, so that it needs no finished chain:
// a request's first-block hash h_0 = chain_step(h_init, its first digest) is the
// group key, and the shared-prefix length is the number of leading blocks
// whose digests equal the leader's. Equal digests from equal previous hashes
// give equal hashes, so the leader's masks serve those blocks exactly.
//
// A stored digest is d_b ^ (d_b >> 30): the chain's first xor-shift
// x ^ (x >> 30) is linear over xor, so the digest's share of it is taken here,
// off the chain's serial path (a bijection, so equal words are equal digests).
__device__ __forceinline__ uint64_t stored_digest(uint64_t d) { return d ^ (d >> 30); }

// h_b before the sentinel remap, from h_{b-1} and the stored digest of block b:
// mix64((h_{b-1} + kGamma) ^ d_b) on 32-bit halves, for the serial chain where
// only latency counts. The high word of each product is the low-by-low high
// half plus the two cross products, the second accumulated onto the first.
__device__ __forceinline__ uint64_t chain_raw(uint64_t hp, uint64_t ds) {
  const uint64_t a = hp + kGamma;
  uint32_t lo = (uint32_t)a, hi = (uint32_t)(a >> 32);
  auto mul = [&](uint64_t c) {
    const uint32_t cl = (uint32_t)c, ch = (uint32_t)(c >> 32);
    const uint32_t x = hi * cl + lo * ch;
    hi = __umulhi(lo, cl) + x;
    lo = lo * cl;
  };
  auto xs = [&](int n, uint32_t xl, uint32_t xh) {
    lo ^= __funnelshift_r(lo, hi, n) ^ xl;
    hi ^= (hi >> n) ^ xh;
  };
  xs(30, (uint32_t)ds, (uint32_t)(ds >> 32));
  mul(0xBF58476D1CE4E5B9ull);
  xs(27, 0, 0);
  mul(0x94D049BB133111EBull);
  xs(31, 0, 0);
  return ((uint64_t)hi << 32) | lo;
}

// One chain step with the sentinel remap.
__device__ __forceinline__ uint64_t chain_step(uint64_t hp, uint64_t ds) {
  const uint64_t h = chain_raw(hp, ds);
  return h < 2 ? (h | 2) : h;
}

// Requests whose first block hashes are equal form a group; its leader is
// the lowest request id. Table of (key, INT32_MAX - leader) word pairs,
// key 0 = empty (block hashes are >= 2), linear probing, at most half full.
__device__ __forceinline__ void group_insert(uint64_t* __restrict__ groups, uint64_t gmask, uint64_t key,
                                             int32_t r) {
  uint64_t s = key & gmask;
  for (uint64_t t = 0; t <= gmask; ++t) {
    unsigned long long* const slot = reinterpret_cast<unsigned long long*>(groups + 2 * s);
    const unsigned long long k = atomicCAS(slot, 0ull, (unsigned long long)key);
    if (k == 0ull || k == key) {
      atomicMax(slot + 1, (unsigned long long)(INT32_MAX - r));
      return;
    }
    s = (s + 1) & gmask;
  }
}

// request_of by a whole warp (f warp-uniform), 32 points a step: two or three
// dependent loads instead of up to fifteen.
__device__ __forceinline__ int32_t request_of_warp(const int64_t* __restrict__ block_off, int32_t lo, int32_t n,
                                                     int64_t f) {
  const int lane = threadIdx.x & 31;
  int32_t hi = n;
  while (hi - lo > 1) {
    const int32_t step = (hi - lo + 31) / 32;
    const int64_t at = (int64_t)lo + (int64_t)lane * step;
    const unsigned m = __ballot_sync(kFull, at < hi && __ldg(block_off + at) <= f);  // a prefix of the lanes, lane 0 in it
    const int last = 31 - __clz(m);
    hi = (int32_t)min((int64_t)hi, (int64_t)lo + (int64_t)(last + 1) * step);
    lo += last * step;
  }
  return lo;
}

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// Digest of one block from its shared-memory row. `row` points at the 8-byte
// word holding the block's first token (its low half when the block starts on
// an even token, its high half when on an odd one).
template <int HB>
__device__ __forceinline__ uint64_t digest_row(const uint64_t* row, bool odd, int hb, uint64_t d) {
  const int n = HB > 0 ? HB : hb;
  if (!odd) {
#pragma unroll 16
    for (int k = 0; k < n; ++k) d = mix64(d ^ row[k]);
  } else {
    uint64_t x = row[0];
#pragma unroll 16
    for (int k = 0; k < n; ++k) {
      const uint64_t y = row[k + 1];
      d = mix64(d ^ ((x >> 32) | (y << 32)));
      x = y;
    }
  }
  return d;
}

// 16 bytes of the token buffer at byte offset `a`, of which only the first
// `avail` bytes (a multiple of 4) are read when fewer than 16 remain.
__device__ __forceinline__ uint4 load_piece(const char* base, int64_t a, int64_t avail) {
  if (avail >= 16) return __ldg(reinterpret_cast<const uint4*>(base + a));
  uint32_t w[4] = {0, 0, 0, 0};
#pragma unroll
  for (int q = 0; q < 4; ++q)
    if (4 * q < avail) w[q] = __ldg(reinterpret_cast<const uint32_t*>(base + a) + q);
  return make_uint4(w[0], w[1], w[2], w[3]);
}

// Row layout shared by both digest kernels: row j holds the bytes of block j
// rounded out to 16-byte boundaries, [a_j, a_j + 16*NP) with
// a_j = (4*first token) & ~15, so lane j reading word k of its own block hits
// bank group (row stride * j + 8k) mod 128 and rows of 16*NP bytes keep the
// 32 lanes spread over the banks.

// B = 2*HB with B % 4 == 0 (HB even). A chunk whose 32 blocks belong to one
// request is one contiguous byte span; the warp loads it with coalesced
// 16-byte loads (piece p = lane + 32 i) into registers one chunk ahead, and
// scatters each piece into the row(s) that contain it: piece p lies in row
// p / PB and, when it starts a block, also ends row p / PB - 1.
template <int HB>
__global__ void __launch_bounds__(kDigestWarps * 32)
    k_digest(const int32_t* __restrict__ tokens, int64_t n_tokens, const int64_t* __restrict__ off,
             const int64_t* __restrict__ block_off, int32_t n, uint64_t d_init,
             const int32_t* __restrict__ batch_ok, uint64_t* __restrict__ digest,
             uint64_t* __restrict__ groups, uint64_t gmask, uint64_t h_init) {
  pdl_enter();
  constexpr int B = 2 * HB;
  constexpr int PB = HB > 0 ? HB / 2 : 1;  // 16-byte pieces per block (k_digest<0> is never launched)
  constexpr int NP = PB + 1;  // pieces per row (the block plus its misalignment)
  extern __shared__ uint4 dsm[];
  if (!*batch_ok) return;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, warps = blockDim.x >> 5;
  const int64_t total = block_off[n];
  const int64_t n_chunks = (total + kChunk - 1) / kChunk;
  const int64_t tw = (int64_t)gridDim.x * warps;
  const int64_t per = (n_chunks + tw - 1) / tw;
  const int64_t c_lo = ((int64_t)blockIdx.x * warps + warp) * per;
  const int64_t c_hi = min(n_chunks, c_lo + per);
  if (c_lo >= c_hi) return;
  uint4* const st = dsm + (size_t)warp * kChunk * NP;
  const int64_t token_bytes = 4 * n_tokens;
  const char* const tb = reinterpret_cast<const char*>(tokens);

  int32_t r = request_of(block_off, 0, n, min(c_lo * kChunk + lane, total - 1));

  struct Chunk {
    int64_t tok0;  // this lane's first token
    int64_t a0;    // byte offset of piece 0 (fast path)
    int nv;        // valid lanes (a prefix of the warp)
    int32_t req;   // this lane's request
    bool valid, fast, head;  // head: the lane's block is its request's block 0
  };
  uint4 buf[NP];
  // locate chunk c and load its bytes into registers
  auto load = [&](int64_t c, Chunk& ch) {
    const int64_t f = c * kChunk + lane;
    ch.valid = f < total;
    ch.head = false;
    ch.req = r;
    if (ch.valid) {
      if (__ldg(block_off + r + 1) <= f) r = request_of(block_off, r + 1, n, f);
      ch.tok0 = __ldg(off + r) + (f - __ldg(block_off + r)) * B;
      ch.head = f == __ldg(block_off + r);
      ch.req = r;
    } else {
      ch.tok0 = 0;
    }
    ch.nv = __popc(__ballot_sync(kFull, ch.valid));
    const int32_t r0 = __shfl_sync(kFull, r, 0);
    ch.a0 = (4 * __shfl_sync(kFull, ch.tok0, 0)) & ~(int64_t)15;
    const int npieces = ch.nv * PB + 1;
    ch.fast = __all_sync(kFull, !ch.valid || r == r0) && ch.a0 + 16 * (int64_t)npieces <= token_bytes;
    if (ch.fast) {
#pragma unroll
      for (int i = 0; i < NP; ++i) {
        const int p = lane + 32 * i;
        if (p < npieces) buf[i] = __ldg(reinterpret_cast<const uint4*>(tb + ch.a0) + p);
      }
    } else if (ch.valid) {
      const int64_t a = (4 * ch.tok0) & ~(int64_t)15;
#pragma unroll
      for (int i = 0; i < NP; ++i) buf[i] = load_piece(tb, a + 16 * i, token_bytes - (a + 16 * i));
    }
  };
  auto store = [&](const Chunk& ch) {
    if (ch.fast) {
      const int npieces = ch.nv * PB + 1;
#pragma unroll
      for (int i = 0; i < NP; ++i) {
        const int p = lane + 32 * i;
        if (p < npieces) {
          const int j = p / PB, q = p - j * PB;
          if (j < ch.nv) st[j * NP + q] = buf[i];
          if (q == 0 && j >= 1) st[(j - 1) * NP + PB] = buf[i];
        }
      }
    } else if (ch.valid) {
#pragma unroll
      for (int i = 0; i < NP; ++i) st[lane * NP + i] = buf[i];
    }
  };

  Chunk cur, nxt;
  load(c_lo, cur);
  for (int64_t c = c_lo; c < c_hi; ++c) {
    store(cur);
    __syncwarp();
    if (c + 1 < c_hi) load(c + 1, nxt);  // in flight during this chunk's arithmetic
    if (cur.valid) {
      const int delta = (int)((cur.tok0 * 4) & 15);  // 0, 4, 8 or 12
      const uint64_t* row = reinterpret_cast<const uint64_t*>(st + lane * NP) + (delta >> 3);
      const uint64_t d = stored_digest(digest_row<HB>(row, (delta & 4) != 0, HB, d_init));
      digest[c * kChunk + lane] = d;
      if (groups && cur.head) group_insert(groups, gmask, chain_step(h_init, d), cur.req);
    }
    __syncwarp();
    cur = nxt;
  }
}

// ---- TMA tensor path -------------------------------------------------------
//
// For B % 4 == 0, block j of a request starts 4B*j bytes after block 0, so the
// rows a_j = (4*first token of block j) & ~15 of one request form a strided
// 2D region: rows of 4B+16 bytes at stride 4B. A 2D tensor map with row stride
// 4B lets one TMA tile load of 32 rows bring a whole chunk into the padded
// layout. Up to B = 64 there is a map per 16-byte phase k of a_0 (base = tokens +
// 16k, rows of 4B+16 bytes). For B = 128, rows of 8B bytes serve every phase, at
// column 16k: one map from the buffer's start, and one whose rows end with the
// buffer, for the chunk that the first one's last rows do not reach. (With 32
// maps a call took 2.2 us more on the host; without the second, batches of 235
// requests 1 us more, for their last chunk's lane copies; with such maps at B =
// 32 the digest of 205M tokens 1.4 us more.)
// Every row of a map lies inside the token buffer; rows past its end are
// zero-filled by the TMA unit, and a chunk that needs such a row is copied by its
// lanes instead.

constexpr uint32_t kSpinLimit = 1u << 22;  // bounded mbarrier waits

template <int HB>
struct TokenMaps {
  static constexpr int kPhases = HB > 0 ? HB / 2 : 1;  // 4B / 16
  static constexpr bool kWide = kPhases > 16;  // two maps for every phase
  static constexpr int kMaps = kWide ? 2 : kPhases;
  CUtensorMap map[kMaps];
  uint32_t rows[kMaps];  // rows addressable through map k
  uint32_t base[kMaps];  // its first byte in the token buffer
};

__device__ __forceinline__ void mbar_init(uint32_t mbar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(mbar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint32_t mbar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(mbar), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t mbar, uint32_t parity) {
  uint32_t done;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(done) : "r"(mbar), "r"(parity) : "memory");
  return done != 0;
}
// Bounded wait for the phase with the given parity; false on timeout.
__device__ __forceinline__ bool mbar_wait(uint32_t mbar, uint32_t parity) {
  for (uint32_t i = 0; i < kSpinLimit; ++i)
    if (mbar_try_wait(mbar, parity)) return true;
  return false;
}
__device__ __forceinline__ void tma_rows(uint32_t dst, const CUtensorMap* map, int32_t x, int32_t y, uint32_t mbar,
                                         uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.L2::cache_hint"
      " [%0], [%1, {%2, %3}], [%4], %5;\n" ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(x),
      "r"(y), "r"(mbar), "l"(policy)
      : "memory");
}

template <int HB, int STAGES>
__global__ void __launch_bounds__(tma_warps(HB) * 32)
    k_digest_tma(const __grid_constant__ TokenMaps<HB> maps, const int32_t* __restrict__ tokens,
                 int64_t n_tokens, const int64_t* __restrict__ off, const int64_t* __restrict__ block_off,
                 const int64_t* __restrict__ chunk_off, int32_t n, uint64_t d_init, const int32_t* __restrict__ batch_ok,
                 uint64_t* __restrict__ digest, int32_t* status, uint64_t* __restrict__ groups, uint64_t gmask,
                 uint64_t h_init) {
  pdl_enter();
  constexpr int B = 2 * HB;
  constexpr int NP = HB / 2 + 1;           // 16-byte pieces per row
  constexpr uint32_t ROW = 16u * NP;       // = 4B + 16
  constexpr uint32_t STAGE = kChunk * ROW;
  extern __shared__ __align__(128) unsigned char dsm_raw[];
  if (!*batch_ok) return;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, warps = blockDim.x >> 5;
  // chunk c is chunk q of request r: its blocks 32q .. 32q+31, so a chunk
  // never spans two requests
  const int64_t n_chunks = chunk_off[n];
  // A CTA takes a contiguous range of chunks and its warps interleave over it
  // (warp w: chunks w, w + warps, ...), so that the copies a CTA has in flight
  // cover one stretch of consecutive tokens.
  const int64_t per = (n_chunks + gridDim.x - 1) / gridDim.x;  // chunks per CTA
  const int64_t k_lo = (int64_t)blockIdx.x * per;
  const int64_t c_hi = min(n_chunks, k_lo + per);
  const int64_t c_lo = k_lo + warp;  // then every warps-th chunk of the CTA's range
  if (c_lo >= c_hi) return;
  unsigned char* const stages = dsm_raw + (size_t)warp * STAGES * STAGE;
  const uint32_t mbar0 = smem_u32(dsm_raw + (size_t)warps * STAGES * STAGE) + 8u * STAGES * (uint32_t)warp;
  if (lane == 0) {
#pragma unroll
    for (int s = 0; s < STAGES; ++s) mbar_init(mbar0 + 8u * s, 1);
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  __syncwarp();
  uint64_t policy;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;\n" : "=l"(policy));
  const int64_t token_bytes = 4 * n_tokens;
  const char* const tb = reinterpret_cast<const char*>(tokens);
  int32_t r = request_of_warp(chunk_off, 0, n, c_lo);

  // Start the copy of chunk c into stage s; returns this lane's first token
  // and sets its digest index and its request (`head` when the lane has the
  // request's block 0, whose digest also gives the request's group key).
  auto issue = [&](int64_t c, int s, bool& valid, int64_t& gidx, int32_t& req, bool& head) -> int64_t {
    for (int i = 0; i < 4 && __ldg(chunk_off + r + 1) <= c; ++i) ++r;  // usually a step or two
    if (__ldg(chunk_off + r + 1) <= c) r = request_of(chunk_off, r + 1, n, c);
    const int64_t bo = __ldg(block_off + r), nbr = __ldg(block_off + r + 1) - bo;
    const int64_t b = (c - __ldg(chunk_off + r)) * kChunk + lane;  // block of request r
    valid = b < nbr;
    const int64_t tok0 = __ldg(off + r) + b * B;
    gidx = bo + b;
    req = r;
    head = b == 0;
    const int nv = (int)min((int64_t)kChunk, nbr - (b - lane));
    const int64_t a0 = (4 * __shfl_sync(kFull, tok0, 0)) & ~(int64_t)15;
    int k = (int)((a0 % (4 * B)) >> 4), x = 0;  // map, and column (in tokens, a multiple of 16 bytes)
    int64_t y0 = a0 / (4 * B);
    if constexpr (TokenMaps<HB>::kWide) {
      x = 4 * k;
      k = 0;
      if (y0 + nv > (int64_t)maps.rows[0] && a0 >= (int64_t)maps.base[1]) {
        const uint64_t e = (uint64_t)a0 - maps.base[1];
        k = 1;
        x = (int)((uint32_t)e % (4 * B)) >> 2;
        y0 = (int64_t)(e / (4 * B));
      }
    }
    unsigned char* const st = stages + (size_t)s * STAGE;
    const uint32_t mbar = mbar0 + 8u * (uint32_t)s;
    if (y0 + nv <= (int64_t)maps.rows[k]) {
      if (lane == 0) {
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
        mbar_arrive_expect_tx(mbar, STAGE);
        tma_rows(smem_u32(st), &maps.map[k], x, (int32_t)y0, mbar, policy);
      }
    } else {
      // lanes copy their own rows; the stage's barrier completes on lane 0's
      // arrival with no bytes expected
      if (valid) {
        const int64_t a = (4 * tok0) & ~(int64_t)15;
        uint4* row = reinterpret_cast<uint4*>(st + lane * ROW);
#pragma unroll
        for (int i = 0; i < NP; ++i) row[i] = load_piece(tb, a + 16 * i, token_bytes - (a + 16 * i));
      }
      __syncwarp();
      if (lane == 0) mbar_arrive_expect_tx(mbar, 0);
    }
    return tok0;
  };

  uint32_t phase = 0;
  bool failed = false;
  bool v[STAGES], hd[STAGES];
  int64_t t[STAGES], gi[STAGES];
  int32_t rq[STAGES];
#pragma unroll
  for (int s = 0; s < STAGES; ++s)
    if (c_lo + s * warps < c_hi) t[s] = issue(c_lo + s * warps, s, v[s], gi[s], rq[s], hd[s]);
  int s = 0;
  for (int64_t c = c_lo; c < c_hi; c += warps) {
    if (!mbar_wait(mbar0 + 8u * (uint32_t)s, (phase >> s) & 1)) { failed = true; break; }
    phase ^= 1u << s;
    bool vc = false, hc = false;
    int64_t tc = 0, gc = 0;
    int32_t rc = 0;
#pragma unroll
    for (int q = 0; q < STAGES; ++q) if (q == s) { vc = v[q]; tc = t[q]; gc = gi[q]; rc = rq[q]; hc = hd[q]; }
    if (vc) {
      const int delta = (int)((tc * 4) & 15);  // 0, 4, 8 or 12
      const uint64_t* row = reinterpret_cast<const uint64_t*>(stages + (size_t)s * STAGE + lane * ROW) + (delta >> 3);
      const uint64_t d = stored_digest(digest_row<HB>(row, (delta & 4) != 0, HB, d_init));
      digest[gc] = d;
      if (groups && hc) group_insert(groups, gmask, chain_step(h_init, d), rc);
    }
    __syncwarp();
    if (c + STAGES * warps < c_hi) {
      bool vn, hn;
      int64_t gn = 0;
      int32_t rn = 0;
      const int64_t tn = issue(c + STAGES * warps, s, vn, gn, rn, hn);
#pragma unroll
      for (int q = 0; q < STAGES; ++q) if (q == s) { v[q] = vn; t[q] = tn; gi[q] = gn; rq[q] = rn; hd[q] = hn; }
    }
    s = s + 1 == STAGES ? 0 : s + 1;
  }
  if (failed) {
    // a copy never completed: report it and give copies in flight a bounded
    // chance to land before the shared memory is released
    if (lane == 0) latch_error(status, SMETRIC_ERR_CUDA);
#pragma unroll
    for (int q = 0; q < STAGES; ++q) mbar_wait(mbar0 + 8u * q, (phase >> q) & 1);
  }
}

// Any even B: each lane copies its own row straight from global memory.
__global__ void __launch_bounds__(kDigestWarps * 32)
    k_digest_any(const int32_t* __restrict__ tokens, int64_t n_tokens, const int64_t* __restrict__ off,
                 const int64_t* __restrict__ block_off, int32_t n, int B, int nch, uint64_t d_init,
                 const int32_t* __restrict__ batch_ok, uint64_t* __restrict__ digest,
                 uint64_t* __restrict__ groups, uint64_t gmask, uint64_t h_init) {
  pdl_enter();
  extern __shared__ uint4 dsm[];
  if (!*batch_ok) return;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, warps = blockDim.x >> 5;
  const int64_t total = block_off[n];
  const int64_t n_chunks = (total + kChunk - 1) / kChunk;
  const int64_t tw = (int64_t)gridDim.x * warps;
  const int64_t per = (n_chunks + tw - 1) / tw;
  const int64_t c_lo = ((int64_t)blockIdx.x * warps + warp) * per;
  const int64_t c_hi = min(n_chunks, c_lo + per);
  if (c_lo >= c_hi) return;
  uint4* const row = dsm + ((size_t)warp * kChunk + lane) * nch;
  const int64_t token_bytes = 4 * n_tokens;
  const char* const tb = reinterpret_cast<const char*>(tokens);
  int32_t r = request_of(block_off, 0, n, min(c_lo * kChunk + lane, total - 1));
  for (int64_t c = c_lo; c < c_hi; ++c) {
    const int64_t f = c * kChunk + lane;
    if (f >= total) continue;
    if (__ldg(block_off + r + 1) <= f) r = request_of(block_off, r + 1, n, f);
    const int64_t tok0 = __ldg(off + r) + (f - __ldg(block_off + r)) * B;
    const int64_t a = (4 * tok0) & ~(int64_t)15;
    for (int i = 0; i < nch; ++i) row[i] = load_piece(tb, a + 16 * i, token_bytes - (a + 16 * i));
    const int delta = (int)((tok0 * 4) & 15);
    const uint64_t d = stored_digest(digest_row<0>(reinterpret_cast<const uint64_t*>(row) + (delta >> 3),
                                                   (delta & 4) != 0, B >> 1, d_init));
    digest[f] = d;
    if (groups && f == __ldg(block_off + r)) group_insert(groups, gmask, chain_step(h_init, d), r);
  }
}

// ---------------------------------------------------------------------------
// match
// ---------------------------------------------------------------------------

// Tier masks of key h (zeros when absent) from the read-only table: the home
// bucket's 15 tags, then the entry of each tag match, then later buckets while
// the bucket just read has keys stored past it (its overflow count).
template <int W>
__device__ __forceinline__ void probe_one(const uint8_t* __restrict__ tags, const uint64_t* __restrict__ table,
                                          uint64_t n_buckets, uint64_t h, uint64_t (&M)[W]) {
  constexpr int EW = entry_words(W);
  constexpr int NV = (W + 2) / 2;  // 16-byte loads covering key + W mask words
#pragma unroll
  for (int w = 0; w < W; ++w) M[w] = 0;
  const uint32_t tg = key_tag(h);
  uint64_t b = home_bucket(h, n_buckets);
  const uint64_t mb = max_buckets(n_buckets);
  for (uint64_t t = 0; t < mb; ++t) {
    const uint4 tv = __ldg(reinterpret_cast<const uint4*>(tags + b * kBucket));
    uint32_t cand = slot_match(tv, tg);
    while (cand) {
      const int sl = next_slot(cand);
      const ulonglong2* e = reinterpret_cast<const ulonglong2*>(table + (b * kSlots + sl) * EW);
      ulonglong2 v[NV];
#pragma unroll
      for (int q = 0; q < NV; ++q) v[q] = __ldg(e + q);
      if (v[0].x == h) {
#pragma unroll
        for (int w = 0; w < W; ++w) M[w] = (w & 1) ? v[(w + 1) >> 1].x : v[(w + 1) >> 1].y;
        return;
      }
    }
    if (overflow_count(tv) == 0) return;
    if (++b == n_buckets) b = 0;
  }
}

// ---------------------------------------------------------------------------
// chain, shared prefix and probe in one kernel
// ---------------------------------------------------------------------------
//
// The chain is bound by the latency of its dependent steps and the probe by
// random memory accesses, so one kernel runs both at once: one CTA of
// kCpWarps warps per SM. Chain warps (lane = request, warps 0 ..
// chain_warps - 1, one per scheduler) only turn digests into hashes, in place
// in a ring of 32-block chunks in shared memory; every other access is a probe
// warp's. Why the ring: a chain step's own latency is ~75 cycles, any number
// of chain warps up to one per scheduler, but ~147 with four chain warps that
// store their hashes per lane to global memory (32 sectors an instruction).
// Measured, N = 64, B = 32, 24k tokens a prompt: a step takes 88 cycles with few
// requests an SM and ~140 beside the probes of 8,192 requests (before: 145 and
// ~205); the kernel 31 us instead of 46 for 16 requests, 53 instead of 83 for
// 777, 99 instead of 138 for 8,192 and 245 instead of 460 for 32,768, where
// 6.4M probes at 29 G/s are what random reads allow.
//
// Lane j of the CTA chains a stream of requests, one after another; position q
// of the stream is a 32-block chunk of one of them, kept in slot q mod slots
// of lane j's part of the ring. Item (q, j), taken by the probe warps in
// position-major order: once the chain warp has chained position q, read its
// hashes, put the digests of position q + slots into the slot, then probe the
// index with the hashes, store masks and the chunk's AND, and (where wanted)
// store the hashes, coalesced. Two mbarriers per chain warp and slot carry the
// order: `full` (one arrival per lane in use) and `ready` (the chain warp's).
// A slot's barriers cannot run ahead of an item that still waits, since its
// own refill is one of the arrivals that the next phase needs; an item taken
// more than `slots` positions ahead first polls the chain warp's position
// counter, so that the parity it then waits for is that of its own phase.
//
// Chunk q of request r is its blocks 32q .. 32q + 31; the chunk ANDs the walk reads are kept per such
// request-aligned chunk, at index chunk_off[r] + q.
constexpr int kCpWarps = 32;
// Without an index (32 requests an SM at most: one chain warp). 4,096 prompts of
// 750 blocks: 45.6 us, with 24 warps 48.7, with 32 49.7; 1,024 prompts 40.2, 41.2, 41.2.
constexpr int kHashWarps = 16;
__host__ __device__ constexpr int cp_warps(int W) { return W == 0 ? kHashWarps : kCpWarps; }
constexpr int kCpMaxChainWarps = 4;  // warps 0 .. 3, one per scheduler
constexpr int kCpMaxLanes = 32 * kCpMaxChainWarps;
// Bytes of a slot: 32 words, and 16 bytes that make the distance between the
// lanes' rows of one slot an odd number of 16-byte units, so that a chain
// warp's 16-byte accesses meet no bank conflict.
constexpr int kCpRow = 272;
constexpr int kCpMaxSlots = 8;       // 8 with one or two chain warps, 4 with more
constexpr size_t kCpMaxRing = (size_t)kCpMaxLanes * (kCpMaxSlots / 2) * kCpRow;  // 139,264 bytes, and with two warps too
constexpr int kCpRound = 512;        // requests a CTA takes at a time

__device__ __forceinline__ void mbar_arrive(uint32_t mbar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(mbar) : "memory");
}

// Bounded poll until a chain warp's position counter reaches v (which only says
// which phase its barriers are in: the barriers order the data); positions
// take about a microsecond each, so the sleep grows with the distance.
__device__ __forceinline__ bool poll_at_least(const int32_t* p, int32_t v, volatile int* failed) {
  bool ok = false;
  for (uint32_t i = 0; i < kSpinLimit; ++i) {
    const int32_t at = *reinterpret_cast<const volatile int32_t*>(p);
    ok = at >= v;
    if (ok || ((i & 15) == 15 && *failed)) break;
    __nanosleep(400u * (uint32_t)min(v - at, 8));
  }
  ok = __all_sync(kFull, ok);
  if (!ok) *failed = 1;
  return ok;
}

// As mbar_try_wait, suspended for up to `ns` (a hint) before it answers no: a
// warp that asks again and again takes issue slots from the chain warps.
__device__ __forceinline__ bool mbar_try_wait_for(uint32_t mbar, uint32_t parity, uint32_t ns) {
  uint32_t done;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n"
      " selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(done) : "r"(mbar), "r"(parity), "r"(ns) : "memory");
  return done != 0;
}

// A warp's bounded wait for a phase; false when it gave up, or when another warp of the
// CTA did (*failed), after which every wait of the CTA ends at once.
__device__ __forceinline__ bool mbar_wait_or(uint32_t mbar, uint32_t parity, volatile int* failed) {
  bool ok = false;
  for (uint32_t i = 0; i < kSpinLimit; ++i) {
    ok = mbar_try_wait_for(mbar, parity, 4000);
    if (ok || ((i & 15) == 15 && *failed)) break;
  }
  ok = __all_sync(kFull, ok);  // the warp goes on together
  if (!ok) *failed = 1;
  return ok;
}

// Eight chain steps: digests c in, hashes to o (which may be where c came from).
template <bool EXACT>
__device__ __forceinline__ uint64_t chain8(uint64_t h, const ulonglong2 (&c)[4], ulonglong2* o) {
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const uint64_t x = EXACT ? chain_step(h, c[i].x) : chain_raw(h, c[i].x);
    h = EXACT ? chain_step(x, c[i].y) : chain_raw(x, c[i].y);
    o[i] = make_ulonglong2(x, h);
  }
  return h;
}

__device__ __forceinline__ void load8(ulonglong2 (&c)[4], const ulonglong2* p) {
#pragma unroll
  for (int i = 0; i < 4; ++i) c[i] = p[i];
}

// Tier masks of a warp's keys, one per lane: the home-bucket tags, then the
// tag matches' entries in turn for the whole warp (the first is the key's own
// for all but ~4 % of the keys held), then probe_one for a key not in its
// home bucket where that has keys stored past it.
template <int W>
__device__ __forceinline__ void probe_warp(const uint8_t* __restrict__ tags, const uint64_t* __restrict__ table,
                                           uint64_t n_buckets, bool act, uint64_t h, uint64_t (&M)[W]) {
  constexpr int EW = entry_words(W);
  constexpr int NV = (W + 2) / 2;
  const uint64_t bk = home_bucket(h, n_buckets);
  uint4 tv = make_uint4(0, 0, 0, 0);
  if (act) tv = __ldg(reinterpret_cast<const uint4*>(tags + bk * kBucket));
  uint32_t cand = act ? slot_match(tv, key_tag(h)) : 0;
  bool found = false;
#pragma unroll
  for (int w = 0; w < W; ++w) M[w] = 0;
  while (__any_sync(kFull, cand != 0)) {
    if (cand) {
      const ulonglong2* e = reinterpret_cast<const ulonglong2*>(table + (bk * kSlots + next_slot(cand)) * EW);
      ulonglong2 v[NV];
#pragma unroll
      for (int q = 0; q < NV; ++q) v[q] = __ldg(e + q);
      if (v[0].x == h) {
#pragma unroll
        for (int w = 0; w < W; ++w) M[w] = (w & 1) ? v[(w + 1) >> 1].x : v[(w + 1) >> 1].y;
        found = true;
        cand = 0;
      }
    }
  }
  if (act && !found && overflow_count(tv) != 0) probe_one<W>(tags, table, n_buckets, h, M);
  __syncwarp();
}

// The group stage, a warp per request: its leader (the lowest request with the
// same first block, from the group table), the shared prefix (leading blocks
// with the leader's digests) and whether the chain kernel takes the request.
// With `defer`, a member with a short tail past its shared prefix is left to
// the walk kernel, which chains only the tail, from the leader's hash: the
// chain kernel then has the leaders and a few others.
constexpr int kDeferTail = 256;  // blocks; the walk's steps take ~100 cycles each
// The line: with four or fewer requests an SM nothing is deferred; with more, a
// tail of a quarter of the prompt at most. 8,192 requests of the burst trace:
// k_lead 14 us instead of 4, the chain kernel 99 instead of 165 (all requests
// chained there), the walk 18.5 instead of 15.7.
__device__ __forceinline__ bool short_tail(int64_t nb, int64_t sh) {
  return nb - sh <= kDeferTail && 4 * (nb - sh) <= nb;
}

__global__ void __launch_bounds__(256)
    k_lead(const int64_t* __restrict__ block_off, int32_t n, const int32_t* __restrict__ batch_ok,
           const uint64_t* __restrict__ D, uint64_t h_init, const uint64_t* __restrict__ groups, uint64_t gmask,
           bool defer, int32_t* __restrict__ lead, int32_t* __restrict__ share, uint8_t* __restrict__ active) {
  pdl_enter();
  const int32_t r = (int32_t)((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5);
  const int lane = threadIdx.x & 31;
  if (r >= n || !*batch_ok) return;
  const int64_t bo = __ldg(block_off + r), nb = __ldg(block_off + r + 1) - bo;
  int32_t l = r;
  int64_t sh = 0;
  // the request's own leading digests, on their way while its leader is sought
  uint64_t own[kGroupAhead];
#pragma unroll
  for (int u = 0; u < kGroupAhead; ++u) own[u] = 32 * u + lane < nb ? __ldg(D + bo + 32 * u + lane) : 0;
  if (nb > 0) {
    const uint64_t key = chain_step(h_init, __shfl_sync(kFull, own[0], 0));
    const uint64_t s0 = key & gmask;
    for (uint64_t t = 0; t <= gmask; t += 32) {
      const uint64_t sl = (s0 + t + lane) & gmask;
      const ulonglong2 e = *reinterpret_cast<const ulonglong2*>(groups + 2 * sl);
      const unsigned hit = __ballot_sync(kFull, e.x == key), stop = hit | __ballot_sync(kFull, e.x == 0);
      if (stop) {
        const int first = __ffs(stop) - 1;
        const int32_t who = __shfl_sync(kFull, INT32_MAX - (int32_t)e.y, first);
        if (hit & (1u << first)) l = who;
        break;
      }
    }
    if (l != r && l >= 0 && l < n) {
      const int64_t lo = __ldg(block_off + l), nl = __ldg(block_off + l + 1) - lo;
      const int64_t m = nb < nl ? nb : nl;
      sh = m;
      for (int64_t b = 0; b < m; b += 32 * kGroupAhead) {
        bool ne[kGroupAhead];
        uint64_t other[kGroupAhead];
#pragma unroll
        for (int u = 0; u < kGroupAhead; ++u) {
          const int64_t bb = b + 32 * u + lane;
          other[u] = bb < m ? __ldg(D + lo + bb) : 0;
          if (b > 0) own[u] = bb < m ? __ldg(D + bo + bb) : 0;
        }
#pragma unroll
        for (int u = 0; u < kGroupAhead; ++u) ne[u] = b + 32 * u + lane < m && own[u] != other[u];
        int64_t first = -1;
#pragma unroll
        for (int u = 0; u < kGroupAhead; ++u) {
          const unsigned x = __ballot_sync(kFull, ne[u]);
          if (x && first < 0) first = 32 * u + __ffs(x) - 1;
        }
        if (first >= 0) {
          sh = b + first;
          break;
        }
      }
    } else {
      l = r;
    }
  }
  if (lane == 0) {
    lead[r] = l;
    share[r] = (int32_t)sh;
    active[r] = !(defer && sh > 0 && short_tail(nb, sh));
  }
}

struct ChainArgs {
  const int64_t* block_off;
  const int64_t* chunk_off;
  int32_t n;
  int S;
  uint64_t h_init;
  const int32_t* batch_ok;
  const uint64_t* D;
  uint64_t* hashes;  // NULL: nobody reads them
  uint64_t* sk_out;
  const int32_t* share;    // leading blocks whose masks the walk reads from the group leader
  const uint8_t* active;   // requests the kernel takes (the walk kernel chains the others' tails)
  const uint8_t* tags;
  const uint64_t* table;
  uint64_t n_buckets;
  uint64_t* masks;
  uint64_t* chunk_and;
  int32_t* status;
  int deal;  // requests dealt by `active`
  int chain_warps;
  int slots;  // per lane of the ring, a power of two
};

// One chain warp's part of a round: its 32 lanes' streams, slot after slot, in
// place: 32 digests become 32 hashes. The eight digests after those in work
// are always loaded ahead, across slots too: whether the next slot is full is
// asked eight steps before its first digests are loaded (slots are filled well
// ahead, so the answer is nearly always yes; else the warp waits). The
// sentinel remap of hashes 0 and 1 is left out unless
// EXACT (~15 cycles a step): the probe warps look at every hash anyway, and
// a round in which one is below 2 (once in 2^63 blocks) runs again, exactly.
template <bool EXACT>
__device__ __forceinline__ void chain_lanes(const ChainArgs& a, unsigned char* ring, const int32_t* s_at,
                                            uint64_t* s_full, uint64_t* s_ready, int32_t* s_pos, int32_t len, int32_t m,
                                            int* failed) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, lanes = 32 * a.chain_warps;
  const int smask = a.slots - 1, sshift = 31 - __clz(a.slots);
  const int32_t j = 32 * warp + lane;
  unsigned char* const mine = ring + (size_t)j * kCpRow;
  const uint32_t full = smem_u32(s_full + warp * kCpMaxSlots), ready = smem_u32(s_ready + warp * kCpMaxSlots);
  if (len == 0) return;
  int32_t i = j;                               // the stream's next request,
  int32_t next = i < m ? s_at[i] : INT32_MAX;  // and the position where it begins
  uint64_t h = a.h_init;
  ulonglong2 c[4], x[4];
  if (!mbar_wait_or(full, 0, failed)) {
    if (lane == 0) latch_error(a.status, SMETRIC_ERR_CUDA);
    return;
  }
  ulonglong2* row = reinterpret_cast<ulonglong2*>(mine);
  load8(c, row);
  for (int32_t q = 0; q < len; ++q) {
    while (q == next) {  // (an empty request begins where the next one does)
      h = a.h_init;
      i += lanes;
      next = i < m ? s_at[i] : INT32_MAX;
    }
    load8(x, row + 4);
    h = chain8<EXACT>(h, c, row);
    load8(c, row + 8);
    h = chain8<EXACT>(h, x, row + 4);
    const int32_t qn = q + 1 < len ? q + 1 : q;
    const uint32_t bar = full + 8u * (uint32_t)(qn & smask), par = (uint32_t)(qn >> sshift) & 1u;
    ulonglong2* const next_row = reinterpret_cast<ulonglong2*>(mine + (size_t)((qn & smask) * lanes) * kCpRow);
    const bool there = mbar_try_wait(bar, par);
    load8(x, row + 12);
    h = chain8<EXACT>(h, c, row + 8);
    // (the loads come after the answer: nothing else holds them back)
    if (!__all_sync(kFull, there) && !mbar_wait_or(bar, par, failed)) {
      if (lane == 0) latch_error(a.status, SMETRIC_ERR_CUDA);
      return;
    }
    load8(c, next_row);
    h = chain8<EXACT>(h, x, row + 12);
    __syncwarp();
    if (lane == 0) {
      mbar_arrive(ready + 8u * (uint32_t)(q & smask));
      *reinterpret_cast<volatile int32_t*>(s_pos + warp) = q + 1;
    }
    row = next_row;
  }
}

struct __align__(16) ChainReq {
  int64_t bo;     // first block in the batch
  int64_t cb;     // first request-aligned chunk
  int32_t nb;     // full blocks
  int32_t share;  // leading blocks whose masks the group leader's probes give
  int32_t req;
};

// W = 0: chain only (no index): hashes and session keys.
template <int W>
__global__ void __launch_bounds__(cp_warps(W) * 32, 1) k_chain_probe(const ChainArgs a) {
  extern __shared__ __align__(128) unsigned char csm[];  // the ring: slot s of lane j at (s * lanes + j) * kCpRow
  // per request of the round, in lane order (request k of a round is the
  // k / lanes-th of a lane's stream)
  __shared__ ChainReq s_rq[kCpRound];
  __shared__ int32_t s_at[kCpRound];    // first position in the lane's stream
  __shared__ int32_t s_dead[kCpRound];  // first chunk whose AND is empty (INT32_MAX until one is)
  __shared__ int32_t s_mine[kCpRound];
  __shared__ int32_t s_len0[kCpRound];  // full blocks, in the order taken
  __shared__ int32_t s_len[kCpMaxLanes];  // positions of each lane's stream
  __shared__ int32_t s_most[kCpMaxChainWarps];  // and the most of a chain warp's lanes
  __shared__ int32_t s_pos[kCpMaxChainWarps];   // positions each chain warp has chained
  __shared__ int32_t s_nmine;
  __shared__ int32_t s_wsum[kCpWarps];
  __shared__ int s_failed;
  __shared__ int s_redo;  // this round has met a hash below 2
  __shared__ __align__(8) uint64_t s_full[kCpMaxChainWarps * kCpMaxSlots];
  __shared__ __align__(8) uint64_t s_ready[kCpMaxChainWarps * kCpMaxSlots];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int32_t stride = (int32_t)gridDim.x, n = a.n;
  const int lanes = 32 * a.chain_warps;
  const int smask = a.slots - 1;
  const int sshift = 31 - __clz(a.slots);
  pdl_enter();
  if (!*a.batch_ok) {
    for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < n; r += (int64_t)stride * blockDim.x)
      a.sk_out[r] = 0;
    return;
  }
  // The CTAs' requests: those k_lead left to this kernel are dealt round robin
  // in request order, so that every CTA gets its share of them. Past 32
  // requests a thread, or kCpRound a CTA (no request is left to the walk then),
  // requests are taken as blockIdx.x + k * gridDim.x.
  const int32_t per_t = (n + (int32_t)blockDim.x - 1) / (int32_t)blockDim.x;
  const bool dealt = W > 0 && a.deal;
  if (dealt) {
    if (threadIdx.x == 0) s_nmine = 0;
    const int32_t lo = min(n, (int32_t)threadIdx.x * per_t), hi = min(n, lo + per_t);
    uint32_t bits = 0;  // bit i: request lo + i is this kernel's
    for (int32_t r = lo; r < hi; ++r) bits |= (uint32_t)__ldg(a.active + r) << (r - lo);
    // exclusive scan of the counts over the threads, in request order
    const int32_t cnt = __popc(bits);
    int32_t incl = cnt;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int32_t y = __shfl_up_sync(kFull, incl, d);
      if (lane >= d) incl += y;
    }
    if (lane == 31) s_wsum[warp] = incl;
    __syncthreads();
    int32_t rank = incl - cnt;
    for (int w2 = 0; w2 < warp; ++w2) rank += s_wsum[w2];
    for (; bits; bits &= bits - 1, ++rank)
      if (rank % stride == (int32_t)blockIdx.x) s_mine[atomicAdd(&s_nmine, 1)] = lo + __ffs(bits) - 1;
    __syncthreads();
  }
  const int32_t m_all = dealt ? s_nmine
                              : n > (int32_t)blockIdx.x ? (n - (int32_t)blockIdx.x + stride - 1) / stride : 0;

  bool again = false, used = false;  // the round before met a sentinel; barriers exist
  for (int32_t g0 = 0; g0 < m_all; g0 += again ? 0 : kCpRound) {
    const int32_t m = min(kCpRound, m_all - g0);
    const int act = min(m, lanes);  // lanes in use
    // ---- the round's requests; with more than one per lane, longest first
    int32_t k = -1;  // this thread's request: its place in lane order
    ChainReq x = {};
    if (threadIdx.x < (unsigned)m) {
      k = (int32_t)threadIdx.x;
      x.req = dealt ? s_mine[g0 + k] : (int32_t)blockIdx.x + (g0 + k) * stride;
      x.bo = __ldg(a.block_off + x.req);
      x.nb = (int32_t)(__ldg(a.block_off + x.req + 1) - x.bo);
      if (W > 0) {
        x.cb = __ldg(a.chunk_off + x.req);
        x.share = __ldg(a.share + x.req);
      }
      s_len0[k] = x.nb;
    }
    if (threadIdx.x < kCpMaxLanes) s_len[threadIdx.x] = 0;
    if (threadIdx.x < kCpMaxChainWarps) s_most[threadIdx.x] = s_pos[threadIdx.x] = 0;
    if (threadIdx.x == 0) {
      s_failed = 0;
      s_redo = again;
      for (int i = 0; i < a.chain_warps; ++i) {
        const int in_use = min(32, act - 32 * i);
        for (int s = 0; s < a.slots; ++s) {
          if (used) {
            asm volatile("mbarrier.inval.shared::cta.b64 [%0];\n" ::"r"(smem_u32(s_full + i * kCpMaxSlots + s)) : "memory");
            asm volatile("mbarrier.inval.shared::cta.b64 [%0];\n" ::"r"(smem_u32(s_ready + i * kCpMaxSlots + s)) : "memory");
          }
          mbar_init(smem_u32(s_full + i * kCpMaxSlots + s), (uint32_t)max(1, in_use));
          mbar_init(smem_u32(s_ready + i * kCpMaxSlots + s), 1);
        }
      }
    }
    __syncthreads();
    if (k >= 0) {
      if (m > lanes) {  // by length, each pass over the lanes against the last: long after short
        int32_t rank = 0;
        for (int32_t i = 0; i < m; ++i) {
          const int32_t v = s_len0[i];
          rank += v > x.nb || (v == x.nb && i < (int32_t)threadIdx.x);
        }
        const int32_t pass = rank / lanes, at = rank % lanes;
        k = pass * lanes + ((pass & 1) ? at : min(lanes, m - pass * lanes) - 1 - at);
      }
    }
    __syncthreads();
    if (k >= 0) {
      if (W > 0) s_dead[k] = INT32_MAX;
      s_rq[k] = x;
      if (x.nb == 0) a.sk_out[x.req] = 0;
    }
    __syncthreads();
    if (threadIdx.x < (unsigned)act) {
      int32_t pos = 0;
      for (int32_t i = (int32_t)threadIdx.x; i < m; i += lanes) {
        s_at[i] = pos;
        pos += (s_rq[i].nb + kChunk - 1) / kChunk;
      }
      s_len[threadIdx.x] = pos;
      atomicMax(&s_most[threadIdx.x >> 5], pos);
    }
    if (threadIdx.x == 0) asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    __syncthreads();
    int32_t most = 0;
    for (int i = 0; i < a.chain_warps; ++i) most = max(most, s_most[i]);

    // The request of lane j's stream at position q (q < s_len[j]).
    auto find = [&](int32_t q, int32_t j) {
      int32_t i = j;
      while (i + lanes < m && s_at[i + lanes] <= q) i += lanes;
      return i;
    };
    auto row_of = [&](int32_t q, int32_t j) {
      return reinterpret_cast<uint64_t*>(csm + (size_t)((q & smask) * lanes + j) * kCpRow);
    };
    // Position q of lane j: this lane's stored digest (0 past the request's end).
    auto fill_load = [&](int32_t q, int32_t j) -> uint64_t {
      if (q >= s_len[j]) return 0;
      const int32_t i = find(q, j), b = kChunk * (q - s_at[i]) + lane;
      return b < s_rq[i].nb ? __ldg(a.D + s_rq[i].bo + b) : 0;
    };
    auto fill_store = [&](int32_t q, int32_t j, uint64_t d) {
      row_of(q, j)[lane] = d;
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(s_full + (j >> 5) * kCpMaxSlots + (q & smask)));
    };

    if (warp < a.chain_warps) {
      if (!s_redo)
        chain_lanes<false>(a, csm, s_at, s_full, s_ready, s_pos, s_most[warp], m, &s_failed);
      else
        chain_lanes<true>(a, csm, s_at, s_full, s_ready, s_pos, s_most[warp], m, &s_failed);
    } else {
      // the first positions of every lane
      const int pw = warp - a.chain_warps, npw = cp_warps(W) - a.chain_warps;
      for (int32_t t = pw; t < act * a.slots; t += npw) {
        const int32_t q = t / act, j = t - q * act;
        if (q >= s_most[j >> 5]) continue;
        fill_store(q, j, fill_load(q, j));
      }
      // items in position-major order, every npw-th one
      const int32_t dq = npw / act, dj = npw - dq * act;
      int32_t q = pw / act, j = pw - q * act;
      for (; q < most; q += dq, j += dj) {
        if (j >= act) {
          j -= act;
          if (++q >= most) break;
        }
        const int32_t cw = j >> 5;
        if (q >= s_most[cw]) continue;
        const bool refill = q + a.slots < s_most[cw];
        const uint64_t d = refill ? fill_load(q + a.slots, j) : 0;
        if ((q >= a.slots && !poll_at_least(s_pos + cw, q - a.slots + 1, &s_failed)) ||
            !mbar_wait_or(smem_u32(s_ready + cw * kCpMaxSlots + (q & smask)), (q >> sshift) & 1, &s_failed)) {
          if (lane == 0) latch_error(a.status, SMETRIC_ERR_CUDA);
          break;
        }
        const uint64_t h = row_of(q, j)[lane];
        __syncwarp();
        if (refill) fill_store(q + a.slots, j, d);
        if (q >= s_len[j]) continue;
        const int32_t i = find(q, j);
        const ChainReq x = s_rq[i];
        const int32_t c = q - s_at[i], b = kChunk * c + lane;
        const bool in = b < x.nb;
        if (in) {
          if (h < 2) s_redo = 1;
          if (a.hashes) a.hashes[x.bo + b] = h;
          if (b == min(x.nb, a.S) - 1) a.sk_out[x.req] = h;
        }
        if constexpr (W > 0) {
          // nothing to probe in a chunk wholly inside the shared prefix (the walk reads the
          // leader's), nor after one whose AND is empty (every run has ended there)
          const int32_t dead = __shfl_sync(kFull, *(volatile int32_t*)&s_dead[i], 0);
          if (kChunk * (c + 1) <= x.share || dead < c) continue;
          const bool on = in && b >= x.share;
          uint64_t M[W];
          probe_warp<W>(a.tags, a.table, a.n_buckets, on, h, M);
          if (on) {
            uint64_t* const out = a.masks + (x.bo + b) * W;
#pragma unroll
            for (int w = 0; w < W; ++w) out[w] = M[w];
          }
          bool empty = true;
#pragma unroll
          for (int w = 0; w < W; ++w) {
            const uint64_t y = on ? M[w] : ~0ull;
            const uint64_t v = (uint64_t)__reduce_and_sync(kFull, (unsigned)y) |
                               ((uint64_t)__reduce_and_sync(kFull, (unsigned)(y >> 32)) << 32);
            if (lane == w) a.chunk_and[(x.cb + c) * W + w] = v;
            empty &= v == 0;
          }
          if (empty && lane == 0) atomicMin(&s_dead[i], c);
        }
      }
    }
    __syncthreads();
    used = true;
    again = !again && s_redo && !s_failed;
    __syncthreads();  // the round's shared state is rewritten by the next one
  }
}

// ---------------------------------------------------------------------------
// chain, one thread per request
// ---------------------------------------------------------------------------

// The hash-only calls of more than 32 requests an SM. There the ring is bound by
// its items (a load, two waits and a store each, 20 warps an SM), while enough
// threads hide a step's own loads and stores: at 4,096 requests the ring's call is
// up to 9 % faster than with this kernel; at 8,192 of 1,000 blocks it took 235 us
// and 470 at 16,384, with this one 226 and 352.
constexpr int kChainThreads = 32;  // one warp per CTA: chains spread over every SM
constexpr int kChainAhead = 16;    // digests loaded ahead per request

// 32-byte global load (read-only path) and store of four words, 32-byte aligned.
__device__ __forceinline__ void ld_nc_v4(const uint64_t* p, uint64_t (&v)[4]) {
  asm volatile("ld.global.nc.v4.u64 {%0,%1,%2,%3}, [%4];\n"
               : "=l"(v[0]), "=l"(v[1]), "=l"(v[2]), "=l"(v[3])
               : "l"(p));
}
__device__ __forceinline__ void st_v4(uint64_t* p, uint64_t a, uint64_t b, uint64_t c, uint64_t d) {
  asm volatile("st.global.v4.u64 [%0], {%1,%2,%3,%4};\n" ::"l"(p), "l"(a), "l"(b), "l"(c), "l"(d) : "memory");
}

__global__ void __launch_bounds__(kChainThreads) k_chain(ChainArgs a) {
  pdl_enter();
  const int32_t r = blockIdx.x * kChainThreads + threadIdx.x;
  if (r >= a.n) return;
  if (!*a.batch_ok) {
    a.sk_out[r] = 0;
    return;
  }
  const int64_t bo = __ldg(a.block_off + r), nb = __ldg(a.block_off + r + 1) - bo;
  const uint64_t* const d = a.D + bo;
  uint64_t* const out = a.hashes + bo;
  // Digests are read and hashes written four blocks per 32-byte access (a
  // lane's accesses are its own request's and do not coalesce across the warp,
  // and fewer instructions shorten every serial step): single blocks up to a
  // 32-byte boundary and after the last whole quad. A caller's hash buffer in
  // another 32-byte phase than the digests takes one block per access throughout.
  const bool same_phase = ((reinterpret_cast<uintptr_t>(d) ^ reinterpret_cast<uintptr_t>(out)) & 31) == 0;
  uint64_t h = a.h_init;
  int64_t b = 0;
  while (b < nb && (!same_phase || (reinterpret_cast<uintptr_t>(d + b) & 31))) {
    h = chain_step(h, __ldg(d + b));
    out[b++] = h;
  }
  const uint64_t* const dq = d + b;
  uint64_t* const hq = out + b;
  const int64_t nq = (nb - b) >> 2;  // whole quads
  constexpr int Q = kChainAhead / 4;
  uint64_t c[Q][4], x[Q][4];
#pragma unroll
  for (int j = 0; j < Q; ++j)
    if (j < nq) ld_nc_v4(dq + 4 * j, c[j]);
  for (int64_t q0 = 0; q0 < nq; q0 += Q) {
#pragma unroll
    for (int j = 0; j < Q; ++j)
      if (q0 + Q + j < nq) ld_nc_v4(dq + 4 * (q0 + Q + j), x[j]);
#pragma unroll
    for (int j = 0; j < Q; ++j) {
      if (q0 + j < nq) {
        const uint64_t a0 = chain_step(h, c[j][0]), a1 = chain_step(a0, c[j][1]), a2 = chain_step(a1, c[j][2]);
        h = chain_step(a2, c[j][3]);
        st_v4(hq + 4 * (q0 + j), a0, a1, a2, h);
      }
    }
#pragma unroll
    for (int j = 0; j < Q; ++j)
#pragma unroll
      for (int k = 0; k < 4; ++k) c[j][k] = x[j][k];
  }
  for (b += 4 * nq; b < nb; ++b) {
    h = chain_step(h, __ldg(d + b));
    out[b] = h;
  }
  a.sk_out[r] = nb > 0 ? out[min(nb, (int64_t)a.S) - 1] : 0;
}

// ---------------------------------------------------------------------------
// walk
// ---------------------------------------------------------------------------

// The session-centric policy (Figure 10) as the walk's decision; off for
// the argmin cost of smetric_route_batch.
enum Decide { kArgmin = 0, kSession = 1, kColoc = 2, kBailian = 3, kLMetric = 4 };

struct WalkPolicy {
  int on;    // a Decide value; 0 = the argmin cost
  int summ;  // also record every request's run ends (the sequential variant reads them)
  int64_t c_lin, c_att, d0, d1, hit_num, hit_den;
  int32_t rr_base;
  const int32_t* turn;
  const int64_t* est_hit;
  int32_t* stick;
  const int64_t* tpot;  // colocation: prefill cost each instance's live decodes absorb
  const int64_t* nreq;  // colocation: requests each instance runs; baselines: batch sizes
  int64_t lam_num, lam_den;  // Bailian's weight
};

struct WalkArgs {
  int N, B, S;
  const int64_t* off;
  const int64_t* block_off;
  const int64_t* chunk_off;
  int32_t n;
  const int64_t* load;
  int64_t w_load, w_miss, w_glob;
  const uint64_t* masks;
  const uint64_t* chunk_and;
  const int32_t* batch_ok;
  const int32_t* lead;
  const int32_t* share;
  int32_t* summ;
  int32_t* inst_out;
  int32_t* lhit_out;
  int32_t* ghit_out;
  uint4* groups;
  int64_t group_vecs;
  // k_lead's marks, when it left members' tails to this kernel (NULL: it did not)
  const uint8_t* active;
  const uint64_t* D;
  uint64_t* hashes;
  bool want_hashes;
  uint64_t* sk_out;
  const uint8_t* tags;
  const uint64_t* table;
  uint64_t n_buckets;
};

// One warp per request, lanes = 32 consecutive blocks. The masks are
// AND-scanned across lanes; lane j's "death set" is the local tiers held
// through block j-1 but not through block j. A block where runs end (two or
// three of a request's have any) hands its set to the lanes that hold those
// instances: lane i keeps c of instances i, i + 32, ... in registers. The
// global-tier run is the first lane whose block the global tier lacks. Then
// lanes = instances for the cost and a shuffle argmin with ties to the lowest id.
//
// A member's blocks before `share` are its leader's, whose masks and chunk ANDs
// the probe wrote (the member's own were not probed there): its walk reads them
// from the leader up to block `share` (a 32-block chunk that straddles `share`
// block by block), then its own.
//
// A member that k_lead did not leave to the chain kernel has only its shared
// prefix there. Its tail past `share` is chained here as far as it is needed,
// all lanes in step from the leader's hash: the first block alone, which ends
// most walks (a tail is mostly a request's fresh tokens, which no tier holds),
// then 32 blocks at a time.
template <int W, int DECIDE>
__global__ void __launch_bounds__(kMatchWarps * 32, 4) k_walk(const WalkArgs a, const WalkPolicy pol) {
  pdl_enter();
  const int N = a.N, B = a.B;
  const int32_t n = a.n;
  const int64_t w_load = a.w_load, w_miss = a.w_miss, w_glob = a.w_glob;
  int32_t* const inst_out = a.inst_out;
  int32_t* const lhit_out = a.lhit_out;
  int32_t* const ghit_out = a.ghit_out;
  __shared__ int64_t load_s[SMETRIC_MAX_INSTANCES];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int i = threadIdx.x; i < N; i += blockDim.x) load_s[i] = a.load[i];
  __syncthreads();
  const bool ok = *a.batch_ok != 0;
  const int gword = N >> 6;
  const uint64_t gbit = 1ull << (N & 63);
  const int64_t tw = (int64_t)gridDim.x * kMatchWarps;

  if (!ok)
    for (int64_t r = (int64_t)blockIdx.x * kMatchWarps + warp; r < n; r += tw)
      if (lane == 0) {
        inst_out[r] = -1; lhit_out[r] = 0; ghit_out[r] = 0;
        if (DECIDE == kSession || DECIDE == kColoc) pol.stick[r] = 0;
      }
  for (int64_t r = (int64_t)blockIdx.x * kMatchWarps + warp; ok && r < n; r += tw) {
    const int64_t L = a.off[r + 1] - a.off[r];
    const int64_t nb = L / B;
    const int64_t bo = a.block_off[r];
    const int64_t sh = a.share[r];  // 0 for a leader
    const int32_t l = sh > 0 ? a.lead[r] : (int32_t)r;
    const bool tail = a.active && !a.active[r];
    // chunk ANDs are per request-aligned chunk: blocks 32q .. 32q + 31 of
    // request r at index chunk_off[r] + q; block p < sh of the request is
    // block p of its leader
    const int64_t cbase = __ldg(a.chunk_off + r);
    const int64_t lbo = sh > 0 ? __ldg(a.block_off + l) : bo;
    const int64_t lcb = sh > 0 ? __ldg(a.chunk_off + l) : cbase;
    // masks of the blocks from block p on, lane = block (all ones past `end`)
    auto masks_at = [&](int64_t p, int64_t end, uint64_t (&x)[W]) {
      const int64_t b = p + lane;
      const uint64_t* const m = a.masks + ((b < sh ? lbo : bo) + b) * W;
#pragma unroll
      for (int w = 0; w < W; ++w) x[w] = b < end ? __ldg(m + w) : ~0ull;
    };
    auto and_at = [&](int64_t q, int w) -> uint64_t {  // its chunk q; 0 where the chunk straddles sh
      if (32 * (q + 1) <= sh) return __ldg(a.chunk_and + (lcb + q) * W + w);
      if (32 * q < sh) return 0ull;  // walked block by block
      return __ldg(a.chunk_and + (cbase + q) * W + w);
    };
    constexpr int CT = 2 * W;  // groups of 32 covering the N + 1 <= 64 W tiers
    int32_t c[CT];             // c of instance 32 t + lane
    uint64_t A[W];             // local tiers holding every block so far (warp-uniform)
    bool galive = true;
    int64_t g = 0;
#pragma unroll
    for (int t = 0; t < CT; ++t) c[t] = (int32_t)nb;  // until its run ends
#pragma unroll
    for (int w = 0; w < W; ++w) {
      const int lo = w * 64;
      A[w] = N >= lo + 64 ? ~0ull : (N > lo ? (1ull << (N - lo)) - 1 : 0ull);
    }
    // `len` consecutive blocks from request block `base`, lane j < len holding
    // block base + j (lanes past len hold all ones): records the runs that end
    // there; returns true once no run is alive
    auto span = [&](int64_t base, int len, const uint64_t (&x)[W]) -> bool {
      if (galive) {
        uint64_t mg = 0;
#pragma unroll
        for (int w = 0; w < W; ++w) if (w == gword) mg = x[w];
        const unsigned miss = __ballot_sync(kFull, !(mg & gbit));
        if (miss) { g = base + __ffs(miss) - 1; galive = false; }
        else g = base + len;
      }
      bool dies = false, any = false;
      uint64_t X[W];
#pragma unroll
      for (int w = 0; w < W; ++w) {
        uint64_t v = x[w];
#pragma unroll
        for (int dd = 1; dd < 32; dd <<= 1) {
          const uint64_t y = __shfl_up_sync(kFull, v, dd);
          if (lane >= dd) v &= y;
        }
        v &= A[w];                                     // held through block base + lane
        const uint64_t prev = __shfl_up_sync(kFull, v, 1);
        X[w] = (lane ? prev : A[w]) & ~v;              // runs that end at block base + lane
        dies |= X[w] != 0;
        A[w] = __shfl_sync(kFull, v, 31);
        any |= A[w] != 0;
      }
      for (unsigned ev = __ballot_sync(kFull, dies); ev; ev &= ev - 1) {
        const int at = __ffs(ev) - 1;
#pragma unroll
        for (int w = 0; w < W; ++w) {
          const uint64_t v = __shfl_sync(kFull, X[w], at);
          if (((uint32_t)v >> lane) & 1u) c[2 * w] = (int32_t)base + at;
          if (((uint32_t)(v >> 32) >> lane) & 1u) c[2 * w + 1] = (int32_t)base + at;
        }
      }
      return !any && !galive;
    };
    // 32 chunks per step from their AND summaries (lane = chunk); the first
    // chunk that ends an alive run is walked block by block, and the last
    // partial chunk too (for a tail chained here: the shared prefix's).
    const int64_t summed = tail ? sh : nb;  // blocks with masks and chunk ANDs
    bool dead = false;
    for (int64_t p = 0; !dead && p < summed;) {
      uint64_t x[W];
      const int64_t nfull = (summed - p) >> 5;
      if (nfull > 0) {
#pragma unroll
        for (int w = 0; w < W; ++w) x[w] = lane < nfull ? and_at((p >> 5) + lane, w) : 0;
        bool stop = lane >= nfull;
#pragma unroll
        for (int w = 0; w < W; ++w) {
          stop |= (x[w] & A[w]) != A[w];
          if (w == gword && galive) stop |= !(x[w] & gbit);
        }
        const unsigned sm = __ballot_sync(kFull, stop);
        const int k = sm ? __ffs(sm) - 1 : 32;
        p += 32 * (int64_t)k;  // chunks that keep every alive run
        if (galive) g = p;
        if (k >= nfull || k == 32) continue;
      }
      masks_at(p, summed, x);
      dead = span(p, (int)min((int64_t)32, summed - p), x);
      p += 32;
    }
    if (tail) {
      const int64_t kS = min(nb, (int64_t)a.S) - 1;
      uint64_t h = a.hashes[lbo + sh - 1];
      if (lane == 0 && kS < sh) a.sk_out[r] = a.hashes[lbo + kS];
      if (a.want_hashes)
        for (int64_t b = lane; b < sh; b += 32) a.hashes[bo + b] = a.hashes[lbo + b];
      for (int64_t f = sh; f < nb && (!dead || a.want_hashes || f <= kS);) {
        const int len = (int)min((int64_t)(f == sh ? 1 : 32), nb - f);
        const uint64_t d = lane < len ? __ldg(a.D + bo + f + lane) : 0;
        uint64_t mine = 0;
        for (int i = 0; i < len; ++i) {
          h = chain_step(h, __shfl_sync(kFull, d, i));
          if (lane == i) mine = h;
        }
        if (lane < len) {
          if (a.want_hashes) a.hashes[bo + f + lane] = mine;
          if (f + lane == kS) a.sk_out[r] = mine;
        }
        if (!dead) {
          uint64_t x[W];
          if (lane < len) {
            probe_one<W>(a.tags, a.table, a.n_buckets, mine, x);
          } else {
#pragma unroll
            for (int w = 0; w < W; ++w) x[w] = ~0ull;
          }
          __syncwarp();
          dead = span(f, len, x);
        }
        f += len;
      }
    }
    if (galive) g = nb;  // the global run reaches the last block
    // per instance (lanes = instances): c_i, then the decision
    int64_t best_cost = INT64_MAX;
    int32_t best = N;
    int64_t best_c = 0;
    // policies: prev = argmax c (lowest id); the balance key per instance:
    // 2*estimate_load (Figure 10), or the 128-bit product 2*estimate_load *
    // requests (colocation: over the candidates passing the TPOT check, and
    // over all instances for when none passes); ties rotate from s0
    int64_t pc = -1, pe = INT64_MAX, pec = 0;
    int32_t pi = N, prot = N;
    bool meets_any = false, cand_any = false;
    uint64_t ahi = ~0ull, alo = ~0ull, chi = ~0ull, clo = ~0ull;
    int32_t arot = N, crot = N;
    int64_t ac = 0, cc = 0;
    auto less128 = [](uint64_t h1, uint64_t l1, int32_t r1, uint64_t h2, uint64_t l2, int32_t r2) {
      return h1 < h2 || (h1 == h2 && (l1 < l2 || (l1 == l2 && r1 < r2)));
    };
    int64_t lmax = 0;  // Bailian: the largest batch size
    if (DECIDE == kBailian) {
      for (int i = lane; i < N; i += 32) lmax = max(lmax, __ldg(pol.nreq + i));
#pragma unroll
      for (int dd = 16; dd > 0; dd >>= 1) lmax = max(lmax, __shfl_xor_sync(kFull, lmax, dd));
    }
    const int32_t s0 = DECIDE == kSession || DECIDE == kColoc ? (int32_t)(((int64_t)pol.rr_base + r) % N) : 0;
    const int64_t budget2 = DECIDE == kSession || DECIDE == kColoc ? 2 * (pol.d0 + pol.d1 * L) : 0;
    int32_t* const out_c = a.summ + r * (N + 1);
#pragma unroll
    for (int t = 0; t < CT; ++t) {
      const int i = 32 * t + lane;
      if (i >= N) break;
      const int64_t ci = c[t];
      if (pol.summ) out_c[i] = c[t];
      if (DECIDE == kArgmin) {
        const int64_t gi = ci > g ? ci : g;
        const int64_t cost = w_load * load_s[i] + w_miss * (L - B * gi) + w_glob * B * (gi - ci);
        if (cost < best_cost) { best_cost = cost; best = i; best_c = ci; }
      } else if (DECIDE == kLMetric) {
        // (q_i + L - B c_i) * l_i, below 2^61
        const int64_t f = (load_s[i] + L - B * ci) * __ldg(pol.nreq + i);
        if (less128(0, (uint64_t)f, i, ahi, alo, arot)) { ahi = 0; alo = (uint64_t)f; arot = i; ac = ci; }
      } else if (DECIDE == kBailian) {
        // f_i * LAM_DEN * max l * L = (LAM_DEN - LAM_NUM) l_i L + LAM_NUM (L - B c_i) max l, in 128 bits
        const uint64_t Lm = lmax > 0 ? (uint64_t)lmax : 1, Lr = L > 0 ? (uint64_t)L : 1;
        const uint64_t a1 = lmax > 0 ? (uint64_t)((pol.lam_den - pol.lam_num) * __ldg(pol.nreq + i)) : 0;
        const uint64_t a2 = (uint64_t)pol.lam_num * (L > 0 ? (uint64_t)(L - B * ci) : 1);
        const uint64_t l1 = a1 * Lr, h1 = __umul64hi(a1, Lr), l2 = a2 * Lm, h2 = __umul64hi(a2, Lm);
        const uint64_t lo = l1 + l2, hi = h1 + h2 + (lo < l1 ? 1 : 0);
        if (less128(hi, lo, i, ahi, alo, arot)) { ahi = hi; alo = lo; arot = i; ac = ci; }
      } else {
        // Eq. 1 doubled: 2*c_lin*n + c_att*n*(2L - n), n = new tokens, plus 2*q_i
        const int64_t nn = L - B * ci;
        const int64_t cost2 = 2 * pol.c_lin * nn + pol.c_att * nn * (2 * L - nn);
        const int64_t est2 = 2 * load_s[i] + cost2;
        meets_any |= est2 <= budget2;
        if (ci > pc) { pc = ci; pi = i; }  // lanes see their instances in increasing order
        const int32_t rot = (int32_t)((i - s0 + N) % N);
        if (DECIDE == kSession) {
          if (est2 < pe || (est2 == pe && rot < prot)) { pe = est2; prot = rot; pec = ci; }
        } else {
          const bool cand = cost2 <= 2 * __ldg(pol.tpot + i);
          const uint64_t R = (uint64_t)__ldg(pol.nreq + i);
          const uint64_t lo = (uint64_t)est2 * R, hi = __umul64hi((uint64_t)est2, R);
          cand_any |= cand;
          if (less128(hi, lo, rot, ahi, alo, arot)) { ahi = hi; alo = lo; arot = rot; ac = ci; }
          if (cand && less128(hi, lo, rot, chi, clo, crot)) { chi = hi; clo = lo; crot = rot; cc = ci; }
        }
      }
    }
    if (pol.summ && lane == 0) out_c[N] = (int32_t)g;
    if (DECIDE == kBailian || DECIDE == kLMetric) {
#pragma unroll
      for (int dd = 16; dd > 0; dd >>= 1) {
        const uint64_t oh = __shfl_xor_sync(kFull, ahi, dd), ol = __shfl_xor_sync(kFull, alo, dd);
        const int32_t oi = __shfl_xor_sync(kFull, arot, dd);
        const int64_t oc2 = __shfl_xor_sync(kFull, ac, dd);
        if (less128(oh, ol, oi, ahi, alo, arot)) { ahi = oh; alo = ol; arot = oi; ac = oc2; }
      }
      if (lane == 0) {
        const int64_t gb = ac > g ? ac : g;
        inst_out[r] = arot;
        lhit_out[r] = (int32_t)(B * ac);
        ghit_out[r] = (int32_t)(B * (gb - ac));
      }
    } else if (DECIDE == kArgmin) {
#pragma unroll
      for (int dd = 16; dd > 0; dd >>= 1) {
        const int64_t oc = __shfl_xor_sync(kFull, best_cost, dd);
        const int32_t oi = __shfl_xor_sync(kFull, best, dd);
        const int64_t ocb = __shfl_xor_sync(kFull, best_c, dd);
        if (oc < best_cost || (oc == best_cost && oi < best)) { best_cost = oc; best = oi; best_c = ocb; }
      }
      if (lane == 0) {
        const int64_t gb = best_c > g ? best_c : g;
        inst_out[r] = best;
        lhit_out[r] = (int32_t)(B * best_c);
        ghit_out[r] = (int32_t)(B * (gb - best_c));
      }
    } else {
#pragma unroll
      for (int dd = 16; dd > 0; dd >>= 1) {
        const int64_t oc = __shfl_xor_sync(kFull, pc, dd);
        const int32_t oi = __shfl_xor_sync(kFull, pi, dd);
        if (oc > pc || (oc == pc && oi < pi)) { pc = oc; pi = oi; }
        if (DECIDE == kSession) {
          const int64_t oe = __shfl_xor_sync(kFull, pe, dd);
          const int32_t orot = __shfl_xor_sync(kFull, prot, dd);
          const int64_t oec = __shfl_xor_sync(kFull, pec, dd);
          if (oe < pe || (oe == pe && orot < prot)) { pe = oe; prot = orot; pec = oec; }
        } else {
          uint64_t oh = __shfl_xor_sync(kFull, ahi, dd), ol = __shfl_xor_sync(kFull, alo, dd);
          int32_t orot = __shfl_xor_sync(kFull, arot, dd);
          int64_t oc2 = __shfl_xor_sync(kFull, ac, dd);
          if (less128(oh, ol, orot, ahi, alo, arot)) { ahi = oh; alo = ol; arot = orot; ac = oc2; }
          oh = __shfl_xor_sync(kFull, chi, dd);
          ol = __shfl_xor_sync(kFull, clo, dd);
          orot = __shfl_xor_sync(kFull, crot, dd);
          oc2 = __shfl_xor_sync(kFull, cc, dd);
          if (less128(oh, ol, orot, chi, clo, crot)) { chi = oh; clo = ol; crot = orot; cc = oc2; }
        }
      }
      const bool any = __any_sync(kFull, meets_any);
      const bool cands = __any_sync(kFull, cand_any);
      if (lane == 0) {
        const int64_t np = L - B * pc;
        const int64_t cost2p = 2 * pol.c_lin * np + pol.c_att * np * (2 * L - np);
        const int64_t est2p = 2 * load_s[pi] + cost2p;
        const bool cached = B * pc * pol.hit_den > pol.hit_num * pol.est_hit[r];
        bool stick;
        int32_t to;
        int64_t ct;
        if (DECIDE == kSession) {
          stick = pol.turn[r] != 0 && cached && (est2p <= budget2 || !any);
          to = stick ? pi : (int32_t)((s0 + prot) % N);
          ct = stick ? pc : pec;
        } else {
          const bool prev_cand = !cands || cost2p <= 2 * __ldg(pol.tpot + pi);
          stick = pol.turn[r] != 0 && cached && est2p <= budget2 && prev_cand;
          to = stick ? pi : (int32_t)((s0 + (cands ? crot : arot)) % N);
          ct = stick ? pc : (cands ? cc : ac);
        }
        const int64_t gt = ct > g ? ct : g;
        inst_out[r] = to;
        lhit_out[r] = (int32_t)(B * ct);
        ghit_out[r] = (int32_t)(B * (gt - ct));
        pol.stick[r] = stick ? 1 : 0;
      }
    }
    __syncwarp();
  }
  // the group stage has read the group table: empty it for the next route
  // (it is zero from index creation before the first)
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < a.group_vecs;
       i += (int64_t)gridDim.x * blockDim.x)
    a.groups[i] = make_uint4(0, 0, 0, 0);
}

// ---------------------------------------------------------------------------
// sequential-update variant
// ---------------------------------------------------------------------------

// Requests in batch order: the a4-a5 argmin over the run ends the walk recorded
// (summ: c_i for every instance, then g) with the current loads, then the
// chosen load grows by L_r - B*c_{i*}. One request's choice is the next one's
// input, so the kernel's time is n times the latency of one decision; all that
// does not depend on the loads is taken out of it. kSeqWarps producer warps,
// one request each per stage, write every instance's
//   rest  = w_miss*(L - B*g_i) + w_glob*B*(g_i - c_i) and fresh = L - B*c_i
// to a ring in shared memory; one warp (lane = instances lane, lane + 32, ...,
// w_load*load_i in registers) adds rest, takes the minimum and lets the
// winning lane add w_load*fresh; the outputs are stored stage by stage.
// With costs below 2^55 the instance id sits in the cost's low 8 bits, so that
// the minimum names one instance, the lowest. Then one 32-bit warp reduction
// decides most requests: loads relative to the stage's smallest (loads only
// grow) and rests relative to the request's smallest, both cut off at
// kSeqCut: a minimum below the cut has neither part cut, so it is the true one.
// Otherwise two reductions find the 64-bit minimum (high words, then the low
// words of those that have it), and with wider costs a third the lowest id.
// Bound: ~150 cycles a decision (a reduction takes 22, the branch on it 35).
// Measured, 4,096 requests, N = 64: 292 us; 320 with producers on the deciding
// warp's scheduler too, 379 with rows loaded one stage ahead, 2,347 with one
// warp that also read the rows and reduced (cost, id, c) by shuffles.
constexpr int kSeqWarps = 12;   // producers, and requests of a stage
constexpr int kSeqBlock = 16;   // warps of the CTA: the last decides, the others of its scheduler (3, 7, 11) stay out
constexpr int kSeqStages = 3;   // 147 KB of ring at N = 256
constexpr int kSeqAhead = 4;    // stages
constexpr uint32_t kSeqCut = 0x7fffffffu;

struct __align__(16) SeqEntry {
  uint64_t rest;    // all ones where there is no instance
  uint32_t fresh;
  uint32_t rest32;  // rest less the request's smallest, cut off
};

template <int T, bool UNIQUE>
__device__ __forceinline__ bool seq_decide(int N, int32_t n, uint64_t w_load, const int64_t* __restrict__ load,
                                           const SeqEntry* ring, const int2* lens, uint32_t full, uint32_t empty,
                                           int* failed, int32_t* __restrict__ inst_out,
                                           int32_t* __restrict__ lhit_out, int32_t* __restrict__ ghit_out,
                                           int64_t* __restrict__ load_after) {
  const int lane = threadIdx.x & 31;
  constexpr int SH = UNIQUE ? 8 : 0;
  constexpr int UNROLL = T <= 2 ? kSeqWarps : 5;
  const uint32_t wl = (uint32_t)(w_load << SH);  // w_load <= 2^20
  uint64_t key[T];   // w_load * load_i, and the id below it when UNIQUE
  int64_t q[T];
#pragma unroll
  for (int t = 0; t < T; ++t) {
    const int i = 32 * t + lane;
    q[t] = i < N ? load[i] : 0;
    key[t] = i < N ? (((uint64_t)q[t] * w_load) << SH) | (UNIQUE ? (uint64_t)i : 0ull) : 0;
  }
  for (int32_t r0 = 0, st = 0; r0 < n; r0 += kSeqWarps, ++st) {
    const int slot = st % kSeqStages;
    if (!mbar_wait_or(full + 8u * slot, (uint32_t)(st / kSeqStages) & 1u, failed)) return false;
    // The stage's smallest load, and the loads relative to it.
    uint32_t rel[T];
    if (UNIQUE) {
      uint32_t mh = 0xffffffffu, ml = 0xffffffffu;
#pragma unroll
      for (int t = 0; t < T; ++t)
        if (32 * t + lane < N) mh = min(mh, (uint32_t)(key[t] >> 32));
      mh = __reduce_min_sync(kFull, mh);
#pragma unroll
      for (int t = 0; t < T; ++t)
        if (32 * t + lane < N && (uint32_t)(key[t] >> 32) == mh) ml = min(ml, (uint32_t)key[t]);
      ml = __reduce_min_sync(kFull, ml) & ~0xffu;
      const uint64_t low = ((uint64_t)mh << 32) | ml;
#pragma unroll
      for (int t = 0; t < T; ++t)
        rel[t] = 32 * t + lane < N ? (uint32_t)min(key[t] - low, (uint64_t)kSeqCut) : kSeqCut;
    }
    // All of the stage's places are gone through: those past the last request
    // have fresh = 0. Lane k keeps place k's choice, and writes its outputs
    // once the stage is through.
    const SeqEntry* const e = ring + (size_t)slot * kSeqWarps * 32 * T + lane;
    uint32_t chosen = 0;
    SeqEntry next[T];
#pragma unroll
    for (int t = 0; t < T; ++t) next[t] = e[32 * t];
#pragma unroll UNROLL
    for (int k = 0; k < kSeqWarps; ++k) {
      SeqEntry x[T];
      uint64_t grown[T];
      uint32_t id = 0, least = kSeqCut, grown32[T];
#pragma unroll
      for (int t = 0; t < T; ++t) {
        x[t] = next[t];
        if (k + 1 < kSeqWarps) next[t] = e[((k + 1) * T + t) * 32];
        grown[t] = (uint64_t)x[t].fresh * wl;
        grown32[t] = (uint32_t)min(grown[t], (uint64_t)kSeqCut);
      }
      if (UNIQUE) {
#pragma unroll
        for (int t = 0; t < T; ++t) least = min(least, rel[t] + x[t].rest32);
        least = __reduce_min_sync(kFull, least);
        id = least & 0xffu;
      }
      if (least >= kSeqCut) {  // (the warp's: never taken in the common case)
        uint32_t hi[T], lo[T], mh = 0xffffffffu, ml = 0xffffffffu;
#pragma unroll
        for (int t = 0; t < T; ++t) {
          const uint64_t c = key[t] + x[t].rest;  // (no instance: rest is all ones, key 0)
          hi[t] = (uint32_t)(c >> 32);
          lo[t] = (uint32_t)c;
          mh = min(mh, hi[t]);
        }
        mh = __reduce_min_sync(kFull, mh);
#pragma unroll
        for (int t = 0; t < T; ++t) ml = min(ml, hi[t] == mh ? lo[t] : 0xffffffffu);
        ml = __reduce_min_sync(kFull, ml);
        id = ml & 0xffu;
        if (!UNIQUE) {
          id = 0xffffffffu;
#pragma unroll
          for (int t = T - 1; t >= 0; --t)
            if (hi[t] == mh && lo[t] == ml && 32 * t + lane < N) id = 32 * t + lane;
          id = __reduce_min_sync(kFull, id);
        }
      }
#pragma unroll
      for (int t = 0; t < T; ++t) {
        const bool won = id == (uint32_t)(32 * t + lane);
        if (UNIQUE) rel[t] = won ? min(rel[t] + grown32[t], kSeqCut) : rel[t];
        key[t] += won ? grown[t] : 0ull;
        q[t] += won ? x[t].fresh : 0u;
      }
      if (lane == k) chosen = id;
    }
    if (lane < kSeqWarps && r0 + lane < n) {
      const int at = slot * kSeqWarps + lane;
      const int32_t hit = lens[at].x - (int32_t)ring[(size_t)at * 32 * T + chosen].fresh;  // B * c
      inst_out[r0 + lane] = (int32_t)chosen;
      lhit_out[r0 + lane] = hit;
      ghit_out[r0 + lane] = max(lens[at].y - hit, 0);
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(empty + 8u * slot);
  }
  if (load_after)
#pragma unroll
    for (int t = 0; t < T; ++t)
      if (32 * t + lane < N) load_after[32 * t + lane] = q[t];
  return true;
}

template <int T>
__global__ void __launch_bounds__(kSeqBlock * 32)
    k_seq(int N, int B, const int64_t* __restrict__ off, int32_t n, const int64_t* __restrict__ load,
          int64_t w_load, int64_t w_miss, int64_t w_glob, const int32_t* __restrict__ summ,
          const int32_t* __restrict__ batch_ok, int32_t* __restrict__ inst_out, int32_t* __restrict__ lhit_out,
          int32_t* __restrict__ ghit_out, int64_t* __restrict__ load_after, int32_t* status) {
  extern __shared__ __align__(16) unsigned char seq_sm[];
  SeqEntry* const ring = reinterpret_cast<SeqEntry*>(seq_sm);  // [kSeqStages][kSeqWarps][32 T]
  __shared__ int2 lens[kSeqStages * kSeqWarps];  // L and B * g
  __shared__ __align__(8) uint64_t full[kSeqStages], empty[kSeqStages];
  __shared__ int failed;
  __shared__ int64_t s_top;
  const int lane = threadIdx.x & 31, all = threadIdx.x >> 5;
  const int warp = all == kSeqBlock - 1 ? kSeqWarps : all - (all >> 2);  // producer, or kSeqWarps: the deciding warp
  if (!*batch_ok) return;  // the route already wrote the invalid batch's outputs
  if (threadIdx.x == 0) {
    failed = 0;
    for (int i = 0; i < kSeqStages; ++i) {
      mbar_init(smem_u32(full + i), kSeqWarps);
      mbar_init(smem_u32(empty + i), 1);
    }
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  if (warp == kSeqWarps) {
    int64_t top = 0;
    for (int i = lane; i < N; i += 32) top = max(top, load[i]);
#pragma unroll
    for (int dd = 16; dd > 0; dd >>= 1) top = max(top, __shfl_xor_sync(kFull, top, dd));
    if (lane == 0) s_top = top;
  }
  __syncthreads();
  const int64_t total = off[n] - off[0], top = s_top;
  if (top + total > (1LL << 42)) {
    for (int32_t r = threadIdx.x; r < n; r += blockDim.x) { inst_out[r] = -1; lhit_out[r] = 0; ghit_out[r] = 0; }
    if (threadIdx.x == 0) latch_error(status, SMETRIC_ERR_OVERFLOW);
    return;
  }
  // no cost reaches 2^55: the products are below 2^62 and 2^52
  const uint64_t most = (uint64_t)(top + total) * (uint64_t)w_load +
                        (uint64_t)min(total, (int64_t)INT32_MAX) * (uint64_t)(w_miss + w_glob);
  const bool unique = most < (1ull << 55);
  if (warp == kSeqWarps) {
    const bool ok = unique ? seq_decide<T, true>(N, n, (uint64_t)w_load, load, ring, lens, smem_u32(full), smem_u32(empty),
                                                 &failed, inst_out, lhit_out, ghit_out, load_after)
                           : seq_decide<T, false>(N, n, (uint64_t)w_load, load, ring, lens, smem_u32(full), smem_u32(empty),
                                                  &failed, inst_out, lhit_out, ghit_out, load_after);
    if (!ok && lane == 0) latch_error(status, SMETRIC_ERR_CUDA);
    return;
  }
  if ((all & 3) == 3) return;
  // producers: request r0 + warp of each stage, its row loaded kSeqAhead stages
  // before (a stage is decided faster than a row arrives)
  struct Row {
    int32_t c[T], g;
    int64_t L;
  };
  const uint32_t wm = (uint32_t)w_miss, wg = (uint32_t)w_glob;
  const int sh = unique ? 8 : 0;
  Row rows[kSeqAhead];
  auto load_row = [&](int64_t r, Row& d) {
    d = Row{};  // a place past the last request: fresh = 0
    if (r >= n) return;
    const int32_t* const row = summ + r * (N + 1);
#pragma unroll
    for (int t = 0; t < T; ++t) d.c[t] = 32 * t + lane < N ? row[32 * t + lane] : 0;
    d.g = row[N];
    d.L = off[r + 1] - off[r];
  };
#pragma unroll
  for (int u = 0; u < kSeqAhead; ++u) load_row((int64_t)u * kSeqWarps + warp, rows[u]);
  for (int32_t st0 = 0; (int64_t)st0 * kSeqWarps < n; st0 += kSeqAhead) {
#pragma unroll
    for (int u = 0; u < kSeqAhead; ++u) {
      const int32_t st = st0 + u;
      if ((int64_t)st * kSeqWarps >= n) return;
      const int slot = st % kSeqStages;
      const Row x = rows[u];
      load_row((int64_t)(st + kSeqAhead) * kSeqWarps + warp, rows[u]);
      // (32-bit factors, all within their limits; the smallest rest as the deciding warp finds its minimum)
      uint64_t rest[T];
      uint32_t mh = 0xffffffffu, ml = 0xffffffffu;
      const uint32_t L = (uint32_t)x.L;
#pragma unroll
      for (int t = 0; t < T; ++t) {
        const uint32_t have = (uint32_t)(B * max(x.c[t], x.g)), own = (uint32_t)(B * x.c[t]);
        rest[t] = ((uint64_t)wm * (L - have) + (uint64_t)wg * (have - own)) << sh;
        if (32 * t + lane >= N) rest[t] = ~0ull;
        mh = min(mh, (uint32_t)(rest[t] >> 32));
      }
      mh = __reduce_min_sync(kFull, mh);
#pragma unroll
      for (int t = 0; t < T; ++t)
        if ((uint32_t)(rest[t] >> 32) == mh) ml = min(ml, (uint32_t)rest[t]);
      ml = __reduce_min_sync(kFull, ml);
      const uint64_t low = ((uint64_t)mh << 32) | ml;
      if (st >= kSeqStages && !mbar_wait_or(smem_u32(empty + slot), (uint32_t)(st / kSeqStages - 1) & 1u, &failed)) return;
      SeqEntry* const e = ring + ((size_t)slot * kSeqWarps + warp) * 32 * T + lane;
#pragma unroll
      for (int t = 0; t < T; ++t) {
        SeqEntry y;
        y.rest = rest[t];
        y.fresh = L - (uint32_t)(B * x.c[t]);
        y.rest32 = (uint32_t)min(rest[t] - low, (uint64_t)kSeqCut);
        e[32 * t] = y;
      }
      if (lane == 0) lens[slot * kSeqWarps + warp] = make_int2((int32_t)x.L, B * x.g);
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(full + slot));
    }
  }
}

// ---------------------------------------------------------------------------
// reuse breakdown
// ---------------------------------------------------------------------------

uint64_t reuse_slots_for(int64_t n_blocks) {
  uint64_t g = 64;
  while (g < 2 * (uint64_t)n_blocks) g <<= 1;
  return g;
}

// The first table tried holds an eighth of the window's blocks at load 1/2
// (67 MB for 16M blocks, so it stays in L2); windows whose distinct blocks
// exceed that fall back on the device to the full table, sized for every
// block distinct.
uint64_t reuse_small_slots_for(int64_t n_blocks) { return reuse_slots_for((n_blocks + 7) / 8); }
constexpr int kReuseSmallProbe = 64;  // longer probes in the first table also fall back

// Workspace header after the table: [0] the fallback flag, [1] distinct keys
// in the first table.
struct ReuseHeader {
  int32_t big;
  uint32_t distinct;
  uint32_t next[3];  // work counters of the two inserts and the walk
  uint32_t pad[3];
};

// Warps take requests from a counter in arrival order, so that a warp done
// with a short request takes the next one instead of idling behind a long one.
__device__ __forceinline__ int64_t next_request(uint32_t* ctr, int lane) {
  uint32_t r = 0;
  if (lane == 0) r = atomicAdd(ctr, 1u);
  return __shfl_sync(kFull, r, 0);
}

// Rounds of 32 blocks that a warp loads ahead before it uses them.
constexpr int kReuseAhead = 4;

// Equal chain hashes mean equal prefixes, so the requests that hold a block of r
// hold every block of r before it too: an earlier request that has block b has
// the ones before, and the earliest holders of r's blocks, in order, never go
// back to an earlier request. Both kernels sample 32 of a request's blocks first
// and go through the blocks between samples only where they have to.
__device__ __forceinline__ int64_t sample_block(int lane, int64_t nb) { return nb > 0 ? lane * (nb - 1) / 31 : 0; }

// The table entry of `key` whose home slot holds e (key 0: absent).
__device__ __forceinline__ ulonglong2 reuse_find(const uint64_t* table, uint64_t mask, uint64_t key, ulonglong2 e,
                                                 uint64_t probes) {
  uint64_t s = key & mask;
  for (uint64_t t = 0; t < probes && e.x != key && e.x != 0; ++t) {
    s = (s + 1) & mask;
    e = *reinterpret_cast<const ulonglong2*>(table + 2 * s);
  }
  return e.x == key ? e : make_ulonglong2(0ull, 0ull);
}

// Warp per request, 32 blocks per round: each block's hash into the table
// with the earliest request holding it and that request's session, packed as
// (INT32_MAX - request) << 32 | session so that atomicMax keeps the earliest.
// Blocks up to the last sampled one that names an earlier request already are
// left out: that request has them all, and puts them in (or an earlier one
// does). The earliest holder of a block never leaves it out. Warps take
// requests in arrival order, and only two CTAs an SM run, so that most of a
// turn's blocks are in before the next turn looks. A slot that already names an
// earlier (or the same) request is left alone. The pre-checks are plain loads,
// so a block every request shares (a system prompt) is read from L1; a stale
// copy only shows an empty key or a smaller value, and both fall through to the
// atomics. The order of a request's blocks does not matter, so each request
// starts at a round of its own and wraps around, which spreads the requests in
// flight over the table.
// BIG = false fills the first table and raises the fallback flag when it
// runs full (more distinct keys than limit, or a probe longer than
// kReuseSmallProbe); BIG = true runs only after that, on the cleared full
// table. Bound: dependent reads of the table. 8,192 requests of 750 blocks in 8
// turns: 142 us (two CTAs an SM; one 135, four 164), against 217 with every
// block looked up and its claims one after another, 185 with the claims of four
// rounds in flight together.
template <bool BIG>
__global__ void __launch_bounds__(256)
    k_reuse_insert(const int64_t* __restrict__ block_off, int32_t n, const int32_t* __restrict__ batch_ok,
                   const uint64_t* __restrict__ H, const int32_t* __restrict__ sessions,
                   uint64_t* __restrict__ table, uint64_t mask, ReuseHeader* hdr, uint32_t limit) {
  if (!*batch_ok) return;
  if (BIG && !__ldcg(&hdr->big)) return;
  const int lane = threadIdx.x & 31;
  for (int64_t r = next_request(&hdr->next[BIG], lane); r < n; r = next_request(&hdr->next[BIG], lane)) {
    if (!BIG && __shfl_sync(kFull, lane == 0 ? __ldcg(&hdr->big) : 0, 0)) return;
    const int64_t bo = block_off[r], nb = block_off[r + 1] - bo;
    const unsigned long long val = ((unsigned long long)(INT32_MAX - r) << 32) | (uint32_t)sessions[r];
    int64_t b0 = 0;  // blocks before it are in
    {
      const int64_t p = sample_block(lane, nb);
      const uint64_t key = nb > 0 ? H[bo + p] : 0;
      bool in = false;
      if (nb > 0) {
        const ulonglong2 e = reuse_find(table, mask, key, *reinterpret_cast<const ulonglong2*>(table + 2 * (key & mask)),
                                        kReuseSmallProbe);
        in = e.x == key && e.y >= val;
      }
      const unsigned m = __ballot_sync(kFull, in);
      if (m) b0 = __shfl_sync(kFull, p, 31 - __clz(m)) + 1;
    }
    const int64_t rounds = (nb - b0 + 31) >> 5;
    const int64_t start = rounds ? r % rounds : 0;
    uint32_t fresh_n = 0;
    for (int64_t i = 0; i < rounds; i += kReuseAhead) {
      int64_t b[kReuseAhead];
      uint64_t key[kReuseAhead];
      ulonglong2 sl[kReuseAhead];
#pragma unroll
      for (int u = 0; u < kReuseAhead; ++u) {
        int64_t rd = start + i + u;
        rd = rd >= rounds ? rd - rounds : rd;
        b[u] = i + u < rounds ? b0 + rd * 32 + lane : nb;
        key[u] = b[u] < nb ? H[bo + b[u]] : 0;
      }
#pragma unroll
      for (int u = 0; u < kReuseAhead; ++u)
        if (b[u] < nb) sl[u] = *reinterpret_cast<const ulonglong2*>(table + 2 * (key[u] & mask));
      // Home slots first, all rounds' claims in flight together: a block whose
      // home slot is empty claims it, one whose slot it has raises the value
      // (unless an earlier request is there already); the others walk on.
      bool full = false, on[kReuseAhead];
      unsigned long long got[kReuseAhead];
#pragma unroll
      for (int u = 0; u < kReuseAhead; ++u) {
        on[u] = b[u] < nb && !(sl[u].x == key[u] && sl[u].y >= val);
        got[u] = sl[u].x;
        if (on[u] && sl[u].x == 0ull)
          got[u] = atomicCAS(reinterpret_cast<unsigned long long*>(table + 2 * (key[u] & mask)), 0ull,
                             (unsigned long long)key[u]);
      }
#pragma unroll
      for (int u = 0; u < kReuseAhead; ++u) {
        if (!on[u]) continue;
        uint64_t s = key[u] & mask;
        unsigned long long k = got[u];
        fresh_n += k == 0ull && sl[u].x == 0ull;
        const uint64_t probes = BIG ? mask + 1 : kReuseSmallProbe;
        bool placed = false;
        for (uint64_t t = 0; t < probes; ++t) {
          unsigned long long* const slot = reinterpret_cast<unsigned long long*>(table + 2 * s);
          if (t > 0) {
            k = slot[0];
            if (k == 0ull) {
              k = atomicCAS(slot, 0ull, (unsigned long long)key[u]);
              fresh_n += k == 0ull;
            }
          }
          if (k == 0ull || k == key[u]) {
            atomicMax(slot + 1, val);
            placed = true;
            break;
          }
          s = (s + 1) & mask;
        }
        full |= !placed;
      }
      if (!BIG && __any_sync(kFull, full)) {
        if (lane == 0) atomicExch(&hdr->big, 1);
        return;
      }
    }
    if (!BIG) {
      fresh_n = __reduce_add_sync(kFull, fresh_n);
      if (lane == 0 && fresh_n && atomicAdd(&hdr->distinct, fresh_n) + fresh_n > limit) atomicExch(&hdr->big, 1);
    }
  }
}

// Clears the full table once the first one has run full.
__global__ void __launch_bounds__(256) k_reuse_clear(const ReuseHeader* hdr, uint4* table, int64_t n16) {
  if (!*reinterpret_cast<const volatile int32_t*>(&hdr->big)) return;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n16; i += (int64_t)gridDim.x * blockDim.x)
    table[i] = make_uint4(0, 0, 0, 0);
}

// Warp per request: block b is reused when its earliest holder precedes the
// request; the run stops at the first block that is not. Reused blocks split
// into system prompt (b < sys_r), intra-session (the holder is of r's session)
// and inter-session. Where two samples have one holder, the blocks between them
// have it too; kReuseAhead of the other stretches are looked up at a time. 37 us
// for the window above, against 77 with every reused block looked up.
__global__ void __launch_bounds__(256)
    k_reuse_walk(const int64_t* __restrict__ block_off, int32_t n, const int32_t* __restrict__ batch_ok,
                 const uint64_t* __restrict__ H, const uint64_t* __restrict__ table, uint64_t mask_small,
                 uint64_t mask_big, ReuseHeader* hdr, const int32_t* __restrict__ sessions,
                 const int32_t* __restrict__ sys_blocks,
                 int32_t* __restrict__ hit, int32_t* __restrict__ sys, int32_t* __restrict__ intra,
                 int32_t* __restrict__ inter, int32_t* status) {
  const int lane = threadIdx.x & 31;
  const bool ok = *batch_ok != 0;
  const uint64_t mask = hdr->big ? mask_big : mask_small;
  for (int64_t r = next_request(&hdr->next[2], lane); r < n; r = next_request(&hdr->next[2], lane)) {
    int32_t nh = 0, ns = 0, ni = 0, ne = 0;
    if (ok) {
      const int64_t bo = block_off[r], nb = block_off[r + 1] - bo;
      int64_t sb = sys_blocks[r];
      if (sb < 0) {
        if (lane == 0) latch_error(status, SMETRIC_ERR_INVALID_ARG);
        sb = 0;
      }
      const int32_t sr = sessions[r];
      auto look = [&](int64_t b, uint64_t key, ulonglong2 home, int32_t& holder, int32_t& sess) {
        const ulonglong2 e = reuse_find(table, mask, key, home, mask);
        holder = e.x == key && key ? INT32_MAX - (int32_t)(e.y >> 32) : INT32_MAX;
        sess = (int32_t)(uint32_t)e.y;
      };
      // samples: lane i's stretch is the blocks after lane i - 1's sample up to its own
      const int64_t p = sample_block(lane, nb);
      int32_t holder = INT32_MAX, sess = 0;
      if (nb > 0) {
        const uint64_t key = H[bo + p];
        look(p, key, *reinterpret_cast<const ulonglong2*>(table + 2 * (key & mask)), holder, sess);
      }
      const unsigned miss = __ballot_sync(kFull, holder >= r);
      const int last = miss ? __ffs(miss) - 1 : 32;  // the first sample that is not reused
      const int32_t before = __shfl_up_sync(kFull, holder, 1);
      const int64_t previous = __shfl_up_sync(kFull, p, 1);
      const int64_t from = lane ? previous + 1 : 0;  // the stretch's first block
      // stretches within the run: one holder throughout (a single block has), or looked up
      const bool whole = lane < last && (from >= p || (lane > 0 && before == holder));
      const bool part = !whole && lane <= last && last > 0 && from <= p;
      int64_t end = last == 32 ? nb : last == 0 ? 0 : nb;  // the run's end, once known
      int64_t mine = 0;                                    // this lane's intra-session blocks
      if (whole && sess == sr) mine = max((int64_t)0, p + 1 - max(from, sb));
      unsigned todo = __ballot_sync(kFull, part);
      while (todo) {
        int64_t f[kReuseAhead], t[kReuseAhead];
        uint64_t key[kReuseAhead];
        ulonglong2 home[kReuseAhead];
        int n_at = 0;
#pragma unroll
        for (int u = 0; u < kReuseAhead; ++u) {
          f[u] = t[u] = nb;
          key[u] = 0;
          if (!todo) continue;
          const int l = __ffs(todo) - 1;
          todo &= todo - 1;
          f[u] = __shfl_sync(kFull, from, l);
          t[u] = __shfl_sync(kFull, p, l) + 1;
          n_at = u + 1;
          if (f[u] + lane < t[u]) key[u] = H[bo + f[u] + lane];
        }
#pragma unroll
        for (int u = 0; u < kReuseAhead; ++u)
          if (key[u]) home[u] = *reinterpret_cast<const ulonglong2*>(table + 2 * (key[u] & mask));
#pragma unroll
        for (int u = 0; u < kReuseAhead; ++u) {
          if (u >= n_at) continue;  // warp-uniform
          for (int64_t b = f[u]; b < t[u]; b += 32) {  // (more than 32 blocks past 1,024)
            int32_t h = INT32_MAX, hs = 0;
            if (b + lane < t[u]) {
              if (b > f[u]) {
                key[u] = H[bo + b + lane];
                home[u] = *reinterpret_cast<const ulonglong2*>(table + 2 * (key[u] & mask));
              }
              look(b + lane, key[u], home[u], h, hs);
            }
            const bool reused = b + lane < t[u] && h < r;
            const unsigned gone = __ballot_sync(kFull, b + lane < t[u] && !reused);
            if (gone) end = min(end, b + __ffs(gone) - 1);
            if (reused && b + lane < end && b + lane >= sb && hs == sr) ++mine;
          }
        }
      }
      nh = (int32_t)end;
      ns = (int32_t)min(end, sb);
#pragma unroll
      for (int dd = 16; dd > 0; dd >>= 1) mine += __shfl_xor_sync(kFull, mine, dd);
      ni = (int32_t)mine;
      ne = nh - ns - ni;
    }
    if (lane == 0) {
      hit[r] = ok ? nh : -1;
      sys[r] = ok ? ns : -1;
      intra[r] = ok ? ni : -1;
      inter[r] = ok ? ne : -1;
    }
  }
}

// ---------------------------------------------------------------------------
// session links
// ---------------------------------------------------------------------------

// A request's parent is sought among the requests of its user's turn before:
// k_link_turns lists the requests of each (user, turn) and k_link_parents goes
// through the list that a request's parent must be in, comparing one hash per
// entry. In a trace a list has one request or a few; a request whose list is
// longer than kLinkList is marked instead (parent -2) and found by its prefixes
// in three more kernels, which return at once when there is none. 8,192
// requests of 750 blocks, lists of one: 10 us instead of 156 for a thread per
// (request, prefix length).
constexpr int kLinkList = 64;   // entries, a dependent read each
constexpr int32_t kLinkMarked = -2;

struct LinkState {
  int32_t marked;  // some request is marked
  int32_t deep;    // some chain of parents is longer than kLinkHops
};

__device__ __forceinline__ uint64_t turn_key(int64_t user, int64_t turn) {
  const uint64_t x = mix64(mix64((uint64_t)user ^ kGamma) ^ (uint64_t)turn);
  return x ? x : 1;
}

// Thread per request p: to the front of its (user, turn)'s list. A table entry
// is the turn's fingerprint, the list's head (request + 1) and its length.
__global__ void __launch_bounds__(256)
    k_link_turns(int32_t n, const int32_t* __restrict__ batch_ok, const int64_t* __restrict__ users,
                 const int32_t* __restrict__ turns, uint64_t* __restrict__ table, uint64_t gmask,
                 int32_t* __restrict__ next, LinkState* state) {
  pdl_enter();
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p == 0) *state = LinkState{0, 0};
  if (p >= n || !*batch_ok) return;
  const uint64_t key = turn_key(users[p], turns[p]);
  uint64_t s = key & gmask;
  for (uint64_t t = 0; t <= gmask; ++t) {
    unsigned long long* const slot = reinterpret_cast<unsigned long long*>(table + 2 * s);
    const unsigned long long old = atomicCAS(slot, 0ull, (unsigned long long)key);
    if (old == 0ull || old == key) {
      int32_t* const list = reinterpret_cast<int32_t*>(slot + 1);
      next[p] = atomicExch(list, (int32_t)p + 1);
      atomicAdd(list + 1, 1);
      return;
    }
    s = (s + 1) & gmask;
  }
}

// Thread per request r: the latest earlier request on the list of (user_r,
// turn_r - 1) whose last block is r's block there. (A fingerprint may stand for
// several turns: user and turn are compared.)
__global__ void __launch_bounds__(256)
    k_link_parents(const int64_t* __restrict__ block_off, int32_t n, const int32_t* __restrict__ batch_ok,
                   const uint64_t* __restrict__ H, const int64_t* __restrict__ users,
                   const int32_t* __restrict__ turns, const uint64_t* __restrict__ table, uint64_t gmask,
                   const int32_t* __restrict__ next, int32_t* __restrict__ parent, int32_t* __restrict__ mark,
                   LinkState* state) {
  pdl_enter();
  const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= n || !*batch_ok) return;
  const int64_t user = users[r], turn = (int64_t)turns[r] - 1;
  const int64_t bo = __ldg(block_off + r), nb = __ldg(block_off + r + 1) - bo;
  int32_t best = -1;
  const uint64_t key = turn_key(user, turn);
  uint64_t s = key & gmask;
  for (uint64_t t = 0; t <= gmask; ++t) {
    const ulonglong2 e = __ldg(reinterpret_cast<const ulonglong2*>(table + 2 * s));
    if (e.x == 0) break;
    if (e.x == key) {
      if ((int32_t)(e.y >> 32) > kLinkList) {
        best = kLinkMarked;
        state->marked = 1;
        break;
      }
      for (int32_t p = (int32_t)(uint32_t)e.y - 1; p >= 0; p = __ldg(next + p) - 1) {
        if (p >= r || p <= best || users[p] != user || (int64_t)turns[p] != turn) continue;
        const int64_t pbo = __ldg(block_off + p), k = __ldg(block_off + p + 1) - pbo;
        if (k <= nb && (k == 0 || __ldg(H + pbo + k - 1) == __ldg(H + bo + k - 1))) best = p;
      }
      break;
    }
    s = (s + 1) & gmask;
  }
  parent[r] = best;
  mark[r] = best;  // (the mark outlives a parent found later; the session output until it is written)
}

// With marked requests: empties the table for its use as a multi-map.
__global__ void __launch_bounds__(256) k_link_clear(const LinkState* state, uint4* __restrict__ table, int64_t vecs) {
  pdl_enter();
  if (!state->marked) return;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < vecs; i += (int64_t)gridDim.x * blockDim.x)
    table[i] = make_uint4(0, 0, 0, 0);
}

// Fingerprint of (user, turn, number of blocks, last block hash) for the
// multi-map; 0 marks an empty slot.
__device__ __forceinline__ uint64_t link_key(int64_t user, int64_t turn, int64_t nb, uint64_t last) {
  uint64_t x = mix64((uint64_t)user ^ kGamma);
  x = mix64(x ^ (uint64_t)turn);
  x = mix64(x ^ (uint64_t)nb);
  x = mix64(x ^ last);
  return x ? x : 1;
}

// With marked requests, thread per request p: (key, p) into the table (a
// multi-map: every request takes its own slot).
__global__ void __launch_bounds__(256)
    k_link_insert(const int64_t* __restrict__ block_off, int32_t n, const int32_t* __restrict__ batch_ok,
                  const uint64_t* __restrict__ H, const int64_t* __restrict__ users,
                  const int32_t* __restrict__ turns, uint64_t* __restrict__ table, uint64_t gmask,
                  const LinkState* state) {
  pdl_enter();
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= n || !*batch_ok || !state->marked) return;
  const int64_t bo = block_off[p], nb = block_off[p + 1] - bo;
  const uint64_t key = link_key(users[p], turns[p], nb, nb ? H[bo + nb - 1] : 0);
  uint64_t s = key & gmask;
  for (uint64_t t = 0; t <= gmask; ++t) {
    unsigned long long* const slot = reinterpret_cast<unsigned long long*>(table + 2 * s);
    if (atomicCAS(slot, 0ull, (unsigned long long)key) == 0ull) {
      slot[1] = (unsigned long long)p;
      return;
    }
    s = (s + 1) & gmask;
  }
}

// Thread per (marked request r, prefix length k <= n_r): the latest earlier
// request of r's user, of turn turn_r - 1, with exactly k blocks, the last equal
// to r's block k - 1, raises parent[r] to it (any request is above the mark; one
// without a parent keeps it). Candidates from the table are checked field by
// field.
__global__ void __launch_bounds__(256)
    k_link_find(const int64_t* __restrict__ block_off, int32_t n, const int32_t* __restrict__ batch_ok,
                const uint64_t* __restrict__ H, const int64_t* __restrict__ users,
                const int32_t* __restrict__ turns, const uint64_t* __restrict__ table, uint64_t gmask,
                int32_t* parent, const int32_t* __restrict__ mark, const LinkState* state) {
  pdl_enter();
  if (!*batch_ok || !state->marked) return;
  const int64_t total = block_off[n] + n;  // sum over r of n_r + 1
  int32_t r = 0;
  for (int64_t f = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; f < total;
       f += (int64_t)gridDim.x * blockDim.x) {
    int32_t lo = r, hi = n;  // largest r with block_off[r] + r <= f
    while (hi - lo > 1) {
      const int32_t mid = (lo + hi) >> 1;
      if (__ldg(block_off + mid) + mid <= f) lo = mid; else hi = mid;
    }
    r = lo;
    if (mark[r] != kLinkMarked) continue;
    const int64_t bo = __ldg(block_off + r), k = f - (bo + r);
    const int64_t user = users[r], turn = (int64_t)turns[r] - 1;
    const uint64_t last = k ? __ldg(H + bo + k - 1) : 0;
    const uint64_t key = link_key(user, turn, k, last);
    int32_t best = -1;
    uint64_t s = key & gmask;
    for (uint64_t t = 0; t <= gmask; ++t) {
      const uint64_t kk = __ldg(table + 2 * s);
      if (kk == 0) break;
      if (kk == key) {
        const int32_t p = (int32_t)__ldg(table + 2 * s + 1);
        const int64_t pbo = __ldg(block_off + p);
        if (p < r && p > best && users[p] == user && (int64_t)turns[p] == turn &&
            __ldg(block_off + p + 1) - pbo == k && (k == 0 || __ldg(H + pbo + k - 1) == last))
          best = p;
      }
      s = (s + 1) & gmask;
    }
    if (best >= 0) atomicMax(parent + r, best);
  }
}

// Thread per request: up the chain of parents, kLinkHops of them at most; then
// session[r] is the head, or an ancestor on the way to it. (Parents are earlier
// requests, so every chain ends.) A parent left at the mark is none.
constexpr int kLinkHops = 64;
__global__ void __launch_bounds__(256)
    k_link_chase(int32_t n, const int32_t* __restrict__ batch_ok, const int32_t* __restrict__ parent,
                 int32_t* __restrict__ session, LinkState* state) {
  pdl_enter();
  const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= n || !*batch_ok) return;
  int32_t s = (int32_t)r;
  for (int k = 0; k < kLinkHops; ++k) {
    const int32_t p = __ldg(parent + s);
    if (p < 0) break;
    s = p;
  }
  if (__ldg(parent + s) >= 0) state->deep = 1;
  session[r] = s;
}

// CTA 0: the heads of longer chains by pointer jumping (session[r] an ancestor
// of r throughout), -1 everywhere after invalid offsets, and no parent where
// one is still marked. The other CTAs empty the table for the next call.
__global__ void __launch_bounds__(1024)
    k_link_heads(int32_t n, const int32_t* __restrict__ batch_ok, int32_t* __restrict__ parent,
                 int32_t* __restrict__ session, uint4* __restrict__ table, int64_t table_vecs,
                 const LinkState* state) {
  pdl_enter();
  if (blockIdx.x > 0) {
    for (int64_t i = (int64_t)(blockIdx.x - 1) * blockDim.x + threadIdx.x; i < table_vecs;
         i += (int64_t)(gridDim.x - 1) * blockDim.x)
      table[i] = make_uint4(0, 0, 0, 0);
    return;
  }
  if (!*batch_ok) {
    for (int32_t r = threadIdx.x; r < n; r += blockDim.x) { parent[r] = -1; session[r] = -1; }
    return;
  }
  if (state->deep) {
    for (int64_t span = 1; span < n; span <<= 1) {
      int moved = 0;
      for (int32_t r = threadIdx.x; r < n; r += blockDim.x) {
        const int32_t a = session[r], b = session[a];
        if (a != b) {
          session[r] = b;  // an ancestor either way: the heads are reached all the same
          moved = 1;
        }
      }
      if (!__syncthreads_or(moved)) break;
    }
  }
  if (state->marked)
    for (int32_t r = threadIdx.x; r < n; r += blockDim.x)
      if (parent[r] == kLinkMarked) parent[r] = -1;
}

// ---------------------------------------------------------------------------
// commit
// ---------------------------------------------------------------------------

// Checks of a batch to commit and the queue drain, on an index without an LRU
// (with one, its first kernel does both).
__global__ void __launch_bounds__(1024)
    k_drain(const int64_t* __restrict__ off, int32_t n, int N, const int32_t* __restrict__ instance,
            const int32_t* __restrict__ local_hit, int32_t* __restrict__ batch_ok,
            int64_t* __restrict__ load, int32_t* status) {
  pdl_enter();
  drain_batch(off, n, N, instance, local_hit, batch_ok, load, status);
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------

void profile_mark(smetric_index* idx, int k, cudaStream_t s);

// How a batch shares the GPU with the batch after it (smetric_route_batches
// on two scratch sets): an event recorded once its chain and probe are
// enqueued, which the next batch's first kernel waits for.
struct Overlap {
  cudaEvent_t after_chain;
};

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*,
                                  CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                                  CUtensorMapFloatOOBfill);

// The driver's tensor-map encoder, looked up once (thread-safe static init).
EncodeTiledFn tensor_map_encoder() {
  static const EncodeTiledFn fn = [] {
    EncodeTiledFn f = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", reinterpret_cast<void**>(&f), 12000,
                                         cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      f = nullptr;
    return f;
  }();
  return fn;
}

// The maps of a token buffer: as many rows as fit inside it from each map's base.
template <int HB>
bool make_token_maps(TokenMaps<HB>& m, const int32_t* tokens, int64_t n_tokens) {
  using Maps = TokenMaps<HB>;
  constexpr int B = 2 * HB, width = Maps::kWide ? 2 * B : B + 4;
  EncodeTiledFn enc = tensor_map_encoder();
  if (!enc) return false;
  memset(&m, 0, sizeof(m));
  const int64_t bytes = 4 * n_tokens, row = 4 * width, stride = 4 * B;
  for (int k = 0; k < Maps::kMaps; ++k) {
    const int64_t base = !Maps::kWide ? 16 * k : k == 0 || bytes < row ? 0 : (bytes - row) % stride & ~(int64_t)15;
    m.base[k] = (uint32_t)base;
    if (bytes < base + row) continue;  // rows[k] = 0: chunks fall back to lane copies
    int64_t rows = (bytes - base - row) / stride + 1;
    if (rows > INT32_MAX) rows = INT32_MAX;
    const cuuint64_t dims[2] = {(cuuint64_t)width, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)stride};
    const cuuint32_t box[2] = {(cuuint32_t)(B + 4), (cuuint32_t)kChunk};
    const cuuint32_t es[2] = {1, 1};
    if (enc(&m.map[k], CU_TENSOR_MAP_DATA_TYPE_UINT32, 2,
            const_cast<char*>(reinterpret_cast<const char*>(tokens)) + base, dims, strides, box, es,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
      return false;
    m.rows[k] = (uint32_t)rows;
  }
  return true;
}

// Group-table slots a batch of n requests uses: a power of two >= 2n.
uint64_t group_slots_for(int32_t n) {
  uint64_t g = 64;
  while (g < 2 * (uint64_t)n) g <<= 1;
  return g;
}

// Empties the group table of a call of n requests whose last kernel, which does
// that, could not be launched.
void empty_groups(smetric_index* idx, int32_t n, cudaStream_t s) {
  (void)cudaMemsetAsync(idx->groups, 0, 2 * sizeof(uint64_t) * group_slots_for(n), s);
  (void)cudaGetLastError();  // (the call returns the first error)
}

// The digest kernel for the index's block size; with `group` it also puts
// each request's first-block hash into the group table.
template <int HB>
int launch_digest(smetric_index* idx, const int32_t* d_tokens, int64_t n_tokens,
                  const int64_t* d_offsets, int32_t n, cudaStream_t s, bool group) {
  const int B = idx->cfg.block_size;
  const uint64_t d_init = mix64(idx->cfg.hash_seed ^ (uint64_t)B);
  const uint64_t h_init = mix64(idx->cfg.hash_seed + kGamma);
  uint64_t* const groups = group ? idx->groups : nullptr;
  const uint64_t gmask = group_slots_for(n) - 1;
  // request-aligned chunks (TMA kernel) number at most blocks / 32 + n
  const int64_t max_chunks = (n_tokens / B + kChunk - 1) / kChunk + (HB > 0 ? n : 0);
  // rows of 16*nch bytes: a block's 4B bytes start at most 12 bytes past a
  // 16-byte boundary
  const int nch = HB > 0 ? HB / 2 + 1 : (4 * B + 12 + 15) / 16;
  if constexpr (HB > 0) {
    static thread_local TokenMaps<HB> maps;
    if (make_token_maps<HB>(maps, d_tokens, n_tokens)) {
      auto kern = k_digest_tma<HB, kTmaStages>;
      const size_t per_warp = (size_t)kTmaStages * kChunk * nch * 16 + 8 * kTmaStages;
      const int warps = tma_warps(HB);
      const size_t smem = (size_t)warps * per_warp;
      if (idx->digest_occ == 0) {
        if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
          return cuda_status(cudaErrorInvalidValue);
        int occ = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, warps * 32, smem) != cudaSuccess)
          return cuda_status(cudaErrorInvalidValue);
        idx->digest_occ = occ < 1 ? 1 : occ;
      }
      const int64_t want = (max_chunks + warps - 1) / warps;
      const int64_t grid = std::max<int64_t>(1, std::min<int64_t>(want, (int64_t)idx->num_sms * idx->digest_occ));
      idx->launches++;
      return launch_k(kern, dim3((unsigned)grid), dim3(warps * 32), smem, s, !idx->profiling, maps, d_tokens,
                      n_tokens, d_offsets, (const int64_t*)idx->block_off, (const int64_t*)idx->chunk_off, n, d_init,
                      (const int32_t*)idx->batch_ok, idx->digest, idx->status, groups, gmask, h_init);
    }
  }
  const size_t per_warp = (size_t)kChunk * nch * 16;
  const int warps = (int)std::max<size_t>(1, std::min<size_t>(kDigestWarps, kDigestSmem / per_warp));
  const size_t smem = (size_t)warps * per_warp;
  auto kern = HB > 0 ? k_digest<HB> : nullptr;
  const void* fn = HB > 0 ? (const void*)kern : (const void*)k_digest_any;
  if (idx->digest_occ == 0) {  // once per index: B, and so the plan, is fixed
    if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kDigestSmem) != cudaSuccess)
      return cuda_status(cudaErrorInvalidValue);
    int occ = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, fn, warps * 32, smem) != cudaSuccess)
      return cuda_status(cudaErrorInvalidValue);
    idx->digest_occ = occ < 1 ? 1 : occ;
  }
  const int64_t want = (max_chunks + warps - 1) / warps;
  const int64_t grid = std::max<int64_t>(1, std::min<int64_t>(want, (int64_t)idx->num_sms * idx->digest_occ));
  idx->launches++;
  if (HB > 0)
    return launch_k(kern, dim3((unsigned)grid), dim3(warps * 32), smem, s, !idx->profiling, d_tokens, n_tokens,
                    d_offsets, (const int64_t*)idx->block_off, n, d_init, (const int32_t*)idx->batch_ok,
                    idx->digest, groups, gmask, h_init);
  return launch_k(k_digest_any, dim3((unsigned)grid), dim3(warps * 32), smem, s, !idx->profiling, d_tokens,
                  n_tokens, d_offsets, (const int64_t*)idx->block_off, n, B, nch, d_init,
                  (const int32_t*)idx->batch_ok, idx->digest, groups, gmask, h_init);
}

int dispatch_digest(smetric_index* idx, const int32_t* d_tokens, int64_t n_tokens,
                    const int64_t* d_offsets, int32_t n, cudaStream_t s, bool group) {
  switch (idx->cfg.block_size) {
    case 16: return launch_digest<8>(idx, d_tokens, n_tokens, d_offsets, n, s, group);
    case 32: return launch_digest<16>(idx, d_tokens, n_tokens, d_offsets, n, s, group);
    case 64: return launch_digest<32>(idx, d_tokens, n_tokens, d_offsets, n, s, group);
    case 128: return launch_digest<64>(idx, d_tokens, n_tokens, d_offsets, n, s, group);
    default: return launch_digest<0>(idx, d_tokens, n_tokens, d_offsets, n, s, group);
  }
}

// Chain, shared prefixes and probe (W > 0), or the chain alone (W = 0): one CTA
// per SM, a chain lane for each request a CTA owns (1 to 4 warps; more requests
// share lanes). The ring's slots per lane fit 139 KB: 8 with one or two chain
// warps, 4 with three or four.
template <int W>
int launch_chain_probe(ChainArgs a, int num_sms, cudaStream_t s, bool pdl) {
  const int grid = (int)std::min<int64_t>(num_sms, a.n);
  const int64_t per_cta = ((int64_t)a.n + grid - 1) / grid;
  a.chain_warps = (int)std::max<int64_t>(1, std::min<int64_t>(kCpMaxChainWarps, (per_cta + 31) / 32));
  a.slots = a.chain_warps <= 2 ? kCpMaxSlots : kCpMaxSlots / 2;
  const size_t smem = (size_t)32 * a.chain_warps * a.slots * kCpRow;
  return launch_k(k_chain_probe<W>, dim3((unsigned)grid), dim3(cp_warps(W) * 32), smem, s, pdl, a);
}

// The limits on dynamic shared memory of the chain kernel and of the sequential
// decisions. A limit belongs to the kernel and not to the index or the call, so
// it is set to the most that any call takes, once per index (the call without an
// index sets it itself), and never lowered: a call on another index and thread
// may come between any two of this one's.
template <int W>
bool chain_limit() {
  return cudaFuncSetAttribute(k_chain_probe<W>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kCpMaxRing) == cudaSuccess;
}
template <int T>
constexpr size_t seq_smem() { return (size_t)kSeqStages * kSeqWarps * 32 * T * sizeof(SeqEntry); }
template <int T>
bool seq_limit() {
  return cudaFuncSetAttribute(k_seq<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)seq_smem<T>()) == cudaSuccess;
}

// The hash-only calls' chain.
int launch_chain(const ChainArgs& a, int num_sms, cudaStream_t s, bool pdl) {
  if (a.n <= 32 * (int64_t)num_sms) return launch_chain_probe<0>(a, num_sms, s, pdl);
  return launch_k(k_chain, dim3((unsigned)((a.n + kChainThreads - 1) / kChainThreads)), dim3(kChainThreads), 0, s, pdl, a);
}

// The arguments that every chain launch of an index has.
ChainArgs chain_args(const smetric_index* idx, int32_t n, uint64_t* sk) {
  ChainArgs a = {};
  a.block_off = idx->block_off;
  a.n = n;
  a.S = idx->cfg.session_blocks;
  a.h_init = mix64(idx->cfg.hash_seed + kGamma);
  a.batch_ok = idx->batch_ok;
  a.D = idx->digest;
  a.sk_out = sk;
  a.status = idx->status;
  return a;
}

template <int W>
int launch_match(smetric_index* idx, const int64_t* d_offsets, int32_t n, const int64_t* d_load,
                 smetric_weights w, int32_t* inst, int32_t* lhit, int32_t* ghit, uint64_t* hashes,
                 uint64_t* sk, const WalkPolicy& pol, cudaStream_t s, const Overlap* ov) {
  const cudaEvent_t after_chain = ov ? ov->after_chain : nullptr;
  const int N = idx->cfg.num_instances;
  int rc;
  // Short tails are left to the walk where the chain warps would have several
  // lanes in use otherwise (with few requests an SM a tail chained after its
  // leader only adds to the batch's time), and while the chain kernel can deal
  // the rest out by k_lead's flags: 32 requests a thread, kCpRound a CTA.
  const bool defer = n > 4 * idx->num_sms && n <= 32 * kCpWarps * 32 &&
                     (n + idx->num_sms - 1) / idx->num_sms <= kCpRound;
  // one byte a request, in the scratch words k_link_sessions uses for its keys
  uint8_t* const flags = reinterpret_cast<uint8_t*>(idx->sk_tmp);
  idx->launches++;
  if ((rc = launch_k(k_lead, dim3((unsigned)((n + 7) / 8)), dim3(256), 0, s, !idx->profiling,
                     (const int64_t*)idx->block_off, n, (const int32_t*)idx->batch_ok, (const uint64_t*)idx->digest,
                     mix64(idx->cfg.hash_seed + kGamma), (const uint64_t*)idx->groups, group_slots_for(n) - 1, defer,
                     idx->lead, idx->share, flags)))
    return rc;
  ChainArgs chain = chain_args(idx, n, sk);
  chain.chunk_off = idx->chunk_off;
  chain.hashes = hashes ? hashes : defer ? idx->hashes : nullptr;
  chain.share = idx->share;
  chain.active = flags;
  chain.deal = defer;
  chain.tags = idx->tags;
  chain.table = idx->table;
  chain.n_buckets = idx->n_buckets;
  chain.masks = idx->masks;
  chain.chunk_and = idx->chunk_and;
  idx->launches++;
  if ((rc = launch_chain_probe<W>(chain, idx->num_sms, s, !idx->profiling))) return rc;
  if (after_chain && cudaEventRecord(after_chain, s) != cudaSuccess) return cuda_status(cudaErrorUnknown);
  profile_mark(idx, kChainProbe, s);
  const int64_t want = ((int64_t)n + kMatchWarps - 1) / kMatchWarps;
  const int64_t grid = std::max<int64_t>(1, std::min<int64_t>(want, (int64_t)idx->num_sms * 8));
  // every request in one pass (members read their leaders' probes)
  using WalkKernel = decltype(&k_walk<W, kArgmin>);  // every instantiation has this signature
  const WalkKernel kerns[5] = {k_walk<W, kArgmin>, k_walk<W, kSession>, k_walk<W, kColoc>, k_walk<W, kBailian>,
                               k_walk<W, kLMetric>};
  const WalkKernel kern = kerns[pol.on];
  idx->launches++;
  WalkArgs a = {};
  a.N = N;
  a.B = idx->cfg.block_size;
  a.S = idx->cfg.session_blocks;
  a.off = d_offsets;
  a.block_off = idx->block_off;
  a.chunk_off = idx->chunk_off;
  a.n = n;
  a.load = d_load;
  a.w_load = w.w_load;
  a.w_miss = w.w_miss;
  a.w_glob = w.w_glob;
  a.masks = idx->masks;
  a.chunk_and = idx->chunk_and;
  a.batch_ok = idx->batch_ok;
  a.lead = idx->lead;
  a.share = idx->share;
  a.summ = idx->summ;
  a.inst_out = inst;
  a.lhit_out = lhit;
  a.ghit_out = ghit;
  a.groups = reinterpret_cast<uint4*>(idx->groups);
  a.group_vecs = (int64_t)group_slots_for(n);
  if (defer) {
    a.active = flags;
    a.D = idx->digest;
    a.hashes = hashes ? hashes : idx->hashes;
    a.want_hashes = hashes != nullptr;
    a.sk_out = sk;
    a.tags = idx->tags;
    a.table = idx->table;
    a.n_buckets = idx->n_buckets;
  }
  if ((rc = launch_k(kern, dim3((unsigned)grid), dim3(kMatchWarps * 32), 0, s, !idx->profiling, a, pol))) return rc;
  return SMETRIC_OK;
}

int dispatch_match(smetric_index* idx, const int64_t* d_offsets, int32_t n, const int64_t* d_load,
                   smetric_weights w, int32_t* inst, int32_t* lhit, int32_t* ghit, uint64_t* hashes,
                   uint64_t* sk, const WalkPolicy& pol, cudaStream_t s, const Overlap* ov) {
  switch (idx->W) {
    case 1: return launch_match<1>(idx, d_offsets, n, d_load, w, inst, lhit, ghit, hashes, sk, pol, s, ov);
    case 2: return launch_match<2>(idx, d_offsets, n, d_load, w, inst, lhit, ghit, hashes, sk, pol, s, ov);
    case 3: return launch_match<3>(idx, d_offsets, n, d_load, w, inst, lhit, ghit, hashes, sk, pol, s, ov);
    case 4: return launch_match<4>(idx, d_offsets, n, d_load, w, inst, lhit, ghit, hashes, sk, pol, s, ov);
    case 5: return launch_match<5>(idx, d_offsets, n, d_load, w, inst, lhit, ghit, hashes, sk, pol, s, ov);
    default: return SMETRIC_ERR_INVALID_ARG;
  }
}

void profile_begin(smetric_index* idx, cudaStream_t s) {
  if (!idx->profiling) return;
  ProfileSlot slot;
  if (!idx->prof_pool.empty()) {
    slot = idx->prof_pool.back();
    idx->prof_pool.pop_back();
  } else {
    for (auto& e : slot.ev)
      if (cudaEventCreate(&e) != cudaSuccess) return;
  }
  idx->prof_used.push_back(slot);
  cudaEventRecord(idx->prof_used.back().ev[0], s);
}

void profile_mark(smetric_index* idx, int k, cudaStream_t s) {
  if (idx->profiling && !idx->prof_used.empty()) cudaEventRecord(idx->prof_used.back().ev[k + 1], s);
}

bool weights_ok(const smetric_weights& w) {
  auto in = [](int64_t v) { return v >= 0 && v <= SMETRIC_MAX_WEIGHT; };
  return in(w.w_load) && in(w.w_miss) && in(w.w_glob);
}

template <bool PROBE>
int route_common(smetric_index* idx, const int32_t* d_tokens, int64_t n_tokens, const int64_t* d_offsets,
                 int32_t n, const int64_t* d_load, smetric_weights w, int32_t* inst, int32_t* lhit,
                 int32_t* ghit, uint64_t* sk, uint64_t* hashes, int64_t hashes_cap, cudaStream_t s,
                 const WalkPolicy* pol = nullptr, const Overlap* ov = nullptr) {
  int rc = check_device(idx);
  if (rc) return rc;
  const smetric_index_config& c = idx->cfg;
  if (n < 0 || n > c.max_batch_requests || n_tokens < 0 || n_tokens > c.max_batch_tokens)
    return SMETRIC_ERR_INVALID_ARG;
  if (n == 0) return SMETRIC_OK;
  if (!d_offsets || !sk || (n_tokens > 0 && !d_tokens)) return SMETRIC_ERR_INVALID_ARG;
  if (d_tokens && (reinterpret_cast<uintptr_t>(d_tokens) & 15)) return SMETRIC_ERR_INVALID_ARG;
  if (PROBE && (!d_load || !inst || !lhit || !ghit || !weights_ok(w))) return SMETRIC_ERR_INVALID_ARG;
  if (hashes && hashes_cap < n_tokens / c.block_size) return SMETRIC_ERR_INVALID_ARG;
  if (!PROBE && !hashes) return SMETRIC_ERR_INVALID_ARG;

  profile_begin(idx, s);
  // the policies' Eq. 1 arithmetic has its own limits on queues and lengths
  const bool eq1 = pol && (pol->on == kSession || pol->on == kColoc);
  k_prep<<<prep_grid(n), kPrepThreads, 0, s>>>((int)prep_passes(n), d_offsets, n, n_tokens, c.block_size, d_load, PROBE ? c.num_instances : 0,
                            idx->block_off, idx->chunk_off, idx->batch_ok, idx->status,
                            eq1 ? SMETRIC_POLICY_MAX_QUEUED : SMETRIC_MAX_LOAD,
                            eq1 ? SMETRIC_POLICY_MAX_LEN : (int64_t)INT32_MAX, pol ? pol->est_hit : nullptr,
                            pol ? pol->tpot : nullptr, SMETRIC_POLICY_MAX_TPOT,
                            pol ? pol->nreq : nullptr, SMETRIC_POLICY_MAX_REQUESTS);
  idx->launches++;
  if ((rc = cuda_status(cudaGetLastError()))) return rc;
  profile_mark(idx, kPrep, s);
  // a route's digests also fill the group table (each request's first-block hash)
  if (n_tokens / c.block_size > 0) {
    if ((rc = dispatch_digest(idx, d_tokens, n_tokens, d_offsets, n, s, PROBE)))
      return rc;
  }
  profile_mark(idx, kDigest, s);
  if (PROBE) {
    const WalkPolicy off_pol = {};
    if ((rc = dispatch_match(idx, d_offsets, n, d_load, w, inst, lhit, ghit, hashes, sk, pol ? *pol : off_pol, s, ov))) {
      empty_groups(idx, n, s);  // the walk that would have emptied the table was not launched
      return rc;
    }
  } else {
    ChainArgs a = chain_args(idx, n, sk);
    a.hashes = hashes;
    idx->launches++;
    if ((rc = launch_chain(a, idx->num_sms, s, !idx->profiling))) return rc;
    profile_mark(idx, kChainProbe, s);
  }
  profile_mark(idx, kWalk, s);
  return SMETRIC_OK;
}

int route_policy(smetric_index* idx, int mode, const int32_t* d_tokens, int64_t n_tokens,
                 const int64_t* d_offsets, int32_t n_requests, const int64_t* d_queued,
                 const int64_t* d_tpot, const int64_t* d_nreq, const int32_t* d_turn,
                 const int64_t* d_est_hit, smetric_policy p, int32_t* d_instance, int32_t* d_local_hit,
                 int32_t* d_global_hit, int32_t* d_stick, uint64_t* d_session_key, uint64_t* d_block_hashes,
                 int64_t hashes_cap, smetric_stream_t stream) {
  if (!idx) return SMETRIC_ERR_INVALID_ARG;
  const int64_t N = idx->cfg.num_instances;
  if (p.c_lin < 0 || p.c_lin > (1LL << 20) || p.c_att < 0 || p.c_att > (1LL << 12) || p.ttft_d0 < 0 ||
      p.ttft_d0 > (1LL << 60) || p.ttft_d1 < 0 || p.ttft_d1 > (1LL << 35) || p.hit_den < 1 ||
      p.hit_den > (1LL << 20) || p.hit_num < 0 || p.hit_num > p.hit_den || p.rr_base < 0 || p.rr_base >= N ||
      p.reserved != 0)
    return SMETRIC_ERR_INVALID_ARG;
  if (n_requests > 0 && (!d_turn || !d_est_hit || !d_stick)) return SMETRIC_ERR_INVALID_ARG;
  WalkPolicy pol = {};
  pol.on = mode;
  pol.c_lin = p.c_lin;
  pol.c_att = p.c_att;
  pol.d0 = p.ttft_d0;
  pol.d1 = p.ttft_d1;
  pol.hit_num = p.hit_num;
  pol.hit_den = p.hit_den;
  pol.rr_base = p.rr_base;
  pol.turn = d_turn;
  pol.est_hit = d_est_hit;
  pol.stick = d_stick;
  pol.tpot = d_tpot;
  pol.nreq = d_nreq;
  // the argmin weights are unused by the policy; any valid ones pass the checks
  return route_common<true>(idx, d_tokens, n_tokens, d_offsets, n_requests, d_queued, smetric_weights{0, 0, 0},
                            d_instance, d_local_hit, d_global_hit, d_session_key, d_block_hashes, hashes_cap,
                            reinterpret_cast<cudaStream_t>(stream), &pol);
}

}  // namespace

#include <mutex>
#include <new>
#include <unordered_map>

#include "call_range.cuh"

// ---------------------------------------------------------------------------
// batches overlapped on two scratch sets
// ---------------------------------------------------------------------------

namespace smetric {

// Shared-memory limits of the kernels that index x's calls launch with more than
// 48 KB (the digest's is set on its first call, the LRU's by smetric_index_set_lru).
bool kernel_limits(const smetric_index* x) {
  const bool chain = x->W == 1   ? chain_limit<1>()
                     : x->W == 2 ? chain_limit<2>()
                     : x->W == 3 ? chain_limit<3>()
                     : x->W == 4 ? chain_limit<4>()
                                 : chain_limit<5>();
  return chain && chain_limit<0>() && seq_limit<1>() && seq_limit<2>() && seq_limit<4>() && seq_limit<8>();
}

// The second route scratch set of an index created with SMETRIC_FLAG_PIPELINE:
// the same buffers, with the same sizes, as the index's own set.
struct RouteScratchSet {
  int64_t* block_off = nullptr;
  int64_t* chunk_off = nullptr;
  uint64_t* digest = nullptr;
  uint64_t* hashes = nullptr;
  uint64_t* masks = nullptr;
  uint64_t* chunk_and = nullptr;
  uint64_t* groups = nullptr;
  int32_t* lead = nullptr;  // lead, then share at lead + max_batch_requests + 1
  int32_t* summ = nullptr;
  uint64_t* sk_tmp = nullptr;
  int32_t* batch_ok = nullptr;
};

struct Pipeline {
  RouteScratchSet alt;
  cudaStream_t stream = nullptr;                   // runs the batches that use `alt`
  cudaEvent_t chain_done[2] = {nullptr, nullptr};  // per set: its latest batch's chain has finished
  cudaEvent_t start = nullptr, finish = nullptr;   // the caller's stream to `stream`, and back
};

// Both live until the process ends and are never destroyed, so that an index
// destroyed late in process exit still finds them.
static std::mutex& pipeline_mutex() {
  static std::mutex* m = new std::mutex;
  return *m;
}

// Indexes created with SMETRIC_FLAG_PIPELINE and their second sets (kept
// beside the index so that the index's layout stays as it is).
static std::unordered_map<const smetric_index*, Pipeline*>& pipelines() {
  static auto* table = new std::unordered_map<const smetric_index*, Pipeline*>;
  return *table;
}

static Pipeline* pipeline_of(const smetric_index* idx) {
  std::lock_guard<std::mutex> lock(pipeline_mutex());
  auto it = pipelines().find(idx);
  return it == pipelines().end() ? nullptr : it->second;
}

static void free_pipeline(Pipeline* p) {
  RouteScratchSet& a = p->alt;
  cudaFree(a.block_off);
  cudaFree(a.chunk_off);
  cudaFree(a.digest);
  cudaFree(a.hashes);
  cudaFree(a.masks);
  cudaFree(a.chunk_and);
  cudaFree(a.groups);
  cudaFree(a.lead);
  cudaFree(a.summ);
  cudaFree(a.sk_tmp);
  cudaFree(a.batch_ok);
  if (p->stream) cudaStreamDestroy(p->stream);
  for (cudaEvent_t e : {p->chain_done[0], p->chain_done[1], p->start, p->finish})
    if (e) cudaEventDestroy(e);
  delete p;
}

// Exchanges the index's route scratch with set `a` (host pointers only: a
// launch takes the pointers current when it is enqueued).
static void swap_scratch(smetric_index* x, RouteScratchSet& a) {
  std::swap(x->block_off, a.block_off);
  std::swap(x->chunk_off, a.chunk_off);
  std::swap(x->digest, a.digest);
  std::swap(x->hashes, a.hashes);
  std::swap(x->masks, a.masks);
  std::swap(x->chunk_and, a.chunk_and);
  std::swap(x->groups, a.groups);
  std::swap(x->lead, a.lead);
  x->share = x->lead + (x->cfg.max_batch_requests + 1);
  std::swap(x->summ, a.summ);
  std::swap(x->sk_tmp, a.sk_tmp);
  std::swap(x->batch_ok, a.batch_ok);
}

// Allocates the second set of index x (called by smetric_index_create once
// the index's own set exists). The sizes are those of the index's own set.
int pipeline_attach(smetric_index* x) {
  const smetric_index_config& c = x->cfg;
  const size_t R = (size_t)c.max_batch_requests;
  const size_t max_blocks = (size_t)(c.max_batch_tokens / c.block_size);
  const size_t nb = max_blocks > 0 ? max_blocks : 1;
  const size_t W = (size_t)x->W;
  Pipeline* p = new (std::nothrow) Pipeline();
  if (!p) return SMETRIC_ERR_OOM;
  RouteScratchSet& a = p->alt;
  bool ok = cudaMalloc(&a.block_off, (R + 1) * sizeof(int64_t)) == cudaSuccess &&
            cudaMalloc(&a.digest, nb * sizeof(uint64_t)) == cudaSuccess &&
            cudaMalloc(&a.hashes, nb * sizeof(uint64_t)) == cudaSuccess &&
            cudaMalloc(&a.masks, nb * W * sizeof(uint64_t)) == cudaSuccess &&
            cudaMalloc(&a.chunk_and, (max_blocks / 32 + R + 1) * W * sizeof(uint64_t)) == cudaSuccess &&
            cudaMalloc(&a.groups, 2 * x->group_slots * sizeof(uint64_t)) == cudaSuccess &&
            cudaMalloc(&a.lead, 2 * (R + 1) * sizeof(int32_t)) == cudaSuccess &&
            cudaMalloc(&a.chunk_off, (R + 1) * sizeof(int64_t)) == cudaSuccess &&
            cudaMalloc(&a.sk_tmp, (R + 1) * sizeof(uint64_t)) == cudaSuccess &&
            cudaMalloc(&a.summ, (R > 0 ? R : 1) * ((size_t)c.num_instances + 1) * sizeof(int32_t)) == cudaSuccess &&
            cudaMalloc(&a.batch_ok, sizeof(int32_t)) == cudaSuccess &&
            cudaMemset(a.groups, 0, 2 * x->group_slots * sizeof(uint64_t)) == cudaSuccess &&
            cudaStreamCreateWithFlags(&p->stream, cudaStreamNonBlocking) == cudaSuccess;
  for (cudaEvent_t* e : {&p->chain_done[0], &p->chain_done[1], &p->start, &p->finish})
    ok = ok && cudaEventCreateWithFlags(e, cudaEventDisableTiming) == cudaSuccess;
  if (!ok) {
    (void)cudaGetLastError();
    free_pipeline(p);
    return SMETRIC_ERR_OOM;
  }
  std::lock_guard<std::mutex> lock(pipeline_mutex());
  pipelines()[x] = p;
  return SMETRIC_OK;
}

// Frees the second set of index x, if it has one (the device is idle).
void pipeline_release(smetric_index* x) {
  Pipeline* p = nullptr;
  {
    std::lock_guard<std::mutex> lock(pipeline_mutex());
    auto it = pipelines().find(x);
    if (it == pipelines().end()) return;
    p = it->second;
    pipelines().erase(it);
  }
  free_pipeline(p);
}

}  // namespace smetric

namespace {

// smetric_route_batches: the host checks of route_common for every batch
// first, then the batches, alternating between the two sets when the index
// has a second one. Batch j's first kernel waits for batch j - 1's chain and
// probe kernel, so that batch j's prep and digests (bound by the integer
// pipe) run beside batch j - 1's walk (bound by latency), and batch j - 1's
// chain does not share the GPU with batch j's digests.
int route_batches(smetric_index* idx, int32_t nb, const int32_t* const* tok, const int64_t* ntok,
                  const int64_t* const* off, const int32_t* nreq, const int64_t* const* load, smetric_weights w,
                  int32_t* const* inst, int32_t* const* lhit, int32_t* const* ghit, uint64_t* const* sk,
                  cudaStream_t s) {
  int rc = check_device(idx);
  if (rc) return rc;
  if (nb < 0 || (nb > 0 && (!tok || !ntok || !off || !nreq || !load || !inst || !lhit || !ghit || !sk)))
    return SMETRIC_ERR_INVALID_ARG;
  const smetric_index_config& c = idx->cfg;
  for (int32_t j = 0; j < nb; ++j) {
    const int32_t n = nreq[j];
    const int64_t nt = ntok[j];
    if (n < 0 || n > c.max_batch_requests || nt < 0 || nt > c.max_batch_tokens) return SMETRIC_ERR_INVALID_ARG;
    if (n == 0) continue;
    if (!off[j] || !sk[j] || (nt > 0 && !tok[j])) return SMETRIC_ERR_INVALID_ARG;
    if (tok[j] && (reinterpret_cast<uintptr_t>(tok[j]) & 15)) return SMETRIC_ERR_INVALID_ARG;
    if (!load[j] || !inst[j] || !lhit[j] || !ghit[j] || !weights_ok(w)) return SMETRIC_ERR_INVALID_ARG;
  }
  Pipeline* p = pipeline_of(idx);
  if (!p || idx->profiling || nb < 2) {
    for (int32_t j = 0; j < nb; ++j)
      if ((rc = route_common<true>(idx, tok[j], ntok[j], off[j], nreq[j], load[j], w, inst[j], lhit[j], ghit[j],
                                   sk[j], nullptr, 0, s)))
        return rc;
    return SMETRIC_OK;
  }
  // the second stream starts from everything enqueued on the caller's stream
  if (cudaEventRecord(p->start, s) != cudaSuccess || cudaStreamWaitEvent(p->stream, p->start, 0) != cudaSuccess)
    return cuda_status(cudaErrorUnknown);
  for (int32_t j = 0; j < nb && rc == SMETRIC_OK; ++j) {
    const int set = j & 1;
    cudaStream_t sj = set ? p->stream : s;
    if (j > 0 && cudaStreamWaitEvent(sj, p->chain_done[set ^ 1], 0) != cudaSuccess) {
      rc = cuda_status(cudaErrorUnknown);
      break;
    }
    if (set) swap_scratch(idx, p->alt);
    const Overlap ov = {p->chain_done[set]};
    rc = route_common<true>(idx, tok[j], ntok[j], off[j], nreq[j], load[j], w, inst[j], lhit[j], ghit[j], sk[j],
                            nullptr, 0, sj, nullptr, &ov);
    if (set) swap_scratch(idx, p->alt);
  }
  // the caller's stream continues after the second stream's batches
  if (cudaEventRecord(p->finish, p->stream) != cudaSuccess || cudaStreamWaitEvent(s, p->finish, 0) != cudaSuccess)
    return rc ? rc : cuda_status(cudaErrorUnknown);
  return rc;
}

// smetric_index_commit_batch's steps; with prep the batch's block offsets
// and validity are computed here, else a route call just left them.
int commit_common(smetric_index* idx, const int64_t* d_offsets, int32_t n_requests, const int32_t* d_instance,
                  const int32_t* d_local_hit, const uint64_t* d_block_hashes, int32_t flags, int64_t* d_load,
                  cudaStream_t s, bool prep) {
  int rc = check_device(idx);
  if (rc) return rc;
  const smetric_index_config& c = idx->cfg;
  if (n_requests < 0 || n_requests > c.max_batch_requests || (flags & ~SMETRIC_COMMIT_GLOBAL))
    return SMETRIC_ERR_INVALID_ARG;
  if (n_requests == 0) return SMETRIC_OK;
  if (!d_offsets || !d_instance || !d_block_hashes || (d_load && !d_local_hit)) return SMETRIC_ERR_INVALID_ARG;
  if (prep) {
    // block offsets of the batch (and the offsets' checks) into the index's scratch
    k_prep<<<prep_grid(n_requests), kPrepThreads, 0, s>>>((int)prep_passes(n_requests), d_offsets, n_requests, c.max_batch_tokens, c.block_size, nullptr, 0, idx->block_off,
                              nullptr, idx->batch_ok, idx->status, SMETRIC_MAX_LOAD, (int64_t)INT32_MAX, nullptr);
    idx->launches++;
    if ((rc = cuda_status(cudaGetLastError()))) return rc;
  }
  const bool global = (flags & SMETRIC_COMMIT_GLOBAL) != 0;
  if (idx->lru)
    return lru_commit(idx, d_offsets, d_instance, d_local_hit, d_block_hashes, n_requests, global, d_load, s);
  // the checks (and the drain) first: a bad output commits nothing
  idx->launches++;
  if ((rc = launch_k(k_drain, dim3(1), dim3(1024), 0, s, true, d_offsets, n_requests, c.num_instances, d_instance,
                     d_local_hit, idx->batch_ok, d_load, idx->status)))
    return rc;
  return launch_commit(idx, d_instance, d_block_hashes, n_requests, c.max_batch_tokens / c.block_size, global, s);
}

}  // namespace

extern "C" {

int smetric_route_batch(smetric_index* idx, const int32_t* d_tokens, int64_t n_tokens,
                        const int64_t* d_offsets, int32_t n_requests, const int64_t* d_load,
                        smetric_weights w, int32_t* d_instance, int32_t* d_local_hit,
                        int32_t* d_global_hit, uint64_t* d_session_key, uint64_t* d_block_hashes,
                        int64_t hashes_cap, smetric_stream_t stream) {
  CallRange range("smetric_route_batch");
  return route_common<true>(idx, d_tokens, n_tokens, d_offsets, n_requests, d_load, w, d_instance,
                            d_local_hit, d_global_hit, d_session_key, d_block_hashes, hashes_cap,
                            reinterpret_cast<cudaStream_t>(stream));
}

int smetric_route_batches(smetric_index* idx, int32_t n_batches, const int32_t* const* d_tokens,
                          const int64_t* n_tokens, const int64_t* const* d_offsets, const int32_t* n_requests,
                          const int64_t* const* d_load, smetric_weights w, int32_t* const* d_instance,
                          int32_t* const* d_local_hit, int32_t* const* d_global_hit,
                          uint64_t* const* d_session_key, smetric_stream_t stream) {
  CallRange range("smetric_route_batches");
  return route_batches(idx, n_batches, d_tokens, n_tokens, d_offsets, n_requests, d_load, w, d_instance,
                       d_local_hit, d_global_hit, d_session_key, reinterpret_cast<cudaStream_t>(stream));
}

int smetric_route_batch_sequential(smetric_index* idx, const int32_t* d_tokens, int64_t n_tokens,
                                   const int64_t* d_offsets, int32_t n_requests, const int64_t* d_load,
                                   smetric_weights w, int32_t* d_instance, int32_t* d_local_hit,
                                   int32_t* d_global_hit, uint64_t* d_session_key, uint64_t* d_block_hashes,
                                   int64_t hashes_cap, int64_t* d_load_after, smetric_stream_t stream) {
  CallRange range("smetric_route_batch_sequential");
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  WalkPolicy pol = {};
  pol.summ = 1;
  int rc = route_common<true>(idx, d_tokens, n_tokens, d_offsets, n_requests, d_load, w, d_instance, d_local_hit,
                              d_global_hit, d_session_key, d_block_hashes, hashes_cap, s, &pol);
  if (rc || n_requests == 0) return rc;
  idx->launches++;
  const int N = idx->cfg.num_instances;
  auto launch = [&](auto kern, size_t smem) {
    kern<<<1, kSeqBlock * 32, smem, s>>>(N, idx->cfg.block_size, d_offsets, n_requests, d_load, w.w_load,
                                               w.w_miss, w.w_glob, idx->summ, idx->batch_ok, d_instance, d_local_hit,
                                               d_global_hit, d_load_after, idx->status);
    return cuda_status(cudaGetLastError());
  };
  return N <= 32    ? launch(k_seq<1>, seq_smem<1>())
         : N <= 64  ? launch(k_seq<2>, seq_smem<2>())
         : N <= 128 ? launch(k_seq<4>, seq_smem<4>())
                    : launch(k_seq<8>, seq_smem<8>());
}

int smetric_route_batch_baseline(smetric_index* idx, const int32_t* d_tokens, int64_t n_tokens,
                                 const int64_t* d_offsets, int32_t n_requests, int32_t scorer,
                                 const int64_t* d_queued, const int64_t* d_batch, int64_t lam_num,
                                 int64_t lam_den, int32_t* d_instance, int32_t* d_local_hit,
                                 int32_t* d_global_hit, uint64_t* d_session_key, uint64_t* d_block_hashes,
                                 int64_t hashes_cap, smetric_stream_t stream) {
  CallRange range("smetric_route_batch_baseline");
  if (!idx || !d_batch || (scorer != SMETRIC_SCORER_BAILIAN && scorer != SMETRIC_SCORER_LMETRIC) ||
      lam_den < 1 || lam_den > (1LL << 20) || lam_num < 0 || lam_num > lam_den)
    return SMETRIC_ERR_INVALID_ARG;
  WalkPolicy pol = {};
  pol.on = scorer == SMETRIC_SCORER_BAILIAN ? kBailian : kLMetric;
  pol.nreq = d_batch;
  pol.lam_num = lam_num;
  pol.lam_den = lam_den;
  return route_common<true>(idx, d_tokens, n_tokens, d_offsets, n_requests, d_queued, smetric_weights{0, 0, 0},
                            d_instance, d_local_hit, d_global_hit, d_session_key, d_block_hashes, hashes_cap,
                            reinterpret_cast<cudaStream_t>(stream), &pol);
}

int smetric_route_batch_policy_coloc(smetric_index* idx, const int32_t* d_tokens, int64_t n_tokens,
                                     const int64_t* d_offsets, int32_t n_requests, const int64_t* d_queued,
                                     const int64_t* d_tpot_budget, const int64_t* d_num_requests,
                                     const int32_t* d_turn, const int64_t* d_est_hit, smetric_policy p,
                                     int32_t* d_instance, int32_t* d_local_hit, int32_t* d_global_hit,
                                     int32_t* d_stick, uint64_t* d_session_key, uint64_t* d_block_hashes,
                                     int64_t hashes_cap, smetric_stream_t stream) {
  CallRange range("smetric_route_batch_policy_coloc");
  if (!idx || !d_tpot_budget || !d_num_requests) return SMETRIC_ERR_INVALID_ARG;
  return route_policy(idx, kColoc, d_tokens, n_tokens, d_offsets, n_requests, d_queued, d_tpot_budget,
                      d_num_requests, d_turn, d_est_hit, p, d_instance, d_local_hit, d_global_hit, d_stick,
                      d_session_key, d_block_hashes, hashes_cap, stream);
}

int smetric_route_batch_policy(smetric_index* idx, const int32_t* d_tokens, int64_t n_tokens,
                               const int64_t* d_offsets, int32_t n_requests, const int64_t* d_queued,
                               const int32_t* d_turn, const int64_t* d_est_hit, smetric_policy p,
                               int32_t* d_instance, int32_t* d_local_hit, int32_t* d_global_hit,
                               int32_t* d_stick, uint64_t* d_session_key, uint64_t* d_block_hashes,
                               int64_t hashes_cap, smetric_stream_t stream) {
  CallRange range("smetric_route_batch_policy");
  return route_policy(idx, kSession, d_tokens, n_tokens, d_offsets, n_requests, d_queued, nullptr, nullptr,
                      d_turn, d_est_hit, p, d_instance, d_local_hit, d_global_hit, d_stick, d_session_key,
                      d_block_hashes, hashes_cap, stream);
}


int smetric_index_commit_batch(smetric_index* idx, const int64_t* d_offsets, int32_t n_requests,
                               const int32_t* d_instance, const int32_t* d_local_hit,
                               const uint64_t* d_block_hashes, int32_t flags, int64_t* d_load,
                               smetric_stream_t stream) {
  CallRange range("smetric_index_commit_batch");
  return commit_common(idx, d_offsets, n_requests, d_instance, d_local_hit, d_block_hashes, flags, d_load,
                       reinterpret_cast<cudaStream_t>(stream), true);
}

int smetric_route_commit_batch(smetric_index* idx, const int32_t* d_tokens, int64_t n_tokens,
                               const int64_t* d_offsets, int32_t n_requests, int64_t* d_load,
                               smetric_weights w, int32_t* d_instance, int32_t* d_local_hit,
                               int32_t* d_global_hit, uint64_t* d_session_key, uint64_t* d_block_hashes,
                               int64_t hashes_cap, int32_t flags, smetric_stream_t stream) {
  CallRange range("smetric_route_commit_batch");
  if ((flags & ~SMETRIC_COMMIT_GLOBAL) || !d_block_hashes) return SMETRIC_ERR_INVALID_ARG;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  const int rc = route_common<true>(idx, d_tokens, n_tokens, d_offsets, n_requests, d_load, w, d_instance,
                                    d_local_hit, d_global_hit, d_session_key, d_block_hashes, hashes_cap, s);
  if (rc) return rc;
  // the route's prep left this batch's block offsets and validity in the scratch
  return commit_common(idx, d_offsets, n_requests, d_instance, d_local_hit, d_block_hashes, flags, d_load, s,
                       false);
}

int64_t smetric_reuse_workspace_bytes(int64_t n_blocks) {
  return n_blocks < 0 ? 0 : (int64_t)(2 * sizeof(uint64_t) * reuse_slots_for(n_blocks) + sizeof(ReuseHeader));
}

int smetric_reuse_breakdown(smetric_index* idx, const int32_t* d_tokens, int64_t n_tokens,
                            const int64_t* d_offsets, int32_t n_requests, const int32_t* d_sessions,
                            const int32_t* d_sys_blocks, void* d_workspace, int64_t workspace_bytes,
                            int32_t* d_hit, int32_t* d_sys, int32_t* d_intra, int32_t* d_inter,
                            smetric_stream_t stream) {
  CallRange range("smetric_reuse_breakdown");
  int rc = check_device(idx);
  if (rc) return rc;
  if (n_requests < 0 || n_requests > idx->cfg.max_batch_requests || n_tokens < 0) return SMETRIC_ERR_INVALID_ARG;
  if (n_requests == 0) return SMETRIC_OK;
  const int64_t n_blocks = n_tokens / idx->cfg.block_size;
  if (!d_sessions || !d_sys_blocks || !d_hit || !d_sys || !d_intra || !d_inter || !d_workspace ||
      workspace_bytes < smetric_reuse_workspace_bytes(n_blocks) || (reinterpret_cast<uintptr_t>(d_workspace) & 15))
    return SMETRIC_ERR_INVALID_ARG;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  if ((rc = route_common<false>(idx, d_tokens, n_tokens, d_offsets, n_requests, nullptr, smetric_weights{0, 0, 0},
                                nullptr, nullptr, nullptr, idx->sk_tmp, idx->hashes, n_blocks, s)))
    return rc;
  const uint64_t slots = reuse_slots_for(n_blocks), small = reuse_small_slots_for(n_blocks);
  uint64_t* table = static_cast<uint64_t*>(d_workspace);
  ReuseHeader* hdr = reinterpret_cast<ReuseHeader*>(table + 2 * slots);
  if (cudaMemsetAsync(table, 0, 2 * sizeof(uint64_t) * small, s) != cudaSuccess ||
      cudaMemsetAsync(hdr, 0, sizeof(ReuseHeader), s) != cudaSuccess)
    return cuda_status(cudaErrorUnknown);
  const unsigned wgrid = (unsigned)std::max<int64_t>(1, std::min<int64_t>(((int64_t)n_requests + 7) / 8,
                                                                          (int64_t)idx->num_sms * 8));
  // few enough in flight that a turn is mostly in before the next one looks
  const unsigned igrid = std::min<unsigned>(wgrid, 2u * (unsigned)idx->num_sms);
  k_reuse_insert<false><<<igrid, 256, 0, s>>>(idx->block_off, n_requests, idx->batch_ok, idx->hashes, d_sessions,
                                              table, small - 1, hdr, (uint32_t)(small / 2));
  k_reuse_clear<<<idx->num_sms * 8, 256, 0, s>>>(hdr, reinterpret_cast<uint4*>(table), (int64_t)slots);
  k_reuse_insert<true><<<igrid, 256, 0, s>>>(idx->block_off, n_requests, idx->batch_ok, idx->hashes, d_sessions,
                                             table, slots - 1, hdr, 0);
  k_reuse_walk<<<wgrid, 256, 0, s>>>(idx->block_off, n_requests, idx->batch_ok, idx->hashes, table, small - 1,
                                     slots - 1, hdr, d_sessions, d_sys_blocks, d_hit, d_sys, d_intra, d_inter,
                                     idx->status);
  idx->launches += 4;
  return cuda_status(cudaGetLastError());
}

int smetric_link_sessions(smetric_index* idx, const int32_t* d_tokens, int64_t n_tokens,
                          const int64_t* d_offsets, int32_t n_requests, const int64_t* d_users,
                          const int32_t* d_turns, int32_t* d_parent, int32_t* d_session,
                          smetric_stream_t stream) {
  CallRange range("smetric_link_sessions");
  int rc = check_device(idx);
  if (rc) return rc;
  if (n_requests < 0 || n_requests > idx->cfg.max_batch_requests) return SMETRIC_ERR_INVALID_ARG;
  if (n_requests == 0) return SMETRIC_OK;
  if (!d_users || !d_turns || !d_parent || !d_session) return SMETRIC_ERR_INVALID_ARG;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  // block hashes of the batch into the index's scratch
  if ((rc = route_common<false>(idx, d_tokens, n_tokens, d_offsets, n_requests, nullptr, smetric_weights{0, 0, 0},
                                nullptr, nullptr, nullptr, idx->sk_tmp, idx->hashes,
                                n_tokens / idx->cfg.block_size, s)))
    return rc;
  const uint64_t gmask = group_slots_for(n_requests) - 1;
  const dim3 g((unsigned)((n_requests + 255) / 256)), t(256);
  const int64_t want = (n_tokens / idx->cfg.block_size + n_requests + 255) / 256;
  const dim3 grid((unsigned)std::max<int64_t>(1, std::min<int64_t>(want, (int64_t)idx->num_sms * 8)));
  const int64_t* const bo = idx->block_off;
  const int32_t* const ok = idx->batch_ok;
  const uint64_t* const H = idx->hashes;
  uint64_t* const table = idx->groups;
  int32_t* const next = idx->lead;  // per request: the next of its turn's list
  LinkState* const st = reinterpret_cast<LinkState*>(idx->share);
  uint4* const vecs = reinterpret_cast<uint4*>(table);
  idx->launches += 7;
  if ((rc = launch_k(k_link_turns, g, t, 0, s, true, n_requests, ok, d_users, d_turns, table, gmask, next, st)) ||
      (rc = launch_k(k_link_parents, g, t, 0, s, true, bo, n_requests, ok, H, d_users, d_turns,
                     (const uint64_t*)table, gmask, (const int32_t*)next, d_parent, d_session, st)) ||
      (rc = launch_k(k_link_clear, dim3((unsigned)idx->num_sms), t, 0, s, true, (const LinkState*)st, vecs,
                     (int64_t)(gmask + 1))) ||
      (rc = launch_k(k_link_insert, g, t, 0, s, true, bo, n_requests, ok, H, d_users, d_turns, table, gmask,
                     (const LinkState*)st)) ||
      (rc = launch_k(k_link_find, grid, t, 0, s, true, bo, n_requests, ok, H, d_users, d_turns,
                     (const uint64_t*)table, gmask, d_parent, (const int32_t*)d_session, (const LinkState*)st)) ||
      (rc = launch_k(k_link_chase, g, t, 0, s, true, n_requests, ok, (const int32_t*)d_parent, d_session, st)) ||
      (rc = launch_k(k_link_heads, dim3((unsigned)std::min<int64_t>(1 + ((int64_t)gmask + 1024) / 1024, idx->num_sms)),
                     dim3(1024), 0, s, true, n_requests, ok, d_parent, d_session, vecs, (int64_t)(gmask + 1),
                     (const LinkState*)st))) {
    empty_groups(idx, n_requests, s);
    return rc;
  }
  return SMETRIC_OK;
}

int smetric_block_hashes(smetric_index* idx, const int32_t* d_tokens, int64_t n_tokens,
                         const int64_t* d_offsets, int32_t n_requests, uint64_t* d_session_key,
                         uint64_t* d_block_hashes, int64_t hashes_cap, smetric_stream_t stream) {
  CallRange range("smetric_block_hashes");
  smetric_weights w{0, 0, 0};
  return route_common<false>(idx, d_tokens, n_tokens, d_offsets, n_requests, nullptr, w, nullptr,
                             nullptr, nullptr, d_session_key, d_block_hashes, hashes_cap,
                             reinterpret_cast<cudaStream_t>(stream));
}

int smetric_route_batch_host(smetric_index* idx, const int32_t* h_tokens, int64_t n_tokens,
                             const int64_t* h_offsets, int32_t n_requests, const int64_t* h_load,
                             smetric_weights w, int32_t* h_instance, int32_t* h_local_hit,
                             int32_t* h_global_hit, uint64_t* h_session_key, smetric_stream_t stream) {
  CallRange range("smetric_route_batch_host");
  int rc = check_device(idx);
  if (rc) return rc;
  if (!(idx->cfg.flags & SMETRIC_FLAG_HOST_STAGING)) return SMETRIC_ERR_INVALID_ARG;
  const smetric_index_config& c = idx->cfg;
  if (n_requests < 0 || n_requests > c.max_batch_requests || n_tokens < 0 || n_tokens > c.max_batch_tokens)
    return SMETRIC_ERR_INVALID_ARG;
  if (n_requests == 0) return SMETRIC_OK;
  if (!h_offsets || !h_load || !h_instance || !h_local_hit || !h_global_hit || !h_session_key ||
      (n_tokens > 0 && !h_tokens))
    return SMETRIC_ERR_INVALID_ARG;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  const size_t R = (size_t)n_requests, N = (size_t)c.num_instances;
  const bool small = n_requests <= kHostSmall;
  int64_t* const d_load = idx->st_in;
  int64_t* const d_offsets = idx->st_in + N;
  uint64_t* const d_sk = idx->st_out;
  int32_t* const o = reinterpret_cast<int32_t*>(idx->st_out + R);
  // The caller's arrays are read when the stream gets there: pinned ones may still be written by what is enqueued
  // before this call.
  bool ok = true;
  if (n_tokens > 0)
    ok = ok && cudaMemcpyAsync(idx->st_tokens, h_tokens, (size_t)n_tokens * sizeof(int32_t),
                               cudaMemcpyHostToDevice, s) == cudaSuccess;
  ok = ok && cudaMemcpyAsync(d_offsets, h_offsets, (R + 1) * sizeof(int64_t), cudaMemcpyHostToDevice, s) == cudaSuccess &&
       cudaMemcpyAsync(d_load, h_load, N * sizeof(int64_t), cudaMemcpyHostToDevice, s) == cudaSuccess;
  if (!ok) return cuda_status(cudaErrorUnknown);
  rc = smetric_route_batch(idx, idx->st_tokens, n_tokens, d_offsets, n_requests, d_load, w, o, o + R, o + 2 * R,
                           d_sk, nullptr, 0, stream);
  if (rc) return rc;
  if (small) {
    // the status and every output, then one wait
    ok = cudaMemcpyAsync(idx->st_pin, idx->status, kStatusBytes + R * 20, cudaMemcpyDeviceToHost, s) == cudaSuccess;
    if (cudaStreamSynchronize(s) != cudaSuccess || !ok) return cuda_status(cudaErrorUnknown);
    const int32_t status = *reinterpret_cast<const int32_t*>(idx->st_pin);
    const unsigned char* const keys = idx->st_pin + kStatusBytes;
    const unsigned char* const p = keys + R * sizeof(uint64_t);
    memcpy(h_session_key, keys, R * sizeof(uint64_t));
    memcpy(h_instance, p, R * sizeof(int32_t));
    memcpy(h_local_hit, p + R * sizeof(int32_t), R * sizeof(int32_t));
    memcpy(h_global_hit, p + 2 * R * sizeof(int32_t), R * sizeof(int32_t));
    if (status != 0 && cudaMemset(idx->status, 0, sizeof(int32_t)) != cudaSuccess) return cuda_status(cudaErrorUnknown);
    return status;
  }
  ok = cudaMemcpyAsync(h_instance, o, R * sizeof(int32_t), cudaMemcpyDeviceToHost, s) == cudaSuccess &&
       cudaMemcpyAsync(h_local_hit, o + R, R * sizeof(int32_t), cudaMemcpyDeviceToHost, s) == cudaSuccess &&
       cudaMemcpyAsync(h_global_hit, o + 2 * R, R * sizeof(int32_t), cudaMemcpyDeviceToHost, s) == cudaSuccess &&
       cudaMemcpyAsync(h_session_key, d_sk, R * sizeof(uint64_t), cudaMemcpyDeviceToHost, s) == cudaSuccess;
  if (!ok) return cuda_status(cudaErrorUnknown);
  return smetric_status(idx, stream);
}

int smetric_profile_enable(smetric_index* idx, int32_t on) {
  if (!idx) return SMETRIC_ERR_INVALID_ARG;
  idx->profiling = on != 0;
  return SMETRIC_OK;
}

int smetric_profile_read(smetric_index* idx, int32_t max_kernels, double* ms, int64_t* launches) {
  if (!idx || max_kernels < 0 || (max_kernels > 0 && (!ms || !launches))) return SMETRIC_ERR_INVALID_ARG;
  const int k = std::min<int>(max_kernels, kNumRouteKernels);
  for (int i = 0; i < k; ++i) { ms[i] = 0; launches[i] = 0; }
  int rc = SMETRIC_OK;
  for (auto& slot : idx->prof_used) {
    if (cudaEventSynchronize(slot.ev[kNumRouteKernels]) != cudaSuccess) { rc = cuda_status(cudaErrorUnknown); continue; }
    for (int i = 0; i < k; ++i) {
      float t = 0;
      if (cudaEventElapsedTime(&t, slot.ev[i], slot.ev[i + 1]) == cudaSuccess) {
        ms[i] += t;
        launches[i] += 1;
      } else {
        (void)cudaGetLastError();
      }
    }
    idx->prof_pool.push_back(slot);
  }
  idx->prof_used.clear();
  return rc ? rc : kNumRouteKernels;
}

const char* smetric_profile_kernel_name(int32_t k) {
  switch (k) {
    case kPrep: return "k_prep";
    case kDigest: return "k_digest";
    case kChainProbe: return "k_chain_probe";
    case kWalk: return "k_walk";
    default: return "";
  }
}

}  // extern "C"

// ---------------------------------------------------------------------------
// block hashes with fixed scratch and no allocation
// ---------------------------------------------------------------------------

namespace {

// Word layout of the fixed scratch: the batch-valid flag, the per-request
// first-block offsets, the per-block digests. Each part starts on a 256-byte
// boundary. Nothing in it needs an initial value: every call writes the flag
// and the offsets before any kernel reads them, and the digests of exactly
// the blocks the chain reads.
constexpr int64_t kNaFlagWords = 32;
constexpr int64_t kNaOffWords = (SMETRIC_NOALLOC_MAX_REQUESTS + 1 + 31) / 32 * 32;
constexpr int64_t kNaWords = kNaFlagWords + kNaOffWords + SMETRIC_NOALLOC_MAX_BLOCKS;
static_assert(kNaWords * 8 == 295424, "the header states the scratch size");

static __device__ __align__(256) uint64_t na_scratch[kNaWords];

constexpr int kNaMaxDevices = 64;
std::atomic<uint64_t*> na_addr[kNaMaxDevices];

// Device address of na_scratch on the current device, looked up once per
// device (the first call on a device should not be under stream capture).
// The cached address is not refreshed after a device reset (a reset
// recreates the context and reloads the module).
int na_scratch_for(int dev, uint64_t** out) {
  if (dev < 0 || dev >= kNaMaxDevices) return SMETRIC_ERR_INVALID_ARG;
  uint64_t* p = na_addr[dev].load(std::memory_order_acquire);
  if (!p) {
    if (cudaGetSymbolAddress(reinterpret_cast<void**>(&p), na_scratch) != cudaSuccess)
      return cuda_status(cudaErrorInvalidSymbol);
    na_addr[dev].store(p, std::memory_order_release);
  }
  *out = p;
  return SMETRIC_OK;
}

template <int HB>
int na_digest(const int32_t* d_tokens, int64_t n_tokens, const int64_t* d_offsets, const int64_t* block_off,
              int32_t n, int B, int num_sms, uint64_t d_init, const int32_t* ok, uint64_t* digest,
              cudaStream_t s) {
  const int64_t max_chunks = (n_tokens / B + kChunk - 1) / kChunk;
  const int nch = HB > 0 ? HB / 2 + 1 : (4 * B + 12 + 15) / 16;
  const size_t per_warp = (size_t)kChunk * nch * 16;
  const int warps = (int)std::max<size_t>(1, std::min<size_t>(kDigestWarps, kDigestSmem / per_warp));
  const size_t smem = (size_t)warps * per_warp;
  const void* fn = HB > 0 ? (const void*)k_digest<(HB > 0 ? HB : 2)> : (const void*)k_digest_any;
  int occ = 0;
  if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kDigestSmem) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, fn, warps * 32, smem) != cudaSuccess)
    return cuda_status(cudaErrorInvalidValue);
  const int64_t want = (max_chunks + warps - 1) / warps;
  const int64_t grid = std::max<int64_t>(1, std::min<int64_t>(want, (int64_t)num_sms * std::max(occ, 1)));
  if (HB > 0)
    k_digest<(HB > 0 ? HB : 2)><<<(unsigned)grid, warps * 32, smem, s>>>(d_tokens, n_tokens, d_offsets,
                                                                        block_off, n, d_init, ok, digest,
                                                                        nullptr, 0, 0);
  else
    k_digest_any<<<(unsigned)grid, warps * 32, smem, s>>>(d_tokens, n_tokens, d_offsets, block_off, n, B, nch,
                                                          d_init, ok, digest, nullptr, 0, 0);
  return cuda_status(cudaGetLastError());
}

}  // namespace

extern "C" int smetric_block_hashes_noalloc(const int32_t* d_tokens, int64_t n_tokens,
                                            const int64_t* d_offsets, int32_t n_requests, int32_t block_size,
                                            int32_t session_blocks, uint64_t hash_seed,
                                            uint64_t* d_session_key, uint64_t* d_block_hashes,
                                            int64_t hashes_cap, int32_t* d_status, smetric_stream_t stream) {
  const int B = block_size;
  if (B < 2 || B > 256 || (B & 1) || session_blocks < 1 || n_requests < 0 || n_tokens < 0)
    return SMETRIC_ERR_INVALID_ARG;
  if (n_requests > SMETRIC_NOALLOC_MAX_REQUESTS || n_tokens / B > SMETRIC_NOALLOC_MAX_BLOCKS)
    return SMETRIC_ERR_TOO_LARGE;
  if (n_requests == 0) return SMETRIC_OK;
  if (!d_offsets || !d_session_key || !d_block_hashes || !d_status || (n_tokens > 0 && !d_tokens))
    return SMETRIC_ERR_INVALID_ARG;
  if (d_tokens && (reinterpret_cast<uintptr_t>(d_tokens) & 15)) return SMETRIC_ERR_INVALID_ARG;
  if (hashes_cap < n_tokens / B) return SMETRIC_ERR_INVALID_ARG;
  int dev = 0, num_sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&num_sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return cuda_status(cudaErrorInvalidDevice);
  uint64_t* scratch = nullptr;
  int rc = na_scratch_for(dev, &scratch);
  if (rc) return rc;
  int32_t* ok = reinterpret_cast<int32_t*>(scratch);
  int64_t* block_off = reinterpret_cast<int64_t*>(scratch + kNaFlagWords);
  uint64_t* digest = scratch + kNaFlagWords + kNaOffWords;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);

  k_prep<<<prep_grid(n_requests), kPrepThreads, 0, s>>>((int)prep_passes(n_requests), d_offsets, n_requests, n_tokens, B, nullptr, 0, block_off, nullptr, ok, d_status,
                            SMETRIC_MAX_LOAD, (int64_t)INT32_MAX, nullptr);
  if ((rc = cuda_status(cudaGetLastError()))) return rc;
  if (n_tokens / B > 0) {
    const uint64_t d_init = mix64(hash_seed ^ (uint64_t)B);
    switch (B) {
      case 16: rc = na_digest<8>(d_tokens, n_tokens, d_offsets, block_off, n_requests, B, num_sms, d_init, ok, digest, s); break;
      case 32: rc = na_digest<16>(d_tokens, n_tokens, d_offsets, block_off, n_requests, B, num_sms, d_init, ok, digest, s); break;
      case 64: rc = na_digest<32>(d_tokens, n_tokens, d_offsets, block_off, n_requests, B, num_sms, d_init, ok, digest, s); break;
      default: rc = na_digest<0>(d_tokens, n_tokens, d_offsets, block_off, n_requests, B, num_sms, d_init, ok, digest, s);
    }
    if (rc) return rc;
  }
  ChainArgs a = {};
  a.block_off = block_off;
  a.n = n_requests;
  a.S = session_blocks;
  a.h_init = mix64(hash_seed + kGamma);
  a.batch_ok = ok;
  a.D = digest;
  a.hashes = d_block_hashes;
  a.sk_out = d_session_key;
  a.status = d_status;
  if (!chain_limit<0>()) return cuda_status(cudaErrorInvalidValue);
  return launch_chain(a, num_sms, s, false);
}
