// Shared device helpers of the column-oriented Datalog kernels (sm_103a).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/cdl.h"

namespace cdl {

constexpr int kMaxK = CDL_MAX_ARITY;
constexpr uint32_t kEmpty = CDL_EMPTY_KEY;

// Column sets passed by value to kernels: column k of a relation is c[k].
struct ColsIn {
  const uint32_t* c[kMaxK];
};
struct ColsOut {
  uint32_t* c[kMaxK];
};

// Error bits a kernel may raise in the engine's device status word.
enum : uint32_t {
  kErrTimeout = 1u,   // a bounded wait ran out
  kErrCapacity = 2u,  // an output cursor passed its capacity
  kErrValue = 4u,     // the reserved value was seen in input
  kErrTable = 8u,     // a hash table had no free slot
  kErrState = 16u     // a write whose count was another one (join_begin)
};

// 32-bit finaliser of MurmurHash3 (Austin Appleby, public domain): a
// bijective mixer, so distinct keys never collide before masking.
__host__ __device__ __forceinline__ uint32_t mix32(uint32_t k) {
  k ^= k >> 16;
  k *= 0x85ebca6bu;
  k ^= k >> 13;
  k *= 0xc2b2ae35u;
  k ^= k >> 16;
  return k;
}

__host__ __device__ __forceinline__ uint32_t hash_key(uint32_t k0, uint32_t k1) {
  return mix32(k0 ^ mix32(k1 + 0x9e3779b9u));
}

// Hash slot of the hybrid index: key (one or two words) -> (start, count) in
// the build side sorted by key.  An empty slot has k0 == k1 == 0xFFFFFFFF.
struct __align__(16) Slot {
  uint32_t k0, k1, start, count;
};

__device__ __forceinline__ Slot load_slot(const Slot* t, uint64_t i) {
  const uint4 v = __ldg(reinterpret_cast<const uint4*>(t) + i);
  return Slot{v.x, v.y, v.z, v.w};
}

// Linear-probing lookup; returns count (0 if absent) and start.
__device__ __forceinline__ uint32_t probe_table(const Slot* t, uint64_t mask, uint32_t k0,
                                                uint32_t k1, uint32_t* start) {
  uint64_t i = hash_key(k0, k1) & mask;
  for (uint64_t step = 0; step <= mask; ++step) {
    const Slot s = load_slot(t, i);
    if (s.k0 == k0 && s.k1 == k1) {
      *start = s.start;
      return s.count;
    }
    if (s.k0 == kEmpty && s.k1 == kEmpty) break;
    i = (i + 1) & mask;
  }
  *start = 0;
  return 0;
}

// An index over build rows sorted by key, in one of three forms.  Hash form
// (range 0): the hybrid index's slots.  Direct form, for one-word keys whose
// values lie below a range not much larger than the rows: entry k of an
// array of `range` (start, end) pairs, both 0 for an absent key, so that a
// lookup is one 8-byte read with nothing to compare.  With `last` (the
// largest key, in device memory) the launches take the direct form, of
// *last + 1 entries, where *last < range and else the hash form: a caller
// that does not know the keys' bound spares the wait for it.  (A join call
// of 16M rows with an index of 16M rows over 2^25 keys: 2.73 ms with hash
// slots built and looked up in its size query and again in its write, 0.86 ms
// with entries built once and the rows' starts kept from the count.)
// Offset form (rows > 0, with last): entry k is the number of keys below k,
// *last + 2 of them, so that key k's rows are [entry k, entry k + 1): half the
// bytes of the direct form and nothing to clear first, but two reads a lookup
// and a split search before it is filled.  It pays once the direct form's
// array is larger than L2 (the join above: 838 us with entries, 735 with
// offsets).
struct KeyIndex {
  const Slot* table;
  uint64_t slots;  // hash form: slots, a power of two
  uint32_t range;
  const uint32_t* last;
  uint32_t rows;   // offset form: the build rows
};

// Rows [*start, *start + count) of key k < range in the direct or offset
// form.  (An entry of a build side that is not sorted may be anything: it is
// held within the rows.)
__device__ __forceinline__ uint32_t find_entry(const KeyIndex& x, uint32_t k, uint32_t* start) {
  uint2 e;
  if (x.rows) {
    const uint32_t* t = reinterpret_cast<const uint32_t*>(x.table) + k;
    e.x = min(__ldg(t), x.rows);
    e.y = min(__ldg(t + 1), x.rows);
  } else {
    e = __ldg(reinterpret_cast<const uint2*>(x.table) + k);
  }
  *start = e.x;
  return e.y > e.x ? e.y - e.x : 0u;
}

// The direct form's range as it applies: 0 for the hash form.
__device__ __forceinline__ uint32_t direct_range(const KeyIndex& x) {
  return x.last ? (__ldg(x.last) < x.range ? __ldg(x.last) + 1u : 0u) : x.range;
}

// Build rows of key (k0, k1); range as direct_range gives it.
__device__ __forceinline__ uint32_t find_key(const KeyIndex& x, uint32_t range, uint32_t k0,
                                             uint32_t k1, uint32_t* start) {
  if (range) {
    *start = 0;
    return k0 < range ? find_entry(x, k0, start) : 0u;
  }
  return probe_table(x.table, x.slots - 1, k0, k1, start);
}

// Lexicographic comparison of tuples held in registers.
template <int K>
__device__ __forceinline__ bool tuple_le(const uint32_t (&a)[K], const uint32_t (&b)[K]) {
#pragma unroll
  for (int k = 0; k < K; ++k) {
    if (a[k] != b[k]) return a[k] < b[k];
  }
  return true;
}
template <int K>
__device__ __forceinline__ bool tuple_eq(const uint32_t (&a)[K], const uint32_t (&b)[K]) {
  bool e = true;
#pragma unroll
  for (int k = 0; k < K; ++k) e &= a[k] == b[k];
  return e;
}
template <int K>
__device__ __forceinline__ void load_tuple(const ColsIn& c, uint64_t i, uint32_t (&t)[K]) {
#pragma unroll
  for (int k = 0; k < K; ++k) t[k] = c.c[k][i];
}

__device__ __forceinline__ uint32_t lane_id() { return threadIdx.x & 31u; }
__device__ __forceinline__ uint32_t lanemask_lt() {
  uint32_t m;
  asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
  return m;
}

// Block-wide exclusive sum over THREADS threads (values per thread), with
// the block total in *total.  smem: THREADS/32 words.
template <int THREADS, typename T>
__device__ __forceinline__ T block_exclusive_sum(T v, T* smem, T* total) {
  constexpr int W = THREADS / 32;
  const uint32_t lane = lane_id(), warp = threadIdx.x >> 5;
  T inc = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const T n = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= (uint32_t)o) inc += n;
  }
  if (lane == 31) smem[warp] = inc;
  __syncthreads();
  if (warp == 0) {
    T w = lane < (uint32_t)W ? smem[lane] : T(0);
    T winc = w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const T n = __shfl_up_sync(0xffffffffu, winc, o);
      if (lane >= (uint32_t)o) winc += n;
    }
    if (lane < (uint32_t)W) smem[lane] = winc - w;
    if (lane == W - 1) smem[W] = winc;
  }
  __syncthreads();
  const T res = smem[warp] + inc - v;
  *total = smem[W];
  __syncthreads();
  return res;
}

// Exclusive max-scan over the block's threads (0 for thread 0).  smem:
// THREADS/32 words.  Ends with a barrier.
template <int THREADS>
__device__ __forceinline__ uint32_t block_exclusive_max(uint32_t v, uint32_t* smem) {
  static_assert(THREADS % 32 == 0 && THREADS <= 1024, "whole warps");
  const uint32_t lane = lane_id(), warp = threadIdx.x >> 5;
  uint32_t inc = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t n = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= (uint32_t)o) inc = n > inc ? n : inc;
  }
  const uint32_t ex_in_warp = __shfl_up_sync(0xffffffffu, inc, 1);
  if (lane == 31) smem[warp] = inc;
  __syncthreads();
  uint32_t before = 0;  // max over the earlier warps
  for (uint32_t w = 0; w < warp; ++w) before = smem[w] > before ? smem[w] : before;
  __syncthreads();
  const uint32_t own = lane > 0 ? ex_in_warp : 0u;
  return own > before ? own : before;
}

// Places for a block's outputs in `mask`, packed at *cursor with one claim:
// output q goes to *pos + at[q].  wsum: THREADS / 32 + 2 words.  false (for
// the whole block) where there are none.
template <int THREADS, int N>
__device__ __forceinline__ bool claim_places(uint32_t mask, unsigned long long* cursor,
                                             uint32_t* wsum, uint32_t (&at)[N], uint64_t* pos) {
  constexpr int W = THREADS / 32;
  const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5, lt = (1u << lane) - 1u;
  uint32_t n = 0;
#pragma unroll
  for (int q = 0; q < N; ++q) {
    const uint32_t bal = __ballot_sync(0xffffffffu, (mask >> q) & 1u);
    at[q] = n + __popc(bal & lt);
    n += __popc(bal);
  }
  if (lane == 0) wsum[warp] = n;
  __syncthreads();
  unsigned long long* claim = reinterpret_cast<unsigned long long*>(wsum + W);
  uint32_t before = 0, total = 0;
#pragma unroll
  for (int w = 0; w < W; ++w) {
    const uint32_t c = wsum[w];
    before += w < (int)warp ? c : 0u;
    total += c;
  }
  if (total == 0) return false;
  if (threadIdx.x == 0) *claim = atomicAdd(cursor, (unsigned long long)total);
  __syncthreads();
  *pos = *claim + before;
  return true;
}

// A relation of arity k whose columns need T = bits_0 + ... + bits_{k-1}
// bits in all can also be held as a bitmap of 2^T bits: tuple (v_0..v_{k-1})
// is bit sum_k v_k << shift_k, with shift_k the bits of the columns after k.
// Increasing bit order is then the tuples' lexicographic order, and setting
// a bit twice is a no-op, so the bitmap is a sorted set.
//
// Two uses: the new tuples of one round (append == 0: join outputs only set
// bits, which are read back in order), and Full itself (append == 1: a join
// output whose bit was not set yet is new, and is appended to the round's
// delta rows by whoever set it).
struct DenseSet {
  uint32_t* words;  // nbits / 32 words (at least one)
  uint64_t nbits;   // 2^T
  uint32_t k;
  uint32_t append;
  uint32_t shift[kMaxK];
  uint32_t mask[kMaxK];  // 2^bits_k - 1
  // Hash form, for Full in tuple spaces too large for a bitmap (at most 2^62
  // tuples): open addressing over the packed tuples, words unused.
  unsigned long long* keys;  // kmask + 1 slots (a power of two), or null
  uint64_t kmask;
};
constexpr unsigned long long kSetEmpty = ~0ull;     // a free slot
constexpr unsigned long long kSetGone = ~0ull - 1;  // a tuple taken out again
constexpr uint32_t kSetProbes = 4096;  // slots looked at before the table counts as full

// Position of tuple v in the packed tuple space of d; kNoTuple when v lies
// outside it.
constexpr uint64_t kNoTuple = ~0ull;
__device__ __forceinline__ uint64_t set_pack(const DenseSet& d, const uint32_t (&v)[kMaxK]) {
  uint64_t idx = 0;
  bool out = false;
#pragma unroll
  for (int k = 0; k < kMaxK; ++k)
    if (k < (int)d.k) {
      idx |= (uint64_t)v[k] << d.shift[k];
      out |= v[k] > d.mask[k];
    }
  return out || idx >= d.nbits ? kNoTuple : idx;
}
__device__ __forceinline__ uint32_t set_column(const DenseSet& d, uint64_t idx, int k) {
  return (uint32_t)(idx >> d.shift[k]) & d.mask[k];
}

// Adds the tuples idx[0..N) (kNoTuple: none) to Full's bitmap; bit q of the
// result tells that this call set tuple q's bit, i.e. the tuple is new.  A
// bit seen set by a plain read (of any age, from L1 or L2) needs no atomic: a
// set bit is cleared again only where a new tuple found no room (set_store),
// and then the round's rules for the relation run again.  The N reads, then
// the N atomics, are in flight together.
template <int N>
__device__ __forceinline__ uint32_t set_add(const DenseSet& d, const uint64_t (&idx)[N]) {
  uint32_t seen[N];
#pragma unroll
  for (int q = 0; q < N; ++q)
    seen[q] = idx[q] != kNoTuple ? d.words[idx[q] >> 5] >> (idx[q] & 31) & 1u : 1u;
#pragma unroll
  for (int q = 0; q < N; ++q)
    if (!seen[q]) seen[q] = atomicOr(d.words + (idx[q] >> 5), 1u << (idx[q] & 31)) >> (idx[q] & 31) & 1u;
  uint32_t fresh = 0;
#pragma unroll
  for (int q = 0; q < N; ++q) fresh |= (seen[q] ^ 1u) << q;
  return fresh;
}

// 64-bit finaliser of SplitMix64 (Steele, Lea & Flood, 2014).
__device__ __forceinline__ uint64_t mix64(uint64_t k) {
  k = (k ^ (k >> 30)) * 0xbf58476d1ce4e5b9ull;
  k = (k ^ (k >> 27)) * 0x94d049bb133111ebull;
  return k ^ (k >> 31);
}

// set_add for the hash form.  A slot goes from empty to one key (to gone)
// and never to another, so a key seen by a plain read is there.  Where no
// free slot turns up *full is set and the tuple is left out.
template <int N>
__device__ __forceinline__ uint32_t set_add_hash(const DenseSet& d, const uint64_t (&key)[N],
                                                 bool* full) {
  unsigned long long v[N];
#pragma unroll
  for (int q = 0; q < N; ++q)
    v[q] = key[q] != kNoTuple ? d.keys[mix64(key[q]) & d.kmask] : kNoTuple;
  uint32_t fresh = 0;
#pragma unroll
  for (int q = 0; q < N; ++q)
    if (key[q] != kNoTuple && v[q] == kSetEmpty) {
      v[q] = atomicCAS(d.keys + (mix64(key[q]) & d.kmask), kSetEmpty, key[q]);
      if (v[q] == kSetEmpty) {
        fresh |= 1u << q;
        v[q] = key[q];
      }
    }
  // the others look on, one after another (code for one, not for N)
  uint32_t left = 0;
#pragma unroll
  for (int q = 0; q < N; ++q) left |= (key[q] != kNoTuple && v[q] != key[q] ? 1u : 0u) << q;
  while (left) {
    const uint32_t b = left & (0u - left);
    left ^= b;
    uint64_t k = key[0];
#pragma unroll
    for (int q = 1; q < N; ++q) k = (b >> q) & 1u ? key[q] : k;
    uint64_t at = mix64(k) & d.kmask;
    bool done = false;
    for (uint32_t step = 1; step < kSetProbes && !done; ++step) {
      at = (at + 1) & d.kmask;
      unsigned long long x = d.keys[at];
      if (x == kSetEmpty) {
        x = atomicCAS(d.keys + at, kSetEmpty, k);
        if (x == kSetEmpty) fresh |= b;
      }
      done = x == kSetEmpty || x == k;
    }
    if (!done) *full = true;
  }
  return fresh;
}

// Takes a tuple that is in the set out again.
__device__ __forceinline__ void set_remove(const DenseSet& d, uint64_t idx) {
  if (!d.keys) {
    atomicAnd(d.words + (idx >> 5), ~(1u << (idx & 31)));
    return;
  }
  uint64_t at = mix64(idx) & d.kmask;
  for (uint32_t step = 0; step < kSetProbes; ++step) {
    if (d.keys[at] == idx) {
      d.keys[at] = kSetGone;
      return;
    }
    at = (at + 1) & d.kmask;
  }
}

// Writes a block's new tuples (bit q of fresh: tuple idx[q] is new) packed at
// *cursor.  wsum as for claim_places.  Rows past cap are dropped; false tells
// the caller.
template <int THREADS, int N>
__device__ __forceinline__ bool set_emit(const DenseSet& d, const uint64_t (&idx)[N],
                                         uint32_t fresh, ColsOut out, unsigned long long* cursor,
                                         uint64_t cap, uint32_t* wsum) {
  uint32_t at[N];
  uint64_t pos;
  if (!claim_places<THREADS, N>(fresh, cursor, wsum, at, &pos)) return true;
  bool ok = true;
#pragma unroll
  for (int q = 0; q < N; ++q) {
    if (!((fresh >> q) & 1u)) continue;
    const uint64_t p = pos + at[q];
    if (p < cap) {
#pragma unroll
      for (int k = 0; k < kMaxK; ++k)
        if (k < (int)d.k) out.c[k][p] = set_column(d, idx[q], k);
    } else {
      ok = false;
    }
  }
  return ok;
}

// The word and bit of tuple v in d; false when v lies outside d.
__device__ __forceinline__ bool dense_locate(const DenseSet& d, const uint32_t (&v)[kMaxK],
                                             uint32_t* word, uint32_t* bit) {
  uint64_t idx = 0;
  bool out = false;
#pragma unroll
  for (int k = 0; k < kMaxK; ++k)
    if (k < (int)d.k) {
      idx |= (uint64_t)v[k] << d.shift[k];
      out |= v[k] > d.mask[k];
    }
  *word = (uint32_t)(idx >> 5);
  *bit = 1u << (idx & 31);
  return !out && idx < d.nbits;
}

// Bits only go from 0 to 1 while tuples are added, so a bit seen set (in a
// value read at any time, from L1 or L2) is set: only a missing bit needs an
// atomic.  Repeated outputs of a join mostly stop at the read.  (Merging a
// warp's bits per word first, by match and reduce, costs more than it
// saves: those warp instructions then bound the join's write pass.)
__device__ __forceinline__ bool dense_missing(const DenseSet& d, uint32_t word, uint32_t bit) {
  return (d.words[word] & bit) == 0u;
}

// Sets the bit of tuple v (keep = the thread has one); a tuple outside the
// bitmap raises kErrCapacity and sets nothing.
__device__ __forceinline__ void dense_set_bits(const DenseSet& d, const uint32_t (&v)[kMaxK],
                                               bool keep, uint32_t* err) {
  uint32_t word = 0, bit = 0;
  if (!keep) return;
  if (!dense_locate(d, v, &word, &bit)) {
    atomicOr(err, kErrCapacity);
    return;
  }
  if (dense_missing(d, word, bit)) atomicOr(d.words + word, bit);
}

// Device-sized launches (a round captured in a CUDA graph): the grid is
// sized for a capacity known to the host, the actual size is read from
// device memory and clamped to that capacity, so no access can leave the
// buffers the capacity describes.  dn == nullptr: the size is `cap` itself.
__device__ __forceinline__ uint64_t dev_size(const uint64_t* dn, uint64_t cap) {
  if (!dn) return cap;
  const uint64_t v = *dn;
  return v < cap ? v : cap;
}

// Grid of a launch over `tiles` tiles.  A device-sized launch (dn set: a
// captured round, its tiles counted for a capacity) gets at most kDevGrid
// blocks, which loop over the tiles the actual size gives, so that rounds
// far below the capacity do not launch blocks by the hundred thousand;
// other launches get one block per tile (one iteration of the loop).
constexpr uint64_t kDevGrid = 152 * 8;
inline unsigned dev_grid(uint64_t tiles, const void* dn) {
  return (unsigned)(dn && tiles > kDevGrid ? kDevGrid : (tiles ? tiles : 1));
}

}  // namespace cdl
