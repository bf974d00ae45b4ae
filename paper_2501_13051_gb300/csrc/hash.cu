// Step (a): the hybrid index of Section 3.  Over a column (or column pair)
// sorted by value, every distinct key gets one open-addressing slot holding
// (key, start, count): the first position of the key in the sorted order and
// its run length (the run-length encoding the paper stores in its "unique
// hashmap").  Linear probing over a power-of-two table; the hash is the
// MurmurHash3 finaliser.
//
// One pass: the thread at a run head finds the end of its run by galloping
// (exponential then binary search over the sorted keys, O(log run) reads,
// so a hot key with a long run costs one thread a few dozen reads rather
// than a walk), then claims a slot with a 64-bit compare-and-swap on the
// key words.  Keys are distinct, so an insert never meets its own key.
#include "kernels.h"

namespace cdl {

namespace {

constexpr int kThreads = 256;
constexpr unsigned long long kEmpty64 = ~0ull;

template <bool TWO>
__device__ __forceinline__ bool key_ne(const uint32_t* k0, const uint32_t* k1, uint64_t i,
                                       uint32_t a0, uint32_t a1) {
  if (TWO) return __ldg(k0 + i) != a0 || __ldg(k1 + i) != a1;
  return __ldg(k0 + i) != a0;
}

// Row i's part of the hash form.
template <bool TWO>
__device__ __forceinline__ void hash_row(const uint32_t* __restrict__ k0,
                                         const uint32_t* __restrict__ k1, uint64_t i, uint64_t n,
                                         Slot* __restrict__ t, uint64_t mask, uint32_t* err) {
  const uint32_t a0 = __ldg(k0 + i);
  const uint32_t a1 = TWO ? __ldg(k1 + i) : 0u;
  if (i > 0 && !key_ne<TWO>(k0, k1, i - 1, a0, a1)) return;  // not a run head
  // gallop to the first position past the run
  uint64_t lo = i + 1, hi = n, step = 1;
  while (true) {
    const uint64_t j = i + step;
    if (j >= n) break;
    if (key_ne<TWO>(k0, k1, j, a0, a1)) {
      hi = j;
      break;
    }
    lo = j + 1;
    step <<= 1;
  }
  while (lo < hi) {
    const uint64_t mid = lo + ((hi - lo) >> 1);
    if (key_ne<TWO>(k0, k1, mid, a0, a1))
      hi = mid;
    else
      lo = mid + 1;
  }
  const uint64_t end = lo;
  const unsigned long long packed = ((unsigned long long)a1 << 32) | a0;
  uint64_t s = hash_key(a0, a1) & mask;
  for (uint64_t probe = 0; probe <= mask; ++probe) {
    const unsigned long long prev =
        atomicCAS(reinterpret_cast<unsigned long long*>(t + s), kEmpty64, packed);
    if (prev == kEmpty64) {
      t[s].start = (uint32_t)i;
      t[s].count = (uint32_t)(end - i);
      return;
    }
    s = (s + 1) & mask;
  }
  if (err) atomicOr(err, kErrTable);
}

template <bool TWO>
__global__ void __launch_bounds__(kThreads) k_hash_build(const uint32_t* __restrict__ k0,
                                                         const uint32_t* __restrict__ k1,
                                                         uint64_t n, Slot* __restrict__ t,
                                                         uint64_t mask, uint32_t* err) {
  const uint64_t i = (uint64_t)blockIdx.x * kThreads + threadIdx.x;
  if (i < n) hash_row<TWO>(k0, k1, i, n, t, mask, err);
}

// Direct form: the row that starts a key's run stores the run's start, the
// row that ends it the end, so nothing is searched and, the keys being
// sorted, the writes go up the array.  Bound by memory: keys read, 8 bytes
// per entry cleared and 8 per distinct key written.  (A key at or past the
// range -- of a build side that is not sorted -- is left out.)
__global__ void __launch_bounds__(kThreads) k_index_build(const uint32_t* __restrict__ k0,
                                                          uint64_t n, KeyIndex x, uint32_t* err) {
  const uint64_t i = (uint64_t)blockIdx.x * kThreads + threadIdx.x;
  if (i >= n) return;
  const uint32_t range = direct_range(x);
  Slot* t = const_cast<Slot*>(x.table);
  if (!range) return hash_row<false>(k0, nullptr, i, n, t, x.slots - 1, err);
  const uint32_t a = __ldg(k0 + i);
  if (a >= range) return;
  uint32_t* e = reinterpret_cast<uint32_t*>(t) + 2ull * a;
  const bool first = i == 0 || __ldg(k0 + i - 1) != a, last = i + 1 == n || __ldg(k0 + i + 1) != a;
  if (first && last) {
    *reinterpret_cast<uint2*>(e) = make_uint2((uint32_t)i, (uint32_t)(i + 1));
  } else {
    if (first) e[0] = (uint32_t)i;
    if (last) e[1] = (uint32_t)(i + 1);
  }
}

// Offset form.  The keys and the entries 0 .. range are merged (an entry
// after the keys below it) and cut into equal shares by merge-path splits, so
// that a run of one key or a gap between two costs a block no more than its
// share; a row then writes the entries from the key before it up to its own.
// 63 us for 16.8M keys and 33.5M entries (201 MB): bound by the caches, which
// take every entry as a store of its own (L1 65 %, L2 52 %, DRAM 26 % busy).
constexpr int kOffTile = 4096;
__global__ void __launch_bounds__(kThreads) k_offset_splits(const uint32_t* __restrict__ k0,
                                                            uint64_t n, KeyIndex x,
                                                            uint64_t* __restrict__ splits) {
  const uint32_t range = direct_range(x);
  if (!range) return;
  const uint64_t b = (uint64_t)blockIdx.x * kThreads + threadIdx.x, total = n + range + 1ull;
  if (b > (total + kOffTile - 1) / kOffTile) return;
  const uint64_t d = b * kOffTile < total ? b * kOffTile : total;
  uint64_t lo = d > range + 1ull ? d - (range + 1ull) : 0, hi = d < n ? d : n;
  while (lo < hi) {
    const uint64_t mid = lo + ((hi - lo) >> 1);
    if (__ldg(k0 + mid) < d - mid - 1)  // key mid comes before entry d - mid - 1
      lo = mid + 1;
    else
      hi = mid;
  }
  splits[b] = lo;
}

__global__ void __launch_bounds__(kThreads) k_offset_fill(const uint32_t* __restrict__ k0,
                                                          uint64_t n, KeyIndex x,
                                                          const uint64_t* __restrict__ splits,
                                                          uint32_t* err) {
  const uint32_t range = direct_range(x);
  Slot* table = const_cast<Slot*>(x.table);
  if (!range) {  // the hash form
    for (uint64_t i = (uint64_t)blockIdx.x * kThreads + threadIdx.x; i < n;
         i += (uint64_t)gridDim.x * kThreads)
      hash_row<false>(k0, nullptr, i, n, table, x.slots - 1, err);
    return;
  }
  uint32_t* t = reinterpret_cast<uint32_t*>(table);
  const uint64_t total = n + range + 1ull, tiles = (total + kOffTile - 1) / kOffTile;
  for (uint64_t b = blockIdx.x; b < tiles; b += gridDim.x) {
    const uint64_t d1 = (b + 1) * kOffTile < total ? (b + 1) * kOffTile : total;
    const uint64_t a0 = splits[b], a1 = splits[b + 1];
    const uint64_t e0 = b * kOffTile - a0, e1 = d1 - a1;  // the tile's entries
    // row i writes the tile's entries in (key i - 1, key i]; row a1 (of the
    // next tile, or past the end) those behind the tile's last key
    for (uint64_t i = a0 + threadIdx.x; i <= a1; i += kThreads) {
      uint64_t lo = i > 0 ? (uint64_t)__ldg(k0 + i - 1) + 1 : 0;
      uint64_t hi = i < a1 ? (uint64_t)__ldg(k0 + i) + 1 : e1;
      lo = lo > e0 ? lo : e0;
      hi = hi < e1 ? hi : e1;
      for (uint64_t e = lo; e < hi; ++e) t[e] = (uint32_t)i;
    }
  }
}

// Clears the form that *x.last gives (the offset form needs none).
__global__ void __launch_bounds__(kThreads) k_index_clear(KeyIndex x) {
  const uint32_t range = direct_range(x);
  if (range && x.rows) return;
  const uint64_t words = range ? ((uint64_t)range + 1) / 2 : x.slots;  // 16 bytes each
  const uint32_t v = range ? 0u : 0xFFFFFFFFu;
  uint4* t = reinterpret_cast<uint4*>(const_cast<Slot*>(x.table));
  for (uint64_t i = (uint64_t)blockIdx.x * kThreads + threadIdx.x; i < words;
       i += (uint64_t)gridDim.x * kThreads)
    t[i] = make_uint4(v, v, v, v);
}

template <bool TWO>
__global__ void __launch_bounds__(kThreads) k_count_heads(const uint32_t* __restrict__ k0,
                                                          const uint32_t* __restrict__ k1,
                                                          uint64_t n, unsigned long long* out) {
  uint32_t mine = 0;
  for (uint64_t i = (uint64_t)blockIdx.x * kThreads + threadIdx.x; i < n;
       i += (uint64_t)gridDim.x * kThreads) {
    const uint32_t a0 = __ldg(k0 + i), a1 = TWO ? __ldg(k1 + i) : 0u;
    mine += (i == 0 || key_ne<TWO>(k0, k1, i - 1, a0, a1)) ? 1u : 0u;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) mine += __shfl_xor_sync(0xffffffffu, mine, o);
  if (lane_id() == 0 && mine) atomicAdd(out, (unsigned long long)mine);
}

}  // namespace

uint64_t table_slots(uint64_t n_keys, double load) {
  if (load <= 0.0 || load > 0.9) load = 0.5;
  uint64_t want = (uint64_t)((double)(n_keys ? n_keys : 1) / load) + 1;
  uint64_t s = 16;
  while (s < want) s <<= 1;
  return s;
}

cudaError_t hash_build(Ctx& c, const uint32_t* k0, const uint32_t* k1, uint64_t n, Slot* table,
                       uint64_t slots) {
  cudaError_t e = cudaMemsetAsync(table, 0xFF, slots * sizeof(Slot), c.st);
  if (e != cudaSuccess || n == 0) return e;
  ProfScope p(c, kHashBuild, (k1 ? 8.0 : 4.0) * n);
  const unsigned grid = (unsigned)((n + kThreads - 1) / kThreads);
  if (k1)
    k_hash_build<true><<<grid, kThreads, 0, c.st>>>(k0, k1, n, table, slots - 1, c.d_err);
  else
    k_hash_build<false><<<grid, kThreads, 0, c.st>>>(k0, k1, n, table, slots - 1, c.d_err);
  return cudaGetLastError();
}

cudaError_t index_build(Ctx& c, const uint32_t* k0, uint64_t n, const KeyIndex& x) {
  if (!x.range) return hash_build(c, k0, nullptr, n, const_cast<Slot*>(x.table), x.slots);
  const unsigned grid = (unsigned)((n + kThreads - 1) / kThreads);
  if (x.last) {
    uint64_t blocks = (x.slots + kThreads * 4 - 1) / (kThreads * 4);
    if (blocks > 152 * 16) blocks = 152 * 16;
    k_index_clear<<<(unsigned)blocks, kThreads, 0, c.st>>>(x);
  } else {
    cudaError_t e = cudaMemsetAsync(const_cast<Slot*>(x.table), 0, 8ull * x.range, c.st);
    if (e != cudaSuccess) return e;
  }
  if (n == 0) return cudaGetLastError();
  ProfScope p(c, kHashBuild, 4.0 * n);
  if (x.rows) {
    auto* splits = reinterpret_cast<uint64_t*>(reinterpret_cast<char*>(const_cast<Slot*>(x.table)) +
                                               8 * x.slots + 256);
    const uint64_t tiles = (n + x.range + 1ull + kOffTile - 1) / kOffTile;  // at most
    k_offset_splits<<<(unsigned)((tiles + 1 + kThreads - 1) / kThreads), kThreads, 0, c.st>>>(k0, n, x,
                                                                                              splits);
    k_offset_fill<<<(unsigned)(tiles < 152 * 64 ? tiles : 152 * 64), kThreads, 0, c.st>>>(
        k0, n, x, splits, c.d_err);
    return cudaGetLastError();
  }
  k_index_build<<<grid, kThreads, 0, c.st>>>(k0, n, x, c.d_err);
  return cudaGetLastError();
}

cudaError_t count_heads(Ctx& c, const uint32_t* k0, const uint32_t* k1, uint64_t n,
                        uint64_t* d_out) {
  cudaError_t e = cudaMemsetAsync(d_out, 0, sizeof(uint64_t), c.st);
  if (e != cudaSuccess || n == 0) return e;
  ProfScope p(c, kCountHeads, (k1 ? 8.0 : 4.0) * n);
  uint64_t blocks = (n + kThreads * 8 - 1) / (kThreads * 8);
  if (blocks > 152 * 16) blocks = 152 * 16;
  auto* out = reinterpret_cast<unsigned long long*>(d_out);
  if (k1)
    k_count_heads<true><<<(unsigned)blocks, kThreads, 0, c.st>>>(k0, k1, n, out);
  else
    k_count_heads<false><<<(unsigned)blocks, kThreads, 0, c.st>>>(k0, k1, n, out);
  return cudaGetLastError();
}

}  // namespace cdl
