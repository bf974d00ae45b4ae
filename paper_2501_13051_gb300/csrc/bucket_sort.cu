// Step (c) beside the LSD radix sort (sort.cu): two sorts for tuples whose
// number and distribution let shared memory do the work.
//
// Small sort: up to kSmallSort tuples in one block and one launch.  The
// columns sit in shared memory and a permutation of 16-bit row numbers is
// radix-sorted, 8 bits of the packed key per pass; the significant bits come
// from the columns' maxima, found in the same kernel.
//
// Bucket sort: tuples are thrown by the top bits of a packed key (the first
// columns, up to 64 bits) into buckets of a few thousand (one histogram pass
// over the columns that hold those bits, one scatter of packed keys, order
// within a bucket left open), then each block sorts one bucket in shared
// memory by the remaining bits (and wide tuples by the columns past the key,
// through row numbers scattered with the keys).  Against the LSD sort every tuple crosses HBM twice instead
// of once per 8 or 9 bits, and the input is left as it is.  It needs the
// buckets to come out below kBucketCap: a bucket above (a value that repeats,
// a range of values far denser than the rest) is seen in the histogram, and
// the caller takes the LSD sort.
// sort_unique of 16.7M pairs of 18-bit values: 1,429 us by LSD passes, 657 us
// so; of 1M pairs of 32-bit values 716 and 172 us; of 1M tuples of eight
// 32-bit values 1,440 us (the first four columns alone) and 270 us.
#include "kernels.h"

namespace cdl {

namespace {

// ------------------------------------------------------------- small sort
constexpr int kST = 1024;
constexpr int kSItems = (int)(kSmallSort / kST);

template <int K>
size_t small_smem(uint32_t n) {
  return ((size_t)K * n * 4 + 15) / 16 * 16 + 2 * kSmallSort * 2;
}

// head (may be null): head[0] = 0 (no error), head[1] = number of tuples
// written.  out may be in: every tuple is in shared memory before the first
// is written.  Bound by the latency of its passes (about five block barriers
// each): 1,000 pairs of 36 bits take 5 passes, 16 us; a sort_unique call on
// them 148 us before (eight launches, two waits), 74 us now.
template <int K, bool UNIQUE>
__global__ void __launch_bounds__(kST) k_sort_small(ColsIn in, uint32_t n, ColsOut out,
                                                    uint64_t* head) {
  extern __shared__ __align__(16) uint32_t sm[];
  __shared__ uint32_t wh[kST / 32][256];  // per-warp digit counts, then offsets
  __shared__ uint32_t red[kST / 32 + 1];
  __shared__ uint32_t smax[K];
  uint32_t* col = sm;
  uint16_t* idx = reinterpret_cast<uint16_t*>(sm + ((size_t)K * n + 3) / 4 * 4);
  uint16_t* alt = idx + kSmallSort;
  const uint32_t t = threadIdx.x, warp = t >> 5, lane = t & 31u, lt = lanemask_lt();
  if (t < K) smax[t] = 0;
  __syncthreads();
#pragma unroll
  for (int k = 0; k < K; ++k) {
    uint32_t m = 0;
    for (uint32_t i = t; i < n; i += kST) {
      const uint32_t v = in.c[k][i];
      col[k * n + i] = v;
      m = v > m ? v : m;
    }
    m = __reduce_max_sync(0xffffffffu, m);
    if (lane == 0 && m) atomicMax(&smax[k], m);
  }
  for (uint32_t i = t; i < n; i += kST) idx[i] = (uint16_t)i;
  __syncthreads();
  uint32_t pos[K], bits[K], total = 0;
#pragma unroll
  for (int k = K - 1; k >= 0; --k) {
    pos[k] = total;
    bits[k] = 32u - __clz(smax[k]);
    total += bits[k];
  }
  const uint32_t items = (n + kST - 1) / kST;
  const uint32_t wbase = warp * 32 * items;
  for (uint32_t lo = 0; lo < total; lo += 8) {
    for (int i = t; i < kST / 32 * 256; i += kST) (&wh[0][0])[i] = 0;
    __syncthreads();
    uint32_t dg[kSItems], rk[kSItems];
    uint16_t row[kSItems];
#pragma unroll
    for (int it = 0; it < kSItems; ++it) {
      if (it >= (int)items) break;
      const uint32_t i = wbase + it * 32 + lane;
      uint32_t d = 256u;
      row[it] = 0;
      if (i < n) {
        row[it] = idx[i];
        d = 0;
#pragma unroll
        for (int k = 0; k < K; ++k) {
          const uint32_t s = lo > pos[k] ? lo : pos[k];
          const uint32_t e = lo + 8 < pos[k] + bits[k] ? lo + 8 : pos[k] + bits[k];
          if (s < e) d |= ((col[k * n + row[it]] >> (s - pos[k])) & ((1u << (e - s)) - 1u)) << (s - lo);
        }
      }
      const uint32_t peers = __match_any_sync(0xffffffffu, d);
      const uint32_t leader = (uint32_t)__ffs(peers) - 1u;
      uint32_t b = 0;
      if (d < 256u && lane == leader) b = atomicAdd(&wh[warp][d], (uint32_t)__popc(peers));
      b = __shfl_sync(0xffffffffu, b, leader);
      dg[it] = d;
      rk[it] = b + __popc(peers & lt);
    }
    __syncthreads();
    uint32_t sum = 0;  // digit t: its tuples, and each warp's offset among them
    if (t < 256) {
#pragma unroll 8
      for (int w = 0; w < kST / 32; ++w) {
        const uint32_t x = wh[w][t];
        wh[w][t] = sum;
        sum += x;
      }
    }
    uint32_t tot;
    const uint32_t start = block_exclusive_sum<kST, uint32_t>(sum, red, &tot);
    if (t < 256) {
#pragma unroll 8
      for (int w = 0; w < kST / 32; ++w) wh[w][t] += start;
    }
    __syncthreads();
#pragma unroll
    for (int it = 0; it < kSItems; ++it) {
      if (it >= (int)items) break;
      if (dg[it] < 256u) alt[wh[warp][dg[it]] + rk[it]] = row[it];
    }
    __syncthreads();
    uint16_t* x = idx;
    idx = alt;
    alt = x;
  }
  uint32_t written = 0;
  for (uint32_t i0 = 0; i0 < n; i0 += kST) {
    const uint32_t i = i0 + t;
    bool keep = i < n;
    const uint32_t r = keep ? idx[i] : 0u;
    uint32_t at = i;
    if constexpr (UNIQUE) {
      if (keep && i > 0) {
        const uint32_t p = idx[i - 1];
        bool eq = true;
#pragma unroll
        for (int k = 0; k < K; ++k) eq &= col[k * n + r] == col[k * n + p];
        keep = !eq;
      }
      uint32_t tot;
      at = written + block_exclusive_sum<kST, uint32_t>(keep ? 1u : 0u, red, &tot);
      written += tot;
    }
    if (keep) {
#pragma unroll
      for (int k = 0; k < K; ++k) out.c[k][at] = col[k * n + r];
    }
  }
  if (head && t == 0) {
    head[0] = 0;
    head[1] = UNIQUE ? written : n;
  }
}

template <int K>
cudaError_t small_k(Ctx& c, ColsIn in, uint32_t n, ColsOut out, bool unique, uint64_t* head) {
  auto run = [&](auto kernel) -> cudaError_t {
    const size_t smem = small_smem<K>(n);
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)small_smem<K>(kSmallSort));
    if (e != cudaSuccess) return e;
    ProfScope ps(c, kRadixScatter, 8.0 * K * n);
    kernel<<<1, kST, smem, c.st>>>(in, n, out, head);
    return cudaGetLastError();
  };
  return unique ? run(k_sort_small<K, true>) : run(k_sort_small<K, false>);
}

// ------------------------------------------------------------ bucket sort
constexpr int kBT = 512;
constexpr int kBItems = 16;
constexpr uint32_t kBTile = kBT * kBItems;
constexpr int kLItems = (int)kBucketCap / kBT;  // a bucket in a block's registers

struct Pack {
  uint32_t shift[kMaxK], mask[kMaxK];
};

template <int K>
__device__ __forceinline__ uint64_t pack_row(const ColsIn& in, const Pack& p, uint64_t i) {
  uint64_t key = 0;
#pragma unroll
  for (int k = 0; k < K; ++k) key |= (uint64_t)__ldg(in.c[k] + i) << p.shift[k];
  return key;
}

template <int K>
__device__ __forceinline__ void unpack_row(const ColsOut& out, const Pack& p, uint64_t i,
                                           uint64_t key) {
#pragma unroll
  for (int k = 0; k < K; ++k) out.c[k][i] = (uint32_t)(key >> p.shift[k]) & p.mask[k];
}

// The bucket of a key (values past the columns' bounds, which no caller has,
// would fall in the last one).
__device__ __forceinline__ uint32_t bucket_of(uint64_t key, uint32_t low, uint32_t nb) {
  const uint64_t b = key >> low;
  return b < nb ? (uint32_t)b : nb - 1;
}

// Rows per bucket.  Reads the columns that reach into the top bits only
// (need, a bit per column).
template <int K>
__global__ void __launch_bounds__(kBT) k_bucket_count(ColsIn in, uint64_t n, Pack p, uint32_t low,
                                                      uint32_t need, uint32_t nb,
                                                      uint32_t* __restrict__ bins) {
  extern __shared__ uint32_t h[];
  for (uint32_t i = threadIdx.x; i < nb; i += kBT) h[i] = 0;
  __syncthreads();
  constexpr int kU = 8;
  const uint64_t step = (uint64_t)gridDim.x * kBT * kU;
  for (uint64_t i0 = (uint64_t)blockIdx.x * kBT * kU + threadIdx.x; i0 < n; i0 += step) {
    uint64_t key[kU];
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      key[u] = 0;
      const uint64_t i = i0 + (uint64_t)u * kBT;
      if (i < n) {
#pragma unroll
        for (int k = 0; k < K; ++k)
          if ((need >> k) & 1u) key[u] |= (uint64_t)__ldg(in.c[k] + i) << p.shift[k];
      }
    }
#pragma unroll
    for (int u = 0; u < kU; ++u)
      if (i0 + (uint64_t)u * kBT < n) atomicAdd(&h[bucket_of(key[u], low, nb)], 1u);
  }
  __syncthreads();
  for (uint32_t i = threadIdx.x; i < nb; i += kBT)
    if (h[i]) atomicAdd(bins + i, h[i]);
}

// One block: bucket starts into off[0..nb] and cursor, the largest bucket
// into *d_max.
__global__ void __launch_bounds__(1024) k_bucket_starts(const uint32_t* __restrict__ bins,
                                                        uint32_t nb, uint32_t* __restrict__ off,
                                                        uint32_t* __restrict__ cursor,
                                                        uint64_t* d_max) {
  __shared__ uint32_t red[33];
  __shared__ uint32_t m;
  if (threadIdx.x == 0) m = 0;
  __syncthreads();
  uint32_t carry = 0, mx = 0;
  for (uint32_t b = 0; b < nb; b += 1024) {
    const uint32_t i = b + threadIdx.x;
    const uint32_t v = i < nb ? bins[i] : 0u;
    mx = v > mx ? v : mx;
    uint32_t tot;
    const uint32_t ex = carry + block_exclusive_sum<1024, uint32_t>(v, red, &tot);
    if (i < nb) off[i] = cursor[i] = ex;
    carry += tot;
  }
  mx = __reduce_max_sync(0xffffffffu, mx);
  if ((threadIdx.x & 31) == 0) atomicMax(&m, mx);
  __syncthreads();
  if (threadIdx.x == 0) {
    off[nb] = carry;
    *d_max = m;
  }
}

// Packed keys (and, with rows, their row numbers) into their buckets: a tile
// counts its rows per bucket in shared memory, claims that many places of each
// bucket with one atomic, and stores every key by itself; the stores of the
// tiles meet in L2, where a bucket's sector fills up before it is written
// back.  16.7M pairs into 8,192 buckets 189 us: bound by the latency of the
// claims and column reads in two blocks per SM (64 registers, 26 of 39 cycles
// an instruction on long scoreboard; L2 42 %, DRAM 19 % busy).
template <int K>
__global__ void __launch_bounds__(kBT, 2) k_bucket_scatter(ColsIn in, uint64_t n, Pack p,
                                                           uint32_t low, uint32_t nb,
                                                           uint32_t* __restrict__ cursor,
                                                           uint64_t* __restrict__ packed,
                                                           uint32_t* __restrict__ rows) {
  extern __shared__ uint32_t h[];
  for (uint32_t i = threadIdx.x; i < nb; i += kBT) h[i] = 0;
  __syncthreads();
  const uint64_t base = (uint64_t)blockIdx.x * kBTile;
  uint64_t key[kBItems];
  uint32_t rank[kBItems];
#pragma unroll
  for (int it = 0; it < kBItems; ++it) {
    const uint64_t i = base + (uint64_t)it * kBT + threadIdx.x;
    key[it] = i < n ? pack_row<K>(in, p, i) : 0ull;
  }
#pragma unroll
  for (int it = 0; it < kBItems; ++it) {
    const uint64_t i = base + (uint64_t)it * kBT + threadIdx.x;
    if (i < n) rank[it] = atomicAdd(&h[bucket_of(key[it], low, nb)], 1u);
  }
  __syncthreads();
  for (uint32_t i = threadIdx.x; i < nb; i += kBT)
    if (h[i]) h[i] = atomicAdd(cursor + i, h[i]);
  __syncthreads();
#pragma unroll
  for (int it = 0; it < kBItems; ++it) {
    const uint64_t i = base + (uint64_t)it * kBT + threadIdx.x;
    if (i < n) {
      const uint64_t at = (uint64_t)h[bucket_of(key[it], low, nb)] + rank[it];
      packed[at] = key[it];
      if (rows) rows[at] = (uint32_t)i;
    }
  }
}

// Columns past the packed key (wide tuples): the order of rows x and y of
// equal keys; 0 where they are the same tuple.
struct Rest {
  ColsIn in;
  uint32_t first, k;  // columns [first, k)
};
__device__ __forceinline__ int rest_order(const Rest& w, uint32_t x, uint32_t y) {
  for (uint32_t c = w.first; c < w.k; ++c) {
    const uint32_t a = __ldg(w.in.c[c] + x), b = __ldg(w.in.c[c] + y);
    if (a != b) return a < b ? -1 : 1;
  }
  return 0;
}

// One bucket per block, sorted in shared memory by its low bits.  A counting
// step by the next 12 bits leaves sub-buckets of a tuple or two, and every
// tuple finds its place among the few of its own by comparing with each.
// Where a sub-bucket holds more than kFine (repeats, uneven values) the block
// takes an LSD radix sort of 8 bits a pass instead, ranked as the global sort
// ranks (match within a warp, warps in order).  Bound by shared memory: the
// radix passes alone took 133 us each for 16.7M keys, so three of them for
// 18-bit pairs 400 of the kernel's 508 us; with the counting step 171 us, L1
// and shared memory 79 % busy, DRAM 16 %.
// UNIQUE: repeats dropped, the keys left packed at the bucket's start and
// counted; else the rows go to out.  WIDE (with UNIQUE): tuples of equal keys
// are ordered by the columns past the key, read through their row numbers,
// and the row numbers are left in place of the keys; a bucket that would need
// the radix sort raises *uneven and the caller sorts another way.
constexpr uint32_t kFine = 24;
constexpr int kFineBits = 12;
template <int K, bool UNIQUE, bool WIDE>
__global__ void __launch_bounds__(kBT, WIDE ? 2 : 3)
    k_bucket_sort(uint64_t* __restrict__ packed, uint32_t* __restrict__ rows,
                  const uint32_t* __restrict__ off, uint32_t low, Pack p, ColsOut out,
                  uint32_t* __restrict__ counts, const Rest rest, uint64_t* uneven) {
  static_assert(UNIQUE || !WIDE, "wide tuples leave as unique rows");
  constexpr int kW = kBT / 32, kFines = 1 << kFineBits, kPer = kFines / kBT;
  static_assert(kW * 256 == kFines, "one table serves both sorts");
  extern __shared__ __align__(16) uint64_t s[];  // kBucketCap keys (then as many row numbers)
  uint32_t* srow = reinterpret_cast<uint32_t*>(s + kBucketCap);
  __shared__ uint32_t tab[kFines + 1];
  __shared__ uint32_t red[kW + 1];
  __shared__ uint32_t smax;
  const uint32_t lo = off[blockIdx.x], m = off[blockIdx.x + 1] - lo;
  if (m == 0) {
    if (UNIQUE && threadIdx.x == 0) counts[blockIdx.x] = 0;
    return;
  }
  if (m > kBucketCap) return;  // (the caller has seen the largest bucket)
  const uint32_t t = threadIdx.x, warp = t >> 5, lane = t & 31u, lt = lanemask_lt();
  const uint32_t items = (m + kBT - 1) / kBT;
  uint64_t key[kLItems];
  uint32_t row[WIDE ? kLItems : 1];
#pragma unroll
  for (int it = 0; it < kLItems; ++it) {
    if (it >= (int)items) break;
    const uint32_t i = it * kBT + t;
    key[it] = i < m ? packed[(uint64_t)lo + i] : 0ull;
    if (WIDE) row[it] = i < m ? rows[(uint64_t)lo + i] : 0u;
  }
  const uint32_t fsh = low > kFineBits ? low - kFineBits : 0u;
  const uint32_t fmask = low > kFineBits ? kFines - 1 : (1u << low) - 1u;
  for (int i = t; i <= kFines; i += kBT) tab[i] = 0;
  if (t == 0) smax = 0;
  __syncthreads();
  uint32_t rk[kLItems];
#pragma unroll
  for (int it = 0; it < kLItems; ++it) {
    if (it >= (int)items) break;
    if (it * kBT + t < m) rk[it] = atomicAdd(&tab[(uint32_t)(key[it] >> fsh) & fmask], 1u);
  }
  __syncthreads();
  {
    uint32_t v[kPer], sum = 0, mx = 0;
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
      v[q] = tab[t * kPer + q];
      sum += v[q];
      mx = v[q] > mx ? v[q] : mx;
    }
    mx = __reduce_max_sync(0xffffffffu, mx);
    if (lane == 0) atomicMax(&smax, mx);
    uint32_t tot;
    uint32_t ex = block_exclusive_sum<kBT, uint32_t>(sum, red, &tot);
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
      tab[t * kPer + q] = ex;
      ex += v[q];
    }
    if (t == 0) tab[kFines] = m;
  }
  __syncthreads();
  if (smax <= kFine) {
#pragma unroll
    for (int it = 0; it < kLItems; ++it) {
      if (it >= (int)items) break;
      if (it * kBT + t < m) {
        const uint32_t at = tab[(uint32_t)(key[it] >> fsh) & fmask] + rk[it];
        s[at] = key[it];
        if (WIDE) srow[at] = row[it];
      }
    }
    __syncthreads();
#pragma unroll
    for (int it = 0; it < kLItems; ++it) {
      if (it >= (int)items) break;
      if (it * kBT + t < m) {
        const uint32_t d = (uint32_t)(key[it] >> fsh) & fmask;
        const uint32_t a = tab[d], e = tab[d + 1], me = a + rk[it];
        uint32_t at = a;
        for (uint32_t j = a; j < e; ++j) {
          const uint64_t x = s[j];
          bool before = x < key[it];
          if (x == key[it] && j != me) {
            int o = 0;
            if constexpr (WIDE) o = rest_order(rest, srow[j], row[it]);
            before = o ? o < 0 : j < me;
          }
          at += before ? 1u : 0u;
        }
        rk[it] = at;
      }
    }
    __syncthreads();
#pragma unroll
    for (int it = 0; it < kLItems; ++it) {
      if (it >= (int)items) break;
      if (it * kBT + t < m) {
        s[rk[it]] = key[it];
        if (WIDE) srow[rk[it]] = row[it];
      }
    }
    __syncthreads();
  } else if constexpr (WIDE) {
    if (t == 0) {
      *uneven = 1;
      counts[blockIdx.x] = 0;
    }
    return;
  } else {
    uint32_t(*wh)[256] = reinterpret_cast<uint32_t(*)[256]>(tab);
    const uint32_t wbase = warp * 32 * items;
    for (uint32_t sh = 0; sh < low; sh += 8) {
      const uint32_t dm = low - sh < 8 ? (1u << (low - sh)) - 1u : 255u;
      for (int i = t; i < kW * 256; i += kBT) tab[i] = 0;
      __syncthreads();
#pragma unroll
      for (int it = 0; it < kLItems; ++it) {
        if (it >= (int)items) break;
        // (the first pass takes the keys in the order they were loaded)
        const bool valid = (sh ? wbase + it * 32 + lane : it * kBT + t) < m;
        const uint32_t d = valid ? (uint32_t)(key[it] >> sh) & dm : 256u;
        const uint32_t peers = __match_any_sync(0xffffffffu, d);
        const uint32_t leader = (uint32_t)__ffs(peers) - 1u;
        uint32_t b = 0;
        if (valid && lane == leader) b = atomicAdd(&wh[warp][d], (uint32_t)__popc(peers));
        b = __shfl_sync(0xffffffffu, b, leader);
        rk[it] = b + __popc(peers & lt);
      }
      __syncthreads();
      uint32_t sum = 0;
      if (t < 256) {
#pragma unroll
        for (int w = 0; w < kW; ++w) {
          const uint32_t x = wh[w][t];
          wh[w][t] = sum;
          sum += x;
        }
      }
      uint32_t tot;
      const uint32_t start = block_exclusive_sum<kBT, uint32_t>(sum, red, &tot);
      if (t < 256) {
#pragma unroll
        for (int w = 0; w < kW; ++w) wh[w][t] += start;
      }
      __syncthreads();
#pragma unroll
      for (int it = 0; it < kLItems; ++it) {
        if (it >= (int)items) break;
        if ((sh ? wbase + it * 32 + lane : it * kBT + t) < m)
          s[wh[warp][(uint32_t)(key[it] >> sh) & dm] + rk[it]] = key[it];
      }
      __syncthreads();
      if (sh + 8 < low) {
#pragma unroll
        for (int it = 0; it < kLItems; ++it) {
          if (it >= (int)items) break;
          const uint32_t i = wbase + it * 32 + lane;
          if (i < m) key[it] = s[i];
        }
      }
    }
  }
  if constexpr (!UNIQUE) {
    for (uint32_t i = t; i < m; i += kBT) unpack_row<K>(out, p, (uint64_t)lo + i, s[i]);
  } else {
    // a chunk of kBT keys per step: every warp's count first, then their
    // places (the tables are free)
    uint32_t* cnt = tab;
    const uint32_t steps = (m + kBT - 1) / kBT;
    uint32_t keep = 0;
    for (uint32_t q = 0; q < steps; ++q) {
      const uint32_t i = q * kBT + t;
      bool k = i < m;
      if (k && i > 0 && s[i] == s[i - 1]) {
        k = false;
        if constexpr (WIDE) k = rest_order(rest, srow[i], srow[i - 1]) != 0;
      }
      const uint32_t bal = __ballot_sync(0xffffffffu, k);
      keep |= (k ? 1u : 0u) << q;
      if (lane == 0) cnt[q * kW + warp] = __popc(bal);
    }
    __syncthreads();
    const uint32_t v = t < steps * kW ? cnt[t] : 0u;  // (at most 8 x 16 of them)
    uint32_t tot;
    const uint32_t ex = block_exclusive_sum<kBT, uint32_t>(v, red, &tot);
    if (t < steps * kW) cnt[t] = ex;
    __syncthreads();
    for (uint32_t q = 0; q < steps; ++q) {
      const uint32_t i = q * kBT + t;
      const uint32_t bal = __ballot_sync(0xffffffffu, (keep >> q) & 1u);
      if ((keep >> q) & 1u) {
        const uint64_t at = (uint64_t)lo + cnt[q * kW + warp] + __popc(bal & lt);
        if constexpr (WIDE)
          rows[at] = srow[i];
        else
          packed[at] = s[i];
      }
    }
    if (t == 0) counts[blockIdx.x] = tot;
  }
}

// The buckets' unique keys side by side, as columns.
template <int K>
__global__ void __launch_bounds__(kBT) k_bucket_unpack(const uint64_t* __restrict__ packed,
                                                       const uint32_t* __restrict__ off,
                                                       const uint32_t* __restrict__ counts,
                                                       const uint64_t* __restrict__ pre, Pack p,
                                                       ColsOut out) {
  const uint64_t lo = off[blockIdx.x], at = pre[blockIdx.x];
  const uint32_t m = counts[blockIdx.x];
  for (uint32_t i = threadIdx.x; i < m; i += kBT) unpack_row<K>(out, p, at + i, packed[lo + i]);
}

// The same for wide tuples: whole rows gathered by their numbers.
__global__ void __launch_bounds__(kBT) k_bucket_gather(const uint32_t* __restrict__ rows,
                                                       const uint32_t* __restrict__ off,
                                                       const uint32_t* __restrict__ counts,
                                                       const uint64_t* __restrict__ pre, ColsIn in,
                                                       uint32_t k, ColsOut out) {
  const uint64_t lo = off[blockIdx.x], at = pre[blockIdx.x];
  const uint32_t m = counts[blockIdx.x];
  for (uint32_t i = threadIdx.x; i < m; i += kBT) {
    const uint32_t r = rows[lo + i];
#pragma unroll
    for (int c = 0; c < kMaxK; ++c)
      if (c < (int)k) out.c[c][at + i] = __ldg(in.c[c] + r);
  }
}

template <int K>
cudaError_t bucket_count_k(Ctx& c, const BucketPlan& b, const Pack& p, ColsIn in, uint64_t n,
                           uint32_t* bins) {
  uint32_t need = 0;
  for (int k = 0; k < K; ++k)
    if (p.mask[k] && ((uint64_t)p.mask[k] << p.shift[k]) >> b.low) need |= 1u << k;
  const size_t smem = 4ull * b.buckets;
  cudaError_t e = cudaFuncSetAttribute(k_bucket_count<K>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  uint64_t blocks = (n + kBT * 32 - 1) / (kBT * 32);
  if (blocks > 152 * 2) blocks = 152 * 2;
  ProfScope ps(c, kRadixUpsweep, 4.0 * __builtin_popcount(need) * n);
  k_bucket_count<K><<<(unsigned)blocks, kBT, smem, c.st>>>(in, n, p, b.low, need, b.buckets, bins);
  return cudaGetLastError();
}

template <int K>
cudaError_t bucket_run_k(Ctx& c, const BucketPlan& b, const Pack& p, ColsIn in, uint64_t n,
                         ColsOut out, uint64_t* packed, uint32_t* off, uint32_t* cursor,
                         uint32_t* counts, uint64_t* pre, void* scan_ws, uint64_t* d_unique) {
  const bool wide = b.k > b.keys;
  if (wide && !d_unique) return cudaErrorInvalidValue;
  uint32_t* rows = wide ? reinterpret_cast<uint32_t*>(packed + n) : nullptr;
  const size_t sc = 4ull * b.buckets, ss = (wide ? 12ull : 8ull) * kBucketCap;
  cudaError_t e = cudaFuncSetAttribute(k_bucket_scatter<K>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sc);
  auto sort = wide ? k_bucket_sort<1, true, true>  // (K unused: whole rows are gathered later)
                   : d_unique ? k_bucket_sort<K, true, false> : k_bucket_sort<K, false, false>;
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(sort, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ss);
  if (e != cudaSuccess) return e;
  {
    ProfScope ps(c, kRadixScatter, (4.0 * K + 8.0) * n);
    k_bucket_scatter<K><<<(unsigned)((n + kBTile - 1) / kBTile), kBT, sc, c.st>>>(
        in, n, p, b.low, b.buckets, cursor, packed, rows);
  }
  {
    ProfScope ps(c, kRadixScatter, (8.0 + 4.0 * K) * n);
    sort<<<b.buckets, kBT, ss, c.st>>>(packed, rows, off, b.low, p, out, counts,
                                       Rest{in, b.keys, b.k}, wide ? d_unique + 1 : nullptr);
  }
  e = cudaGetLastError();
  if (e != cudaSuccess || !d_unique) return e;
  e = exclusive_scan(c, counts, b.buckets, pre, d_unique, scan_ws);
  if (e != cudaSuccess) return e;
  ProfScope ps(c, kDiffMerge, (8.0 + 4.0 * b.k) * n);
  if (wide)
    k_bucket_gather<<<b.buckets, kBT, 0, c.st>>>(rows, off, counts, pre, in, b.k, out);
  else
    k_bucket_unpack<K><<<b.buckets, kBT, 0, c.st>>>(packed, off, counts, pre, p, out);
  return cudaGetLastError();
}

size_t up256(size_t b) { return (b + 255) & ~size_t(255); }

}  // namespace

cudaError_t sort_small(Ctx& c, uint32_t k, ColsIn in, uint64_t n, ColsOut out, bool unique,
                       uint64_t* head) {
  if (n > kSmallSort) return cudaErrorInvalidValue;
  switch (k) {
    case 1: return small_k<1>(c, in, (uint32_t)n, out, unique, head);
    case 2: return small_k<2>(c, in, (uint32_t)n, out, unique, head);
    case 3: return small_k<3>(c, in, (uint32_t)n, out, unique, head);
    case 4: return small_k<4>(c, in, (uint32_t)n, out, unique, head);
    case 5: return small_k<5>(c, in, (uint32_t)n, out, unique, head);
    case 6: return small_k<6>(c, in, (uint32_t)n, out, unique, head);
    case 7: return small_k<7>(c, in, (uint32_t)n, out, unique, head);
    case 8: return small_k<8>(c, in, (uint32_t)n, out, unique, head);
    default: return cudaErrorInvalidValue;
  }
}

bool bucket_plan(uint32_t k, const uint32_t* col_bits, const uint32_t* col_max, uint64_t n,
                 BucketPlan& b) {
  b = BucketPlan{};
  b.k = k;
  if (k < 1 || k > (uint32_t)kMaxK || n > 0xFFFFFFFFull) return false;
  uint32_t total = 0;
  while (b.keys < k && total + col_bits[b.keys] <= 64) total += col_bits[b.keys++];
  uint32_t sh = 0;
  for (int c = (int)b.keys - 1; c >= 0; --c) {
    if (col_bits[c]) b.shift[c] = sh;
    b.mask[c] = (uint32_t)((1ull << col_bits[c]) - 1);
    sh += col_bits[c];
  }
  // the largest key, or without the columns' maxima the largest there could
  // be (it may be twice the real one, so fewer rows a bucket are aimed at)
  uint64_t top = total >= 64 ? ~0ull : (1ull << total) - 1;
  uint64_t rows = kBucketRows * 3 / 4;
  if (col_max) {
    top = 0;
    for (uint32_t c = 0; c < b.keys; ++c) top |= (uint64_t)col_max[c] << b.shift[c];
    rows = kBucketRows;
  }
  for (b.low = total; b.low > 1;) {
    if ((top >> (b.low - 1)) >= 1ull << kBucketMaxBits) break;
    --b.low;
    if (n / ((top >> b.low) + 1) <= rows) break;
  }
  if (b.low >= total || n / ((top >> b.low) + 1) > kBucketCap * 7 / 8) return false;
  b.buckets = (uint32_t)(top >> b.low) + 1;
  return true;
}

size_t bucket_workspace(const BucketPlan& b) {
  return 3 * up256(4ull * b.buckets + 4) + up256(4ull * b.buckets) + up256(8ull * b.buckets) +
         scan_workspace(b.buckets);
}

// The workspace: bins (then the buckets' unique counts), off, cursor, pre, scan.
struct BucketWs {
  uint32_t *bins, *off, *cursor, *counts;
  uint64_t* pre;
  void* scan;
  BucketWs(const BucketPlan& b, void* ws) {
    char* p = static_cast<char*>(ws);
    auto take = [&](size_t n) {
      void* r = p;
      p += up256(n);
      return r;
    };
    bins = static_cast<uint32_t*>(take(4ull * b.buckets + 4));
    off = static_cast<uint32_t*>(take(4ull * b.buckets + 4));
    cursor = static_cast<uint32_t*>(take(4ull * b.buckets + 4));
    counts = static_cast<uint32_t*>(take(4ull * b.buckets));
    pre = static_cast<uint64_t*>(take(8ull * b.buckets));
    scan = p;
  }
};

static Pack pack_of(const BucketPlan& b) {
  Pack p{};
  for (uint32_t k = 0; k < b.keys; ++k) {
    p.shift[k] = b.shift[k];
    p.mask[k] = b.mask[k];
  }
  return p;
}

cudaError_t bucket_count(Ctx& c, const BucketPlan& b, ColsIn in, uint64_t n, void* ws,
                         uint64_t* d_max) {
  const BucketWs w(b, ws);
  const Pack p = pack_of(b);
  cudaError_t e = cudaMemsetAsync(w.bins, 0, 4ull * b.buckets, c.st);
  if (e != cudaSuccess) return e;
  switch (b.keys) {
    case 1: e = bucket_count_k<1>(c, b, p, in, n, w.bins); break;
    case 2: e = bucket_count_k<2>(c, b, p, in, n, w.bins); break;
    case 3: e = bucket_count_k<3>(c, b, p, in, n, w.bins); break;
    case 4: e = bucket_count_k<4>(c, b, p, in, n, w.bins); break;
    case 5: e = bucket_count_k<5>(c, b, p, in, n, w.bins); break;
    case 6: e = bucket_count_k<6>(c, b, p, in, n, w.bins); break;
    case 7: e = bucket_count_k<7>(c, b, p, in, n, w.bins); break;
    case 8: e = bucket_count_k<8>(c, b, p, in, n, w.bins); break;
    default: return cudaErrorInvalidValue;
  }
  if (e != cudaSuccess) return e;
  ProfScope ps(c, kScan, 12.0 * b.buckets);
  k_bucket_starts<<<1, 1024, 0, c.st>>>(w.bins, b.buckets, w.off, w.cursor, d_max);
  return cudaGetLastError();
}

cudaError_t bucket_sort(Ctx& c, const BucketPlan& b, ColsIn in, uint64_t n, ColsOut out,
                        uint64_t* packed, void* ws, uint64_t* d_unique) {
  const BucketWs w(b, ws);
  const Pack p = pack_of(b);
#define CDL_BUCKET(K)                                                                       \
  case K:                                                                                   \
    return bucket_run_k<K>(c, b, p, in, n, out, packed, w.off, w.cursor, w.counts, w.pre,   \
                           w.scan, d_unique)
  switch (b.keys) {
    CDL_BUCKET(1);
    CDL_BUCKET(2);
    CDL_BUCKET(3);
    CDL_BUCKET(4);
    CDL_BUCKET(5);
    CDL_BUCKET(6);
    CDL_BUCKET(7);
    CDL_BUCKET(8);
    default: return cudaErrorInvalidValue;
  }
#undef CDL_BUCKET
}

}  // namespace cdl
