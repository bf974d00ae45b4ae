// Step (b): the join of Algorithm 1 in three passes.
//
// Pass 1 (count): every probe row looks its key up in the build side's
// hybrid index and stores the matched range length (0 when absent), and
// each tile of rows also sums its lengths -- the first half of the scan.
// Pass 2 (scan): exclusive scan of the lengths into 64-bit output offsets
// (pos_buf) and the total join size (Algorithm 1's reduce).
// Pass 3 (write): output-partitioned, the variant Section 4 chooses for
// skew: each block owns an equal share of the merged sequence of (row
// starts, output positions) -- a merge-path split found by binary search
// over the offsets, so a block's work is bounded whether its rows match
// nothing or one row matches a hundred thousand tuples.  The block re-probes
// the index once per row it covers, then every output position finds its row
// by binary search in shared memory (the search of Algorithm 1's write loop,
// over the non-empty ranges only) and gathers the build row
// start + (n - pos_buf[j]).  Projection, constant head columns, equalities
// beyond the hashed key and inequalities (x != y) are applied in the same
// pass, so the join result is written directly as head columns (Section 4:
// the join result is materialised only at projection).
#include "kernels.h"

namespace cdl {

namespace {

constexpr int kCT = 256;  // count pass: threads; tiles of kScanTile rows
constexpr int kCItems = kScanTile / kCT;
constexpr int kJT = 256;  // write pass threads
constexpr int kDU = 4;    // write pass into a bitmap: outputs per thread in flight
constexpr uint32_t kDRows = 8;  // ... and the most probe rows a block walks one by one
constexpr int kJItems = 8;
constexpr int kJTile = kJT * kJItems;  // merged items per block

// Column v of a column set held in registers: a chain of selects with
// constant indices, so that a run-time column number does not send the set
// to local memory.
__device__ __forceinline__ const uint32_t* col_of(const ColsIn& c, uint32_t v) {
  const uint32_t* p = c.c[0];
#pragma unroll
  for (int k = 1; k < kMaxK; ++k)
    if (v == (uint32_t)k) p = c.c[k];
  return p;
}

__device__ __forceinline__ uint32_t probe_key1(const JoinSpec& j, const ColsIn& probe,
                                              uint64_t row) {
  return j.pk1 == 0xFFu ? 0u : __ldg(col_of(probe, j.pk1) + row);
}

// Range of build rows matching probe row `row`: the hybrid index lookup, or
// every build row for a join without shared variables.
// (range: direct_range of the index)
__device__ __forceinline__ uint32_t lookup(const JoinSpec& j, const ColsIn& probe, uint32_t range,
                                          uint64_t row, uint32_t* start) {
  if (j.cross) {
    *start = 0;
    return j.n_build;
  }
  return find_key(j.ix, range, __ldg(col_of(probe, j.pk0) + row), probe_key1(j, probe, row), start);
}

// Range of second-build-side rows matching probe row `row` (star joins).
__device__ __forceinline__ uint32_t lookup2(const JoinSpec& j, const ColsIn& probe, uint64_t row,
                                           uint32_t* start) {
  const uint32_t k1 = j.qk1 == 0xFFu ? 0u : __ldg(col_of(probe, j.qk1) + row);
  return find_key(j.ix2, direct_range(j.ix2), __ldg(col_of(probe, j.qk0) + row), k1, start);
}

// The probe side of a launch: the spec's columns and row count, or (inside
// a captured round) the ones device memory holds, the count clamped to the
// capacity the spec's n_probe then gives.
__device__ __forceinline__ ColsIn probe_cols(const JoinSpec& j) {
  return j.dprobe ? *j.dprobe : j.probe;
}

// Ranges of a thread's N probe rows.  The direct form's reads go out
// together; the hash form's probes are a loop each.
template <int N>
__device__ __forceinline__ void set_lookup(const JoinSpec& j, const KeyIndex& x, uint32_t range,
                                           const uint32_t* c0, const uint32_t* c1, uint64_t base,
                                           uint32_t live, uint32_t (&st)[N], uint32_t (&cnt)[N]) {
  uint32_t k0[N];
#pragma unroll
  for (int q = 0; q < N; ++q) {
    k0[q] = 0;
    st[q] = cnt[q] = 0;
    if ((live >> q) & 1u) k0[q] = __ldg(c0 + base + (uint64_t)q * kCT + threadIdx.x);
  }
  if (range) {
#pragma unroll
    for (int q = 0; q < N; ++q)
      if (((live >> q) & 1u) && k0[q] < range) cnt[q] = find_entry(x, k0[q], &st[q]);
    return;
  }
#pragma unroll
  for (int q = 0; q < N; ++q)
    if ((live >> q) & 1u) {
      const uint32_t k1 = c1 ? __ldg(c1 + base + (uint64_t)q * kCT + threadIdx.x) : 0u;
      cnt[q] = probe_table(x.table, x.slots - 1, k0[q], k1, &st[q]);
    }
}

// Key columns of the probe side, for set_lookup.
__device__ __forceinline__ const uint32_t* key_col(const ColsIn& probe, uint32_t v) {
  return v == 0xFFu ? nullptr : col_of(probe, v);
}

// A thread's eight rows of a tile are looked up together: their keys, then
// their entries, are in flight at once.  Points-to's 17 counts 421 -> 270 us;
// 16M rows over 2^25 entries by key stay at 252 us, bound by the 256 MB
// array's sectors (a read of one in 64 bytes of HBM for each row).
__global__ void __launch_bounds__(kCT) k_join_count(const JoinSpec j, uint32_t* __restrict__ counts,
                                                    uint64_t* __restrict__ tile_sums,
                                                    uint32_t* err) {
  __shared__ uint64_t red[kCT / 32 + 1];
  const uint64_t n = dev_size(j.dn, j.n_probe);
  const ColsIn probe = probe_cols(j);
  const uint32_t *pk0 = key_col(probe, j.pk0), *pk1 = key_col(probe, j.pk1);
  const uint32_t *qk0 = nullptr, *qk1 = nullptr;
  if (j.star) {
    qk0 = key_col(probe, j.qk0);
    qk1 = key_col(probe, j.qk1);
  }
  const uint32_t range = direct_range(j.ix), range2 = j.star ? direct_range(j.ix2) : 0u;
  // tile 0 is written even for n == 0; blocks loop over the tiles
  const uint64_t ntiles = n ? (n + kScanTile - 1) / kScanTile : 1;
  for (uint64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const uint64_t base = tile * kScanTile;
    uint32_t live = 0, st[kCItems], cnt[kCItems];
#pragma unroll
    for (int i = 0; i < kCItems; ++i)
      live |= (base + (uint64_t)i * kCT + threadIdx.x < n ? 1u : 0u) << i;
    if (j.cross) {
#pragma unroll
      for (int i = 0; i < kCItems; ++i) {
        st[i] = 0;
        cnt[i] = (live >> i) & 1u ? j.n_build : 0u;
      }
    } else {
      set_lookup<kCItems>(j, j.ix, range, pk0, pk1, base, live, st, cnt);
    }
    if (j.starts) {
#pragma unroll
      for (int i = 0; i < kCItems; ++i)
        if ((live >> i) & 1u) j.starts[base + (uint64_t)i * kCT + threadIdx.x] = st[i];
    }
    if (j.hub_min) {  // hub_or's
#pragma unroll
      for (int i = 0; i < kCItems; ++i)
        if (cnt[i] >= j.hub_min) cnt[i] = 0;
    }
    if (j.star) {
      uint32_t found = 0, cnt2[kCItems];
#pragma unroll
      for (int i = 0; i < kCItems; ++i) found |= (cnt[i] ? 1u : 0u) << i;
      set_lookup<kCItems>(j, j.ix2, range2, qk0, qk1, base, found, st, cnt2);
#pragma unroll
      for (int i = 0; i < kCItems; ++i) {
        const uint64_t prod = (uint64_t)cnt[i] * cnt2[i];
        if (prod > 0xFFFFFFFFull && err) atomicOr(err, kErrCapacity);
        cnt[i] = prod > 0xFFFFFFFFull ? 0u : (uint32_t)prod;
      }
    }
    uint64_t s = 0;
#pragma unroll
    for (int i = 0; i < kCItems; ++i)
      if ((live >> i) & 1u) {
        counts[base + (uint64_t)i * kCT + threadIdx.x] = cnt[i];
        s += cnt[i];
      }
    uint64_t total;
    block_exclusive_sum<kCT, uint64_t>(s, red, &total);  // ends with a barrier
    if (threadIdx.x == 0) tile_sums[tile] = total;
  }
}

__global__ void __launch_bounds__(kCT) k_join_count_only(const JoinSpec j,
                                                         uint32_t* __restrict__ counts) {
  const uint64_t row = (uint64_t)blockIdx.x * kCT + threadIdx.x;
  uint32_t start;
  if (row < j.n_probe) counts[row] = lookup(j, j.probe, direct_range(j.ix), row, &start);
}

// Number of probe rows among the first d items of the merge of the row
// starts off[0..n) with the output positions 0..total-1 (a row start goes
// before the output positions it is <=).
__device__ __forceinline__ uint64_t merge_split(const uint64_t* off, uint64_t n, uint64_t total,
                                                uint64_t d) {
  uint64_t lo = d > total ? d - total : 0, hi = d < n ? d : n;
  while (lo < hi) {
    const uint64_t mid = lo + ((hi - lo) >> 1);
    if (__ldg(off + mid) <= d - mid - 1)
      lo = mid + 1;
    else
      hi = mid;
  }
  return lo;
}

// All blocks' splits at once, one thread per split, so that no block
// waits on a chain of dependent global loads before its first useful one.
// Inside a captured round an unfiltered join's output range is claimed here
// too (thread 0): *d_base = *cursor, *cursor += the join's size, and a range
// past cap raises *overflow.
// A count's mark and its check (kernels.h).  The check costs the write no
// launch and no wait of its own: the splits bear its result (kClosed), and
// only a write that searches its splits itself has it from a launch before.
constexpr uint64_t kMarkTag = 0x6a6f696e636f756eull, kClosed = ~0ull;
__device__ __forceinline__ bool marked(const uint64_t* head, const JoinMark& m, uint64_t total) {
  return head[1] == total && head[4] == kMarkTag && head[5] == m.probe && head[6] == m.build &&
         head[7] == m.form;
}
__device__ __forceinline__ void open_write(uint64_t* head, bool open) {
  head[0] = open ? 0 : kErrState;
  head[2] = 0;
  head[3] = open;
}
__global__ void k_join_begin(uint64_t* head, JoinMark m) {
  head[0] = head[1] = head[2] = head[3] = 0;
  head[4] = kMarkTag;
  head[5] = m.probe;
  head[6] = m.build;
  head[7] = m.form;
}
__global__ void k_join_open(uint64_t* head, JoinMark m, uint64_t total) {
  open_write(head, marked(head, m, total));
}

__global__ void k_write_splits(const uint64_t* __restrict__ off, uint64_t n, uint64_t total,
                               uint64_t* __restrict__ splits, uint64_t nblocks,
                               const uint64_t* dn, const uint64_t* dtotal,
                               unsigned long long* cursor, uint64_t* d_base, uint64_t cap,
                               uint32_t* overflow, uint64_t* head, JoinMark mark) {
  const uint64_t b = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  bool open = true;
  if (head) {
    open = marked(head, mark, total);
    if (b == 0) open_write(head, open);
  }
  if (d_base && b == 0) {
    const uint64_t b0 = *cursor, t = *dtotal;
    *d_base = b0;
    *cursor = b0 + t;
    if (b0 + t > cap) atomicOr(overflow, 1u);
  }
  if (dn) {  // sizes from device memory (nblocks was sized for the capacities)
    n = dev_size(dn, n);
    total = dev_size(dtotal, total);
    nblocks = (n + total + kJTile - 1) / kJTile;
  }
  if (b > nblocks) return;
  const uint64_t d = b * kJTile < n + total ? b * kJTile : n + total;
  splits[b] = open ? merge_split(off, n, total, d) : kClosed;
}

__device__ __forceinline__ uint32_t ref_value(const JoinSpec& j, const ColsIn& probe, const Ref& r,
                                              uint64_t row, uint64_t brow, uint64_t brow2 = 0) {
  if (r.side == 0) return __ldg(col_of(probe, r.v) + row);
  if (r.side == 1) return __ldg(j.build.c[r.v] + brow);
  if (r.side == 3) return __ldg(j.build2.c[r.v] + brow2);
  return r.v;
}

// Where a launch's values come from, staged once per block: the head
// columns, then the pairs of the equalities and of the inequalities.  The
// loops over columns read this table and are not unrolled; only the loop over
// a thread's outputs is, so that its loads are in flight together.  (With the
// columns unrolled as well -- eight outputs times eight columns times the
// sides a value may come from -- half of all warp cycles waited for
// instructions: same generation on 200,000 nodes took 98 ms, 68 so.)
struct SetRefs {
  const uint32_t* p[kMaxK + 16];
  uint32_t side[kMaxK + 16], v[kMaxK + 16];
  uint32_t* out[kMaxK];
  uint32_t shift[kMaxK], mask[kMaxK];
};

__device__ __forceinline__ void stage_refs(const JoinSpec& j, const DenseSet& d, const ColsOut& out,
                                           SetRefs& s) {
  const uint32_t t = threadIdx.x;
  if (t < kMaxK + 16) {
    Ref f{2, 0};
    if (t < kMaxK) {
      if (t < j.out_k) f = j.out[t];
      s.out[t] = j.dout ? j.dout->c[t] : out.c[t];
      s.shift[t] = d.shift[t];
      s.mask[t] = d.mask[t];
    } else {
      const uint32_t i = t - kMaxK;
      if (i < 2 * j.n_eq)
        f = j.eq[i >> 1][i & 1];
      else if (i < 2 * (j.n_eq + j.n_neq))
        f = j.neq[(i >> 1) - j.n_eq][i & 1];
    }
    s.side[t] = f.side;
    s.v[t] = f.v;
    s.p[t] = f.side == 0 ? (j.dprobe ? j.dprobe->c[f.v] : j.probe.c[f.v])
             : f.side == 1 ? j.build.c[f.v]
             : f.side == 3 ? j.build2.c[f.v]
                           : nullptr;
  }
  __syncthreads();
}

// Value i of the table for the N outputs in `live`: probe row base + row[q],
// build rows b1[q] and b2[q].
template <int N>
__device__ __forceinline__ void set_values(const SetRefs& s, uint32_t i, uint32_t live,
                                           uint64_t base, const uint32_t (&row)[N],
                                           const uint32_t (&b1)[N], const uint32_t (&b2)[N],
                                           uint32_t (&v)[N]) {
  const uint32_t side = s.side[i];
  const uint32_t* p = s.p[i] + (side == 0 ? base : 0ull);
#pragma unroll
  for (int q = 0; q < N; ++q) {
    v[q] = s.v[i];
    if (side != 2 && ((live >> q) & 1u)) v[q] = __ldg(p + (side == 0 ? row[q] : side == 1 ? b1[q] : b2[q]));
  }
}

// The outputs in `live` that pass the equalities and inequalities.
template <int N>
__device__ __forceinline__ uint32_t filter_outputs(const JoinSpec& j, const SetRefs& s,
                                                   uint32_t live, uint64_t base,
                                                   const uint32_t (&row)[N],
                                                   const uint32_t (&b1)[N],
                                                   const uint32_t (&b2)[N]) {
#pragma unroll 1
  for (uint32_t f = 0; f < j.n_eq + j.n_neq; ++f) {
    uint32_t x[N], y[N];
    set_values<N>(s, kMaxK + 2 * f, live, base, row, b1, b2, x);
    set_values<N>(s, kMaxK + 2 * f + 1, live, base, row, b1, b2, y);
#pragma unroll
    for (int q = 0; q < N; ++q)
      if ((x[q] == y[q]) != (f < j.n_eq)) live &= ~(1u << q);
  }
  return live;
}

// Packed tuples of the outputs in `live` (kNoTuple: none, dropped by a filter
// or outside the set's space, which sets bad).
template <bool FILTER, int N>
__device__ __forceinline__ void set_tuples(const JoinSpec& j, const SetRefs& s, uint32_t live,
                                           uint64_t base, const uint32_t (&row)[N],
                                           const uint32_t (&b1)[N], const uint32_t (&b2)[N],
                                           uint64_t (&idx)[N], bool& bad) {
  if (FILTER) live = filter_outputs<N>(j, s, live, base, row, b1, b2);
  uint32_t out = 0;
#pragma unroll
  for (int q = 0; q < N; ++q) idx[q] = 0;
#pragma unroll 1
  for (uint32_t k = 0; k < j.out_k; ++k) {
    uint32_t v[N];
    set_values<N>(s, k, live, base, row, b1, b2, v);
    const uint32_t sh = s.shift[k], mask = s.mask[k];
#pragma unroll
    for (int q = 0; q < N; ++q) {
      idx[q] |= (uint64_t)v[q] << sh;
      out |= (v[q] > mask ? 1u : 0u) << q;
    }
  }
  bad |= (out & live) != 0;
#pragma unroll
  for (int q = 0; q < N; ++q)
    if (!((live & ~out) >> q & 1u)) idx[q] = kNoTuple;
}

// New tuples (bit q of fresh) to the head's columns; those past cap are taken
// out of the set again and true is returned to their threads.
template <int THREADS, int N>
__device__ __forceinline__ bool set_store(const JoinSpec& j, const DenseSet& d, const SetRefs& s,
                                          const uint64_t (&idx)[N], uint32_t fresh,
                                          unsigned long long* cursor, uint64_t cap, uint32_t* wsum) {
  uint32_t at[N];
  uint64_t pos;
  if (!claim_places<THREADS, N>(fresh, cursor, wsum, at, &pos)) return false;
  const uint64_t room = cap > pos ? cap - pos : 0;
#pragma unroll 1
  for (uint32_t k = 0; k < j.out_k; ++k) {
    uint32_t* o = s.out[k] + pos;
    const uint32_t sh = s.shift[k], mask = s.mask[k];
#pragma unroll
    for (int q = 0; q < N; ++q)
      if (((fresh >> q) & 1u) && at[q] < room) o[at[q]] = (uint32_t)(idx[q] >> sh) & mask;
  }
  bool over = false;
  if (room < (uint64_t)N * 32) {  // (rare: near or past the buffer's end)
#pragma unroll
    for (int q = 0; q < N; ++q)
      if (((fresh >> q) & 1u) && at[q] >= room) {
        set_remove(d, idx[q]);
        over = true;
      }
  }
  return over;
}

// Row heads: five resident blocks per SM (registers capped at 51).  Bitmap
// heads: registers capped at 32, eight blocks per SM (seven for star joins,
// bounded by shared memory); the bit-setting loop is latency-bound, and on
// points-to at 2^-5 this cap took the write from 6.6 s to 5.6 s per
// fixpoint against four or five blocks.
// FORM kBits: each output tuple sets its bit in dset instead of being written.
// FORM kSet: dset is Full itself; an output whose bit was clear is new and is
// appended to the delta rows (out, packed at *cursor, one claim per block),
// so the round needs no sort and no merge.  Bound by the random accesses to
// the bitmap: a block's outputs are taken in one sweep, eight per thread,
// all reads and then all atomics in flight.  Same generation on 200,000
// nodes, where the bitmap is 8 GB: 1.6e9 outputs in 62 ms when all of its
// joins were written by this form (the sorts, merges and writes it replaced
// took 231 ms of 267); k_join_set has since taken most of them over.
enum Form : int { kRows = 0, kBits = 1, kSet = 2 };
template <bool FILTER, int FORM, bool STAR>
__global__ void __launch_bounds__(kJT, FORM == kBits ? 8 : FORM == kSet ? 4 : 5) k_join_write(const JoinSpec j, const uint64_t* __restrict__ off,
                                                    uint64_t total, ColsOut out, uint64_t base,
                                                    unsigned long long* cursor, uint64_t out_cap,
                                                    const uint64_t* __restrict__ splits,
                                                    uint32_t* err, const uint64_t* dtotal,
                                                    const uint64_t* dbase, const DenseSet dset) {
  constexpr bool DENSE = FORM == kBits;
  // row r's first output: the carried-in row 0 keeps its global start,
  // every later row starts inside the block's window of at most kJTile
  // outputs and keeps its start relative to the window
  __shared__ uint16_t s_loc[kJTile + 1];
  __shared__ uint64_t s_a0;
  __shared__ uint32_t s_start[kJTile + 1];
  __shared__ uint32_t s_start2[STAR ? kJTile + 1 : 1];  // second range: start, length
  __shared__ uint32_t s_cnt2[STAR ? kJTile + 1 : 1];
  __shared__ uint16_t s_row[DENSE ? 1 : kJTile];  // staged row of each of the block's outputs
  __shared__ uint64_t s_split[2];
  __shared__ __align__(8) uint32_t red[kJT / 32 + 2];
  __shared__ unsigned long long s_base;
  __shared__ SetRefs refs;
  if constexpr (FORM == kSet) stage_refs(j, dset, out, refs);
  const uint64_t n_probe = dev_size(j.dn, j.n_probe);
  const ColsIn probe = probe_cols(j);
  // a device-given join size past the capacity the launch was sized for:
  // the outputs past it are not written, so the round must be redone (a
  // filtered join's survivors may still have fit: the flag is conservative)
  if (dtotal && blockIdx.x == 0 && threadIdx.x == 0 && *dtotal > total && err)
    atomicOr(err, kErrCapacity);
  total = dev_size(dtotal, total);
  const uint64_t wbase = dbase ? *dbase : base;  // rows of this join start here
  (void)wbase;  // (a bitmap head writes no rows)
  const uint64_t nm = n_probe + total;
  const uint64_t ntiles = (nm + kJTile - 1) / kJTile;  // a device-given size may be below the grid's
  for (uint64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
  {
  const uint64_t d0 = tile * kJTile;
  const uint64_t d1 = d0 + kJTile < nm ? d0 + kJTile : nm;
  if (splits) {
    if (threadIdx.x < 2) s_split[threadIdx.x] = splits[tile + threadIdx.x];
  } else {
    if (threadIdx.x == 0)
      s_split[0] = FORM == kRows && j.head && !j.head[3] ? kClosed : merge_split(off, n_probe, total, d0);
    if (threadIdx.x == 32) s_split[1] = merge_split(off, n_probe, total, d1);
  }
  // (a device-sized launch had its range claimed by the split kernel)
  if (!FILTER && FORM == kRows && !dbase && tile == 0 && threadIdx.x == 0)
    atomicAdd(cursor, (unsigned long long)total);
  __syncthreads();
  if constexpr (FORM == kRows)
    if (s_split[0] == kClosed) return;
  const uint64_t j0 = s_split[0], j1 = s_split[1];
  const uint64_t o0 = d0 - j0, o1 = d1 - j1;
  const uint64_t r_lo = j0 > 0 ? j0 - 1 : 0;
  const uint32_t nrows = (uint32_t)(j1 - r_lo);
  const uint32_t range = direct_range(j.ix);
  // the outputs' rows come from a table where the head is written as rows
  // (a bitmap head's block searches the staged starts, or walks its rows
  // one by one when it has a few: there the table's barriers cost more
  // than the searches they save)
  constexpr bool table = !DENSE;
  const uint32_t no = (uint32_t)(o1 - o0);
  if constexpr (table) {
    for (uint32_t i = threadIdx.x; i < no; i += kJT) s_row[i] = 0;
    __syncthreads();
  }
  for (uint32_t r = threadIdx.x; r < nrows; r += kJT) {
    const uint64_t row = r_lo + r;
    const uint64_t a = __ldg(off + row);
    const uint64_t b = row + 1 < n_probe ? __ldg(off + row + 1) : total;
    uint32_t st = 0;
    if (b > a) {
      if (!STAR && j.starts)
        st = __ldg(j.starts + row);
      else
        lookup(j, probe, range, row, &st);
    }
    if (r == 0)
      s_a0 = a;
    else
      s_loc[r] = (uint16_t)(a - o0);
    s_start[r] = st;
    // a row with outputs in the block's window marks its first one there
    // (such rows start at distinct outputs; the row carried in from the
    // block before may end at the window's start)
    const uint64_t first = a > o0 ? a : o0;
    if (table && b > first && first < o1) s_row[first - o0] = (uint16_t)r;
    if constexpr (STAR) {
      uint32_t st2 = 0, c2 = 1;
      if (b > a) c2 = lookup2(j, probe, row, &st2);
      s_start2[r] = st2;
      s_cnt2[r] = c2;
    }
  }
  __syncthreads();
  auto off_of = [&](uint32_t r) -> uint64_t { return r == 0 ? s_a0 : o0 + s_loc[r]; };
  // head values of probe row `row` matched with build row `brow`; false
  // when a filter drops the pair
  auto tuple_of = [&](uint64_t row, uint64_t brow, uint64_t brow2,
                      uint32_t (&vals)[kMaxK]) -> bool {
#pragma unroll
    for (int k = 0; k < kMaxK; ++k)
      if (k < (int)j.out_k) vals[k] = ref_value(j, probe, j.out[k], row, brow, brow2);
    bool keep = true;
    if (FILTER) {
      for (uint32_t q = 0; q < j.n_eq; ++q)
        keep &= ref_value(j, probe, j.eq[q][0], row, brow, brow2) ==
                ref_value(j, probe, j.eq[q][1], row, brow, brow2);
      for (uint32_t q = 0; q < j.n_neq; ++q)
        keep &= ref_value(j, probe, j.neq[q][0], row, brow, brow2) !=
                ref_value(j, probe, j.neq[q][1], row, brow, brow2);
    }
    return keep;
  };
  // output l of staged row r (l < its range length, or the product of both)
  auto tuple_in = [&](uint32_t r, uint64_t l, uint32_t (&vals)[kMaxK]) -> bool {
    if constexpr (STAR) {
      const uint32_t c2 = s_cnt2[r];
      const uint32_t l1 = (uint32_t)l / c2;
      return tuple_of(r_lo + r, (uint64_t)s_start[r] + l1,
                      (uint64_t)s_start2[r] + ((uint32_t)l - l1 * c2), vals);
    } else {
      return tuple_of(r_lo + r, (uint64_t)s_start[r] + l, 0, vals);
    }
  };
  // every output takes the last mark at or before it: its row (the
  // load-balanced search of Algorithm 1's write loop, a max-scan over the
  // block's outputs instead of a binary search per output)
  if constexpr (table) {
    const uint32_t q0 = threadIdx.x * kJItems;
    uint16_t loc[kJItems];
    uint32_t m = 0;
#pragma unroll
    for (int q = 0; q < kJItems; ++q) {
      loc[q] = q0 + q < no ? s_row[q0 + q] : (uint16_t)0;
      m = loc[q] > m ? loc[q] : m;
    }
    uint32_t run = block_exclusive_max<kJT>(m, red);
#pragma unroll
    for (int q = 0; q < kJItems; ++q) {
      run = loc[q] > run ? loc[q] : run;
      if (q0 + q < no) s_row[q0 + q] = (uint16_t)run;
    }
    __syncthreads();
  }
  // output o of the block: its probe row from the table, or the last staged
  // row starting at or before it
  auto tuple_at = [&](uint64_t o, uint32_t (&vals)[kMaxK]) -> bool {
    uint32_t r;
    if constexpr (table) {
      r = s_row[o - o0];
    } else {
      uint32_t lo = 0, hi = nrows;
      while (hi - lo > 1) {
        const uint32_t mid = (lo + hi) >> 1;
        if (o0 + s_loc[mid] <= o)
          lo = mid;
        else
          hi = mid;
      }
      r = lo;
    }
    return tuple_in(r, o - off_of(r), vals);
  };
  if constexpr (DENSE) {
   if (nrows <= kDRows) {
    // a few probe rows with long ranges (the hot keys): the block walks
    // each row's outputs in turn, with no search for the row
    bool bad = false;
    for (uint32_t r = 0; r < nrows; ++r) {
      const uint64_t ra = off_of(r);
      const uint64_t a = ra > o0 ? ra : o0;
      const uint64_t e = r + 1 < nrows ? off_of(r + 1) : o1;
      const uint64_t b = e < o1 ? e : o1;
      for (uint64_t o = a + threadIdx.x; o < b; o += kJT) {
        uint32_t vals[kMaxK] = {0, 0, 0, 0};
        if (!tuple_in(r, o - ra, vals)) continue;
        uint32_t word, bit;
        if (!dense_locate(dset, vals, &word, &bit)) {
          bad = true;
          continue;
        }
        if (dense_missing(dset, word, bit)) atomicOr(dset.words + word, bit);
      }
    }
    if (bad && err) atomicOr(err, kErrCapacity);
   } else {
    // kDU outputs per thread at a time, each stage's loads all in flight:
    // the gathers, the words' reads, the atomics of missing bits
    bool bad = false;
    for (uint64_t ob = o0; ob < o1; ob += (uint64_t)kJT * kDU) {
      uint32_t word[kDU], bit[kDU];
      bool need[kDU];
#pragma unroll
      for (int u = 0; u < kDU; ++u) {
        const uint64_t o = ob + (uint64_t)u * kJT + threadIdx.x;
        uint32_t vals[kMaxK] = {0, 0, 0, 0};
        word[u] = bit[u] = 0;
        need[u] = o < o1 && tuple_at(o, vals);
        if (need[u] && !dense_locate(dset, vals, &word[u], &bit[u])) bad = true, need[u] = false;
      }
#pragma unroll
      for (int u = 0; u < kDU; ++u)
        if (need[u]) need[u] = dense_missing(dset, word[u], bit[u]);
#pragma unroll
      for (int u = 0; u < kDU; ++u)
        if (need[u]) atomicOr(dset.words + word[u], bit[u]);
    }
    if (bad && err) atomicOr(err, kErrCapacity);
   }
  }
  if constexpr (FORM == kSet) {
    // the block's outputs in one sweep, eight per thread side by side
    uint32_t row[kJItems], b1[kJItems], b2[kJItems], live = 0;
#pragma unroll
    for (int q = 0; q < kJItems; ++q) {
      const uint64_t o = o0 + (uint64_t)q * kJT + threadIdx.x;
      row[q] = b1[q] = b2[q] = 0;
      if (o < o1) {
        live |= 1u << q;
        const uint32_t r = s_row[o - o0], l = (uint32_t)(o - off_of(r));
        row[q] = r;
        if constexpr (STAR) {
          const uint32_t c2 = s_cnt2[r], l1 = l / c2;
          b1[q] = s_start[r] + l1;
          b2[q] = s_start2[r] + (l - l1 * c2);
        } else {
          b1[q] = s_start[r] + l;
        }
      }
    }
    uint64_t idx[kJItems];
    bool bad = false;
    set_tuples<FILTER, kJItems>(j, refs, live, r_lo, row, b1, b2, idx, bad);
    const uint32_t fresh = set_add<kJItems>(dset, idx);
    bad |= set_store<kJT, kJItems>(j, dset, refs, idx, fresh, cursor, out_cap, red);
    if (bad && err) atomicOr(err, kErrCapacity);
  }
  if constexpr (FORM == kRows)
  for (uint64_t ob = o0; ob < o1; ob += kJT) {
    const uint64_t o = ob + threadIdx.x;
    const bool valid = o < o1;
    uint32_t vals[kMaxK] = {0, 0, 0, 0};
    const bool keep = valid && tuple_at(o, vals);
    uint64_t pos;
    if (FILTER) {
      uint32_t cnt;
      const uint32_t local = block_exclusive_sum<kJT, uint32_t>(keep ? 1u : 0u, red, &cnt);
      if (threadIdx.x == 0) s_base = cnt ? atomicAdd(cursor, (unsigned long long)cnt) : 0ull;
      __syncthreads();
      pos = s_base + local;
      __syncthreads();
    } else {
      pos = wbase + o;
    }
    if (keep) {
      if (pos < out_cap) {
#pragma unroll
        for (int k = 0; k < kMaxK; ++k)
          if (k < (int)j.out_k) out.c[k][pos] = vals[k];
      } else {
        if (err) atomicOr(err, kErrCapacity);
      }
    }
  }
  }
  __syncthreads();  // the next tile restages the offsets and splits
  }
}

}  // namespace

cudaError_t join_count_only(Ctx& c, const JoinSpec& j, uint32_t* counts) {
  if (j.n_probe == 0) return cudaSuccess;
  ProfScope p(c, kJoinCount, (j.pk1 == 0xFFu ? 4.0 : 8.0) * j.n_probe + 20.0 * j.n_probe);
  k_join_count_only<<<(unsigned)((j.n_probe + kCT - 1) / kCT), kCT, 0, c.st>>>(j, counts);
  return cudaGetLastError();
}

size_t join_count_workspace(uint64_t n_probe) {
  const size_t counts = ((n_probe * sizeof(uint32_t)) + 255) & ~size_t(255);
  return counts + scan_workspace(n_probe);
}

cudaError_t join_count_scan(Ctx& c, const JoinSpec& j, uint64_t* d_off, uint64_t* d_total,
                            void* ws) {
  if (j.n_probe == 0) return cudaMemsetAsync(d_total, 0, sizeof(uint64_t), c.st);
  uint32_t* counts = static_cast<uint32_t*>(ws);
  void* scan_ws = static_cast<char*>(ws) + (((j.n_probe * sizeof(uint32_t)) + 255) & ~size_t(255));
  const uint64_t tiles = (j.n_probe + kScanTile - 1) / kScanTile;
  {
    // per row: its key, the slot probed, the count written (a star join's
    // second key and slot are read for rows its first range matches)
    double keyb = j.pk1 == 0xFFu ? 4.0 : 8.0;
    if (j.star) keyb += (j.qk1 == 0xFFu ? 4.0 : 8.0) + 16.0;
    ProfScope p(c, kJoinCount, (keyb + 16.0 + 4.0) * j.n_probe);
    k_join_count<<<dev_grid(tiles, j.dn), kCT, 0, c.st>>>(j, counts,
                                                           static_cast<uint64_t*>(scan_ws), c.d_err);
  }
  return scan_finish(c, counts, j.n_probe, d_off, d_total, scan_ws, j.dn);
}

// ------------------------------------------------------------- hub keys
// Numbers the build index's keys with at least hub_min rows and cuts each
// one's probe rows into tasks of kHubRows.
constexpr uint32_t kHubRows = 64;
struct HubTask {
  uint32_t hub, row, rows;
};

__global__ void __launch_bounds__(kCT) k_hub_list(const JoinSpec j, const KeyIndex pix, uint2* __restrict__ hubs,
                                                  uint64_t cap, HubTask* __restrict__ tasks,
                                                  uint64_t task_cap, unsigned long long* n) {
  const uint32_t range = direct_range(j.ix), prange = direct_range(pix);
  const uint64_t entries = range ? range : j.ix.slots;
  for (uint64_t i = (uint64_t)blockIdx.x * kCT + threadIdx.x; i < entries;
       i += (uint64_t)gridDim.x * kCT) {
    Slot s;
    if (range) {
      s.k0 = (uint32_t)i;
      s.k1 = 0;
      s.count = find_key(j.ix, range, s.k0, 0u, &s.start);
    } else {
      s = load_slot(j.ix.table, i);
      if (s.k0 == kEmpty && s.k1 == kEmpty) continue;
    }
    if (s.count < j.hub_min) continue;
    uint32_t prow;
    const uint32_t pn = find_key(pix, prange, s.k0, s.k1, &prow);
    if (pn == 0) continue;
    const uint64_t h = atomicAdd(n, 1ull);
    if (h >= cap) continue;  // (cannot happen: cap counts every such key)
    hubs[h] = make_uint2(s.start, s.count);
    const uint32_t nt = (pn + kHubRows - 1) / kHubRows;
    const uint64_t t0 = atomicAdd(n + 1, (unsigned long long)nt);
    for (uint32_t t = 0; t < nt && t0 + t < task_cap; ++t)
      tasks[t0 + t] = HubTask{(uint32_t)h, prow + t * kHubRows,
                              pn - t * kHubRows < kHubRows ? pn - t * kHubRows : kHubRows};
  }
}

// A hub's values as bits; gridDim.y blocks share a hub's rows.
__global__ void __launch_bounds__(kCT) k_hub_render(const uint2* __restrict__ hubs,
                                                    const unsigned long long* n_hubs, uint64_t cap,
                                                    const uint32_t* __restrict__ col,
                                                    uint32_t* __restrict__ bits, uint32_t words) {
  const uint64_t n = *n_hubs < cap ? *n_hubs : cap;
  for (uint64_t h = blockIdx.x; h < n; h += gridDim.x) {
    const uint2 u = hubs[h];
    for (uint32_t i = blockIdx.y * kCT + threadIdx.x; i < u.y; i += gridDim.y * kCT) {
      const uint32_t v = __ldg(col + u.x + i);
      if ((v >> 5) < words) atomicOr(bits + h * words + (v >> 5), 1u << (v & 31));
    }
  }
}

// One task per block: a thread holds four words of the hub's bitmap row and
// walks the task's head rows (kHubU of them in flight), reading the four
// words there and setting only what is missing.  A hub of d build rows costs
// a probe row 2^b / 128 coalesced 16-byte reads (b the bits of the last head
// column) instead of d scattered bit reads; bound by the latency of those
// reads (L2 hits 90 to 96 %, L2 9 to 14 % busy) and by the barriers between
// tasks, at four blocks per SM.  Points-to at scale 2^-7: the joins on hubs took 137 ms
// pair by pair, 6.8 ms here (the fixpoint 143 -> 15.4 ms); one word per
// output inside the write kernel took 92 ms (row searches per word).
constexpr int kHubU = 4;
template <bool APPEND>
__global__ void __launch_bounds__(kCT) k_hub_or(const JoinSpec j, const DenseSet d,
                                                const HubTask* __restrict__ tasks,
                                                uint64_t task_cap, const unsigned long long* n_tasks,
                                                const uint32_t* __restrict__ bits, uint32_t words,
                                                ColsOut out, unsigned long long* cursor,
                                                uint64_t out_cap, uint32_t* err) {
  __shared__ uint32_t s_word[kHubRows];  // first word of each head row
  const uint64_t n = *n_tasks < task_cap ? *n_tasks : task_cap;
  const uint32_t quads = words / 4, lane = lane_id();
  // threads side by side on a row's quads; with few quads, several rows at once
  const uint32_t across = quads < kCT ? quads : kCT;
  const uint32_t q0 = threadIdx.x % across, r0 = threadIdx.x / across, rstep = kCT / across;
  for (uint64_t t = blockIdx.x; t < n; t += gridDim.x) {
    const HubTask k = tasks[t];
    __syncthreads();  // the last task's rows are done
    if (threadIdx.x < k.rows) {
      uint32_t v[kMaxK] = {0, 0, 0, 0};
#pragma unroll
      for (int c = 0; c < kMaxK; ++c)
        if (c + 1 < (int)j.out_k)
          v[c] = ref_value(j, j.probe, j.out[c], (uint64_t)k.row + threadIdx.x, 0);
      const uint64_t idx = set_pack(d, v);  // (last column 0: the row's first bit)
      if (idx == kNoTuple) atomicOr(err, kErrCapacity);
      s_word[threadIdx.x] = idx == kNoTuple ? 0xFFFFFFFFu : (uint32_t)(idx >> 5);
    }
    __syncthreads();
    // the loops' bounds are the same for a warp's threads (rounded up), so
    // that the warp packs its new tuples together
    for (uint32_t qb = 0; qb < quads; qb += across) {
      const uint32_t q = qb + q0;
      uint4 h = make_uint4(0u, 0u, 0u, 0u);
      if (q < quads && r0 < rstep)
        h = __ldg(reinterpret_cast<const uint4*>(bits + (uint64_t)k.hub * words) + q);
      const bool any_h = (h.x | h.y | h.z | h.w) != 0u;
      if (!__any_sync(0xffffffffu, any_h)) continue;
      for (uint32_t rb = 0; rb < k.rows; rb += rstep * kHubU) {
        uint4 m[kHubU];
        uint32_t w[kHubU];
#pragma unroll
        for (int u = 0; u < kHubU; ++u) {
          const uint32_t r = rb + u * rstep + r0;
          m[u] = make_uint4(0u, 0u, 0u, 0u);
          w[u] = any_h && r < k.rows ? s_word[r] : 0xFFFFFFFFu;
          if (w[u] != 0xFFFFFFFFu) {
            w[u] += 4 * q;
            const uint4 cur = *reinterpret_cast<const uint4*>(d.words + w[u]);
            m[u] = make_uint4(h.x & ~cur.x, h.y & ~cur.y, h.z & ~cur.z, h.w & ~cur.w);
          }
        }
#pragma unroll
        for (int u = 0; u < kHubU; ++u) {
          if (m[u].x) m[u].x &= ~atomicOr(d.words + w[u], m[u].x);
          if (m[u].y) m[u].y &= ~atomicOr(d.words + w[u] + 1, m[u].y);
          if (m[u].z) m[u].z &= ~atomicOr(d.words + w[u] + 2, m[u].z);
          if (m[u].w) m[u].w &= ~atomicOr(d.words + w[u] + 3, m[u].w);
        }
        if constexpr (APPEND) {
          uint32_t c = 0;
#pragma unroll
          for (int u = 0; u < kHubU; ++u)
            c += __popc(m[u].x) + __popc(m[u].y) + __popc(m[u].z) + __popc(m[u].w);
          if (!__any_sync(0xffffffffu, c)) continue;
          uint32_t inc = c;
#pragma unroll
          for (int o = 1; o < 32; o <<= 1) {
            const uint32_t x = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= (uint32_t)o) inc += x;
          }
          unsigned long long at = 0;
          if (lane == 31) at = atomicAdd(cursor, (unsigned long long)inc);
          uint64_t pos = __shfl_sync(0xffffffffu, at, 31) + inc - c;
          auto emit = [&](uint32_t word, uint32_t x) {
            while (x) {
              const uint64_t idx = ((uint64_t)word << 5) | (uint64_t)(__ffs(x) - 1);
              x &= x - 1;
              if (pos < out_cap) {
#pragma unroll
                for (int c2 = 0; c2 < kMaxK; ++c2)
                  if (c2 < (int)d.k) out.c[c2][pos] = set_column(d, idx, c2);
              } else {
                atomicOr(err, kErrCapacity);  // (cannot happen: the caller gives room for all)
              }
              ++pos;
            }
          };
#pragma unroll
          for (int u = 0; u < kHubU; ++u) {
            emit(w[u], m[u].x);
            emit(w[u] + 1, m[u].y);
            emit(w[u] + 2, m[u].z);
            emit(w[u] + 3, m[u].w);
          }
        }
      }
    }
  }
}

static uint64_t hub_tasks_cap(const JoinSpec& j, const HubPlan& h) {
  return j.n_probe / kHubRows + h.cap;
}

size_t hub_workspace(const JoinSpec& j, const HubPlan& h) {
  auto up = [](uint64_t b) { return (b + 255) & ~uint64_t(255); };
  return 256 + up(8 * h.cap) + up(4ull * h.cap * h.words) + up(sizeof(HubTask) * hub_tasks_cap(j, h));
}

cudaError_t hub_or(Ctx& c, const JoinSpec& j, const HubPlan& h, const DenseSet& d, ColsOut out,
                   uint64_t* d_cursor, uint64_t out_cap, void* ws) {
  auto up = [](uint64_t b) { return (b + 255) & ~uint64_t(255); };
  char* p = static_cast<char*>(ws);
  auto* n = reinterpret_cast<unsigned long long*>(p);  // hubs, tasks
  p += 256;
  uint2* hubs = reinterpret_cast<uint2*>(p);
  p += up(8 * h.cap);
  uint32_t* bits = reinterpret_cast<uint32_t*>(p);
  p += up(4ull * h.cap * h.words);
  HubTask* tasks = reinterpret_cast<HubTask*>(p);
  const uint64_t task_cap = hub_tasks_cap(j, h);
  cudaError_t e = cudaMemsetAsync(n, 0, 256, c.st);
  if (e == cudaSuccess) e = cudaMemsetAsync(bits, 0, 4ull * h.cap * h.words, c.st);
  if (e != cudaSuccess) return e;
  {
    const uint64_t entries = j.ix.range ? j.ix.range : j.ix.slots;
    ProfScope ps(c, kDense, (j.ix.range ? 8.0 : 16.0) * entries);
    uint64_t blocks = (entries + kCT - 1) / kCT;
    if (blocks > 152 * 8) blocks = 152 * 8;
    k_hub_list<<<(unsigned)blocks, kCT, 0, c.st>>>(j, h.probe, hubs, h.cap, tasks,
                                                   task_cap, n);
  }
  {
    ProfScope ps(c, kDense, 4.0 * h.cap * h.words);
    k_hub_render<<<dim3((unsigned)(h.cap < 1024 ? h.cap : 1024), 4), kCT, 0, c.st>>>(
        hubs, n, h.cap, h.col, bits, h.words);
  }
  ProfScope ps(c, kJoinWrite, 0.0);  // (its reads are of L2-resident words)
  const unsigned grid = (unsigned)(task_cap < 152 * 8 ? task_cap : 152 * 8);
  auto* cur = reinterpret_cast<unsigned long long*>(d_cursor);
  if (d.append)
    k_hub_or<true><<<grid, kCT, 0, c.st>>>(j, d, tasks, task_cap, n + 1, bits, h.words, out, cur,
                                           out_cap, c.d_err);
  else
    k_hub_or<false><<<grid, kCT, 0, c.st>>>(j, d, tasks, task_cap, n + 1, bits, h.words, out, cur,
                                            out_cap, c.d_err);
  return cudaGetLastError();
}

// ------------------------------------------------------------ single pass
// The write without count and scan, for joins sized by the estimator: a
// block takes 256 probe rows at a time, scans their range lengths in shared
// memory, claims the rows' outputs with one atomic on the cursor and writes
// them together -- thread t writes outputs t, t + 256, ..., each finding its
// row by binary search over the block's offsets, as the exact write does.
// A row with more than kHeavyChunk outputs goes to the heavy list instead,
// so a hot key never holds one block.
constexpr int kDirT = 256;

// Writes the outputs [o_begin, o_end) of probe row prow (build rows from
// brow0) as one warp: unfiltered outputs go to pos0 + o, filtered ones are
// packed with a ballot and one cursor claim per 32.
template <bool FILTER>
__device__ __forceinline__ void warp_emit(const JoinSpec& j, ColsOut out, uint64_t prow,
                                          uint64_t brow0, uint64_t len, uint64_t pos0,
                                          unsigned long long* cursor, uint64_t cap,
                                          uint32_t* overflow) {
  const uint32_t lane = lane_id();
  const uint32_t lt = lanemask_lt();
  for (uint64_t ob = 0; ob < len; ob += 32) {
    const uint64_t o = ob + lane;
    const bool valid = o < len;
    uint32_t vals[kMaxK] = {0, 0, 0, 0};
    bool keep = valid;
    if (valid) {
#pragma unroll
      for (int k = 0; k < kMaxK; ++k)
        if (k < (int)j.out_k) vals[k] = ref_value(j, j.probe, j.out[k], prow, brow0 + o);
      if (FILTER) {
        for (uint32_t q = 0; q < j.n_eq; ++q)
          keep &= ref_value(j, j.probe, j.eq[q][0], prow, brow0 + o) ==
                  ref_value(j, j.probe, j.eq[q][1], prow, brow0 + o);
        for (uint32_t q = 0; q < j.n_neq; ++q)
          keep &= ref_value(j, j.probe, j.neq[q][0], prow, brow0 + o) !=
                  ref_value(j, j.probe, j.neq[q][1], prow, brow0 + o);
      }
    }
    uint64_t pos;
    if (FILTER) {
      const uint32_t bal = __ballot_sync(0xffffffffu, keep);
      uint64_t cb = 0;
      if (lane == 0 && bal) cb = atomicAdd(cursor, (unsigned long long)__popc(bal));
      cb = __shfl_sync(0xffffffffu, cb, 0);
      pos = cb + __popc(bal & lt);
      if (bal && cb + __popc(bal) > cap && lane == 0) atomicOr(overflow, 1u);
    } else {
      pos = pos0 + o;
    }
    if (keep && pos < cap) {
#pragma unroll
      for (int k = 0; k < kMaxK; ++k)
        if (k < (int)j.out_k) out.c[k][pos] = vals[k];
    }
  }
}

template <bool FILTER>
__global__ void __launch_bounds__(kDirT) k_join_direct(const JoinSpec j, ColsOut out,
                                                       unsigned long long* cursor, uint64_t cap,
                                                       unsigned long long* total,
                                                       uint32_t* overflow, HeavyList heavy) {
  __shared__ uint32_t s_off[kDirT];    // block-local exclusive offsets of the rows
  __shared__ uint32_t s_start[kDirT];  // first build row of each row's range
  __shared__ uint32_t red[kDirT / 32 + 1];
  __shared__ unsigned long long s_base;
  const uint32_t range = direct_range(j.ix);
  for (uint64_t b0 = (uint64_t)blockIdx.x * kDirT; b0 < j.n_probe;
       b0 += (uint64_t)gridDim.x * kDirT) {
    const uint64_t row = b0 + threadIdx.x;
    uint32_t st = 0, cnt = 0;
    if (row < j.n_probe) cnt = lookup(j, j.probe, range, row, &st);
    if (cnt > kHeavyChunk) {  // a long range becomes chunks of the heavy list
      atomicAdd(total, (unsigned long long)cnt);
      uint64_t out0 = 0;
      bool ok = true;
      if (!FILTER) {
        out0 = atomicAdd(cursor, (unsigned long long)cnt);
        ok = out0 + cnt <= cap;
      }
      const uint32_t nch = (cnt + kHeavyChunk - 1) / kHeavyChunk;
      const uint64_t at = ok ? atomicAdd((unsigned long long*)heavy.n, (unsigned long long)nch) : 0;
      ok &= at + nch <= heavy.cap;
      if (ok) {
        for (uint32_t q = 0; q < nch; ++q) {
          HeavyChunk h;
          h.prow = row;
          h.out0 = out0 + (uint64_t)q * kHeavyChunk;
          h.brow = st + q * kHeavyChunk;
          h.len = q + 1 < nch ? kHeavyChunk : cnt - q * kHeavyChunk;
          heavy.e[at + q] = h;
        }
      } else {
        atomicOr(overflow, 1u);
      }
      cnt = 0;
    }
    uint32_t tot;
    const uint32_t ex = block_exclusive_sum<kDirT, uint32_t>(cnt, red, &tot);
    s_off[threadIdx.x] = ex;
    s_start[threadIdx.x] = st;
    if (threadIdx.x == 0 && tot) {
      atomicAdd(total, (unsigned long long)tot);
      if (!FILTER) {
        s_base = atomicAdd(cursor, (unsigned long long)tot);
        if (s_base + tot > cap) atomicOr(overflow, 1u);
      }
    }
    __syncthreads();
    if (tot == 0) continue;  // uniform: nothing of this block reads s_off
    for (uint32_t ob = 0; ob < tot; ob += kDirT) {
      const uint32_t o = ob + threadIdx.x;
      const bool valid = o < tot;
      uint32_t vals[kMaxK] = {0, 0, 0, 0};
      bool keep = valid;
      if (valid) {
        uint32_t lo = 0, hi = kDirT;  // the last row whose range starts at or before o
        while (hi - lo > 1) {
          const uint32_t mid = (lo + hi) >> 1;
          if (s_off[mid] <= o)
            lo = mid;
          else
            hi = mid;
        }
        const uint64_t prow = b0 + lo;
        const uint64_t brow = (uint64_t)s_start[lo] + (o - s_off[lo]);
#pragma unroll
        for (int k = 0; k < kMaxK; ++k)
          if (k < (int)j.out_k) vals[k] = ref_value(j, j.probe, j.out[k], prow, brow);
        if (FILTER) {
          for (uint32_t q = 0; q < j.n_eq; ++q)
            keep &= ref_value(j, j.probe, j.eq[q][0], prow, brow) ==
                    ref_value(j, j.probe, j.eq[q][1], prow, brow);
          for (uint32_t q = 0; q < j.n_neq; ++q)
            keep &= ref_value(j, j.probe, j.neq[q][0], prow, brow) !=
                    ref_value(j, j.probe, j.neq[q][1], prow, brow);
        }
      }
      uint64_t pos;
      if (FILTER) {  // survivors packed with one claim per 256 outputs
        uint32_t n_keep;
        const uint32_t local = block_exclusive_sum<kDirT, uint32_t>(keep ? 1u : 0u, red, &n_keep);
        if (threadIdx.x == 0) {
          s_base = n_keep ? atomicAdd(cursor, (unsigned long long)n_keep) : 0ull;
          if (n_keep && s_base + n_keep > cap) atomicOr(overflow, 1u);
        }
        __syncthreads();
        pos = s_base + local;
        __syncthreads();
      } else {
        pos = s_base + o;
      }
      if (keep && pos < cap) {
#pragma unroll
        for (int k = 0; k < kMaxK; ++k)
          if (k < (int)j.out_k) out.c[k][pos] = vals[k];
      }
    }
    __syncthreads();  // s_off, s_start and s_base are rewritten by the next rows
  }
}

// The heavy list: one warp per chunk, grid-stride over the chunks the
// direct kernel listed (their number is read from device memory).
template <bool FILTER>
__global__ void __launch_bounds__(kDirT) k_join_heavy(const JoinSpec j, ColsOut out,
                                                      unsigned long long* cursor, uint64_t cap,
                                                      uint32_t* overflow, HeavyList heavy) {
  const uint64_t nwarps = ((uint64_t)gridDim.x * kDirT) >> 5;
  uint64_t n = *heavy.n;
  if (n > heavy.cap) n = heavy.cap;
  for (uint64_t w = ((uint64_t)blockIdx.x * kDirT + threadIdx.x) >> 5; w < n; w += nwarps) {
    const HeavyChunk h = heavy.e[w];
    warp_emit<FILTER>(j, out, h.prow, h.brow, h.len, h.out0, cursor, cap, overflow);
  }
}

cudaError_t join_direct(Ctx& c, const JoinSpec& j, ColsOut out, uint64_t* d_cursor,
                        uint64_t out_cap, uint64_t* d_total, uint32_t* d_overflow,
                        const HeavyList& heavy) {
  if (j.star) return cudaErrorInvalidValue;  // star joins keep the count pass
  if (j.n_probe == 0) return cudaSuccess;
  uint64_t blocks = (j.n_probe + kDirT - 1) / kDirT;
  if (blocks > 152 * 8) blocks = 152 * 8;
  const bool filter = j.n_neq > 0 || j.n_eq > 0;
  ProfScope p(c, kJoinDirect, (4.0 + 16.0 + 4.0 * j.out_k) * j.n_probe);
  auto* cur = reinterpret_cast<unsigned long long*>(d_cursor);
  auto* tot = reinterpret_cast<unsigned long long*>(d_total);
  if (filter) {
    k_join_direct<true><<<(unsigned)blocks, kDirT, 0, c.st>>>(j, out, cur, out_cap, tot, d_overflow,
                                                              heavy);
    k_join_heavy<true><<<152 * 8, kDirT, 0, c.st>>>(j, out, cur, out_cap, d_overflow, heavy);
  } else {
    k_join_direct<false><<<(unsigned)blocks, kDirT, 0, c.st>>>(j, out, cur, out_cap, tot,
                                                               d_overflow, heavy);
    k_join_heavy<false><<<152 * 8, kDirT, 0, c.st>>>(j, out, cur, out_cap, d_overflow, heavy);
  }
  return cudaGetLastError();
}

// ------------------------------------------------ single pass into a set
// Where Full is a bitmap a join needs no place computed for its outputs: the
// new ones are packed as they come.  So no count and no scan run; a block
// takes a tile of probe rows (four per thread; fewer where that leaves
// blocks idle), looks them up, scans their output counts in shared memory
// and walks the outputs in windows of four per thread as k_join_write does.
// Rows with more than kHeavyChunk outputs are listed and taken in chunks by
// a second kernel, so that one hot key does not hold one block.
// Bound by the latency of its random reads, of entries and of the set (one
// launch of 53M rows into a 2 GB bitmap: DRAM 8 %, L2 18 % busy; of 0.3M rows
// into a hash set: DRAM 41 %, L2 23 %, 25 of 39 cycles an instruction waiting
// for them).  Same generation on 200,000 nodes: 25 ms of counts and scans and
// 66 of writes became 52 ms, all joins' writes together; a round of a small
// closure takes one launch and one wait (4,001 nodes, 46 rounds: 4.9 ->
// 2.3 ms).  Four rows and outputs a thread in 48 registers and five blocks per
// SM: 57.1 ms for the run on 200,000 nodes (six blocks, 40 registers, 57.4;
// eight rows in four blocks 62.7, in five blocks, spilling, 77.8).
constexpr int kSJT = 256, kSJI = 4, kSJH = 8;
static_assert(kSJT == kCT, "set_lookup's rows lie kCT apart");
constexpr uint32_t kSJTile = kSJT * kSJI;

// Both forms of the set; a full table is noted in *total.
template <bool HASH, int N>
__device__ __forceinline__ uint32_t set_add_any(const DenseSet& d, const uint64_t (&idx)[N],
                                                unsigned long long* total) {
  if constexpr (!HASH) return set_add<N>(d, idx);
  bool full = false;
  const uint32_t fresh = set_add_hash<N>(d, idx, &full);
  if (full) atomicOr(total, (unsigned long long)kSetListFull);
  return fresh;
}

template <bool FILTER, bool STAR, bool HASH>
__global__ void __launch_bounds__(kSJT, 5) k_join_set(const JoinSpec j, const DenseSet d, ColsOut out,
                                                      unsigned long long* cursor, uint64_t cap,
                                                      unsigned long long* total, uint32_t* err,
                                                      uint32_t per, HeavyList heavy) {
  // row q of thread t is slot kSJI t + q; slots lie in the order of their outputs
  __shared__ uint32_t s_off[kSJTile], s_start[kSJTile];
  __shared__ uint32_t s_start2[STAR ? kSJTile : 1], s_cnt2[STAR ? kSJTile : 1];
  __shared__ uint16_t s_slot[kSJTile];
  __shared__ __align__(8) uint32_t red[kSJT / 32 + 2];
  __shared__ SetRefs refs;
  stage_refs(j, d, out, refs);
  const uint64_t n = dev_size(j.dn, j.n_probe);
  const ColsIn* probe = j.dprobe ? j.dprobe : &j.probe;
  const uint32_t* pk0 = j.cross ? nullptr : probe->c[j.pk0];
  const uint32_t* pk1 = j.cross || j.pk1 == 0xFFu ? nullptr : probe->c[j.pk1];
  const uint32_t *qk0 = nullptr, *qk1 = nullptr;
  if constexpr (STAR) {
    qk0 = probe->c[j.qk0];
    qk1 = j.qk1 == 0xFFu ? nullptr : probe->c[j.qk1];
  }
  const uint32_t range = direct_range(j.ix), range2 = STAR ? direct_range(j.ix2) : 0u;
  const uint32_t t = threadIdx.x;
  const uint32_t rows = kSJT * per;
  for (uint64_t base = (uint64_t)blockIdx.x * rows; base < n; base += (uint64_t)gridDim.x * rows) {
    uint32_t cnt[kSJI], st[kSJI];
    uint32_t live = 0;
#pragma unroll
    for (int q = 0; q < kSJI; ++q)
      live |= (q < (int)per && base + (uint64_t)q * kSJT + t < n ? 1u : 0u) << q;
    if (j.cross) {
#pragma unroll
      for (int q = 0; q < kSJI; ++q) {
        st[q] = 0;
        cnt[q] = (live >> q) & 1u ? j.n_build : 0u;
      }
    } else {
      set_lookup<kSJI>(j, j.ix, range, pk0, pk1, base, live, st, cnt);
    }
    uint32_t st2[kSJI], cnt2[kSJI];
    if constexpr (STAR) {
      uint32_t found = 0;
#pragma unroll
      for (int q = 0; q < kSJI; ++q) found |= (cnt[q] ? 1u : 0u) << q;
      set_lookup<kSJI>(j, j.ix2, range2, qk0, qk1, base, found, st2, cnt2);
    }
    uint32_t sum = 0;
#pragma unroll
    for (int q = 0; q < kSJI; ++q) {
      const uint64_t row = base + (uint64_t)q * kSJT + t;
      uint64_t c = cnt[q];
      if constexpr (STAR) {
        s_start2[t * kSJI + q] = st2[q];
        s_cnt2[t * kSJI + q] = cnt2[q];
        c *= cnt2[q];
        if (c > 0xFFFFFFFFull) {
          if (err) atomicOr(err, kErrCapacity);
          c = 0;
        }
      }
      s_start[t * kSJI + q] = st[q];
      if (c > kHeavyChunk) {
        atomicAdd(total, (unsigned long long)c);
        const uint32_t nch = (uint32_t)((c + kHeavyChunk - 1) / kHeavyChunk);
        const uint64_t at = atomicAdd((unsigned long long*)heavy.n, (unsigned long long)nch);
        for (uint32_t i = 0; i < nch && at + i < heavy.cap; ++i) {
          HeavyChunk h;
          h.prow = row;
          h.out0 = (uint64_t)i * kHeavyChunk;  // first output of the row
          h.brow = 0;
          h.len = i + 1 < nch ? kHeavyChunk : (uint32_t)(c - (uint64_t)i * kHeavyChunk);
          heavy.e[at + i] = h;
        }
        if (at + nch > heavy.cap) atomicOr(total, (unsigned long long)kSetListFull);
        c = 0;
      }
      s_off[t * kSJI + q] = sum;
      sum += (uint32_t)c;
    }
    uint32_t tot;
    const uint32_t ex = block_exclusive_sum<kSJT, uint32_t>(sum, red, &tot);
#pragma unroll
    for (int q = 0; q < kSJI; ++q) s_off[t * kSJI + q] += ex;
    if (t == 0 && tot) atomicAdd(total, (unsigned long long)tot);
    __syncthreads();
    for (uint32_t w = 0; w < tot; w += kSJTile) {
      // every output takes the last slot that starts at or before it among
      // those with outputs: marks at their first outputs, then a max-scan
#pragma unroll
      for (int q = 0; q < kSJI; ++q) s_slot[q * kSJT + t] = 0;
      __syncthreads();
#pragma unroll
      for (int q = 0; q < kSJI; ++q) {
        const uint32_t sl = t * kSJI + q, a = s_off[sl];
        const uint32_t b = sl + 1 < kSJTile ? s_off[sl + 1] : tot;
        const uint32_t first = a > w ? a : w;
        if (b > first && first - w < kSJTile) s_slot[first - w] = (uint16_t)sl;
      }
      __syncthreads();
      uint32_t m = 0, loc[kSJI];
#pragma unroll
      for (int q = 0; q < kSJI; ++q) {
        loc[q] = s_slot[t * kSJI + q];
        m = loc[q] > m ? loc[q] : m;
      }
      uint32_t run = block_exclusive_max<kSJT>(m, red);
#pragma unroll
      for (int q = 0; q < kSJI; ++q) {
        run = loc[q] > run ? loc[q] : run;
        s_slot[t * kSJI + q] = (uint16_t)run;
      }
      __syncthreads();
      uint64_t idx[kSJI];
      uint32_t row[kSJI], b1[kSJI], b2[kSJI], have = 0;
      bool bad = false;
#pragma unroll
      for (int q = 0; q < kSJI; ++q) {
        const uint32_t o = w + q * kSJT + t;
        row[q] = b1[q] = b2[q] = 0;
        if (o < tot) {
          have |= 1u << q;
          const uint32_t sl = s_slot[q * kSJT + t], l = o - s_off[sl];
          row[q] = sl % kSJI * kSJT + sl / kSJI;
          if constexpr (STAR) {
            const uint32_t c2 = s_cnt2[sl], l1 = l / c2;
            b1[q] = s_start[sl] + l1;
            b2[q] = s_start2[sl] + (l - l1 * c2);
          } else {
            b1[q] = s_start[sl] + l;
          }
        }
      }
      set_tuples<FILTER, kSJI>(j, refs, have, base, row, b1, b2, idx, bad);
      if (bad && err) atomicOr(err, kErrCapacity);
      const uint32_t fresh = set_add_any<HASH, kSJI>(d, idx, total);
      set_store<kSJT, kSJI>(j, d, refs, idx, fresh, cursor, cap, red);
      __syncthreads();  // the next window rewrites s_slot and red
    }
    __syncthreads();  // the next tile rewrites the slots
  }
}

// The listed chunks, one block at a time (their number from device memory).
template <bool FILTER, bool STAR, bool HASH>
__global__ void __launch_bounds__(kSJT, 4) k_join_set_heavy(const JoinSpec j, const DenseSet d,
                                                            ColsOut out, unsigned long long* cursor,
                                                            uint64_t cap,
                                                            unsigned long long* total,
                                                            uint32_t* err, HeavyList heavy) {
  static_assert(kHeavyChunk <= kSJT * kSJH, "a chunk is one window");
  __shared__ __align__(8) uint32_t red[kSJT / 32 + 2];
  __shared__ SetRefs refs;
  stage_refs(j, d, out, refs);
  const ColsIn probe = probe_cols(j);
  const uint32_t range = direct_range(j.ix);
  const uint64_t n = *heavy.n < heavy.cap ? *heavy.n : heavy.cap;
  for (uint64_t b = blockIdx.x; b < n; b += gridDim.x) {
    const HeavyChunk h = heavy.e[b];
    uint32_t st = 0, st2 = 0, c2 = 1;
    lookup(j, probe, range, h.prow, &st);
    if constexpr (STAR) c2 = lookup2(j, probe, h.prow, &st2);
    uint64_t idx[kSJH];
    uint32_t row[kSJH], b1[kSJH], b2[kSJH], have = 0;
    bool bad = false;
#pragma unroll
    for (int q = 0; q < kSJH; ++q) {
      const uint32_t o = q * kSJT + threadIdx.x;
      row[q] = b1[q] = b2[q] = 0;
      if (o < h.len && c2) {
        have |= 1u << q;
        const uint32_t l = (uint32_t)h.out0 + o, l1 = STAR ? l / c2 : l;
        b1[q] = st + l1;
        b2[q] = st2 + (l - l1 * c2);
      }
    }
    set_tuples<FILTER, kSJH>(j, refs, have, h.prow, row, b1, b2, idx, bad);
    if (bad && err) atomicOr(err, kErrCapacity);
    const uint32_t fresh = set_add_any<HASH, kSJH>(d, idx, total);
    set_store<kSJT, kSJH>(j, d, refs, idx, fresh, cursor, cap, red);
    __syncthreads();  // the next chunk reuses red
  }
}

cudaError_t join_set(Ctx& c, const JoinSpec& j, const DenseSet& d, ColsOut out, uint64_t* d_cursor,
                     uint64_t out_cap, uint64_t* d_total, const HeavyList& heavy, bool run_chunks) {
  if (j.n_probe == 0) return cudaSuccess;
  const bool filter = j.n_neq > 0 || j.n_eq > 0;
  // rows per thread: all once five blocks per SM are busy, else fewer
  uint64_t per = j.n_probe / ((uint64_t)kSJT * 152 * 5);
  per = per < 1 ? 1 : per > (uint64_t)kSJI ? (uint64_t)kSJI : per;
  const unsigned grid = dev_grid((j.n_probe + kSJT * per - 1) / (kSJT * per), j.dn);
  ProfScope p(c, kJoinWrite, ((j.star ? 48.0 : 24.0) + 4.0 * j.out_k) * j.n_probe);
  auto* cur = reinterpret_cast<unsigned long long*>(d_cursor);
  auto* tot = reinterpret_cast<unsigned long long*>(d_total);
  auto launch = [&](auto rows, auto chunks) {
    rows<<<grid, kSJT, 0, c.st>>>(j, d, out, cur, out_cap, tot, c.d_err, (uint32_t)per, heavy);
    if (run_chunks) chunks<<<152, kSJT, 0, c.st>>>(j, d, out, cur, out_cap, tot, c.d_err, heavy);
  };
#define CDL_JOIN_SET(F, S)                                                             \
  d.keys ? launch(k_join_set<F, S, true>, k_join_set_heavy<F, S, true>)                \
         : launch(k_join_set<F, S, false>, k_join_set_heavy<F, S, false>)
  if (j.star)
    if (filter)
      CDL_JOIN_SET(true, true);
    else
      CDL_JOIN_SET(false, true);
  else if (filter)
    CDL_JOIN_SET(true, false);
  else
    CDL_JOIN_SET(false, false);
#undef CDL_JOIN_SET
  return cudaGetLastError();
}

cudaError_t join_begin(Ctx& c, uint64_t* head, const JoinMark& m) {
  k_join_begin<<<1, 1, 0, c.st>>>(head, m);
  return cudaGetLastError();
}

size_t join_write_workspace(uint64_t n_probe, uint64_t total) {
  const uint64_t blocks = (n_probe + total + kJTile - 1) / kJTile;
  return ((blocks + 1) * 8 + 255) & ~uint64_t(255);
}

cudaError_t join_write(Ctx& c, const JoinSpec& j, const uint64_t* d_off, uint64_t total,
                       ColsOut out, uint64_t base, uint64_t* d_cursor, uint64_t out_cap,
                       void* ws, size_t ws_bytes, const uint64_t* d_total, uint64_t* d_base,
                       uint32_t* d_soft_err, const DenseSet* dense) {
  if (total == 0 || j.n_probe == 0) return cudaSuccess;
  const uint64_t nm = j.n_probe + total;
  const uint64_t blocks = (nm + kJTile - 1) / kJTile;
  const bool filter = j.n_neq > 0 || j.n_eq > 0;
  uint64_t* splits = nullptr;
  if (ws && ws_bytes >= join_write_workspace(j.n_probe, total)) {
    splits = static_cast<uint64_t*>(ws);
    k_write_splits<<<(unsigned)((blocks + 1 + 255) / 256), 256, 0, c.st>>>(
        d_off, j.n_probe, total, splits, blocks, j.dn, d_total,
        reinterpret_cast<unsigned long long*>(d_cursor), d_base, out_cap,
        d_soft_err ? d_soft_err : c.d_err, j.head, j.mark);
  } else if (j.head) {
    k_join_open<<<1, 1, 0, c.st>>>(j.head, j.mark, total);
  }
  // per probe row: two offsets, key, re-probed slot (a star join: both
  // keys and slots), its own head columns; per output: the gathered build
  // columns and the written head columns
  uint32_t nbuild = 0, nprobe = 0;
  for (uint32_t k = 0; k < j.out_k; ++k) {
    nbuild += j.out[k].side == 1 || j.out[k].side == 3;
    nprobe += j.out[k].side == 0;
  }
  const double row_b = j.star ? 16.0 + 8.0 + 32.0 : 16.0 + 4.0 + 16.0;
  // (a dense head's bits are set in L2-resident words, not written out)
  const double bytes = (row_b + 4.0 * nprobe) * j.n_probe +
                       (4.0 * nbuild + (dense ? 0.0 : 4.0 * j.out_k)) * total;
  ProfScope p(c, kJoinWrite, bytes);
  auto* cur = reinterpret_cast<unsigned long long*>(d_cursor);
  uint32_t* err = d_soft_err ? d_soft_err : c.d_err;
  const DenseSet ds = dense ? *dense : DenseSet{};
  const unsigned grid = dev_grid(blocks, d_total);
  auto launch = [&](auto kernel) {
    kernel<<<grid, kJT, 0, c.st>>>(j, d_off, total, out, base, cur, out_cap, splits, err, d_total,
                                   d_base, ds);
  };
#define CDL_JOIN_WRITE(FORM)                                                                 \
  if (j.star)                                                                                \
    filter ? launch(k_join_write<true, FORM, true>) : launch(k_join_write<false, FORM, true>); \
  else                                                                                       \
    filter ? launch(k_join_write<true, FORM, false>) : launch(k_join_write<false, FORM, false>)
  if (!dense) {
    CDL_JOIN_WRITE(kRows);
  } else if (!dense->append) {
    CDL_JOIN_WRITE(kBits);
  } else {
    CDL_JOIN_WRITE(kSet);
  }
#undef CDL_JOIN_WRITE
  return cudaGetLastError();
}

}  // namespace cdl
