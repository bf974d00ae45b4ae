// Dense relations as bitmaps, a second form of step (c) of the round
// (Section 4, "Projection and Selection" and the sort + unique that
// follows).  Where a relation's tuples fit in 2^T bits, new tuples set bits
// instead of being written, sorted and deduplicated.  Extraction reads the
// bits back in increasing order: the same sorted unique list the radix sort
// and the unique pass produce, at the cost of one pass over the bitmap.
#include "kernels.h"

namespace cdl {

namespace {

constexpr int kXT = 256;                              // threads per extraction block
constexpr int kXWords = 8;                            // bitmap words per thread
constexpr uint64_t kXTile = (uint64_t)kXT * kXWords;  // words per block

size_t up256(size_t b) { return (b + 255) & ~size_t(255); }

__host__ __device__ __forceinline__ uint64_t words_of(uint64_t nbits) {
  return nbits >= 32 ? nbits >> 5 : 1;
}

__global__ void __launch_bounds__(256) k_dense_insert(DenseSet d, ColsIn rows, uint64_t n,
                                                      uint32_t* err) {
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t b = (uint64_t)blockIdx.x * blockDim.x; b < n; b += stride) {
    const uint64_t i = b + threadIdx.x;
    const bool keep = i < n;
    uint32_t v[kMaxK] = {0, 0, 0, 0};
    if (keep) {
#pragma unroll
      for (int k = 0; k < kMaxK; ++k)
        if (k < (int)d.k) v[k] = __ldg(rows.c[k] + i);
    }
    dense_set_bits(d, v, keep, err);
  }
}

__global__ void __launch_bounds__(256) k_dense_remove(DenseSet d, ColsIn rows, uint64_t n) {
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
    uint32_t v[kMaxK] = {0, 0, 0, 0};
#pragma unroll
    for (int k = 0; k < kMaxK; ++k)
      if (k < (int)d.k) v[k] = __ldg(rows.c[k] + i);
    const uint64_t idx = set_pack(d, v);
    if (idx != kNoTuple) set_remove(d, idx);
  }
}

// Rows appended to Full's bitmap: the new ones (their bit was clear) go out
// packed at *cursor.
// (HASH: Full's hash form; EMIT false: the rows only join the set.)
constexpr int kAT = 256, kAItems = 4;
template <bool HASH, bool EMIT>
__global__ void __launch_bounds__(kAT) k_set_insert(DenseSet d, ColsIn rows, uint64_t n,
                                                    ColsOut out, unsigned long long* cursor,
                                                    uint64_t cap, uint32_t* err) {
  __shared__ __align__(8) uint32_t red[kAT / 32 + 2];
  constexpr uint64_t kTile = (uint64_t)kAT * kAItems;
  for (uint64_t b = blockIdx.x * kTile; b < n; b += gridDim.x * kTile) {
    uint64_t idx[kAItems];
    bool bad = false;
#pragma unroll
    for (int q = 0; q < kAItems; ++q) {
      const uint64_t i = b + (uint64_t)q * kAT + threadIdx.x;
      uint32_t v[kMaxK] = {0, 0, 0, 0};
      idx[q] = kNoTuple;
      if (i < n) {
#pragma unroll
        for (int k = 0; k < kMaxK; ++k)
          if (k < (int)d.k) v[k] = __ldg(rows.c[k] + i);
        idx[q] = set_pack(d, v);
        bad |= idx[q] == kNoTuple;
      }
    }
    uint32_t fresh;
    if constexpr (HASH)
      fresh = set_add_hash<kAItems>(d, idx, &bad);
    else
      fresh = set_add<kAItems>(d, idx);
    if constexpr (EMIT) {
      bad |= !set_emit<kAT, kAItems>(d, idx, fresh, out, cursor, cap, red);
      __syncthreads();  // the next tile reuses red
    }
    if (bad && err) atomicOr(err, kErrCapacity);
  }
}

// The keys of another table into d (a larger table takes over).
__global__ void __launch_bounds__(kAT) k_hash_move(DenseSet d, const unsigned long long* old,
                                                   uint64_t slots, uint32_t* err) {
  constexpr uint64_t kTile = (uint64_t)kAT * kAItems;
  for (uint64_t b = blockIdx.x * kTile; b < slots; b += gridDim.x * kTile) {
    uint64_t idx[kAItems];
#pragma unroll
    for (int q = 0; q < kAItems; ++q) {
      const uint64_t i = b + (uint64_t)q * kAT + threadIdx.x;
      const unsigned long long v = i < slots ? old[i] : kSetEmpty;
      idx[q] = v < kSetGone ? v : kNoTuple;
    }
    bool full = false;
    set_add_hash<kAItems>(d, idx, &full);
    if (full && err) atomicOr(err, kErrTable);
  }
}

// The table's keys, packed in no order, as their high and low words.
__global__ void __launch_bounds__(kAT) k_hash_keys(DenseSet d, uint32_t* __restrict__ hi,
                                                   uint32_t* __restrict__ lo, uint64_t cap,
                                                   unsigned long long* cursor, uint32_t* err) {
  constexpr int kI = 8;
  __shared__ uint32_t red[kAT / 32 + 1];
  __shared__ unsigned long long s_at;
  const uint64_t slots = d.kmask + 1;
  for (uint64_t b = blockIdx.x * (uint64_t)kAT * kI; b < slots; b += gridDim.x * (uint64_t)kAT * kI) {
    unsigned long long v[kI];
    uint32_t n = 0;
#pragma unroll
    for (int q = 0; q < kI; ++q) {
      const uint64_t i = b + (uint64_t)q * kAT + threadIdx.x;
      v[q] = i < slots ? d.keys[i] : kSetEmpty;
      n += v[q] < kSetGone ? 1u : 0u;
    }
    uint32_t tot;
    const uint32_t ex = block_exclusive_sum<kAT, uint32_t>(n, red, &tot);
    if (threadIdx.x == 0) s_at = tot ? atomicAdd(cursor, (unsigned long long)tot) : 0ull;
    __syncthreads();
    uint64_t at = s_at + ex;
#pragma unroll
    for (int q = 0; q < kI; ++q)
      if (v[q] < kSetGone) {
        if (at < cap) {
          hi[at] = (uint32_t)(v[q] >> 32);
          lo[at] = (uint32_t)v[q];
        } else if (err) {
          atomicOr(err, kErrCapacity);
        }
        ++at;
      }
    __syncthreads();  // the next tile rewrites s_at
  }
}

// Keys as high and low words to 8-byte words, and back.
__global__ void __launch_bounds__(256) k_hash_zip(const uint32_t* __restrict__ hi,
                                                  const uint32_t* __restrict__ lo, uint64_t n,
                                                  uint64_t* __restrict__ out) {
  for (uint64_t i = (uint64_t)blockIdx.x * 256 + threadIdx.x; i < n; i += (uint64_t)gridDim.x * 256)
    out[i] = (uint64_t)hi[i] << 32 | lo[i];
}
__global__ void __launch_bounds__(256) k_hash_unzip(const uint64_t* __restrict__ in, uint64_t n,
                                                    uint32_t* __restrict__ hi,
                                                    uint32_t* __restrict__ lo) {
  for (uint64_t i = (uint64_t)blockIdx.x * 256 + threadIdx.x; i < n; i += (uint64_t)gridDim.x * 256) {
    hi[i] = (uint32_t)(in[i] >> 32);
    lo[i] = (uint32_t)in[i];
  }
}

__global__ void __launch_bounds__(256) k_hash_unpack(DenseSet d, const uint32_t* __restrict__ hi,
                                                     const uint32_t* __restrict__ lo, uint64_t n,
                                                     ColsOut out) {
  for (uint64_t i = (uint64_t)blockIdx.x * 256 + threadIdx.x; i < n; i += (uint64_t)gridDim.x * 256) {
    const uint64_t idx = ((uint64_t)__ldg(hi + i) << 32) | __ldg(lo + i);
#pragma unroll
    for (int k = 0; k < kMaxK; ++k)
      if (k < (int)d.k) out.c[k][i] = set_column(d, idx, k);
  }
}

// The words a thread owns: [w0, w0 + kXWords) clipped to nw.
__device__ __forceinline__ void load_words(const uint32_t* words, uint64_t w0, uint64_t nw,
                                           uint32_t (&w)[kXWords]) {
  if (w0 + kXWords <= nw) {  // 32-byte aligned: w0 is a multiple of 8
    const uint4 a = *reinterpret_cast<const uint4*>(words + w0);
    const uint4 b = *reinterpret_cast<const uint4*>(words + w0 + 4);
    w[0] = a.x, w[1] = a.y, w[2] = a.z, w[3] = a.w;
    w[4] = b.x, w[5] = b.y, w[6] = b.z, w[7] = b.w;
  } else {
#pragma unroll
    for (int i = 0; i < kXWords; ++i) w[i] = w0 + i < nw ? words[w0 + i] : 0u;
  }
}

__global__ void __launch_bounds__(kXT) k_dense_count(const uint32_t* __restrict__ words,
                                                     uint64_t nw, uint32_t* __restrict__ counts) {
  __shared__ uint32_t red[kXT / 32 + 1];
  const uint64_t w0 = (uint64_t)blockIdx.x * kXTile + (uint64_t)threadIdx.x * kXWords;
  uint32_t w[kXWords];
  load_words(words, w0, nw, w);
  uint32_t c = 0;
#pragma unroll
  for (int i = 0; i < kXWords; ++i) c += __popc(w[i]);
  uint32_t total;
  block_exclusive_sum<kXT, uint32_t>(c, red, &total);
  if (threadIdx.x == 0) counts[blockIdx.x] = total;
}

// Rows of the set bits at their ranks, in bit order; a round's bitmap is
// cleared behind the read so that it starts the next round empty.  The set
// bits' positions in the block's words (16 bits each) are staged in shared
// memory, kXStage at a time, so that a column's rows leave as contiguous
// stores whatever the density.
constexpr uint32_t kXStage = 4096;
__global__ void __launch_bounds__(kXT) k_dense_write(DenseSet d, uint64_t nw,
                                                     const uint64_t* __restrict__ offs,
                                                     ColsOut out, uint64_t cap, uint32_t* err) {
  static_assert(kXTile * 32 <= 65536, "a staged position has 16 bits");
  __shared__ uint32_t red[kXT / 32 + 1];
  __shared__ uint16_t stage[kXStage];
  const uint64_t w0 = (uint64_t)blockIdx.x * kXTile + (uint64_t)threadIdx.x * kXWords;
  uint32_t w[kXWords];
  load_words(d.words, w0, nw, w);
  uint32_t c = 0;
#pragma unroll
  for (int i = 0; i < kXWords; ++i) c += __popc(w[i]);
  uint32_t total;
  uint32_t pos = block_exclusive_sum<kXT, uint32_t>(c, red, &total);
  if (!d.append) {
#pragma unroll
    for (int i = 0; i < kXWords; ++i)
      if (w[i]) d.words[w0 + i] = 0u;
  }
  const uint64_t first = offs[blockIdx.x];
  const uint64_t bit0 = (uint64_t)blockIdx.x * kXTile * 32;
  for (uint32_t s0 = 0; s0 < total; s0 += kXStage) {
    if (pos < s0 + kXStage) {  // the thread's next positions, up to the stage's end
#pragma unroll
      for (int i = 0; i < kXWords; ++i) {
        while (w[i] && pos < s0 + kXStage) {
          stage[pos - s0] = (uint16_t)(((threadIdx.x * kXWords + i) << 5) | (__ffs(w[i]) - 1));
          w[i] &= w[i] - 1;
          ++pos;
        }
      }
    }
    __syncthreads();
    const uint32_t m = total - s0 < kXStage ? total - s0 : kXStage;
    for (uint32_t i = threadIdx.x; i < m; i += kXT) {
      const uint64_t idx = bit0 + stage[i];
      const uint64_t at = first + s0 + i;
      if (at < cap) {
#pragma unroll
        for (int k = 0; k < kMaxK; ++k)
          if (k < (int)d.k) out.c[k][at] = set_column(d, idx, k);
      } else {
        atomicOr(err, kErrCapacity);
      }
    }
    __syncthreads();
  }
}

}  // namespace

cudaError_t dense_insert(Ctx& c, const DenseSet& d, ColsIn rows, uint64_t n) {
  if (n == 0) return cudaSuccess;
  ProfScope p(c, kDense, 4.0 * d.k * n);
  if (d.keys) {
    uint64_t tiles = (n + kAT * kAItems - 1) / (kAT * kAItems);
    if (tiles > 152 * 16) tiles = 152 * 16;
    k_set_insert<true, false><<<(unsigned)tiles, kAT, 0, c.st>>>(d, rows, n, ColsOut{}, nullptr, 0,
                                                                 c.d_err);
    return cudaGetLastError();
  }
  uint64_t blocks = (n + 255) / 256;
  if (blocks > 152 * 16) blocks = 152 * 16;
  k_dense_insert<<<(unsigned)blocks, 256, 0, c.st>>>(d, rows, n, c.d_err);
  return cudaGetLastError();
}

cudaError_t dense_remove(Ctx& c, const DenseSet& d, ColsIn rows, uint64_t n) {
  if (n == 0) return cudaSuccess;
  ProfScope p(c, kDense, 4.0 * d.k * n);
  uint64_t blocks = (n + 255) / 256;
  if (blocks > 152 * 16) blocks = 152 * 16;
  k_dense_remove<<<(unsigned)blocks, 256, 0, c.st>>>(d, rows, n);
  return cudaGetLastError();
}

cudaError_t set_insert(Ctx& c, const DenseSet& d, ColsIn rows, uint64_t n, ColsOut out,
                       uint64_t* d_cursor, uint64_t out_cap) {
  if (n == 0) return cudaSuccess;
  ProfScope p(c, kDense, 4.0 * d.k * n);
  uint64_t blocks = (n + kAT * kAItems - 1) / (kAT * kAItems);
  if (blocks > 152 * 16) blocks = 152 * 16;
  auto* cur = reinterpret_cast<unsigned long long*>(d_cursor);
  if (d.keys)
    k_set_insert<true, true><<<(unsigned)blocks, kAT, 0, c.st>>>(d, rows, n, out, cur, out_cap, c.d_err);
  else
    k_set_insert<false, true><<<(unsigned)blocks, kAT, 0, c.st>>>(d, rows, n, out, cur, out_cap, c.d_err);
  return cudaGetLastError();
}

cudaError_t hash_move(Ctx& c, const DenseSet& d, const unsigned long long* old, uint64_t slots) {
  ProfScope p(c, kDense, 8.0 * slots);
  uint64_t blocks = (slots + kAT * kAItems - 1) / (kAT * kAItems);
  if (blocks > 152 * 16) blocks = 152 * 16;
  k_hash_move<<<(unsigned)blocks, kAT, 0, c.st>>>(d, old, slots, c.d_err);
  return cudaGetLastError();
}

cudaError_t hash_keys(Ctx& c, const DenseSet& d, uint32_t* hi, uint32_t* lo, uint64_t cap,
                      uint64_t* d_count) {
  ProfScope p(c, kDense, 8.0 * (d.kmask + 1));
  cudaError_t e = cudaMemsetAsync(d_count, 0, 8, c.st);
  if (e != cudaSuccess) return e;
  uint64_t blocks = (d.kmask + 1 + 2047) / 2048;
  if (blocks > 152 * 16) blocks = 152 * 16;
  k_hash_keys<<<(unsigned)blocks, kAT, 0, c.st>>>(
      d, hi, lo, cap, reinterpret_cast<unsigned long long*>(d_count), c.d_err);
  return cudaGetLastError();
}

static unsigned zip_grid(uint64_t n) {
  const uint64_t blocks = (n + 1023) / 1024;
  return (unsigned)(blocks < 152 * 64 ? blocks : 152 * 64);
}

cudaError_t hash_zip(Ctx& c, const uint32_t* hi, const uint32_t* lo, uint64_t n, uint64_t* out) {
  if (n == 0) return cudaSuccess;
  ProfScope p(c, kDense, 16.0 * n);
  k_hash_zip<<<zip_grid(n), 256, 0, c.st>>>(hi, lo, n, out);
  return cudaGetLastError();
}

cudaError_t hash_unzip(Ctx& c, const uint64_t* in, uint64_t n, uint32_t* hi, uint32_t* lo) {
  if (n == 0) return cudaSuccess;
  ProfScope p(c, kDense, 16.0 * n);
  k_hash_unzip<<<zip_grid(n), 256, 0, c.st>>>(in, n, hi, lo);
  return cudaGetLastError();
}

cudaError_t hash_unpack(Ctx& c, const DenseSet& d, const uint32_t* hi, const uint32_t* lo,
                        uint64_t n, ColsOut out) {
  if (n == 0) return cudaSuccess;
  ProfScope p(c, kDense, (8.0 + 4.0 * d.k) * n);
  uint64_t blocks = (n + 1023) / 1024;
  if (blocks > 152 * 64) blocks = 152 * 64;
  k_hash_unpack<<<(unsigned)blocks, 256, 0, c.st>>>(d, hi, lo, n, out);
  return cudaGetLastError();
}

size_t dense_extract_workspace(uint64_t nbits) {
  const uint64_t tiles = (words_of(nbits) + kXTile - 1) / kXTile;
  return up256(tiles * 4) + up256(tiles * 8) + scan_workspace(tiles);
}

cudaError_t dense_extract(Ctx& c, const DenseSet& d, ColsOut out, uint64_t cap,
                          uint64_t* d_count, void* ws) {
  const uint64_t nw = words_of(d.nbits);
  const uint64_t tiles = (nw + kXTile - 1) / kXTile;
  char* w = static_cast<char*>(ws);
  uint32_t* counts = reinterpret_cast<uint32_t*>(w);
  w += up256(tiles * 4);
  uint64_t* offs = reinterpret_cast<uint64_t*>(w);
  w += up256(tiles * 8);
  {
    ProfScope p(c, kDense, 4.0 * nw);
    k_dense_count<<<(unsigned)tiles, kXT, 0, c.st>>>(d.words, nw, counts);
  }
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) e = exclusive_scan(c, counts, tiles, offs, d_count, w);
  if (e != cudaSuccess) return e;
  // the bitmap read again and its set words cleared; the rows are added
  // to the class's bytes once their number is known
  ProfScope p(c, kDense, 4.0 * nw);
  k_dense_write<<<(unsigned)tiles, kXT, 0, c.st>>>(d, nw, offs, out, cap, c.d_err);
  return cudaGetLastError();
}

}  // namespace cdl
