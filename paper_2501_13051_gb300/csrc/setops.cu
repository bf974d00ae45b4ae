// Selection / projection of one body atom (Section 4, "Projection and
// Selection"): rows are filtered on constants, repeated variables and
// inequalities, then projected onto head columns and packed with one atomic
// per block; plus the check of loaded values against the reserved value.
#include "kernels.h"

namespace cdl {

namespace {

// ------------------------------------------------------------- select
constexpr int kST = 256;
constexpr int kSItems = 8;

// Eight rows per thread: their filters, then one claim of the output for the
// block, then the columns one after the other, eight loads in flight.  (With
// a scan and a claim for every 256 rows, one after another, the 270 copies of
// an OWL-RL fixpoint took 10.4 us each; the fixpoint 37.2 -> 35.4 ms.)
__global__ void __launch_bounds__(kST) k_select(const SelectSpec s, ColsOut out,
                                                unsigned long long* cursor, uint64_t cap,
                                                uint32_t* err) {
  __shared__ __align__(8) uint32_t red[kST / 32 + 2];
  const uint64_t base = (uint64_t)blockIdx.x * kST * kSItems + threadIdx.x;
  uint32_t live = 0;
#pragma unroll
  for (int i = 0; i < kSItems; ++i) live |= (base + (uint64_t)i * kST < s.n ? 1u : 0u) << i;
  auto load = [&](const Ref& r, uint32_t (&v)[kSItems]) {
    const uint32_t* p = r.side == 2 ? nullptr : s.in.c[r.v] + base;
#pragma unroll
    for (int i = 0; i < kSItems; ++i) {
      v[i] = r.v;
      if (p && ((live >> i) & 1u)) v[i] = __ldg(p + (uint64_t)i * kST);
    }
  };
  auto filter = [&](const Ref& x, const Ref& y, bool equal) {
    uint32_t a[kSItems], b[kSItems];
    load(x, a);
    load(y, b);
#pragma unroll
    for (int i = 0; i < kSItems; ++i)
      if ((a[i] == b[i]) != equal) live &= ~(1u << i);
  };
#pragma unroll 1
  for (uint32_t q = 0; q < s.n_const; ++q) filter(Ref{0, s.const_col[q]}, Ref{2, s.const_val[q]}, true);
#pragma unroll 1
  for (uint32_t q = 0; q < s.n_same; ++q) filter(Ref{0, s.same[q][0]}, Ref{0, s.same[q][1]}, true);
#pragma unroll 1
  for (uint32_t q = 0; q < s.n_neq; ++q) filter(s.neq[q][0], s.neq[q][1], false);
  uint32_t at[kSItems];
  uint64_t pos;
  if (!claim_places<kST, kSItems>(live, cursor, red, at, &pos)) return;
  const uint64_t room = cap > pos ? cap - pos : 0;
  bool over = false;
#pragma unroll
  for (int i = 0; i < kSItems; ++i)
    if (((live >> i) & 1u) && at[i] >= room) {
      over = true;
      live &= ~(1u << i);
    }
  if (over && err) atomicOr(err, kErrCapacity);
#pragma unroll 1
  for (uint32_t k = 0; k < s.out_k; ++k) {
    uint32_t v[kSItems];
    load(s.out[k], v);
    uint32_t* o = out.c[k] + pos;
#pragma unroll
    for (int i = 0; i < kSItems; ++i)
      if ((live >> i) & 1u) o[at[i]] = v[i];
  }
}

__global__ void k_check_values(ColsIn in, uint32_t k, uint64_t n, uint32_t* d_max,
                               uint32_t* err) {
  for (uint32_t c = 0; c < k; ++c) {
    uint32_t m = 0;
    bool bad = false;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (uint64_t)gridDim.x * blockDim.x) {
      const uint32_t v = __ldg(in.c[c] + i);
      bad |= v == kEmpty;
      m = max(m, v);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (bad && err) atomicOr(err, kErrValue);
    if (lane_id() == 0) atomicMax(d_max + c, m);
  }
}

// The same for the columns of many loads at once: blockIdx.y is the column.
__global__ void __launch_bounds__(256) k_check_columns(const CheckJob* __restrict__ jobs,
                                                       uint32_t* err) {
  const CheckJob j = jobs[blockIdx.y];
  const uint64_t step = (uint64_t)gridDim.x * 256;
  uint32_t m = 0;
  bool bad = false;
  for (uint64_t i = (uint64_t)blockIdx.x * 256 + threadIdx.x; i < j.n; i += 4 * step) {
    uint32_t v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) v[u] = i + u * step < j.n ? __ldg(j.col + i + u * step) : 0u;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      bad |= v[u] == kEmpty;
      m = max(m, v[u]);
    }
  }
  m = __reduce_max_sync(0xffffffffu, m);
  if (bad && err) atomicOr(err, kErrValue);
  if (lane_id() == 0 && m) atomicMax(j.max, m);
}

// Batched fixpoints: every row of a delta whose column 0 is an instance id
// marks its instance as one that derived something in this round; a row whose
// neighbour before it has the same instance leaves the store to that one.
// The rows may be in any order (a delta of sorted rows stores once per
// instance, one that came from a hash set about once per row).
__global__ void k_mark_instances(const uint32_t* __restrict__ inst, uint64_t n,
                                 uint32_t n_instances, uint64_t* __restrict__ last_round,
                                 uint64_t round, const ColsIn* dinst, const uint64_t* dn,
                                 const uint64_t* dround) {
  if (dinst) {  // inside a captured round: the delta and the round from device memory
    inst = dinst->c[0];
    n = dev_size(dn, n);
    round += *dround;
  }
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (uint64_t)gridDim.x * blockDim.x) {
    const uint32_t v = __ldg(inst + i);
    if ((i == 0 || __ldg(inst + i - 1) != v) && v < n_instances) last_round[v] = round;
  }
}

// bounds[i] = the first row whose instance id (column 0, sorted: Full's rows,
// not a delta from a hash set) is >= i, for i in [0, n_instances].
__global__ void k_instance_bounds(const uint32_t* __restrict__ inst, uint64_t n,
                                  uint32_t n_instances, uint64_t* __restrict__ bounds) {
  const uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i > n_instances) return;
  uint64_t lo = 0, hi = n;
  while (lo < hi) {
    const uint64_t mid = (lo + hi) >> 1;
    if ((uint64_t)__ldg(inst + mid) < i)
      lo = mid + 1;
    else
      hi = mid;
  }
  bounds[i] = lo;
}

// Output row j of segment s (out_off[s] <= j < out_off[s + 1]) copies row
// src[s] + (j - out_off[s]) of table a, or of table b when bit 63 of src[s]
// is set.  Consecutive rows of a segment are consecutive source rows, so
// reads and writes stay coalesced.
constexpr int kGT = 256;
constexpr int kGItems = 8;
constexpr uint32_t kGSmem = 2048;  // segment offsets held in shared memory

template <bool SMEM>
__global__ void __launch_bounds__(kGT) k_gather_segments(ColsIn a, ColsIn b, uint32_t k,
                                                         const uint64_t* __restrict__ out_off,
                                                         const uint64_t* __restrict__ src,
                                                         uint32_t nseg, uint64_t total,
                                                         ColsOut out) {
  __shared__ uint64_t s_off[SMEM ? kGSmem + 1 : 1];
  if (SMEM) {
    for (uint32_t i = threadIdx.x; i <= nseg; i += kGT) s_off[i] = out_off[i];
    __syncthreads();
  }
  const uint64_t base = (uint64_t)blockIdx.x * kGT * kGItems;
  for (int it = 0; it < kGItems; ++it) {
    const uint64_t j = base + (uint64_t)it * kGT + threadIdx.x;
    if (j >= total) break;
    uint32_t lo = 0, hi = nseg;  // the last segment whose start is <= j
    while (hi - lo > 1) {
      const uint32_t mid = (lo + hi) >> 1;
      const uint64_t o = SMEM ? s_off[mid] : __ldg(out_off + mid);
      if (o <= j)
        lo = mid;
      else
        hi = mid;
    }
    const uint64_t start = SMEM ? s_off[lo] : __ldg(out_off + lo);
    const uint64_t sv = __ldg(src + lo);
    const uint64_t row = (sv & ~(1ull << 63)) + (j - start);
    const bool from_b = (sv >> 63) != 0;
#pragma unroll
    for (int c = 0; c < kMaxK; ++c)  // constant indices: the column sets stay in registers
      if (c < (int)k) out.c[c][j] = __ldg((from_b ? b.c[c] : a.c[c]) + row);
  }
}

}  // namespace

// col[j] = s for every row j of segment s (rows [off[s], off[s + 1])).
__global__ void k_fill_segments(uint32_t* __restrict__ col, const uint64_t* __restrict__ off,
                                uint32_t nseg, uint64_t total) {
  for (uint64_t j = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; j < total;
       j += (uint64_t)gridDim.x * blockDim.x) {
    uint32_t lo = 0, hi = nseg;  // the last segment starting at or before j
    while (hi - lo > 1) {
      const uint32_t mid = (lo + hi) >> 1;
      if (__ldg(off + mid) <= j)
        lo = mid;
      else
        hi = mid;
    }
    col[j] = lo;
  }
}

cudaError_t fill_segments(Ctx& c, uint32_t* col, const uint64_t* off, uint32_t nseg,
                          uint64_t total) {
  if (total == 0 || nseg == 0) return cudaSuccess;
  ProfScope p(c, kMisc, 4.0 * total);
  uint64_t blocks = (total + 255) / 256;
  if (blocks > 152 * 16) blocks = 152 * 16;
  k_fill_segments<<<(unsigned)blocks, 256, 0, c.st>>>(col, off, nseg, total);
  return cudaGetLastError();
}

// Row j of segment s (rows [off[s], off[s + 1])): out.c[0][j] = s and
// out.c[1 + c][j] = column c of src[s] at row j - off[s].
__global__ void k_concat_segments(ColsOut out, const ColsIn* __restrict__ src, uint32_t k,
                                  const uint64_t* __restrict__ off, uint32_t nseg,
                                  uint64_t total) {
  for (uint64_t j = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; j < total;
       j += (uint64_t)gridDim.x * blockDim.x) {
    uint32_t lo = 0, hi = nseg;  // the last segment starting at or before j
    while (hi - lo > 1) {
      const uint32_t mid = (lo + hi) >> 1;
      if (__ldg(off + mid) <= j)
        lo = mid;
      else
        hi = mid;
    }
    const uint64_t r = j - __ldg(off + lo);
    out.c[0][j] = lo;
#pragma unroll
    for (uint32_t c = 0; c + 1 < (uint32_t)kMaxK; ++c)
      if (c < k) out.c[c + 1][j] = __ldg(src[lo].c[c] + r);
  }
}

// The reverse: row j of segment s goes to row j - off[s] of dst[s].
__global__ void k_split_segments(ColsIn in, const ColsOut* __restrict__ dst, uint32_t k,
                                 const uint64_t* __restrict__ off, uint32_t nseg, uint64_t total) {
  for (uint64_t j = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; j < total;
       j += (uint64_t)gridDim.x * blockDim.x) {
    uint32_t lo = 0, hi = nseg;  // the last segment starting at or before j
    while (hi - lo > 1) {
      const uint32_t mid = (lo + hi) >> 1;
      if (__ldg(off + mid) <= j)
        lo = mid;
      else
        hi = mid;
    }
    const uint64_t r = j - __ldg(off + lo);
#pragma unroll
    for (uint32_t c = 0; c < (uint32_t)kMaxK; ++c)
      if (c < k) dst[lo].c[c][r] = __ldg(in.c[c] + j);
  }
}

cudaError_t split_segments(Ctx& c, ColsIn in, const ColsOut* dst, uint32_t k, const uint64_t* off,
                           uint32_t nseg, uint64_t total) {
  if (total == 0 || nseg == 0) return cudaSuccess;
  ProfScope p(c, kMisc, 8.0 * k * total);
  uint64_t blocks = (total + 255) / 256;
  if (blocks > 152 * 16) blocks = 152 * 16;
  k_split_segments<<<(unsigned)blocks, 256, 0, c.st>>>(in, dst, k, off, nseg, total);
  return cudaGetLastError();
}

cudaError_t concat_segments(Ctx& c, ColsOut out, const ColsIn* src, uint32_t k,
                            const uint64_t* off, uint32_t nseg, uint64_t total) {
  if (total == 0 || nseg == 0) return cudaSuccess;
  ProfScope p(c, kMisc, (8.0 * k + 4.0) * total);
  uint64_t blocks = (total + 255) / 256;
  if (blocks > 152 * 16) blocks = 152 * 16;
  k_concat_segments<<<(unsigned)blocks, 256, 0, c.st>>>(out, src, k, off, nseg, total);
  return cudaGetLastError();
}

cudaError_t instance_bounds(Ctx& c, const uint32_t* inst, uint64_t n, uint32_t n_instances,
                            uint64_t* bounds) {
  ProfScope p(c, kRetire, 8.0 * (n_instances + 1));
  k_instance_bounds<<<(n_instances + 256) / 256, 256, 0, c.st>>>(inst, n, n_instances, bounds);
  return cudaGetLastError();
}

cudaError_t gather_segments(Ctx& c, uint32_t k, ColsIn a, ColsIn b, const uint64_t* out_off,
                            const uint64_t* src, uint32_t nseg, uint64_t total, ColsOut out) {
  if (total == 0 || nseg == 0) return cudaSuccess;
  ProfScope p(c, kRetire, 8.0 * k * total);
  const uint64_t blocks = (total + kGT * kGItems - 1) / (kGT * kGItems);
  if (nseg <= kGSmem)
    k_gather_segments<true><<<(unsigned)blocks, kGT, 0, c.st>>>(a, b, k, out_off, src, nseg, total,
                                                                 out);
  else
    k_gather_segments<false><<<(unsigned)blocks, kGT, 0, c.st>>>(a, b, k, out_off, src, nseg,
                                                                  total, out);
  return cudaGetLastError();
}

cudaError_t mark_instances(Ctx& c, const uint32_t* inst, uint64_t n, uint32_t n_instances,
                           uint64_t* last_round, uint64_t round, const ColsIn* dinst,
                           const uint64_t* dn, const uint64_t* dround) {
  if (n == 0) return cudaSuccess;
  ProfScope p(c, kMisc, 4.0 * n);
  k_mark_instances<<<dev_grid((n + 255) / 256, dinst), 256, 0, c.st>>>(
      inst, n, n_instances, last_round, round, dinst, dn, dround);
  return cudaGetLastError();
}

cudaError_t select_project(Ctx& c, const SelectSpec& s, ColsOut out, uint64_t* d_cursor,
                           uint64_t out_cap, uint32_t* soft_overflow) {
  if (s.n == 0) return cudaSuccess;
  const uint64_t blocks = (s.n + kST * kSItems - 1) / (kST * kSItems);
  ProfScope p(c, kSelect, 4.0 * s.in_k * s.n + 4.0 * s.out_k * s.n);
  k_select<<<(unsigned)blocks, kST, 0, c.st>>>(s, out,
                                               reinterpret_cast<unsigned long long*>(d_cursor),
                                               out_cap,
                                               soft_overflow ? soft_overflow : c.d_err);
  return cudaGetLastError();
}

cudaError_t check_columns(Ctx& c, const CheckJob* jobs, uint32_t njobs, uint64_t most,
                          uint64_t total) {
  if (njobs == 0 || most == 0) return cudaSuccess;
  ProfScope p(c, kMisc, 4.0 * total);
  uint64_t blocks = (most + 4095) / 4096;
  if (blocks > 64) blocks = 64;
  constexpr uint32_t kMost = 65535;  // of a grid's second dimension
  for (uint32_t at = 0; at < njobs; at += kMost)
    k_check_columns<<<dim3((unsigned)blocks, njobs - at < kMost ? njobs - at : kMost), 256, 0, c.st>>>(
        jobs + at, c.d_err);
  return cudaGetLastError();
}

cudaError_t check_values(Ctx& c, ColsIn in, uint32_t k, uint64_t n, uint32_t* d_max) {
  cudaError_t e = cudaMemsetAsync(d_max, 0, sizeof(uint32_t) * k, c.st);
  if (e != cudaSuccess || n == 0) return e;
  ProfScope p(c, kMisc, 4.0 * k * n);
  uint64_t blocks = (n + 2047) / 2048;
  if (blocks > 152 * 8) blocks = 152 * 8;
  k_check_values<<<(unsigned)blocks, 256, 0, c.st>>>(in, k, n, d_max, c.d_err);
  return cudaGetLastError();
}

}  // namespace cdl
