// C ABI of the single steps (include/cdl.h, "Steps of one round"): the
// engine's own kernels on caller-owned device buffers, scratch carved from a
// caller-provided workspace.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>
#include <vector>

#include "../../include/cdl.h"
#include "kernels.h"

using namespace cdl;

namespace {

size_t up(size_t b) { return (b + 255) & ~size_t(255); }

// Carves consecutive 256-byte aligned pieces out of a workspace.
struct Carve {
  char* p;
  size_t used = 0;
  explicit Carve(void* base) : p(static_cast<char*>(base)) {}
  void* take(size_t b) {
    void* r = p ? p + used : nullptr;
    used += up(b);
    return r;
  }
};

constexpr size_t kHead = 256;  // error word, cursor, totals

// cdl_sort_unique: bits of tuple space per row up to which the rows go
// through a bitmap.
constexpr uint64_t kBitmapPerRow = 64;

bool pow2(uint64_t x) { return x && !(x & (x - 1)); }

cdl_status cuda_status(cudaError_t e) { return e == cudaSuccess ? CDL_OK : CDL_E_CUDA; }

cdl_status read_flags(uint64_t* head, cudaStream_t st, uint64_t* host, int n) {
  if (cudaMemcpyAsync(host, head, sizeof(uint64_t) * n, cudaMemcpyDeviceToHost, st) != cudaSuccess)
    return CDL_E_CUDA;
  if (cudaStreamSynchronize(st) != cudaSuccess) return CDL_E_CUDA;
  const uint32_t f = (uint32_t)host[0];
  if (f & kErrState) return CDL_E_INVALID;
  if (f & kErrTimeout) return CDL_E_TIMEOUT;
  if (f & kErrCapacity) return CDL_E_CAPACITY;
  if (f & kErrTable) return CDL_E_CAPACITY;
  if (f & kErrValue) return CDL_E_VALUE;
  return CDL_OK;
}

uint32_t bits_of(uint32_t v) {
  uint32_t b = 0;
  while (v) {
    ++b;
    v >>= 1;
  }
  return b;
}

}  // namespace

extern "C" {

uint64_t cdl_hash_table_bytes(uint64_t n_keys, double load) {
  return table_slots(n_keys, load) * sizeof(Slot);
}

cdl_status cdl_hash_build(const uint32_t* keys, uint64_t n, void* table, uint64_t table_bytes,
                          void* stream) {
  if ((!keys && n) || !table) return CDL_E_INVALID;
  const uint64_t slots = table_bytes / sizeof(Slot);
  if (!pow2(slots) || slots <= n) return CDL_E_INVALID;
  if (n > 0xFFFFFFFFull) return CDL_E_CAPACITY;
  Ctx c;
  c.st = static_cast<cudaStream_t>(stream);
  return cuda_status(hash_build(c, keys, nullptr, n, static_cast<Slot*>(table), slots));
}

cdl_status cdl_join_count(const uint32_t* probe, uint64_t n, const void* table,
                          uint64_t table_bytes, uint32_t* counts, void* stream) {
  if ((!probe || !counts) && n) return CDL_E_INVALID;
  const uint64_t slots = table_bytes / sizeof(Slot);
  if (!table || !pow2(slots)) return CDL_E_INVALID;
  Ctx c;
  c.st = static_cast<cudaStream_t>(stream);
  JoinSpec j{};
  j.probe.c[0] = probe;
  j.n_probe = n;
  j.pk0 = 0;
  j.pk1 = 0xFFu;
  j.ix.table = static_cast<const Slot*>(table);
  j.ix.slots = slots;
  return cuda_status(join_count_only(c, j, counts));
}

cdl_status cdl_exclusive_scan(const uint32_t* in, uint64_t n, uint64_t* out, uint64_t* total_host,
                              void* workspace, size_t* ws_bytes, void* stream) {
  if (!ws_bytes) return CDL_E_INVALID;
  const size_t need = kHead + up(scan_workspace(n));
  if (!workspace) {
    *ws_bytes = need;
    return CDL_OK;
  }
  if (*ws_bytes < need || ((!in || !out) && n)) return CDL_E_INVALID;
  Carve cv(workspace);
  uint64_t* head = static_cast<uint64_t*>(cv.take(kHead));
  void* sws = cv.take(scan_workspace(n));
  Ctx c;
  c.st = static_cast<cudaStream_t>(stream);
  cudaError_t e = cudaMemsetAsync(head, 0, kHead, c.st);
  if (e == cudaSuccess) e = exclusive_scan(c, in, n, out, head + 1, sws);
  if (e != cudaSuccess) return CDL_E_CUDA;
  if (total_host) {
    uint64_t h[2];
    cdl_status s = read_flags(head, c.st, h, 2);
    if (s != CDL_OK) return s;
    *total_host = h[1];
  }
  return CDL_OK;
}

// cdl_join and cdl_join_write: checked arguments and the workspace's parts.
struct JoinCall {
  JoinSpec j{};
  uint64_t* head;  // error word, total, output cursor; gate and mark (join_begin)
  JoinMark mark;
  Slot* table;
  uint64_t* off;
  void* cws;
};

static cdl_status join_setup(const uint32_t* const* probe_cols, uint32_t probe_arity,
                             uint64_t n_probe, uint32_t probe_key,
                             const uint32_t* const* build_cols, uint32_t build_arity,
                             uint64_t n_build, uint32_t build_key, const cdl_colref* spec,
                             uint32_t out_arity, const cdl_colref* neq, uint32_t nneq,
                             void* workspace, size_t ws_bytes, size_t need, JoinCall& jc) {
  if (probe_arity < 1 || probe_arity > CDL_MAX_ARITY || build_arity < 1 ||
      build_arity > CDL_MAX_ARITY || out_arity < 1 || out_arity > CDL_MAX_ARITY ||
      probe_key >= probe_arity || build_key >= build_arity || nneq > 4 || !spec)
    return CDL_E_INVALID;
  if (n_build > 0xFFFFFFFFull) return CDL_E_CAPACITY;
  JoinSpec& j = jc.j;
  for (uint32_t k = 0; k < probe_arity; ++k) j.probe.c[k] = probe_cols[k];
  for (uint32_t k = 0; k < build_arity; ++k) j.build.c[k] = build_cols[k];
  j.n_probe = n_probe;
  j.pk0 = probe_key;
  j.pk1 = 0xFFu;
  auto conv = [&](const cdl_colref& r, Ref& out) {
    if (r.side > 2) return false;
    if (r.side == 0 && r.v >= probe_arity) return false;
    if (r.side == 1 && r.v >= build_arity) return false;
    out = Ref{(uint8_t)r.side, r.v};
    return true;
  };
  j.out_k = out_arity;
  for (uint32_t k = 0; k < out_arity; ++k)
    if (!conv(spec[k], j.out[k])) return CDL_E_INVALID;
  j.n_neq = nneq;
  for (uint32_t q = 0; q < nneq; ++q)
    if (!conv(neq[2 * q], j.neq[q][0]) || !conv(neq[2 * q + 1], j.neq[q][1])) return CDL_E_INVALID;
  const uint64_t slots = table_slots(n_build, 0.5);
  Carve cv(workspace);
  jc.head = static_cast<uint64_t*>(cv.take(kHead));
  jc.table = static_cast<Slot*>(cv.take(slots * sizeof(Slot)));
  jc.off = static_cast<uint64_t*>(cv.take(8 * (n_probe ? n_probe : 1)));
  jc.cws = cv.take(join_count_workspace(n_probe));
  // (a workspace of the size without the rows' starts does as well: the write
  // then looks the keys up again)
  if (ws_bytes >= need) j.starts = static_cast<uint32_t*>(cv.take(4 * (n_probe ? n_probe : 1)));
  // the direct form where the largest key fits the table's memory (4 to 8
  // keys per row: it is then cleared, filled and read for less than the hash
  // form)
  j.ix.table = jc.table;
  j.ix.slots = slots;
  if (n_build) {
    j.ix.range = (uint32_t)std::min<uint64_t>(2 * slots, 0xFFFFFFFFull);
    j.ix.last = build_cols[build_key] + n_build - 1;
    // (from 2^22 rows the entries by key may outgrow L2: offsets instead)
    if (n_build >= 1ull << 22) j.ix.rows = (uint32_t)n_build;
  }
  // what the offsets and the kept starts depend on
  jc.mark = JoinMark{n_probe, n_build, (uint64_t)probe_key | (uint64_t)build_key << 8 |
                                           (uint64_t)(j.starts != nullptr) << 16};
  return CDL_OK;
}

static cdl_status join_output(const JoinCall& jc, uint32_t* const* out_cols, uint32_t out_arity,
                              uint64_t out_cap, uint64_t total, uint64_t* n_out, Ctx& c) {
  ColsOut out;
  for (uint32_t k = 0; k < CDL_MAX_ARITY; ++k) out.c[k] = k < out_arity ? out_cols[k] : nullptr;
  // the count workspace is free again: it holds the write splits if large enough
  cudaError_t e = join_write(c, jc.j, jc.off, total, out, 0, jc.head + 2, out_cap, jc.cws,
                             join_count_workspace(jc.j.n_probe));
  if (e != cudaSuccess) return CDL_E_CUDA;
  uint64_t h[3];
  cdl_status s = read_flags(jc.head, c.st, h, 3);
  if (s != CDL_OK) return s;
  *n_out = h[2];
  return CDL_OK;
}

static size_t join_need(uint64_t n_probe, uint64_t n_build, bool starts) {
  return kHead + up(table_slots(n_build, 0.5) * sizeof(Slot)) + up(8 * (n_probe ? n_probe : 1)) +
         up(join_count_workspace(n_probe)) + (starts ? up(4 * (n_probe ? n_probe : 1)) : 0);
}

cdl_status cdl_join(const uint32_t* const* probe_cols, uint32_t probe_arity, uint64_t n_probe,
                    uint32_t probe_key, const uint32_t* const* build_cols, uint32_t build_arity,
                    uint64_t n_build, uint32_t build_key, const cdl_colref* spec,
                    uint32_t out_arity, const cdl_colref* neq, uint32_t nneq,
                    uint32_t* const* out_cols, uint64_t out_cap, uint64_t* n_out, void* workspace,
                    size_t* ws_bytes, void* stream) {
  if (!ws_bytes) return CDL_E_INVALID;
  const size_t need = join_need(n_probe, n_build, true);
  if (!workspace) {
    *ws_bytes = need;
    return CDL_OK;
  }
  if (*ws_bytes < join_need(n_probe, n_build, false) || !n_out) return CDL_E_INVALID;
  JoinCall jc;
  cdl_status s = join_setup(probe_cols, probe_arity, n_probe, probe_key, build_cols, build_arity,
                            n_build, build_key, spec, out_arity, neq, nneq, workspace, *ws_bytes,
                            need, jc);
  if (s != CDL_OK) return s;
  Ctx c;
  c.st = static_cast<cudaStream_t>(stream);
  c.d_err = reinterpret_cast<uint32_t*>(jc.head);
  cudaError_t e = join_begin(c, jc.head, jc.mark);
  if (e == cudaSuccess) e = index_build(c, build_cols[build_key], n_build, jc.j.ix);
  if (e == cudaSuccess) e = join_count_scan(c, jc.j, jc.off, jc.head + 1, jc.cws);
  if (e != cudaSuccess) return CDL_E_CUDA;
  uint64_t h[2];
  s = read_flags(jc.head, c.st, h, 2);
  if (s != CDL_OK) return s;
  const uint64_t total = h[1];
  *n_out = total;
  if (total == 0) return CDL_OK;
  if (out_cap < total) return CDL_E_CAPACITY;  // (the workspace is ready for cdl_join_write)
  return join_output(jc, out_cols, out_arity, out_cap, total, n_out, c);
}

cdl_status cdl_join_write(const uint32_t* const* probe_cols, uint32_t probe_arity, uint64_t n_probe,
                          uint32_t probe_key, const uint32_t* const* build_cols,
                          uint32_t build_arity, uint64_t n_build, uint32_t build_key,
                          const cdl_colref* spec, uint32_t out_arity, const cdl_colref* neq,
                          uint32_t nneq, uint32_t* const* out_cols, uint64_t out_cap,
                          uint64_t* n_out, void* workspace, const size_t* ws_bytes, void* stream) {
  if (!ws_bytes || !workspace || !n_out) return CDL_E_INVALID;
  if (*ws_bytes < join_need(n_probe, n_build, false)) return CDL_E_INVALID;
  const uint64_t total = *n_out;
  if (total == 0) return CDL_OK;
  if (out_cap < total) return CDL_E_CAPACITY;
  JoinCall jc;
  cdl_status s = join_setup(probe_cols, probe_arity, n_probe, probe_key, build_cols, build_arity,
                            n_build, build_key, spec, out_arity, neq, nneq, workspace, *ws_bytes,
                            join_need(n_probe, n_build, true), jc);
  if (s != CDL_OK) return s;
  Ctx c;
  c.st = static_cast<cudaStream_t>(stream);
  c.d_err = reinterpret_cast<uint32_t*>(jc.head);
  jc.j.head = jc.head;
  jc.j.mark = jc.mark;
  return join_output(jc, out_cols, out_arity, out_cap, total, n_out, c);
}

cdl_status cdl_sort_unique(const uint32_t* const* cols, uint32_t arity, uint64_t n,
                           uint32_t* const* out_cols, uint64_t* n_out, void* workspace,
                           size_t* ws_bytes, void* stream) {
  if (!ws_bytes || arity < 1 || arity > CDL_MAX_ARITY) return CDL_E_INVALID;
  const uint64_t rows = n ? n : 1;
  const size_t col = up(rows * 4);
  const size_t need = kHead + 2 * arity * col + up(radix_workspace(n, 9)) +
                      up(diff_merge_workspace(0, n));
  if (!workspace) {
    *ws_bytes = need;
    return CDL_OK;
  }
  if (*ws_bytes < need || !n_out || ((!cols || !out_cols) && n)) return CDL_E_INVALID;
  if (n > 0xFFFFFFFFull) return CDL_E_CAPACITY;
  Carve cv(workspace);
  uint64_t* head = static_cast<uint64_t*>(cv.take(kHead));
  Ctx c;
  c.st = static_cast<cudaStream_t>(stream);
  c.d_err = reinterpret_cast<uint32_t*>(head);
  ColsIn in{};
  ColsOut out{};
  for (uint32_t k = 0; k < arity && n; ++k) {
    in.c[k] = cols[k];
    out.c[k] = out_cols[k];
  }
  uint64_t h[8];
  auto finish = [&]() {
    cdl_status s = read_flags(head, c.st, h, 2);
    if (s == CDL_OK) *n_out = h[1];
    return s;
  };
  if (n && n <= kSmallSort) {  // one launch
    if (sort_small(c, arity, in, n, out, true, head) != cudaSuccess) return CDL_E_CUDA;
    return finish();
  }
  // room for two copies of the columns, the sort's tables and the difference's
  char* rows_ws = static_cast<char*>(cv.take(2 * arity * col));
  void* rws = cv.take(radix_workspace(n, 9));  // room for 9-bit digits
  void* dws = cv.take(diff_merge_workspace(0, n));
  cudaError_t e = cudaMemsetAsync(head, 0, kHead, c.st);
  uint32_t* dmax = reinterpret_cast<uint32_t*>(head + 4);
  if (e == cudaSuccess) e = column_max(c, in, arity, n, dmax);
  if (e != cudaSuccess) return CDL_E_CUDA;
  cdl_status s = read_flags(head, c.st, h, 8);
  if (s != CDL_OK) return s;
  uint32_t bits[kMaxK] = {0, 0, 0, 0}, max[kMaxK];
  memcpy(max, h + 4, sizeof(max));
  uint32_t total = 0;
  for (uint32_t k = 0; k < arity; ++k) total += bits[k] = bits_of(max[k]);
  // few possible tuples (a bitmap of them takes at most 8 bytes a row): set
  // bits, read back in order (1M pairs of 12-bit values 359 -> 126 us, of
  // 16.7M 14-bit pairs 1,218 -> 502 us; 1M 14-bit pairs, just past the line,
  // take 167 us by buckets)
  if (n && total < 40 && (1ull << total) <= kBitmapPerRow * n) {
    DenseSet d{};
    d.nbits = 1ull << total;
    d.k = arity;
    d.append = 1;  // (the bits need no clearing behind the read)
    d.words = reinterpret_cast<uint32_t*>(rows_ws);
    uint32_t sh = 0;
    for (int k = (int)arity - 1; k >= 0; --k) {
      if (bits[k]) d.shift[k] = sh;
      d.mask[k] = (uint32_t)((1ull << bits[k]) - 1);
      sh += bits[k];
    }
    const size_t bytes = d.nbits >= 32 ? d.nbits >> 3 : 4;
    if (bytes <= 2 * arity * col && dense_extract_workspace(d.nbits) <= radix_workspace(n, 9)) {
      e = cudaMemsetAsync(rows_ws, 0, bytes, c.st);
      if (e == cudaSuccess) e = dense_insert(c, d, in, n);
      if (e == cudaSuccess) e = dense_extract(c, d, out, n, head + 1, rws);
      return e == cudaSuccess ? finish() : CDL_E_CUDA;
    }
  }
  // (wide tuples are read again while the output is written: not over the input)
  bool overlap = false;
  for (uint32_t i = 0; i < arity; ++i)
    for (uint32_t j = 0; j < arity; ++j)
      overlap |= out_cols[i] < cols[j] + n && cols[j] < out_cols[i] + n;
  BucketPlan bp;
  if (bucket_plan(arity, bits, max, n, bp) && (bp.keys == bp.k || !overlap) &&
      bucket_workspace(bp) <= up(radix_workspace(n, 9)) + up(diff_merge_workspace(0, n)) &&
      (bp.keys < bp.k ? 12 : 8) * n <= 2 * arity * col) {
    e = bucket_count(c, bp, in, n, rws, head + 3);
    if (e != cudaSuccess) return CDL_E_CUDA;
    s = read_flags(head, c.st, h, 4);
    if (s != CDL_OK) return s;
    if (h[3] <= kBucketCap) {
      e = bucket_sort(c, bp, in, n, out, reinterpret_cast<uint64_t*>(rows_ws), rws, head + 1);
      if (e != cudaSuccess) return CDL_E_CUDA;
      s = read_flags(head, c.st, h, 3);
      if (s != CDL_OK) return s;
      *n_out = h[1];
      if (!h[2]) return CDL_OK;  // (else too uneven: the radix sort)
    }
  }
  ColsOut a{}, b{};
  for (uint32_t k = 0; k < arity; ++k) {
    a.c[k] = reinterpret_cast<uint32_t*>(rows_ws + k * col);
    b.c[k] = reinterpret_cast<uint32_t*>(rows_ws + (arity + k) * col);
  }
  for (uint32_t k = 0; k < arity && n && e == cudaSuccess; ++k)
    e = cudaMemcpyAsync(a.c[k], cols[k], n * 4, cudaMemcpyDeviceToDevice, c.st);
  if (e != cudaSuccess) return CDL_E_CUDA;
  RadixPlan plan = make_radix_plan(arity, bits, fit_digit_bits(total, 8));
  bool in_b = false;
  e = radix_sort(c, plan, a, b, n, rws, &in_b);
  if (e != cudaSuccess) return CDL_E_CUDA;
  ColsIn sorted;
  for (int k = 0; k < kMaxK; ++k) sorted.c[k] = in_b ? b.c[k] : a.c[k];
  ColsOut none{};
  ColsIn empty{};
  e = diff_merge(c, arity, empty, 0, sorted, n, out, none, head + 1, dws);
  return e == cudaSuccess ? finish() : CDL_E_CUDA;
}

cdl_status cdl_mlp_forward(const float* params, const float* X, uint64_t n, float* out,
                           void* workspace, size_t* ws_bytes, void* stream) {
  if (!ws_bytes) return CDL_E_INVALID;
  const size_t need = mlp_workspace(n);  // (the call's contract; the kernel keeps nothing in it)
  if (!workspace) {
    *ws_bytes = need;
    return CDL_OK;
  }
  if (*ws_bytes < need || !params || ((!X || !out) && n)) return CDL_E_INVALID;
  Ctx c;
  c.st = static_cast<cudaStream_t>(stream);
  return cuda_status(mlp_forward(c, params, X, n, out));
}

cdl_status cdl_mlp_gradient(const float* params, const float* X, const float* y, uint64_t n,
                            float tau, float* out, float* grad, void* workspace, size_t* ws_bytes,
                            void* stream) {
  if (!ws_bytes) return CDL_E_INVALID;
  const size_t need = mlp_workspace(n);
  if (!workspace) {
    *ws_bytes = need;
    return CDL_OK;
  }
  if (*ws_bytes < need || !params || !grad || ((!X || !y || !out) && n)) return CDL_E_INVALID;
  if (!(tau > 0.f && tau < 1.f)) return CDL_E_INVALID;
  Ctx c;
  c.st = static_cast<cudaStream_t>(stream);
  return cuda_status(mlp_gradient(c, params, X, y, n, tau, out, grad, workspace));
}

cdl_status cdl_mlp_infer_bf16(const float* params, const float* X, uint64_t n, float* out,
                              void* workspace, size_t* ws_bytes, void* stream) {
  if (!ws_bytes) return CDL_E_INVALID;
  const size_t need = up(sizeof(uint16_t) * kMlpParams);
  if (!workspace) {
    *ws_bytes = need;
    return CDL_OK;
  }
  if (*ws_bytes < need || !params || ((!X || !out) && n)) return CDL_E_INVALID;
  Ctx c;
  c.st = static_cast<cudaStream_t>(stream);
  cudaError_t e = mlp_to_bf16(c, params, workspace);
  if (e == cudaSuccess) e = mlp_infer_bf16(c, workspace, X, n, out);
  return cuda_status(e);
}

cdl_status cdl_mlp_adam(float* params, const float* grad, float* m, float* v, uint64_t step,
                        float lr, void* stream) {
  if (!params || !grad || !m || !v || step == 0) return CDL_E_INVALID;
  Ctx c;
  c.st = static_cast<cudaStream_t>(stream);
  return cuda_status(mlp_adam(c, params, grad, m, v, step, lr));
}

cdl_status cdl_join_features(const uint32_t* probe_k0, const uint32_t* probe_k1, uint64_t n_probe,
                             const uint32_t* build_k0, const uint32_t* build_k1, uint64_t n_build,
                             const float* host, float* features, void* stream) {
  if (!host || !features || (n_probe && !probe_k0) || (n_build && !build_k0)) return CDL_E_INVALID;
  JoinFeatureHost hf{host[0], host[1], host[2], host[3], host[4], host[5]};
  Ctx c;
  c.st = static_cast<cudaStream_t>(stream);
  return cuda_status(join_features(c, probe_k0, probe_k1, n_probe, build_k0, build_k1, n_build,
                                   hf, features));
}

cdl_status cdl_diff_merge(const uint32_t* const* full, uint64_t n_full,
                          const uint32_t* const* fresh, uint64_t n_fresh, uint32_t arity,
                          uint32_t* const* delta, uint64_t* n_delta, uint32_t* const* merged,
                          void* workspace, size_t* ws_bytes, void* stream) {
  if (!ws_bytes || arity < 1 || arity > CDL_MAX_ARITY) return CDL_E_INVALID;
  const size_t need = kHead + up(diff_merge_workspace(n_full, n_fresh));
  if (!workspace) {
    *ws_bytes = need;
    return CDL_OK;
  }
  if (*ws_bytes < need || !n_delta) return CDL_E_INVALID;
  if ((n_full && !full) || (n_fresh && !fresh) || !delta || !merged) return CDL_E_INVALID;
  Carve cv(workspace);
  uint64_t* head = static_cast<uint64_t*>(cv.take(kHead));
  void* dws = cv.take(diff_merge_workspace(n_full, n_fresh));
  ColsIn f{}, u{};
  ColsOut d{}, m{};
  for (uint32_t k = 0; k < arity; ++k) {
    f.c[k] = n_full ? full[k] : nullptr;
    u.c[k] = n_fresh ? fresh[k] : nullptr;
    d.c[k] = delta[k];
    m.c[k] = merged[k];
  }
  Ctx c;
  c.st = static_cast<cudaStream_t>(stream);
  c.d_err = reinterpret_cast<uint32_t*>(head);
  cudaError_t e = cudaMemsetAsync(head, 0, kHead, c.st);
  if (e == cudaSuccess) e = diff_merge(c, arity, f, n_full, u, n_fresh, d, m, head + 1, dws);
  if (e != cudaSuccess) return CDL_E_CUDA;
  uint64_t h[2];
  cdl_status s = read_flags(head, c.st, h, 2);
  if (s != CDL_OK) return s;
  *n_delta = h[1];
  return CDL_OK;
}

}  // extern "C"
