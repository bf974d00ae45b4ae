// Size rules of the host side that are plain arithmetic (no CUDA headers, so
// that they are checked at sizes no test can allocate).
#pragma once

#include <stdint.h>

namespace cdl {

// The direct form of an index over `rows` rows whose one-word keys lie below
// 2^bits: the number of its entries, or 0 for the hash form.  It is taken
// where its array, 8 bytes an entry, is cleared and read at no more than 32
// bytes per row (hash slots take 32 to 64 per distinct key), or is small
// beside a launch; it also spares the count of the keys and the wait for it:
// points-to at 2^-7 15.6 -> 14.9 ms, a closure of 4,001 nodes 5.26 -> 4.89
// ms.  Past 4 GB (a seventieth of the device's memory) it is not: a relation
// that large may have few distinct keys, and the slots for them are small.
// limited (runs under a memory limit): the small array alone.
constexpr uint64_t kDirectKeysMin = 1ull << 16, kDirectKeysMax = 1ull << 29;
inline uint32_t direct_entries(uint32_t bits, uint64_t rows, bool limited) {
  const uint64_t keys = 1ull << bits;
  if (keys <= kDirectKeysMin) return (uint32_t)keys;
  return !limited && keys <= 4 * rows && keys <= kDirectKeysMax ? (uint32_t)keys : 0u;
}

// Rows that Full, kept as a set, may have at the end of a captured round: with
// more the round leaves the graph and is run by the host, which stops at the
// 2^32 tuples a relation may hold.  times: a hash set's table is for so many
// times the rows there are (0: a bitmap, which has room for every tuple).
inline uint64_t graph_set_rows(uint64_t rows, uint64_t times) {
  constexpr uint64_t kMost = 0xFFFFFFFFull, kLeast = 1ull << 16;
  if (times == 0 || rows > kMost / times) return kMost;
  return times * rows > kLeast ? times * rows : kLeast;
}

}  // namespace cdl
