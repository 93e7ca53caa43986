// agg_rule.h — which way the offsets kernel of the exchange finds a list's
// position at every tile boundary (plain functions, tested on the host).
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define EFS_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define EFS_HOST_DEVICE inline
#endif

namespace efs {

// The scatter reads every index once (32 MB at most, about 8 us), the searches
// take 8 to 12 us whatever the lists hold. Measured, us an exchange, searches
// -> scatter: 16 lists of 256 K entries over 6,240 tiles 61.6 -> 54.8, 4
// LSTM-shaped workers' steps with their exchange (0.9 M entries each) 333.5 ->
// 300.2; one list of 34.6 M entries over 33,779 tiles 159 -> 180.
constexpr uint32_t kScatterEntries = 8u << 20;

// A list's entries as they are summed over all lists: 256 of them fit 32 bits,
// and one list's can pass kScatterEntries.
EFS_HOST_DEVICE uint32_t scatter_share(uint32_t count) {
  return count <= kScatterEntries ? count : kScatterEntries + 1;
}

// Scatter a list of `count` entries over `per` offsets? `all` is the sum of
// the lists' shares.
EFS_HOST_DEVICE bool scatter_offsets(uint32_t count, uint32_t all, uint32_t per) {
  return count >= per / 16 && all <= kScatterEntries;
}

}  // namespace efs
