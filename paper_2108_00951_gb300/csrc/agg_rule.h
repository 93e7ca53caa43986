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

// The scatter's time grows with the entries it reads, the searches' with the
// number of lists and tiles. Measured on a GB300, us an exchange, searches ->
// scatter, by entries a tile and list:
//     41  16 lists over 6,240 tiles 49.3 -> 49.1, over 33,779 218 -> 202,
//         256 lists over 1,954 520 -> 510, 4 over 33,779 122.3 -> 119.2
//      4  64 lists over 33,779 tiles 655 -> 627
//    164  4 lists over 33,779 tiles 147.9 -> 154.8, 16 over 6,240 77.0 -> 83.7,
//         1 over 6,240 29.3 -> 23.6
//   1024  1 list over 33,779 tiles 153 -> 180, 16 over 1,954 80 -> 114
// So a list of up to 64 entries a tile is scattered, and every list while they
// are few together (32 MB of indexes, about 8 us).
constexpr uint32_t kScatterPerTile = 64;
constexpr uint32_t kScatterEntries = 8u << 20;

// A list's entries as they are summed over all lists: 256 of them fit 32 bits,
// and one list's can pass kScatterEntries.
EFS_HOST_DEVICE uint32_t scatter_share(uint32_t count) {
  return count <= kScatterEntries ? count : kScatterEntries + 1;
}

// Scatter a list of `count` entries over `per` offsets? `all` is the sum of
// the lists' shares.
EFS_HOST_DEVICE bool scatter_offsets(uint32_t count, uint32_t all, uint32_t per) {
  const bool few = count / kScatterPerTile < per || all <= kScatterEntries;
  return count >= per / 16 && few;
}

}  // namespace efs
