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
//     41  16 lists over 6,240 tiles 60.2 -> 48.7, over 33,779 217 -> 203,
//         256 lists over 1,954 527 -> 518, 4 over 33,779 122.4 -> 118.3
//      4  64 lists over 33,779 tiles 652 -> 629
//    164  4 lists over 33,779 tiles 148.3 -> 153.5, 1 over 6,240 30.4 -> 23.2
//   1024  1 list over 33,779 tiles 159 -> 180, 4 over 1,954 34.9 -> 36.6
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
