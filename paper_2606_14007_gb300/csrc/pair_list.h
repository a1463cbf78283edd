// pair_list.h -- the entries a record's pairs take in its warp's pair list
// (partition sort + match).  Compiles for the host too.
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define VX_HD __host__ __device__ __forceinline__
#else
#define VX_HD inline
#endif

namespace vx {

// An entry: the first record of the pair, counted from the warp's first
// record (12 bits), and how many records later its partner stands (4 bits).
VX_HD uint16_t pair_entry(uint32_t rec, uint32_t dist) { return (uint16_t)(rec + (dist << 12)); }

// Stores the first min(cnt, 4) entries of record `rec` at w: the places of
// this record's own pairs and no others, since nothing orders the stores of a
// chunk's 32 lanes.
VX_HD void put_nearest_pairs(uint16_t *w, uint32_t rec, uint32_t cnt)
{
    if (cnt > 0u) w[0] = pair_entry(rec, 1u);
    if (cnt > 1u) w[1] = pair_entry(rec, 2u);
    if (cnt > 2u) w[2] = pair_entry(rec, 3u);
    if (cnt > 3u) w[3] = pair_entry(rec, 4u);
}

}  // namespace vx
