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

// Stores the first min(cnt, 4) entries of record `rec` at w (shared memory on
// the device): the places of this record's own pairs and no others, since
// nothing orders the stores of a chunk's 32 lanes.  On the device as predicated
// stores: as branches they cost the sort 4% (2^26 records 752 us, 722 so; 2^31
// 23.9 and 22.9 ms).
VX_HD void put_nearest_pairs(uint16_t *w, uint32_t rec, uint32_t cnt)
{
#ifdef __CUDA_ARCH__
    asm volatile(
        "{ .reg .pred p0, p1, p2, p3;\n\t"
        "setp.gt.u32 p0, %1, 0;\n\t"
        "setp.gt.u32 p1, %1, 1;\n\t"
        "setp.gt.u32 p2, %1, 2;\n\t"
        "setp.gt.u32 p3, %1, 3;\n\t"
        "@p0 st.shared.u16 [%0], %2;\n\t"
        "@p1 st.shared.u16 [%0 + 2], %3;\n\t"
        "@p2 st.shared.u16 [%0 + 4], %4;\n\t"
        "@p3 st.shared.u16 [%0 + 6], %5; }"
        :
        : "r"((uint32_t)__cvta_generic_to_shared(w)), "r"(cnt), "h"(pair_entry(rec, 1u)), "h"(pair_entry(rec, 2u)),
          "h"(pair_entry(rec, 3u)), "h"(pair_entry(rec, 4u))
        : "memory");
#else
    if (cnt > 0u) w[0] = pair_entry(rec, 1u);
    if (cnt > 1u) w[1] = pair_entry(rec, 2u);
    if (cnt > 2u) w[2] = pair_entry(rec, 3u);
    if (cnt > 3u) w[3] = pair_entry(rec, 4u);
#endif
}

}  // namespace vx
