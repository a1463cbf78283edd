// bitmap_sort.cuh -- ranks the records of a partition in shared memory by a
// digit bitmap: the partition sorts of Table 1 and of Table 2.
#pragma once

#include "vx_internal.cuh"

namespace vx {

constexpr uint32_t kDirtyList = 64;  // listed words with a shared digit (2048 records: about 31)
constexpr int kMaxDigitBits = 18;   // sort digit (bitmap of 2^18 bits, 8192 words)

// Words of the digit bitmap of a plan's dbits (log2 of the mean records of a
// partition): 32 digits per expected record, so that two records share a
// digit about once in 64 records (2048 records, 2^16 digits: 32 pairs).
// More digits cost shared memory (three CTAs per SM need 75 KB each), fewer
// double the shared digits.
__host__ __device__ __forceinline__ uint32_t bitmap_words(int dbits)
{
    const int b = dbits + 5 < kMaxDigitBits ? dbits + 5 : kMaxDigitBits;
    return 1u << (b - 5);
}

// The arrays of one partition's ranking (16-byte aligned BM, PF right after
// its words).
struct Bitmap {
    uint32_t *BM;  // digit bitmap
    uint16_t *PF;  // word prefixes
    uint16_t *DL;  // dirty words (the first kDirtyList of them)
    uint32_t *WS;  // scan workspace, 40 words
};
constexpr uint32_t kWsDirty = 36;  // WS word: how many dirty words the scan met
constexpr uint32_t kWsLong = 37;   // WS word: some warp's pairs do not fit its list (match)

// Inclusive scan of one u32 per lane (a shuffle's own predicate says
// whether its source lane exists: two instructions a step).
__device__ __forceinline__ uint32_t warp_incl_scan(uint32_t x)
{
#pragma unroll
    for (int o = 1; o < 32; o <<= 1)
        asm volatile(
            "{ .reg .pred p; .reg .u32 r; shfl.sync.up.b32 r|p, %0, %1, 0, 0xffffffff; @p add.u32 %0, r, %0; }"
            : "+r"(x)
            : "r"(o));
    return x;
}

constexpr uint32_t kDirty = 0x8000u;  // flag of PF: the word holds a shared digit

// Zeroes the bitmap and the extra counts (PF) of W words; no barrier.
template <int NT>
__device__ __forceinline__ void clear_tables(const Bitmap &A, uint32_t W)
{
    if (threadIdx.x == 0) A.WS[kWsDirty] = A.WS[kWsLong] = 0u;
    if (W % 8u == 0) {  // 6 W bytes, a multiple of 16 (PF follows BM)
        uint4 *t = reinterpret_cast<uint4 *>(A.BM);
        for (uint32_t i = threadIdx.x; i < W * 6u / 16u; i += NT) t[i] = make_uint4(0u, 0u, 0u, 0u);
    } else {
        for (uint32_t i = threadIdx.x; i < W; i += NT) {
            A.BM[i] = 0u;
            A.PF[i] = 0;
        }
    }
}

// The sort.  The digit, the key bits below the partition prefix, is wide
// enough (2^16 for 2048 records) that most records have one of their own:
// then a record's place is the number of records in lower digits, i.e. the
// count before its bitmap word plus the word's bits below its own, and the
// record goes there directly.  Words with a shared digit ("dirty") take
// their records in arrival order, which the caller puts right.  One pass
// marks the digits (mark), one places the records (place_of); a counting
// sort's third pass (ranking every record in its digit run) and its second
// set of shared-memory atomics are gone.

// Marks a digit; one already taken counts as an extra of its word.
__device__ __forceinline__ void mark(const Bitmap &A, uint32_t dg)
{
    const uint32_t w = dg >> 5, bit = 1u << (dg & 31u);
    if (atomicOr(&A.BM[w], bit) & bit)
        atomicAdd(reinterpret_cast<uint32_t *>(A.PF) + (w >> 1), 1u << (16u * (w & 1u)));
}

// A record's place (after scan_words).
__device__ __forceinline__ uint32_t place_of(const Bitmap &A, uint32_t dg)
{
    const uint32_t w = dg >> 5, pf = A.PF[w];
    if (pf & kDirty) return (pf & (kDirty - 1u)) + atomicAdd(&A.BM[w], 1u);
    return pf + (uint32_t)__popc(A.BM[w] & ((1u << (dg & 31u)) - 1u));
}

// Exclusive scan of the W words' record counts into PF, `per` consecutive
// words a thread; dirty words are flagged and listed and their bitmap word
// becomes the count of records placed.  Between two barriers of the caller's;
// one inside.
template <int NT>
__device__ __forceinline__ void scan_words(const Bitmap &A, uint32_t W)
{
    constexpr uint32_t NW = NT / 32;
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    const uint32_t per = W > (uint32_t)NT ? W / NT : 1u;
    const uint32_t w0 = threadIdx.x * per;
    const uint32_t sw = lane & 4u;  // every other four lanes read the upper half first: no bank conflicts
    uint32_t local = 0;
    if (per >= 8) {
        for (uint32_t g = 0; g < per; g += 8) {
            const uint4 a = *reinterpret_cast<const uint4 *>(A.BM + w0 + g + sw);
            const uint4 b = *reinterpret_cast<const uint4 *>(A.BM + w0 + g + 4 - sw);
            const uint4 e = *reinterpret_cast<const uint4 *>(A.PF + w0 + g);
            local += __popc(a.x) + __popc(a.y) + __popc(a.z) + __popc(a.w) + __popc(b.x) + __popc(b.y) +
                     __popc(b.z) + __popc(b.w);
            const uint32_t x = e.x + e.y + e.z + e.w;  // extras: 16-bit halves, < 2^15 in all
            local += (x & 0xFFFFu) + (x >> 16);
        }
    } else if (w0 < W) {
        for (uint32_t g = 0; g < per; ++g) local += __popc(A.BM[w0 + g]) + A.PF[w0 + g];
    }
    const uint32_t incl = warp_incl_scan(local);
    if (lane == 31) A.WS[warp] = incl;
    __syncthreads();
    uint32_t run = incl - local;
#pragma unroll
    for (uint32_t w = 0; w < NW; ++w) run += w < warp ? A.WS[w] : 0u;
    auto set_dirty = [&](uint32_t w) {
        A.PF[w] |= (uint16_t)kDirty;
        A.BM[w] = 0u;
        const uint32_t i = atomicAdd(&A.WS[kWsDirty], 1u);
        if (i < kDirtyList) A.DL[i] = (uint16_t)w;
    };
    if (per >= 8) {
        for (uint32_t g = 0; g < per; g += 8) {
            uint4 e = *reinterpret_cast<const uint4 *>(A.PF + w0 + g);
            uint32_t *const ex[4] = {&e.x, &e.y, &e.z, &e.w};
            uint4 a = *reinterpret_cast<const uint4 *>(A.BM + w0 + g + sw);
            uint4 b = *reinterpret_cast<const uint4 *>(A.BM + w0 + g + 4 - sw);
            if (sw) {
                const uint4 t = a;
                a = b;
                b = t;
            }
            const uint32_t bm[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
            uint32_t m = 0;  // bit j: word w0 + g + j is dirty
            if (e.x | e.y | e.z | e.w) {
#pragma unroll
                for (int h = 0; h < 4; ++h)
                    m |= (*ex[h] & 0xFFFFu ? 1u << (2 * h) : 0u) | (*ex[h] >> 16 ? 2u << (2 * h) : 0u);
            }
#pragma unroll
            for (int h = 0; h < 4; ++h) {
                const uint32_t p0 = run;
                run += __popc(bm[2 * h]) + (*ex[h] & 0xFFFFu);
                const uint32_t p1 = run;
                run += __popc(bm[2 * h + 1]) + (*ex[h] >> 16);
                *ex[h] = p0 | (p1 << 16);
            }
            *reinterpret_cast<uint4 *>(A.PF + w0 + g) = e;
            for (; m; m &= m - 1u) set_dirty(w0 + g + (uint32_t)__ffs((int)m) - 1u);
        }
    } else if (w0 < W) {
        for (uint32_t g = 0; g < per; ++g) {
            const uint32_t x = A.PF[w0 + g];
            A.PF[w0 + g] = (uint16_t)run;
            run += __popc(A.BM[w0 + g]) + x;
            if (x) set_dirty(w0 + g);
        }
    }
}

}  // namespace vx
