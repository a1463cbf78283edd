// k_sortmatch.cu -- partition sort fused with the match stage.
//
// Paper: Sec. I-B / III-A / III-B fuse sort and Table-2 generation into one
// kernel that keeps each bucket in shared memory, one block per bucket,
// with a single-thread insertion sort; Sec. V names that O(n^2) sort as the
// K=31 bottleneck and proposes a parallel radix sort.  Kept here: the
// fusion (a partition never leaves shared memory between sort and match).
// Changed: a physical partition (a run of whole logical buckets, ~2048
// records) per work item, and a sort that places nearly every record by one
// bitmap rank: the key bits below the partition prefix, 32 digits per
// expected record, mark a bitmap, and a record's place is the number of
// marked digits below its own; only the records that share a digit's word
// with a collision are ordered by (key64, nonce).  A partition's pairs
// either go to its own slot (kSortSlots, the default wherever the plan shows
// the pair slot safe: no partition waits on another, a scan and the slot
// pair hash place them) or straight to Table 2 at a base found by a
// decoupled look-back over the partitions before it (partition order comes
// from a ticket counter, so every partition an item waits on is held by a
// running CTA; every wait is bounded and a timeout poisons the chain instead
// of hanging).  With the cross-bucket match (HALO instances) the next
// partition's halo is sorted in behind the partition's records.
//
// The sorted records stand in shared memory as Table-1 words, so Table 1
// leaves by one bulk copy.  The match walks them in chunks of 32, one record
// per lane, each warp over its own run of chunks: a lane compares 32 key
// bits with the records after its own (shuffles), warp scans give the pair
// offsets, and the pairs go through a 16-bit list in shared memory, so that
// they are written one per lane, coalesced.
//
// Bound by instruction issue (59%) and the shared-memory data path (65%)
// together at 24 warps per SM: 16.1 k warp instructions per 2048-record
// partition, against 23 k for the counting sort with ranked digit runs, the
// per-thread Table-1 stores and the record-wise pair stores before it: 31.0
// -> 24.1 ms at K=31, 0.97 -> 0.75 ms at K=26, and with the items handed out
// by a counter 22.8 ms (2^31 records; 3.0 of 6.78 TB/s) and 0.72 ms.  By
// phase at K=26, of 0.75 ms: load, mark and scan 0.23 ms, placement 0.14,
// shared digits 0.04, match and lists 0.27, pair stores 0.07.  Tried and
// dropped, against 0.75: half the digits (0.88 ms), the slot read into
// registers with four CTAs per SM (0.78), eleven rows of loads in flight
// instead of four (0.82).
//
// Two front ends feed the same steps:
//  * k_sortmatch_pipe (the default): persistent CTAs, three per SM at the
//    default slot.  A CTA's next partition slot (keys and nonces, two
//    contiguous runs) comes into shared memory by cp.async.bulk once the
//    current one has been placed.
//  * k_sortmatch_gl: one CTA per partition reading its slot from global
//    memory, for slots too large to hold twice in shared memory.
//
// MODE kSortCount: the sort alone (Table 1 + per-partition pair counts),
// used by the split vx_table1 / vx_match path.
// MODE kSortHash: everything in one kernel, pairs hashed here.
// MODE kSortEmit: Table 1, then each pair written as a Table-2 record
// {a, b, 0, 0} at its final offset; the streaming pair-hash kernel fills in
// the hashes (no barriers, full occupancy: the ALU-bound part runs apart
// from the latency-bound sort).
// MODE kSortSlots: Table 1, then the partition's pairs {a, b} in (i, j)
// order into the partition's own level-2 slot, which the kernel has already
// read: cap2 pairs in the key array, cap2 / 2 in the nonce array.  No
// partition waits on another; a scan of the pair counts and the slot pair
// hash place the records.
#include "bitmap_sort.cuh"
#include "pair_list.h"
#include "vx_internal.cuh"

namespace vx {

enum { kSortCount = 0, kSortHash = 1, kSortEmit = 2, kSortSlots = 3 };
constexpr int kPipeThreads = 256;   // persistent front end
constexpr int kGlThreads = 256;     // one-CTA-per-partition front end
// Tickets between a CTA of the global-memory front end and the partition
// whose slot it prefetches into L2: about half of the CTAs resident at once.
constexpr uint32_t kSlotPrefetchAhead = 384;

// Shared layout (bytes from the base), for slots of at most `cap` records
// (a multiple of 4) and a bitmap of at most `words` words:
//   X: key64 [cap] | nonce [cap], the slot (pipelined front end only)
//   Y: the sorted records as Table-1 words {nonce, h0, h1} [cap], starting
//      up to 12 bytes in, so that shared and Table-1 addresses agree mod 16
//   bitmap [words] | word prefixes, 16 bits [words]; dead once the records
//   are sorted, then overlaid by the warps' pair lists (16 bits an entry, at
//   least 2 * cap entries together)
//   dirty words [kDirtyList] | scan workspace | mbarrier
struct SMLayout {
    size_t xk, xn, y, bm, dl, ws, bar, bytes;
    __host__ __device__ SMLayout(uint32_t cap, uint32_t words, bool two)
    {
        cap = (cap + 3u) & ~3u;
        xk = 0;
        xn = xk + (two ? (size_t)cap * 8 : 0);
        y = xn + (two ? (size_t)cap * 4 : 0);
        bm = y + (size_t)cap * 12 + 16;
        dl = bm + tables_bytes(cap, words);
        ws = dl + (size_t)kDirtyList * 2;
        bar = ws + 40 * 4;
        bytes = bar + 8;
    }
    static __host__ __device__ size_t tables_bytes(uint32_t cap, uint32_t words)
    {
        const size_t tab = ((size_t)words * 6 + 15) & ~(size_t)15, lists = (size_t)cap * 4 + 512;
        return tab > lists ? tab : lists;
    }
};

struct Part : Bitmap {
    uint32_t *Y;   // sorted Table-1 words (record r at Y[3 r])
    uint16_t *PL;  // pair lists, over BM and PF: NT / 32 of them, plw entries each
    uint32_t plw;
};
__device__ __forceinline__ bool rec_less(uint64_t ka, uint32_t na, uint64_t kb, uint32_t nb)
{
    return ka < kb || (ka == kb && na < nb);
}

__device__ __forceinline__ uint64_t y_key(const uint32_t *Y, uint32_t r)
{
    return ((uint64_t)bswap32(Y[3 * r + 1]) << 32) | bswap32(Y[3 * r + 2]);
}

// The 32 key bits below the partition prefix (pk bits), pk <= 21.
__device__ __forceinline__ uint32_t sub_key(uint32_t hi, uint32_t lo, int pk)
{
    return __funnelshift_rc(lo, hi, 32 - pk);
}

// ---------------------------------------------------------------- sort

__device__ __forceinline__ void put_record(const Part &A, uint32_t pos, uint64_t key, uint32_t nonce)
{
    uint32_t *o = A.Y + 3 * pos;
    o[0] = nonce;
    o[1] = bswap32((uint32_t)(key >> 32));
    o[2] = bswap32((uint32_t)key);
}

// The dirty words' records in order: eight lanes a listed word, a lane per
// record, each finding its place among the word's records from its
// neighbours' (shuffles); words with more than eight records or past the
// list by one thread's insertion sort.
template <int NT>
__device__ __forceinline__ void order_dirty(const Part &A, uint32_t W)
{
    constexpr uint32_t NW = NT / 32;
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    auto order_word = [&](uint32_t w) {
        uint32_t *const y = A.Y + 3 * (A.PF[w] & (kDirty - 1u));
        const uint32_t cnt = A.BM[w];
        for (uint32_t a = 1; a < cnt; ++a) {
            const uint64_t kx = y_key(y, a);
            const uint32_t nx = y[3 * a], x1 = y[3 * a + 1], x2 = y[3 * a + 2];
            uint32_t b = a;
            for (; b > 0 && rec_less(kx, nx, y_key(y, b - 1), y[3 * b - 3]); --b) {
                y[3 * b] = y[3 * b - 3];
                y[3 * b + 1] = y[3 * b - 2];
                y[3 * b + 2] = y[3 * b - 1];
            }
            y[3 * b] = nx;
            y[3 * b + 1] = x1;
            y[3 * b + 2] = x2;
        }
    };
    const uint32_t nd = A.WS[kWsDirty];
    if (nd <= kDirtyList) {
        const uint32_t sub = lane & 7u;
        for (uint32_t i0 = 4u * warp; i0 < nd; i0 += 4u * NW) {
            const uint32_t i = i0 + (lane >> 3);
            const uint32_t w = i < nd ? A.DL[i] : 0u;
            uint32_t *const y = A.Y + 3 * (A.PF[w] & (kDirty - 1u));
            const uint32_t all = i < nd ? A.BM[w] : 0u;
            const uint32_t cnt = all <= 8u ? all : 0u;
            const bool mine = sub < cnt;
            uint32_t nx = 0, x1 = 0, x2 = 0;
            if (mine) {
                nx = y[3 * sub];
                x1 = y[3 * sub + 1];
                x2 = y[3 * sub + 2];
            }
            const uint64_t k = ((uint64_t)bswap32(x1) << 32) | bswap32(x2);
            const uint32_t most = __reduce_max_sync(0xffffffffu, cnt);
            uint32_t place = 0;
            for (uint32_t o = 0; o < most; ++o) {
                const uint64_t ko = __shfl_sync(0xffffffffu, k, (int)((lane & 24u) + o));
                const uint32_t no = __shfl_sync(0xffffffffu, nx, (int)((lane & 24u) + o));
                place += o < cnt && rec_less(ko, no, k, nx) ? 1u : 0u;
            }
            if (mine) {
                y[3 * place] = nx;
                y[3 * place + 1] = x1;
                y[3 * place + 2] = x2;
            }
            if (all > 8u && sub == 0) order_word(w);
        }
    } else {
        for (uint32_t w = threadIdx.x; w < W; w += NT)
            if (A.PF[w] & kDirty) order_word(w);
    }
}

// Bits of sub_key below a digit of a W-word bitmap (log2(W) + 5 bits).
__device__ __forceinline__ int digit_shift(uint32_t W) { return 27 - (31 - __clz(W)); }

// Sorts the n records of `src` by (key64, nonce) into Y as Table-1 words.
// Starts after a barrier that follows clear_tables; ends with one.
// `before_place` runs on thread 0 before anything is written to Y,
// `after_place` on thread 0 once `src` is no longer read.
template <int NT, class Src, class F1, class F2>
__device__ __forceinline__ void sort_bitmap(const Part &A, uint32_t n, int pk, uint32_t W, const Src &src,
                                            F1 before_place, F2 after_place)
{
    const int ds = digit_shift(W);
    auto digit = [&](uint64_t k) { return sub_key((uint32_t)(k >> 32), (uint32_t)k, pk) >> ds; };
#pragma unroll 4
    for (uint32_t i = threadIdx.x; i < n; i += NT) mark(A, digit(src.key(i)));
    __syncthreads();
    scan_words<NT>(A, W);
    if (threadIdx.x == 0) before_place();
    __syncthreads();
#pragma unroll 4
    for (uint32_t i = threadIdx.x; i < n; i += NT) {
        const uint64_t k = src.key(i);
        put_record(A, place_of(A, digit(k)), k, src.nonce(i));
    }
    __syncthreads();
    if (threadIdx.x == 0) after_place();
    order_dirty<NT>(A, W);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // Y leaves by a bulk copy
    __syncthreads();
}

// ------------------------------------------------ match and the tables

// Everything after the sort, for partition f (n sorted records in Y, Table-1
// offset `off`) of plot d: Table 1, the next partition's halo (HALO), the
// pair counts and their scan, then the mode's Table-2 output.  Starts and
// ends at a barrier; on failure (the status word says why) it skips the
// output, so a persistent caller goes on to its next item.  Table 1 leaves
// Y by thread 0's bulk copy: the caller waits for its reads before Y is
// written again, and for its end before the CTA exits.
template <int MODE, bool HALO, int NT>
__device__ __forceinline__ void match_and_write(const Desc &d, uint32_t f, uint32_t n, uint64_t off,
                                                const Part &A, uint64_t *s_base, int *s_ok, bool quiet)
{
    constexpr bool EMIT = MODE == kSortHash || MODE == kSortEmit;  // look-back placement
    constexpr bool SLOTS = MODE == kSortSlots;
    constexpr uint32_t NW = NT / 32;
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    uint32_t *const Y = A.Y;
    // 1. Table 1: words [0, 3n) of Y to words [3 off, 3 off + 3n) of the
    //    table.  Shared and global addresses agree mod 16 bytes; the whole
    //    16-byte lines go by one bulk copy, the up to three words before and
    //    after them by plain stores.
    if (warp == 0) {
        uint32_t *__restrict__ t1w = reinterpret_cast<uint32_t *>(d.t1) + 3 * off;
        const uint32_t words = 3 * n;
        const uint32_t head = min(words, (4u - ((uint32_t)(3 * off) & 3u)) & 3u);
        const uint32_t body = (words - head) & ~3u;
        if (lane == 0 && body) bulk_s2g(t1w + head, Y + head, body * 4u);
        if (lane < head) t1w[lane] = Y[lane];
        const uint32_t t = head + body + lane;
        if (lane < 4 && t < words) t1w[t] = Y[t];
    }
    // 2. cross-bucket match: the next partition's halo (its records within
    //    D of its lower edge, collected while the slots were filled) goes
    //    sorted right after this partition's records, so the pair scan
    //    below runs on into it; records n .. nt - 1 start no pairs here.
    uint32_t nt = n;
    if (HALO && d.hcap) {
        const uint32_t hcap = d.hcap;
        const uint64_t fn = (uint64_t)f + 1;
        const uint32_t hc = fn < (1ull << d.p) ? min(d.halo_cnt[fn], hcap) : 0u;
        for (uint32_t h = threadIdx.x; h < hc; h += NT) {
            const uint64_t k = d.halo_keys[fn * hcap + h];
            Y[3 * (n + h)] = d.halo_nonces[fn * hcap + h];
            Y[3 * (n + h) + 1] = bswap32((uint32_t)(k >> 32));
            Y[3 * (n + h) + 2] = bswap32((uint32_t)k);
        }
        __syncthreads();
        if (threadIdx.x == 0) {  // a few records (Poisson, mean 2^11 D / 2^(64-p))
            for (uint32_t a = n + 1; a < n + hc; ++a) {
                const uint64_t kx = y_key(Y, a);
                const uint32_t nx = Y[3 * a], x1 = Y[3 * a + 1], x2 = Y[3 * a + 2];
                uint32_t b = a;
                for (; b > n && rec_less(kx, nx, y_key(Y, b - 1), Y[3 * b - 3]); --b) {
                    Y[3 * b] = Y[3 * b - 3];
                    Y[3 * b + 1] = Y[3 * b - 2];
                    Y[3 * b + 2] = Y[3 * b - 1];
                }
                Y[3 * b] = nx;
                Y[3 * b + 1] = x1;
                Y[3 * b + 2] = x2;
            }
        }
        __syncthreads();
        nt = n + hc;
    }
    // 3. per chunk of 32 sorted records (one per lane; warp w takes chunks
    //    [c0, c1)): the pairs starting at each record r, i.e. the later
    //    records j of its logical bucket with key_j - key_r < D (every
    //    bucket with the cross-bucket match), listed in (i, j) order in the
    //    warp's list as (r - 32 c0) | (j - r) << 12.  A list holds about
    //    twice the default plot's pairs of a warp; a partition with more, or
    //    with a record of more than 15, is counted here and recounted when
    //    its pairs are written.
    const uint32_t nch = (n + 31u) >> 5;
    const uint32_t c0 = warp * nch / NW, c1 = (warp + 1) * nch / NW;
    const uint64_t D = d.D;
    const bool global = HALO && d.scope != 0;
    // the exact count of record r, on whole keys
    auto count_exact = [&](uint32_t r) -> uint32_t {
        const uint64_t k = y_key(Y, r);
        const uint64_t last = global ? ~0ull : (k | ((1ull << 40) - 1));
        uint64_t lim = k + (D - 1);
        if (lim < k) lim = ~0ull;  // saturate
        if (lim > last) lim = last;
        uint32_t q = r + 1;
        while (q < nt && y_key(Y, q) <= lim) ++q;
        return q - r - 1;
    };
    uint16_t *const list = A.PL + warp * A.plw;
    uint32_t mine = 0;  // pairs of the warp's chunks
    bool fits = true;   // ... that the list holds
    auto enlist = [&](uint32_t c, uint32_t cnt) {
        const uint32_t incl = warp_incl_scan(cnt);
        const uint32_t total = __shfl_sync(0xffffffffu, incl, 31);
        if (MODE != kSortCount) {
            fits = fits && mine + total <= A.plw;  // the same for the whole warp
            if (fits) {
                uint16_t *w = list + mine + incl - cnt;
                const uint32_t e = 32u * (c - c0) + lane;
                put_nearest_pairs(w, e, cnt);
                if (__any_sync(0xffffffffu, cnt > 4)) {
                    fits = !__any_sync(0xffffffffu, cnt > 15u);
                    for (uint32_t j = 4; fits && j < cnt; ++j) w[j] = pair_entry(e, j + 1u);
                }
            }
        }
        mine += total;
    };
    // On the 32 key bits q below the partition prefix (a partition holds whole
    // buckets): with D = Dq 2^s + rest, q_j - q_r < Dq is a match and
    // q_j - q_r >= Dq + 2 is none; between them, rarely, the whole keys
    // decide.  The records after r (five: 0.06% of a default plot's records
    // have more pairs) come by shuffles from this chunk's lanes and the next
    // one's; past the last record they are whatever follows in shared memory,
    // and the count is cut there.  Halo records lie past the partition's end,
    // so their q has wrapped: q_j - q_r is still their distance unless that
    // is a partition's width or more, which takes an r within D of the lower
    // edge that sees the halo; such an r is counted on whole keys.
    const int pk = d.pk;
    const uint64_t Dw = D >> (32 - pk);
    const uint32_t Dq = Dw < 0xFFFFFFF0ull ? (uint32_t)Dw : 0xFFFFFFF0u;
    if (global && Dw >= 0xFFFFFFF0ull) {  // D about a partition's width
        for (uint32_t c = c0; c < c1; ++c) {
            const uint32_t r = 32u * c + lane;
            enlist(c, r < n ? count_exact(r) : 0u);
        }
    } else {
        const uint32_t bmask = (1u << (8 + pk)) - 1u;  // q's bits inside a bucket
        const uint32_t *y = Y + 3u * (32u * c0 + lane);
        uint32_t q0 = sub_key(bswap32(y[1]), bswap32(y[2]), pk);
        for (uint32_t c = c0; c < c1; ++c) {
            const uint32_t r = 32u * c + lane;
            y += 96;
            const uint32_t q1 = sub_key(bswap32(y[1]), bswap32(y[2]), pk);
            const uint32_t lim = global ? Dq : min(Dq, (~q0 & bmask) + 1u);  // at most to the bucket's end
            auto diff = [&](uint32_t t) -> uint32_t {  // q of record r + t, less q_r (t < 32)
                return __shfl_sync(0xffffffffu, lane < t ? q1 : q0, (lane + t) & 31u) - q0;
            };
            uint32_t df[5];
#pragma unroll
            for (int t = 1; t <= 5; ++t) df[t - 1] = diff(t);
            const bool m1 = df[0] < lim, m2 = m1 && df[1] < lim, m3 = m2 && df[2] < lim, m4 = m3 && df[3] < lim,
                       m5 = m4 && df[4] < lim;
            uint32_t cnt = m5 ? 5u : m4 ? 4u : m3 ? 3u : m2 ? 2u : m1 ? 1u : 0u;
            // the nearest record that is no sure match
            uint32_t dn = m4 ? df[4] : m3 ? df[3] : m2 ? df[2] : m1 ? df[1] : df[0];
            // records after r (none to count for r past the partition)
            const int after = HALO ? (r < n ? (int)(nt - 1u - r) : 0) : (int)(n - 1u - r);
            const bool edge = global && nt > n && q0 <= Dq + 1u && r + 32u >= n;
            if (__any_sync(0xffffffffu, (m5 || edge || dn - Dq <= 1u) && after > 0)) {
                bool more = m5 && after > 0;
                for (uint32_t t = 6; __any_sync(0xffffffffu, more) && t < 32; ++t) {
                    const uint32_t x = diff(t);
                    dn = more ? x : dn;
                    more = more && x < lim;
                    cnt += more ? 1u : 0u;
                }
                if ((more || edge || dn - Dq <= 1u) && after > 0) cnt = count_exact(r);
            }
            enlist(c, min(cnt, (uint32_t)max(after, 0)));
            q0 = q1;
        }
    }
    if (lane == 0) A.WS[warp] = mine;
    if (MODE != kSortCount && !fits) A.WS[kWsLong] = 1u;
    __syncthreads();
    uint32_t P = 0, wbase = 0;  // the partition's pairs; those before this warp's chunks
#pragma unroll
    for (uint32_t w = 0; w < NW; ++w) {
        const uint32_t t = A.WS[w];
        wbase += w < warp ? t : 0u;
        P += t;
    }
    const bool withhold = (d.test_flags & 1u) != 0;
    if (threadIdx.x == 0) {
        d.pairs[f] = P;  // lets vx_match re-run the match alone
        if (EMIT) lb_publish(d.lb, f, P, withhold);
    }
    if (MODE == kSortCount) {
        __syncthreads();
        return;
    }
    // 4. the Table-2 base: the look-back (warp 0), or the partition's slot
    bool ok = true;
    uint64_t base = 0;
    if (EMIT) {
        if (threadIdx.x < 32) {
            uint64_t excl = 0;
            int got = lb_resolve(d.lb, f, P, d.status, d.spin_limit, withhold, &excl) ? 1 : 0;
            if (threadIdx.x == 0) {
                if (got) {
                    const uint64_t np = 1ull << d.p;
                    d.t2off[f] = excl;
                    if (f + 1 == np) d.t2off[np] = d.totals[0] = excl + P;
                    if (excl + P > d.t2cap) {
                        atomicOr(d.status, kStT2Capacity);
                        got = 0;
                    }
                }
                *s_base = excl;
                *s_ok = got;
            }
        }
        __syncthreads();
        ok = *s_ok != 0;
        base = *s_base;
    } else if (P > d.cap2 + d.cap2 / 2u) {
        if (threadIdx.x == 0 && !quiet) atomicOr(d.status, kStPairSlot);
        ok = false;
    }
    // 5. the pairs, in (i, j) order at their places: into the slot (key
    //    array, then nonce array), as records {a, b, 0, 0}, or hashed here
    uint4 *__restrict__ out = reinterpret_cast<uint4 *>(d.t2) + base;
    uint2 *__restrict__ pa = reinterpret_cast<uint2 *>(d.b_keys + (uint64_t)f * d.cap2);
    uint2 *__restrict__ pb = reinterpret_cast<uint2 *>(d.b_nonces + (uint64_t)f * d.cap2);
    const uint32_t capA = d.cap2;
    uint32_t g[16];
    if (MODE == kSortHash) {
#pragma unroll
        for (int i = 0; i < 16; ++i) g[i] = d.pre2[i];
    }
    auto put = [&](uint32_t x, uint32_t a, uint32_t b) {
        if (SLOTS) {
            *(x < capA ? pa + x : pb + (x - capA)) = make_uint2(a, b);
        } else {
            uint32_t h0 = 0, h1 = 0;
            if (MODE == kSortHash) b3_finish<true>(g, a, b, h0, h1);
            out[x] = make_uint4(a, b, h0, h1);
        }
    };
    if (ok && A.WS[kWsLong] == 0u) {  // from the warp's list, a pair per lane
        const uint32_t *const y0 = Y + 3u * 32u * c0;
        if (SLOTS && P <= capA) {
            uint2 *__restrict__ w = pa + wbase;
#pragma unroll 2
            for (uint32_t x = lane; x < mine; x += 32) {
                const uint32_t e = list[x];
                const uint32_t i = e & 0xFFFu, j = i + (e >> 12);
                w[x] = make_uint2(y0[3u * i], y0[3u * j]);
            }
        } else {
            for (uint32_t x = lane; x < mine; x += 32) {
                const uint32_t e = list[x];
                const uint32_t i = e & 0xFFFu, j = i + (e >> 12);
                put(wbase + x, y0[3u * i], y0[3u * j]);
            }
        }
    } else if (ok) {
        uint32_t at = wbase;
        for (uint32_t c = c0; c < c1; ++c) {
            const uint32_t r = 32u * c + lane;
            const uint32_t cnt = r < n ? count_exact(r) : 0u;
            const uint32_t incl = warp_incl_scan(cnt);
            const uint32_t o = at + incl - cnt;
            at += __shfl_sync(0xffffffffu, incl, 31);
            for (uint32_t j = 0; j < cnt; ++j) put(o + j, Y[3 * r], Y[3 * (r + 1 + j)]);
        }
    }
    __syncthreads();
}

// The arrays of a partition with a W-word bitmap; tables: SMLayout's bytes
// for the bitmap and the lists.
template <int NT>
__device__ __forceinline__ Part part_arrays(unsigned char *base, const SMLayout &L, uint32_t W, uint32_t tables)
{
    Part A;
    A.Y = reinterpret_cast<uint32_t *>(base + L.y);
    A.BM = reinterpret_cast<uint32_t *>(base + L.bm);
    A.PF = reinterpret_cast<uint16_t *>(A.BM + W);
    A.PL = reinterpret_cast<uint16_t *>(A.BM);
    A.plw = tables / 2u / (NT / 32);
    A.DL = reinterpret_cast<uint16_t *>(base + L.dl);
    A.WS = reinterpret_cast<uint32_t *>(base + L.ws);
    return A;
}

// A slot in shared memory.
struct SharedSrc {
    const uint64_t *k;
    const uint32_t *n;
    __device__ __forceinline__ uint64_t key(uint32_t i) const { return k[i]; }
    __device__ __forceinline__ uint32_t nonce(uint32_t i) const { return n[i]; }
};

// A slot in global memory, read through the read-only path unless this
// kernel later overwrites it with the partition's pairs (RO false).
template <bool RO>
struct GlobalSrc {
    const uint64_t *k;
    const uint32_t *n;
    __device__ __forceinline__ uint64_t key(uint32_t i) const { return RO ? __ldg(k + i) : k[i]; }
    __device__ __forceinline__ uint32_t nonce(uint32_t i) const { return RO ? __ldg(n + i) : n[i]; }
};

// ------------------------------------------------- persistent front end
// CTA b starts with work item b of the launch and takes the next ones from a
// counter (the first plot's ticket_i of the launch's chunk), so that all end
// together, also when a CTA starts late: CTAs of a dependent launch come onto
// an SM as the kernel before leaves it, in whatever shared memory is free, so
// that a few SMs host two instead of three and the CTAs left over start when
// the others end (K=28, taking b, b + G, b + 2G, ...: two of 456, a sort of
// 5.0 ms instead of 3.0).  Where all start together it evens out the end:
// K=26 0.75 -> 0.72 ms, K=31 24.2 -> 22.8 ms.  Item t belongs to plot find_plot(t); its partition
// is the plot's next ticket (look-back modes) or t - tile_start[plot].  A CTA
// takes its items two ahead (look-back modes: three, with the ticket of the
// second and the fill count of the first read at the start of an item) and
// starts item k + 1's slot copy once item k's records have been placed, so
// the global round trips and the copy overlap item k's match.
// A CTA takes tickets in its processing order and only while running, so
// the lowest unpublished partition is always being worked on: the
// look-back chain cannot stall on a CTA that is not resident.
struct Item {
    int plot;
    uint32_t f;
    bool ok;
};

// Starts an L2 prefetch of the filled part of partition f's slot (f below
// 2^p), so that the reads that come for it later hit L2.  (Two items ahead
// in the persistent front end it measured 1% slower: its bulk copies do not
// wait on DRAM latency.)
__device__ __forceinline__ void prefetch_slot_l2(const Desc &d, uint32_t f)
{
    const uint32_t nf = min(d.cnt2[f], d.cap2);
    if (!nf) return;
    const uint32_t nk = (nf + 1u) & ~1u, nn = (nf + 3u) & ~3u;  // 16-byte multiples
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(d.b_keys + (uint64_t)f * d.cap2),
                 "r"(nk * 8u)
                 : "memory");
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(d.b_nonces + (uint64_t)f * d.cap2),
                 "r"(nn * 4u)
                 : "memory");
}

template <bool EMIT>
__device__ __forceinline__ Item take_item(const Desc *__restrict__ descs, int nplots,
                                          const uint32_t *__restrict__ tile_start, uint32_t t)
{
    Item it;
    it.plot = find_plot(tile_start, nplots, t);
    const Desc &d = descs[it.plot];
    it.f = EMIT ? atomicAdd(d.ticket, 1u) : t - __ldg(tile_start + it.plot);
    it.ok = true;
    return it;
}

template <int MODE, bool HALO>
__global__ void __launch_bounds__(kPipeThreads, MODE == kSortHash ? 2 : 3)
    k_sortmatch_pipe(const Desc *__restrict__ descs, int nplots, const uint32_t *__restrict__ tile_start,
                     uint32_t items, uint32_t max_cap, uint32_t max_words, bool quiet, int chunk)
{
    constexpr bool EMIT = MODE == kSortHash || MODE == kSortEmit;
    constexpr int NT = kPipeThreads;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int s_plot;
    __shared__ uint32_t s_f, s_n;
    __shared__ int s_valid, s_more;
    __shared__ uint64_t s_base;
    __shared__ int s_ok;
    const SMLayout L(max_cap, max_words, true);
    Part A = part_arrays<NT>(smem_raw, L, max_words, (uint32_t)(L.dl - L.bm));
    uint32_t *const Y0 = A.Y;
    uint64_t *const XK = reinterpret_cast<uint64_t *>(smem_raw + L.xk);
    uint32_t *const XN = reinterpret_cast<uint32_t *>(smem_raw + L.xn);
    uint64_t *bar = reinterpret_cast<uint64_t *>(smem_raw + L.bar);
    const uint32_t G = gridDim.x;
    pdl_go();
    pdl_wait();

    // Thread 0's pipeline: the item after the current one (from the start of
    // the current item on with its fill count), in the look-back modes the one
    // after that, and the number of the next.
    Item nx{0, 0, false}, nn{0, 0, false};
    uint32_t nx_n = 0, nt = items;
    auto next_number = [&]() {
        if (nt < items) nt = G + atomicAdd(descs->ticket_i + chunk, 1u);
    };
    auto take = [&]() {  // item nt; its successor's number is on its way
        Item it{0, 0, false};
        if (nt < items) it = take_item<EMIT>(descs, nplots, tile_start, nt);
        next_number();
        return it;
    };
    // Starts the copy of item `it` (n records) into X and publishes it as
    // the next item; an invalid or empty item completes the barrier phase
    // with no copy.
    auto launch_copy = [&](const Item &it, uint32_t n) {
        // Only if the ticket was not reset: report, never index with it.
        const bool valid = it.ok && it.f < (1u << descs[it.plot].p);
        if (it.ok && !valid) atomicOr(descs[it.plot].status, kStBadTicket);
        const uint32_t cnt = valid ? n : 0u;
        const uint32_t nk = (cnt + 1u) & ~1u, nnz = (cnt + 3u) & ~3u;  // 16-byte multiples
        // X was last accessed by ordinary loads: order those before the
        // copy engine's writes.
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        mbar_expect_tx(bar, nk * 8u + nnz * 4u);
        if (cnt) {
            const Desc &d = descs[it.plot];
            bulk_g2s(XK, d.b_keys + (uint64_t)it.f * d.cap2, nk * 8u, bar);
            bulk_g2s(XN, d.b_nonces + (uint64_t)it.f * d.cap2, nnz * 4u, bar);
        }
        s_plot = it.plot;
        s_f = it.f;
        s_n = cnt;
        s_valid = valid ? 1 : 0;
    };
    if (threadIdx.x == 0) {
        mbar_init(bar, 1);
        s_more = blockIdx.x < items ? 1 : 0;
        if (blockIdx.x < items) {
            const Item i0 = take_item<EMIT>(descs, nplots, tile_start, blockIdx.x);
            const uint32_t n0 = i0.f < (1u << descs[i0.plot].p) ? descs[i0.plot].cnt2[i0.f] : 0u;
            nt = 0;
            next_number();
            if (EMIT) nx = take();
            launch_copy(i0, min(n0, descs[i0.plot].cap2));
        }
    }
    __syncthreads();
    uint32_t phase = 0;
    for (; s_more; phase ^= 1u) {
        const int plot = s_plot;
        const uint32_t f = s_f, n = s_n;
        const bool valid = s_valid != 0;
        const Desc &d = descs[plot];
        const uint32_t W = bitmap_words(d.dbits);
        A.PF = reinterpret_cast<uint16_t *>(A.BM + W);
        clear_tables<NT>(A, W);
        const uint64_t off = valid ? d.t1off[f] : 0ull;
        if (threadIdx.x == 0) {
            if (!EMIT) nx = take();
            if (nx.ok) {
                const Desc &dn = descs[nx.plot];
                nx_n = nx.f < (1u << dn.p) ? min(dn.cnt2[nx.f], dn.cap2) : 0u;
            }
            if (EMIT) nn = take();
        }
        // The slot copy was started during the previous item (or above).
        if (!__syncthreads_and(mbar_wait(bar, phase, d.spin_limit))) {
            if (threadIdx.x == 0) {
                atomicOr(d.status, kStTimeout);
                bulk_wait_all<false>();
            }
            mbar_wait(bar, phase, d.spin_limit);  // let it land before the CTA exits
            return;
        }
        // The next item's copy starts once this slot has been placed in Y.
        auto start_next = [&]() {
            if (nx.ok)
                launch_copy(nx, nx_n);
            else
                s_more = 0;
            nx = nn;
        };
        if (valid) {
            A.Y = Y0 + ((uint32_t)(3 * off) & 3u);
            sort_bitmap<NT>(
                A, n, d.pk, W, SharedSrc{XK, XN},
                [&]() { bulk_wait_all<true>(); },  // the previous item's Table 1 has left Y
                start_next);
            match_and_write<MODE, HALO, NT>(d, f, n, off, A, &s_base, &s_ok, quiet);
        } else {
            __syncthreads();
            if (threadIdx.x == 0) start_next();
            __syncthreads();
        }
    }
    if (threadIdx.x == 0) bulk_wait_all<false>();
}

// ------------------------------------- one CTA per partition front end
template <int MODE, bool HALO>
__global__ void __launch_bounds__(kGlThreads, MODE == kSortHash ? 2 : 3)
    k_sortmatch_gl(const Desc *__restrict__ descs, int nplots, const uint32_t *__restrict__ tile_start, bool quiet)
{
    constexpr bool EMIT = MODE == kSortHash || MODE == kSortEmit;
    constexpr int NT = kGlThreads;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ uint32_t s_f;
    __shared__ uint64_t s_base;
    __shared__ int s_ok;
    pdl_go();
    pdl_wait();
    const int plot = find_plot(tile_start, nplots, blockIdx.x);
    const Desc &d = descs[plot];
    if (EMIT) {
        if (threadIdx.x == 0) s_f = atomicAdd(d.ticket, 1u);
        __syncthreads();
    }
    const uint32_t f = EMIT ? s_f : (blockIdx.x - tile_start[plot]);
    if (f >= (1u << d.p)) {  // only if the ticket was not reset: report, never index with it
        if (threadIdx.x == 0) atomicOr(d.status, kStBadTicket);
        return;
    }
    const uint32_t cap = d.cap2;
    const uint32_t W = bitmap_words(d.dbits);
    const SMLayout L(cap + (HALO ? d.hcap : 0u), W, false);
    Part A = part_arrays<NT>(smem_raw, L, W, (uint32_t)(L.dl - L.bm));
    clear_tables<NT>(A, W);
    // Warm L2 with the filled part of the slot kSlotPrefetchAhead tickets
    // ahead, so that its CTA's reads hit L2.
    const uint64_t fa = (uint64_t)f + kSlotPrefetchAhead;
    if (threadIdx.x == 0 && fa < (1ull << d.p)) prefetch_slot_l2(d, (uint32_t)fa);
    const uint32_t n = min(d.cnt2[f], cap);
    const uint64_t off = d.t1off[f];
    A.Y += (uint32_t)(3 * off) & 3u;
    __syncthreads();
    sort_bitmap<NT>(
        A, n, d.pk, W,
        GlobalSrc<MODE != kSortSlots>{d.b_keys + (uint64_t)f * cap, d.b_nonces + (uint64_t)f * cap}, []() {},
        []() {});
    match_and_write<MODE, HALO, NT>(d, f, n, off, A, &s_base, &s_ok, quiet);
    if (threadIdx.x == 0) bulk_wait_all<false>();
}

// What the planner admits a slot by: the layout of k_sortmatch_gl, the smaller
// front end, or 16 bytes a record (at least 4 * 2^dbits for the last four) and
// 8 KB, the sort's need when the limits were set, whichever is more.  The
// second decides near the limit (cap 14004, 13 bits: 232,424 bytes against
// 224,888 of a CTA's 232,448), so what was refused stays refused; the first
// is more in the middle (cap 9296, 13 bits: 161,016 against 157,096).
size_t sortmatch_smem_bytes(uint32_t cap, int dbits)
{
    const size_t gl = SMLayout(cap, bitmap_words(dbits), false).bytes;
    cap = (cap + 3u) & ~3u;
    const size_t digits = (size_t)4 << dbits, recs = (size_t)cap * 4;
    const size_t limit = (size_t)cap * 12 + (digits > recs ? digits : recs) + 8192 + 168;
    return gl > limit ? gl : limit;
}

uint32_t sortmatch_max_cap() { return 16384u; }

template <int MODE, bool HALO>
static cudaError_t launch_sm(const Desc *descs, int nplots, const uint32_t *tile_start,
                             uint32_t total_tiles, On on, uint32_t max_cap, int max_dbits, bool quiet,
                             int chunk)
{
    if (total_tiles == 0) return cudaSuccess;
    const uint32_t words = bitmap_words(max_dbits);
    const size_t pipe = SMLayout(max_cap, words, true).bytes;
    if (pipe <= kMaxSmemPerCta) {
        auto fn = k_sortmatch_pipe<MODE, HALO>;
        static SmemSeen seen;
        // (shared memory, CTAs that fit the device at once) of the last
        // launch on each device: asking again costs as much as a launch
        static std::atomic<uint64_t> fits[kMaxDevices];
        cudaError_t e = allow_smem(fn, pipe, seen);
        if (e != cudaSuccess) return e;
        int dev = 0, sms = 0, per_sm = 0;
        if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
        const bool known = dev >= 0 && dev < kMaxDevices;
        uint64_t fit = known ? fits[dev].load(std::memory_order_acquire) : 0ull;
        if (fit >> 32 != pipe) {
            if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
            if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, kPipeThreads, pipe)) != cudaSuccess)
                return e;
            fit = (uint64_t)pipe << 32 | (uint64_t)((per_sm > 0 ? per_sm : 1) * sms);
            if (known) fits[dev].store(fit, std::memory_order_release);
        }
        const uint32_t want = (uint32_t)fit;
        return launch_on(on, fn, want < total_tiles ? want : total_tiles, kPipeThreads, pipe, descs, nplots,
                         tile_start, total_tiles, max_cap, words, quiet, chunk);
    }
    const size_t smem = SMLayout(max_cap, words, false).bytes;
    auto fn = k_sortmatch_gl<MODE, HALO>;
    static SmemSeen seen_gl;
    const cudaError_t e = allow_smem(fn, smem, seen_gl);
    if (e != cudaSuccess) return e;
    return launch_on(on, fn, total_tiles, kGlThreads, smem, descs, nplots, tile_start, quiet);
}

template <int MODE>
static cudaError_t launch_sm2(const Desc *descs, int nplots, const uint32_t *tile_start,
                              uint32_t total_tiles, On on, uint32_t max_cap, int max_dbits,
                              bool halo, bool quiet, int chunk)
{
    // HALO instances carry the cross-bucket code; plain launches do not.
    return halo ? launch_sm<MODE, true>(descs, nplots, tile_start, total_tiles, on, max_cap, max_dbits, quiet,
                                         chunk)
                : launch_sm<MODE, false>(descs, nplots, tile_start, total_tiles, on, max_cap, max_dbits, quiet,
                                          chunk);
}

cudaError_t launch_sortmatch(const Desc *descs, int nplots, const uint32_t *tile_start,
                             uint32_t total_tiles, On on, uint32_t max_cap, int max_dbits,
                             SortMatchOut out, bool halo, bool quiet, int chunk)
{
    if (out == kOutLookbackHashed)
        return launch_sm2<kSortHash>(descs, nplots, tile_start, total_tiles, on, max_cap, max_dbits, halo, false,
                                      chunk);
    if (out == kOutSlots)
        return launch_sm2<kSortSlots>(descs, nplots, tile_start, total_tiles, on, max_cap, max_dbits, halo, quiet,
                                       chunk);
    return launch_sm2<kSortEmit>(descs, nplots, tile_start, total_tiles, on, max_cap, max_dbits, halo, false, chunk);
}

cudaError_t launch_sort(const Desc *descs, int nplots, const uint32_t *tile_start,
                        uint32_t total_tiles, On on, uint32_t max_cap, int max_dbits,
                        bool halo)
{
    return launch_sm2<kSortCount>(descs, nplots, tile_start, total_tiles, on, max_cap, max_dbits, halo, false, 0);
}

}  // namespace vx
