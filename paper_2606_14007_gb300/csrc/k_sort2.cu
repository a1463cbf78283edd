// k_sort2.cu -- Table 2 sorted by its hash (hash2), for lookups by a prover.
//
// Paper: a plot is searched by hash value (Sec. I-B, the VaultX prover); the
// paper's Table 2 stays in pair order.  This pass orders the same 16-byte
// records {a, b, hash2} by (key2, a, b), key2 = big-endian u64 of hash2,
// with the Table-1 machinery applied to 16-byte records: a first scatter
// level by the top p1 bits of key2, a second level by the next p2 bits into
// 2^p Poisson-sized partitions, a scan of the partition counts, and a
// shared-memory sort of every partition (ranks by a digit bitmap of the next
// key bits) that writes its records straight back into the Table-2 buffer at
// their places.  Table 2 is read completely by the first level before
// anything writes it.
#include "bitmap_sort.cuh"
#include "vx_internal.cuh"
#include "vx_plan.h"

namespace vx {

constexpr int kS2Threads = 512;              // both levels: 512 threads x 8 records
constexpr uint32_t kS2Tile = 4096;
static_assert(kS2Tile == kPlanS2Tile1, "planner and scatter tiles differ");
constexpr int kS2SortThreads = 256;

__device__ __forceinline__ uint64_t sort2_key(uint4 r)
{
    return ((uint64_t)bswap32(r.z) << 32) | bswap32(r.w);
}

// ------------------------------------------------------------------ setup
__global__ void k_s2_setup(Sort2Desc *dp)
{
    pdl_go();
    Sort2Desc &d = *dp;
    const uint64_t n1 = d.p2 > 0 ? (1ull << d.p1) : 0ull;
    const uint64_t n2 = 1ull << d.p;
    const uint64_t nchunks = (n2 + kScanChunk - 1) / kScanChunk;
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    if (blockIdx.x == 0 && threadIdx.x == 0) *d.ticket = *d.status = 0u;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n2; i += stride) {
        d.cnt2[i] = 0u;
        if (i < n1) d.cnt1[i] = 0u;
        if (i < nchunks) d.lbs[i] = 0ull;
    }
}

// ------------------------------------------------------- scatter levels
// A CTA takes a tile of up to kS2Tile records (level 1: of Table 2, level 2:
// of a first-level slot) by one bulk copy, ranks them by their bin, claims
// one run per (CTA, bin) with a global atomic (its result first needed after
// the order is known), and writes the records bin by bin.  Bound by shared
// memory (90% of its wavefronts, most of them the random 16-byte reads on
// the way out), close to HBM: 58.7 M records take 299 and 307 us, 6.3 TB/s
// (543 and 380 with keys and pairs in arrays of their own, held in registers
// over an in-place restage: two CTAs per SM, the first level's loads one
// after the other).  The records stay where the copy left them: a 16-bit
// order says which one goes next, so no registers hold them and three CTAs
// fit an SM up to 9 bits, with the bin counters sized to the level.
struct S2ScatterLayout {
    size_t order, hist, ws, bar, bytes;
    __host__ __device__ explicit S2ScatterLayout(int bits)
    {
        order = (size_t)kS2Tile * 16;
        hist = order + (size_t)kS2Tile * 2;
        ws = hist + ((size_t)4 << bits);
        bar = (ws + (kS2Threads / 32 + 1) * 4 + 7) & ~(size_t)7;
        bytes = bar + 8;
    }
};

template <int LEVEL>
__global__ void __launch_bounds__(kS2Threads, 3) k_s2_scatter(const Sort2Desc *__restrict__ dp)
{
    constexpr int NT = kS2Threads, PER = kS2Tile / NT;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    pdl_go();
    pdl_wait();
    const Sort2Desc &d = *dp;
    const bool last = LEVEL == 2 || d.p2 == 0;  // the level that fills the partitions
    const int bits = LEVEL == 2 ? d.p2 : last ? d.p : d.p1;
    const uint4 *src;
    uint64_t left, bin0 = 0;  // records from the tile on; first bin of the CTA
    if (LEVEL == 1) {
        const uint64_t n = d.count, base = (uint64_t)blockIdx.x * kS2Tile;
        if (base >= n) return;
        src = d.t2 + base;
        left = n - base;
    } else {
        const uint32_t c = blockIdx.x / d.chunks1, start = (blockIdx.x - c * d.chunks1) * kS2Tile;
        const uint32_t filled = min(d.cnt1[c], d.cap1);
        if (start >= filled) return;
        src = d.a_recs + (uint64_t)c * d.cap1 + start;
        left = filled - start;
        bin0 = (uint64_t)c << bits;
    }
    const uint32_t count = (uint32_t)(left < kS2Tile ? left : kS2Tile);
    const S2ScatterLayout L(bits);
    const uint4 *X = reinterpret_cast<const uint4 *>(smem_raw);
    uint16_t *order = reinterpret_cast<uint16_t *>(smem_raw + L.order);
    uint32_t *hist = reinterpret_cast<uint32_t *>(smem_raw + L.hist);
    uint32_t *ws = reinterpret_cast<uint32_t *>(smem_raw + L.ws);
    uint64_t *bar = reinterpret_cast<uint64_t *>(smem_raw + L.bar);
    if (threadIdx.x == 0) {
        mbar_init(bar, 1);
        mbar_expect_tx(bar, count * 16u);
        bulk_g2s(smem_raw, src, count * 16u, bar);
    }
    const int nbins = 1 << bits;
    // the bin: bits of the key's top 32 (d.p <= 20), below the first level's
    const int shift = 32 - (last ? d.p : d.p1);
    const uint32_t bin_mask = (uint32_t)nbins - 1u;
    auto bin_of = [&](uint32_t z) { return bits ? (bswap32(z) >> shift) & bin_mask : 0u; };
    for (int b = threadIdx.x; b < nbins; b += NT) hist[b] = 0u;
    __syncthreads();
    if (!__syncthreads_and(mbar_wait(bar, 0, d.spin_limit))) {  // one answer for all threads
        if (threadIdx.x == 0) atomicOr(d.status, kStTimeout);
        mbar_wait(bar, 0, d.spin_limit);  // let the copy land before leaving
        return;
    }
    uint32_t where[PER];  // bin << 16 | rank in the bin
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        const uint32_t i = (uint32_t)j * NT + threadIdx.x;
        where[j] = 0u;
        if (i < count) {
            const uint32_t bin = bin_of(X[i].z);
            where[j] = bin << 16 | atomicAdd(&hist[bin], 1u);
        }
    }
    __syncthreads();
    constexpr int PB = ((1 << kMaxCoarseBits) + NT - 1) / NT;  // most bins a thread owns
    const int per = (nbins + NT - 1) / NT;
    const int b0 = threadIdx.x * per;
    const uint32_t cap = last ? d.cap2 : d.cap1;
    uint32_t claim[PB];
    {
        uint32_t *cnt = (last ? d.cnt2 : d.cnt1) + bin0;
        uint32_t loc = 0;
        for (int k = 0; k < per; ++k)
            if (b0 + k < nbins) loc += hist[b0 + k];
        uint32_t total;
        uint32_t run = block_exclusive_scan_u32<NT>(loc, ws, &total);
#pragma unroll
        for (int k = 0; k < PB; ++k) {
            const int b = b0 + k;
            claim[k] = 0u;
            if (k < per && b < nbins) {
                const uint32_t h = hist[b];
                if (h) claim[k] = atomicAdd(&cnt[b], h);
                hist[b] = run;
                run += h;
            }
        }
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        const uint32_t i = (uint32_t)j * NT + threadIdx.x;
        if (i < count) order[hist[where[j] >> 16] + (where[j] & 0xFFFFu)] = (uint16_t)i;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < PB; ++k)
        if (k < per && b0 + k < nbins) hist[b0 + k] = claim[k] - hist[b0 + k];  // run's start less its order index
    __syncthreads();
    uint4 *__restrict__ out = (last ? d.b_recs : d.a_recs) + bin0 * cap;
    bool overflow = false;
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        const uint32_t q = (uint32_t)j * NT + threadIdx.x;
        if (q >= count) break;
        const uint4 r = X[order[q]];
        const uint32_t bin = bin_of(r.z);
        const uint32_t g = hist[bin] + q;
        if (g < cap)
            out[(uint64_t)bin * cap + g] = r;
        else
            overflow = true;
    }
    if (overflow) atomicOr(d.status, kStSort2);
}

// --------------------------------------------------------- offsets scan
// Exclusive prefix of the 2^p partition counts (clipped to the slot), 4096
// counters per CTA, chunks chained by decoupled look-back in ticket order;
// the last chunk checks that every record arrived.
__global__ void __launch_bounds__(256) k_s2_scan(const Sort2Desc *__restrict__ dp)
{
    constexpr int NT = 256;
    constexpr uint32_t PER = kScanChunk / NT;
    __shared__ uint32_t ws[NT / 32 + 1];
    __shared__ uint32_t s_c;
    __shared__ uint64_t s_base;
    __shared__ int s_ok;
    pdl_go();
    pdl_wait();
    const Sort2Desc &d = *dp;
    if (threadIdx.x == 0) s_c = atomicAdd(d.ticket, 1u);
    __syncthreads();
    const uint32_t c = s_c;
    const uint64_t np = 1ull << d.p;
    const uint32_t nchunks = (uint32_t)((np + kScanChunk - 1) / kScanChunk);
    if (c >= nchunks) {
        if (threadIdx.x == 0) atomicOr(d.status, kStBadTicket);
        return;
    }
    const uint64_t b0 = (uint64_t)c * kScanChunk + (uint64_t)threadIdx.x * PER;
    uint32_t v[PER];
    uint32_t loc = 0;
#pragma unroll
    for (uint32_t k = 0; k < PER; ++k) {
        v[k] = b0 + k < np ? min(d.cnt2[b0 + k], d.cap2) : 0u;
        loc += v[k];
    }
    uint32_t total;
    const uint32_t run = block_exclusive_scan_u32<NT>(loc, ws, &total);
    if (threadIdx.x < 32) {
        uint64_t excl = 0;
        const int ok = lookback_warp(d.lbs, c, total, d.status, d.spin_limit, false, &excl) ? 1 : 0;
        if (threadIdx.x == 0) {
            s_ok = ok;
            s_base = excl;
        }
    }
    __syncthreads();
    if (!s_ok) return;
    uint64_t at = s_base + run;
#pragma unroll
    for (uint32_t k = 0; k < PER; ++k) {
        if (b0 + k < np) d.off[b0 + k] = at;
        at += v[k];
    }
    if (c + 1 == nchunks && threadIdx.x == 0) {
        const uint64_t all = s_base + total;
        d.off[np] = all;
        if (all != d.count) atomicOr(d.status, kStSort2);
    }
}

// ------------------------------------------------------- partition sort
// One CTA per partition, its slot brought into shared memory by one bulk
// copy.  The records stay there: a digit bitmap ranks them as in Table 1's
// sort, a 16-bit order takes their indices, the few words with a shared digit
// are put in order by (key2, a, b), and the records leave in that order as
// whole 16-byte words at the partition's offset.  Bound by shared memory (73%
// of its wavefronts) and the wait for the slot: 58.7 M records take 449 us
// (502 with a counting sort and every record ranked in its digit run by
// shuffles, 7.3 instructions a record).  512 threads a CTA, or five CTAs of
// half the digits, measured 5 to 10% slower.
constexpr uint32_t kS2PrefetchAhead = 384;  // partitions ahead: ~half the resident CTAs

// Twice the digits of Table 1's sort for the same dbits: a partition holds
// 2^dbits to 2^(dbits + 1) records.
__host__ __device__ __forceinline__ uint32_t sort2_words(int dbits) { return bitmap_words(dbits + 1); }

struct S2SortLayout {
    size_t bm, order, dl, ws, bar, bytes;
    __host__ __device__ S2SortLayout(uint32_t cap, uint32_t words)
    {
        bm = (size_t)cap * 16;
        order = bm + (size_t)words * 6;
        dl = (order + (size_t)cap * 2 + 3) & ~(size_t)3;
        ws = dl + (size_t)kDirtyList * 2;
        bar = (ws + 40 * 4 + 7) & ~(size_t)7;
        bytes = bar + 8;
    }
};

// Puts the dirty words' indices in the order of their records: eight lanes a
// listed word, a lane per record; words with more than eight records or past
// the list by one thread's insertion sort.
template <int NT>
__device__ __forceinline__ void order_dirty_indices(const Bitmap &A, uint32_t W, const uint4 *X, uint16_t *order)
{
    constexpr uint32_t NW = NT / 32;
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    auto less = [](const uint4 &p, const uint4 &q) {
        const uint64_t kp = sort2_key(p), kq = sort2_key(q);
        return kp < kq || (kp == kq && (p.x < q.x || (p.x == q.x && p.y < q.y)));
    };
    auto order_word = [&](uint32_t w) {
        uint16_t *const o = order + (A.PF[w] & (kDirty - 1u));
        const uint32_t cnt = A.BM[w];
        for (uint32_t a = 1; a < cnt; ++a) {
            const uint16_t ix = o[a];
            const uint4 r = X[ix];
            uint32_t b = a;
            for (; b > 0 && less(r, X[o[b - 1]]); --b) o[b] = o[b - 1];
            o[b] = ix;
        }
    };
    const uint32_t nd = A.WS[kWsDirty];
    if (nd > kDirtyList) {
        for (uint32_t w = threadIdx.x; w < W; w += NT)
            if (A.PF[w] & kDirty) order_word(w);
        return;
    }
    const uint32_t sub = lane & 7u;
    for (uint32_t i0 = 4u * warp; i0 < nd; i0 += 4u * NW) {
        const uint32_t i = i0 + (lane >> 3);
        const uint32_t w = i < nd ? A.DL[i] : 0u;
        uint16_t *const o = order + (A.PF[w] & (kDirty - 1u));
        const uint32_t all = i < nd ? A.BM[w] : 0u;
        const uint32_t cnt = all <= 8u ? all : 0u;
        const bool mine = sub < cnt;
        const uint32_t ix = mine ? o[sub] : 0u;
        const uint4 r = X[ix];
        const uint32_t most = __reduce_max_sync(0xffffffffu, cnt);
        uint32_t place = 0;
        for (uint32_t t = 0; t < most; ++t) {
            const uint32_t other = __shfl_sync(0xffffffffu, ix, (int)((lane & 24u) + t));
            place += t < cnt && less(X[other], r) ? 1u : 0u;
        }
        if (mine) o[place] = (uint16_t)ix;
        if (all > 8u && sub == 0) order_word(w);
    }
}

__global__ void __launch_bounds__(kS2SortThreads, 4) k_s2_sort(const Sort2Desc *__restrict__ dp)
{
    constexpr int NT = kS2SortThreads;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    pdl_go();
    pdl_wait();
    const Sort2Desc &d = *dp;
    if (*d.status & (kStSort2 | kStTimeout | kStBadTicket)) return;  // offsets not trusted
    const uint32_t f = blockIdx.x;
    const uint32_t cap = d.cap2;
    const uint32_t n = min(d.cnt2[f], cap);
    if (n == 0) return;
    const uint32_t W = sort2_words(d.dbits);
    const S2SortLayout L(cap, W);
    const uint4 *X = reinterpret_cast<const uint4 *>(smem_raw);
    uint16_t *order = reinterpret_cast<uint16_t *>(smem_raw + L.order);
    uint64_t *bar = reinterpret_cast<uint64_t *>(smem_raw + L.bar);
    Bitmap A;
    A.BM = reinterpret_cast<uint32_t *>(smem_raw + L.bm);
    A.PF = reinterpret_cast<uint16_t *>(A.BM + W);
    A.DL = reinterpret_cast<uint16_t *>(smem_raw + L.dl);
    A.WS = reinterpret_cast<uint32_t *>(smem_raw + L.ws);
    if (threadIdx.x == 0) {
        mbar_init(bar, 1);
        mbar_expect_tx(bar, n * 16u);
        bulk_g2s(smem_raw, d.b_recs + (uint64_t)f * cap, n * 16u, bar);
    }
    // the filled part of the slot kS2PrefetchAhead partitions ahead goes to L2
    const uint64_t fa = (uint64_t)f + kS2PrefetchAhead;
    if (threadIdx.x == 0 && fa < (1ull << d.p)) {
        const uint32_t nfa = min(d.cnt2[fa], cap);
        if (nfa)
            asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(d.b_recs + fa * cap), "r"(nfa * 16u)
                         : "memory");
    }
    const uint64_t o = d.off[f];
    clear_tables<NT>(A, W);
    __syncthreads();
    if (!__syncthreads_and(mbar_wait(bar, 0, d.spin_limit))) {  // one answer for all threads
        if (threadIdx.x == 0) atomicOr(d.status, kStTimeout);
        mbar_wait(bar, 0, d.spin_limit);  // let the copy land before leaving
        return;
    }
    // log2(W) + 5 bits below the partition prefix
    const int shift = 64 - d.p - (36 - __clz(W));
    const uint32_t dmask = 32u * W - 1u;
    auto digit = [&](uint32_t i) {
        const uint2 h = *reinterpret_cast<const uint2 *>(&X[i].z);
        return (uint32_t)((((uint64_t)bswap32(h.x) << 32) | bswap32(h.y)) >> shift) & dmask;
    };
    constexpr int KEEP = 8;  // digits a thread keeps from the marking to the placing (2048 records)
    uint32_t dg[KEEP];
#pragma unroll
    for (int j = 0; j < KEEP; ++j) {
        const uint32_t i = threadIdx.x + (uint32_t)j * NT;
        if (i < n) mark(A, dg[j] = digit(i));
    }
    for (uint32_t i = threadIdx.x + KEEP * NT; i < n; i += NT) mark(A, digit(i));
    __syncthreads();
    scan_words<NT>(A, W);
    __syncthreads();
#pragma unroll
    for (int j = 0; j < KEEP; ++j) {
        const uint32_t i = threadIdx.x + (uint32_t)j * NT;
        if (i < n) order[place_of(A, dg[j])] = (uint16_t)i;
    }
    for (uint32_t i = threadIdx.x + KEEP * NT; i < n; i += NT) order[place_of(A, digit(i))] = (uint16_t)i;
    __syncthreads();
    order_dirty_indices<NT>(A, W, X, order);
    __syncthreads();
    uint4 *__restrict__ out = d.t2 + o;
#pragma unroll 4
    for (uint32_t i = threadIdx.x; i < n; i += NT) out[i] = X[order[i]];
}

size_t sort2_smem_bytes(uint32_t cap, int dbits) { return S2SortLayout(cap, sort2_words(dbits)).bytes; }

cudaError_t launch_sort2(const Sort2Desc *d_desc, const Sort2Launch &g, cudaStream_t s)
{
    static SmemSeen seen1, seen2, seen3;
    // One level (under 2^21 records), bound by the chain of launches: each
    // kernel a programmatic dependent of the one before (K=16 35.9 -> 33.0 us,
    // K=20 47.5 -> 42.0).  Two levels gain as much or lose (K=26 1092 -> 1087
    // us, K=28 4.80 -> 4.94 ms: CTAs of the next kernel take the places of the
    // last ones of this), so those launch plainly.
    const On on(s, g.tiles2 == 0);
    cudaError_t e;
    k_s2_setup<<<64, 256, 0, s>>>(const_cast<Sort2Desc *>(d_desc));
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if (g.tiles1) {
        const size_t sm = S2ScatterLayout(g.p - g.p2).bytes;
        if ((e = allow_smem(k_s2_scatter<1>, sm, seen1)) != cudaSuccess) return e;
        if ((e = launch_on(on, k_s2_scatter<1>, g.tiles1, kS2Threads, sm, d_desc)) != cudaSuccess) return e;
    }
    if (g.tiles2) {
        const size_t sm = S2ScatterLayout(g.p2).bytes;
        if ((e = allow_smem(k_s2_scatter<2>, sm, seen2)) != cudaSuccess) return e;
        if ((e = launch_on(on, k_s2_scatter<2>, g.tiles2, kS2Threads, sm, d_desc)) != cudaSuccess) return e;
    }
    if ((e = launch_on(on, k_s2_scan, g.tiles_scan, 256, 0, d_desc)) != cudaSuccess) return e;
    const size_t sm = sort2_smem_bytes(g.cap2, g.dbits);
    if ((e = allow_smem(k_s2_sort, sm, seen3)) != cudaSuccess) return e;
    return launch_on(on, k_s2_sort, g.parts, kS2SortThreads, sm, d_desc);
}

}  // namespace vx
