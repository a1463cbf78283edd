// k_sort2.cu -- Table 2 sorted by its hash (hash2), for lookups by a prover.
//
// Paper: a plot is searched by hash value (Sec. I-B, the VaultX prover); the
// paper's Table 2 stays in pair order.  This pass orders the same 16-byte
// records {a, b, hash2} by (key2, a, b), key2 = big-endian u64 of hash2,
// with the Table-1 machinery applied to 16-byte records: a first scatter
// level by the top p1 bits of key2, a second level by the next p2 bits into
// 2^p Poisson-sized partitions, a scan of the partition counts, and a
// shared-memory sort of every partition (counting sort on the next
// dbits + 1 key bits, each record ranked inside its digit run by warp
// shuffles) that writes its records straight back into the Table-2 buffer
// at their places.  Table 2 is read completely by
// the first level before anything writes it.
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
    Sort2Desc &d = *dp;
    const uint64_t n1 = d.p2 > 0 ? (1ull << d.p1) : 0ull;
    const uint64_t n2 = 1ull << d.p;
    const uint64_t nchunks = (n2 + kScanChunk - 1) / kScanChunk;
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    if (blockIdx.x == 0 && threadIdx.x == 0) *d.ticket = 0u;
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
    const Sort2Desc &d = *dp;
    const bool last = LEVEL == 2 || d.p2 == 0;  // the level that fills the partitions
    const int bits = LEVEL == 2 ? d.p2 : last ? d.p : d.p1;
    const uint4 *src;
    uint64_t left, bin0 = 0;  // records from the tile on; first bin of the CTA
    if (LEVEL == 1) {
        const uint64_t n = *d.count, base = (uint64_t)blockIdx.x * kS2Tile;
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
        if (all != *d.count) atomicOr(d.status, kStSort2);
    }
}

// In-place exclusive scan of 2M digit counters of 16 bits, two to a word
// (digit 2w in the low half of word w, 2w + 1 in the high half; every
// count and start below 2^16), by a CTA of NT threads: each word's two
// counts become their starts.  Warp w takes a contiguous run of the words,
// 32 at a time; `ws` holds NT/32 words.  Ends with a __syncthreads.
template <int NT>
__device__ __forceinline__ void block_scan_packed16(uint32_t *A, uint32_t M, uint32_t *ws)
{
    constexpr int NW = NT / 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t chunk = (M + NW - 1) / NW;
    const uint32_t lo = min(M, (uint32_t)warp * chunk), hi = min(M, lo + chunk);
    uint32_t sum = 0;
    for (uint32_t i = lo + lane; i < hi; i += 32) sum += (A[i] & 0xFFFFu) + (A[i] >> 16);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if (lane == 0) ws[warp] = sum;
    __syncthreads();
    uint32_t carry = 0;
#pragma unroll
    for (int w = 0; w < NW; ++w) carry += w < warp ? ws[w] : 0u;
    for (uint32_t base = lo; base < hi; base += 32) {
        const uint32_t i = base + lane;
        const uint32_t a = i < hi ? A[i] : 0u, l = a & 0xFFFFu, v = l + (a >> 16);
        uint32_t incl = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        const uint32_t P = carry + incl - v;
        if (i < hi) A[i] = P | ((P + l) << 16);
        carry += __shfl_sync(0xffffffffu, incl, 31);
    }
    __syncthreads();
}

// ------------------------------------------------------- partition sort
// One CTA per partition, its slot brought into shared memory by one bulk
// copy: counting sort of the record indices on the dbits key bits below the
// partition prefix, then each record ranked inside its digit run by
// (key2, a, b) with warp shuffles and written straight to its place at the
// partition's offset.
constexpr uint32_t kS2PrefetchAhead = 384;  // partitions ahead: ~half the resident CTAs

struct S2SortLayout {
    size_t idx, rank, dcnt, ws, bar, bytes;
    __host__ __device__ S2SortLayout(uint32_t cap, int dbits)
    {
        idx = (size_t)cap * 16;
        rank = idx + (size_t)((cap + 1) & ~1u) * 2;
        dcnt = rank + (size_t)((cap + 1) & ~1u) * 2;
        ws = dcnt + ((size_t)1 << dbits) * 4;
        bar = (ws + 40 * 4 + 7) & ~(size_t)7;
        bytes = bar + 8;
    }
};

__global__ void __launch_bounds__(kS2SortThreads, 4) k_s2_sort(const Sort2Desc *__restrict__ dp)
{
    constexpr int NT = kS2SortThreads;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const Sort2Desc &d = *dp;
    if (*d.status & (kStSort2 | kStTimeout | kStBadTicket)) return;  // offsets not trusted
    const uint32_t f = blockIdx.x;
    const uint32_t cap = d.cap2;
    const int dbits = d.dbits;
    const uint32_t ndig = 1u << dbits;
    const S2SortLayout L(cap, dbits);
    const uint4 *X = reinterpret_cast<const uint4 *>(smem_raw);
    uint16_t *SI = reinterpret_cast<uint16_t *>(smem_raw + L.idx);
    uint16_t *RK = reinterpret_cast<uint16_t *>(smem_raw + L.rank);
    uint32_t *DC = reinterpret_cast<uint32_t *>(smem_raw + L.dcnt);
    uint32_t *WS = reinterpret_cast<uint32_t *>(smem_raw + L.ws);
    const uint32_t n = min(d.cnt2[f], cap);
    const uint64_t o = d.off[f];
    uint64_t *bar = reinterpret_cast<uint64_t *>(smem_raw + L.bar);
    if (n && threadIdx.x == 0) {
        mbar_init(bar, 1);
        mbar_expect_tx(bar, n * 16u);
        bulk_g2s(smem_raw, d.b_recs + (uint64_t)f * cap, n * 16u, bar);
    }
    // one more digit bit than the plan's in the same counter words: 16-bit
    // counters, two to a word (n < 2^16), runs of about half the records
    const int shift = 64 - d.p - dbits - 1;
    const uint32_t pdig = ndig << 1, dmask = pdig - 1u;
    const uint16_t *DC16 = reinterpret_cast<const uint16_t *>(DC);
    // the filled part of the slot kS2PrefetchAhead partitions ahead goes to
    // L2 after step 1 (its fill count is read now)
    const uint64_t fa = (uint64_t)f + kS2PrefetchAhead;
    const uint32_t nfa = (threadIdx.x == 0 && fa < (1ull << d.p)) ? min(d.cnt2[fa], cap) : 0u;
    for (uint32_t i = threadIdx.x; i < ndig; i += NT) DC[i] = 0u;
    if (n == 0) return;
    __syncthreads();
    if (!__syncthreads_and(mbar_wait(bar, 0, d.spin_limit))) {  // one answer for all threads
        if (threadIdx.x == 0) atomicOr(d.status, kStTimeout);
        mbar_wait(bar, 0, d.spin_limit);  // let the copy land before leaving
        return;
    }
    auto key_at = [&](uint32_t i) {
        const uint2 h = *reinterpret_cast<const uint2 *>(&X[i].z);
        return ((uint64_t)bswap32(h.x) << 32) | bswap32(h.y);
    };
#pragma unroll 4
    for (uint32_t i = threadIdx.x; i < n; i += NT) {
        const uint32_t g = (uint32_t)(key_at(i) >> shift) & dmask, h = (g & 1u) << 4;
        RK[i] = (uint16_t)(atomicAdd(&DC[g >> 1], 1u << h) >> h);
    }
    if (nfa)
        asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(d.b_recs + fa * cap), "r"(nfa * 16u)
                     : "memory");
    __syncthreads();
    block_scan_packed16<NT>(DC, ndig, WS);
#pragma unroll 4
    for (uint32_t i = threadIdx.x; i < n; i += NT)
        SI[DC16[(uint32_t)(key_at(i) >> shift) & dmask] + RK[i]] = (uint16_t)i;
    __syncthreads();
    // DC16[g] is the start of run g (records of digit g in arrival order);
    // the run ends at DC16[g + 1] (n for the last digit).  Every position, 32
    // per warp step and one per lane, finds its record's rank inside its run
    // and the record goes straight to its place in the sorted table.  A
    // run's records sit in neighbouring lanes, so each lane compares with
    // the lanes up to the longest run's length away (shuffles, every lane
    // in step) on a 32-bit compare key: the key bits below the digit, or
    // their top 32 (records of a run agree above them).  A lane whose run
    // leaves its chunk, or that meets an equal compare key, ranks itself
    // from shared memory on the whole record (key2, a, b).  Two chunks per step so that their work overlaps.
    uint4 *__restrict__ out = d.t2 + o;
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    constexpr uint32_t NW = NT / 32;
    const uint32_t nch = (n + 31u) >> 5;
    const int cs = shift > 32 ? shift - 32 : 0;
    auto run_bounds = [&](uint64_t k, uint32_t &s0, uint32_t &s1) {
        const uint32_t g = (uint32_t)(k >> shift) & dmask;
        s0 = DC16[g];
        s1 = g + 1 < pdig ? DC16[g + 1] : n;
    };
    // place of record r among the run [s0, s1)
    auto rank_slow = [&](uint4 r, uint32_t s0, uint32_t s1) -> uint32_t {
        const uint64_t k = sort2_key(r), v = (uint64_t)r.x << 32 | r.y;
        uint32_t at = s0;
        for (uint32_t q = s0; q < s1; ++q) {
            const uint4 x = X[SI[q]];
            const uint64_t kq = sort2_key(x);
            at += kq < k || (kq == k && ((uint64_t)x.x << 32 | x.y) < v) ? 1u : 0u;
        }
        return at;
    };
    for (uint32_t c = warp; c < nch; c += 2 * NW) {
        const uint32_t pa = 32u * c + lane, pb = pa + 32u * NW;
        const bool va = pa < n, vb = pb < n;
        const uint32_t xa = va ? pa : 0u, xb = vb ? pb : 0u;
        const uint4 ra = X[SI[xa]], rb = X[SI[xb]];
        const uint64_t ka = sort2_key(ra), kb = sort2_key(rb);
        uint32_t sa, ea, sb, eb;
        run_bounds(ka, sa, ea);
        run_bounds(kb, sb, eb);
        if (!va) sa = ea = 0u;
        if (!vb) sb = eb = 0u;
        const uint32_t lmax = __reduce_max_sync(0xffffffffu, max(ea - sa, eb - sb));
        uint32_t da = sa, db = sb;
        if (lmax > 1) {
            const uint32_t qa = (uint32_t)(ka >> cs), qb = (uint32_t)(kb >> cs);
            bool slow_a = va && (sa < 32u * c || ea > 32u * c + 32u);
            bool slow_b = vb && (sb < 32u * (c + NW) || eb > 32u * (c + NW) + 32u);
            for (uint32_t t = 1; t < lmax; ++t) {
                const uint32_t da_ = __shfl_down_sync(0xffffffffu, qa, t), ua = __shfl_up_sync(0xffffffffu, qa, t);
                const uint32_t db_ = __shfl_down_sync(0xffffffffu, qb, t), ub = __shfl_up_sync(0xffffffffu, qb, t);
                const bool ina_d = pa + t < ea, ina_u = lane >= t && pa - t >= sa;
                const bool inb_d = pb + t < eb, inb_u = lane >= t && pb - t >= sb;
                da += (ina_d && da_ < qa ? 1u : 0u) + (ina_u && ua < qa ? 1u : 0u);
                db += (inb_d && db_ < qb ? 1u : 0u) + (inb_u && ub < qb ? 1u : 0u);
                slow_a = slow_a || (ina_d && da_ == qa) || (ina_u && ua == qa);
                slow_b = slow_b || (inb_d && db_ == qb) || (inb_u && ub == qb);
            }
            if (va && slow_a) da = rank_slow(ra, sa, ea);
            if (vb && slow_b) db = rank_slow(rb, sb, eb);
        }
        if (va) out[da] = ra;
        if (vb) out[db] = rb;
    }
}

size_t sort2_smem_bytes(uint32_t cap, int dbits) { return S2SortLayout(cap, dbits).bytes; }

cudaError_t launch_sort2(const Sort2Desc *d_desc, const Sort2Launch &g, cudaStream_t s)
{
    static SmemSeen seen1, seen2, seen3;
    cudaError_t e;
    k_s2_setup<<<64, 256, 0, s>>>(const_cast<Sort2Desc *>(d_desc));
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if (g.tiles1) {
        const size_t sm = S2ScatterLayout(g.p - g.p2).bytes;
        if ((e = allow_smem(k_s2_scatter<1>, sm, seen1)) != cudaSuccess) return e;
        k_s2_scatter<1><<<g.tiles1, kS2Threads, sm, s>>>(d_desc);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    if (g.tiles2) {
        const size_t sm = S2ScatterLayout(g.p2).bytes;
        if ((e = allow_smem(k_s2_scatter<2>, sm, seen2)) != cudaSuccess) return e;
        k_s2_scatter<2><<<g.tiles2, kS2Threads, sm, s>>>(d_desc);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    k_s2_scan<<<g.tiles_scan, 256, 0, s>>>(d_desc);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    const size_t sm = sort2_smem_bytes(g.cap2, g.dbits);
    if ((e = allow_smem(k_s2_sort, sm, seen3)) != cudaSuccess) return e;
    k_s2_sort<<<g.parts, kS2SortThreads, sm, s>>>(d_desc);
    return cudaGetLastError();
}

}  // namespace vx
