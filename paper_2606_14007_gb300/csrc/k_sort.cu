// k_sort.cu -- second bucketing scatter level, prefix scans, and the
// logical bucket offsets of Table 1.
//
// Paper: Sec. III-A/III-B (Table 1 bucketed by hash prefix, 2^24 buckets).
// The partition sort itself lives in k_sortmatch.cu.
#include "vx_internal.cuh"

namespace vx {

// ------------------------------------------------ second scatter level
// One CTA takes a tile of up to kScatterTile records of one first-level
// slot.  The tile's keys and nonces are contiguous, so two TMA bulk copies
// bring them into shared memory (one mbarrier, bounded wait); ranks within
// the second-level bins come from shared-memory atomics; one global atomic
// per (CTA, bin) claims a run of the final partition slot.  The records stay
// where the copies left them: a 16-bit order says which one goes next, and
// they are written out in that order, so that consecutive threads store
// consecutive addresses of each run.  Bound by HBM: 2^28 records take 1.13
// ms, 5.7 TB/s, 2^31 10.6 ms.  (Restaged in place through registers, with
// two CTAs per SM for their 64 registers a thread, 1.49 and 13.0 ms.)
struct Scatter2Layout {
    size_t nonces, order, hist, ws, bar, bytes;
    __host__ __device__ explicit Scatter2Layout(int bits)
    {
        nonces = (size_t)kScatterTile * 8;
        order = nonces + (size_t)kScatterTile * 4;
        hist = order + (size_t)kScatterTile * 2;
        ws = hist + ((size_t)4 << bits);
        bar = (ws + (kScatterThreads / 32 + 1) * 4 + 7) & ~(size_t)7;
        bytes = bar + 8;
    }
};

// FB: the most second-level bits the instance handles (10; 11 for the
// 2^21 partitions of K = 32); bits: the launch's most.
template <bool HALO, int FB>
__global__ void __launch_bounds__(kScatterThreads, 3) k_scatter2(const Desc *__restrict__ descs,
                                                                int nplots,
                                                                const uint32_t *__restrict__ tile_start,
                                                                int chunk, int bits)
{
    constexpr int NT = kScatterThreads;
    constexpr int PER = kScatterTile / NT;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const Scatter2Layout L(bits);
    uint64_t *keys = reinterpret_cast<uint64_t *>(smem_raw);
    uint32_t *nonces = reinterpret_cast<uint32_t *>(smem_raw + L.nonces);
    uint16_t *order = reinterpret_cast<uint16_t *>(smem_raw + L.order);
    uint32_t *hist = reinterpret_cast<uint32_t *>(smem_raw + L.hist);
    uint32_t *ws = reinterpret_cast<uint32_t *>(smem_raw + L.ws);
    uint64_t *bar = reinterpret_cast<uint64_t *>(smem_raw + L.bar);

    pdl_go();
    pdl_wait();
    const int plot = find_plot(tile_start, nplots, blockIdx.x);
    const Desc &d = descs[plot];
    const uint32_t local = blockIdx.x - tile_start[plot];
    const uint32_t c = local / d.chunks1;              // level-1 bin of this nonce chunk
    const uint32_t part = local - c * d.chunks1;       // tile of the slot
    const uint64_t cs = ((uint64_t)chunk << d.p1) + c; // the slot
    const uint32_t filled = min(d.cnt1[cs], d.cap1);
    const uint32_t start = part * (uint32_t)kScatterTile;
    if (start >= filled) return;
    const uint32_t count = min((uint32_t)kScatterTile, filled - start);
    const int p2 = d.p2;
    const int nbins = 1 << p2;
    const int shift = 32 - d.pk;                       // fine index: of the key's top 32 bits
    const uint32_t bin_mask = (uint32_t)nbins - 1u;
    // Copy a multiple of 4 records: the slot (cap1 % 4 == 0) always holds them.
    const uint32_t ncopy = (count + 3u) & ~3u;
    if (threadIdx.x == 0) {
        mbar_init(bar, 1);
        mbar_expect_tx(bar, ncopy * 12u);
        bulk_g2s(keys, d.a_keys + cs * d.cap1 + start, ncopy * 8u, bar);
        bulk_g2s(nonces, d.a_nonces + cs * d.cap1 + start, ncopy * 4u, bar);
    }
    for (int b = threadIdx.x; b < nbins; b += NT) hist[b] = 0u;
    __syncthreads();
    if (!__syncthreads_and(mbar_wait(bar, 0, d.spin_limit))) {  // one answer for all threads
        // The copy did not land in time: report, give it one more bounded
        // wait so it does not write into a successor's shared memory, stop.
        if (threadIdx.x == 0) atomicOr(d.status, kStTimeout);
        mbar_wait(bar, 0, d.spin_limit);
        return;
    }

    uint32_t where[PER];  // bin << 16 | rank in the bin
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        const uint32_t i = (uint32_t)j * NT + threadIdx.x;
        where[j] = 0u;
        if (i < count) {
            const uint32_t bin = (reinterpret_cast<const uint32_t *>(keys)[2 * i + 1] >> shift) & bin_mask;
            where[j] = bin << 16 | atomicAdd(&hist[bin], 1u);
        }
    }
    __syncthreads();
    constexpr int PB = ((1 << FB) + NT - 1) / NT;  // most bins a thread owns
    const int per = (nbins + NT - 1) / NT;
    const int b0 = threadIdx.x * per;
    uint32_t claim[PB];
    {
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
                // the claim's result is first needed after the order below
                if (h) claim[k] = atomicAdd(&d.cnt2[((uint64_t)c << p2) + b], h);
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
    const uint32_t cap = d.cap2;
    const uint64_t f0 = (uint64_t)c << p2;
    uint64_t *__restrict__ okeys = d.b_keys + f0 * cap;
    uint32_t *__restrict__ ononces = d.b_nonces + f0 * cap;
    bool overflow = false, hover = false;
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        const uint32_t q = (uint32_t)j * NT + threadIdx.x;
        if (q >= count) break;
        const uint32_t i = order[q];
        const uint64_t k = keys[i];
        const uint32_t nonce = nonces[i];
        const uint32_t bin = ((uint32_t)(k >> 32) >> shift) & bin_mask;
        const uint32_t g = hist[bin] + q;
        if (g < cap) {
            const uint64_t at = (uint64_t)bin * cap + g;
            okeys[at] = k;
            ononces[at] = nonce;
        } else {
            overflow = true;
        }
        if (HALO) halo_add(d, f0 + bin, k, nonce, hover);
    }
    if (overflow) atomicOr(d.status, kStSlot2Overflow);
    if (hover) atomicOr(d.status, kStHaloOverflow);
}

cudaError_t launch_scatter2(const Desc *descs, int nplots, const uint32_t *tile_start,
                            uint32_t total_tiles, int chunk, On on, bool halo, int fine_bits)
{
    if (total_tiles == 0) return cudaSuccess;
    const bool wide = fine_bits > kMaxFineBits;
    const size_t smem = Scatter2Layout(fine_bits).bytes;
    auto fn = wide ? (halo ? k_scatter2<true, kMaxFineBitsWide> : k_scatter2<false, kMaxFineBitsWide>)
                   : (halo ? k_scatter2<true, kMaxFineBits> : k_scatter2<false, kMaxFineBits>);
    static SmemSeen seen[4];
    const cudaError_t e = allow_smem(fn, smem, seen[(wide ? 2 : 0) + (halo ? 1 : 0)]);
    if (e != cudaSuccess) return e;
    return launch_on(on, fn, total_tiles, kScatterThreads, smem, descs, nplots, tile_start, chunk, fine_bits);
}

// ------------------------------- Table-1 / Table-2 offsets (counts scan)
// Exclusive prefix of 2^p per-partition counts in chunks of kScanChunk
// counters, one CTA per chunk (taken in ticket order), the chunks chained by
// decoupled look-back.
constexpr int kScanCtaThreads = 256;

// SRC 0: level-2 fill counters (clipped to the slot) -> Table-1 offsets,
// chunk ticket ticket_s, look-back words lbs; the last chunk checks that
// every nonce arrived.
// SRC 1: per-partition pair counts of the slot placement -> Table-2
// offsets, chunk ticket `ticket` and look-back words `lb` (both unused by
// the slot sort, zeroed by the key setup); counts are clipped to one more
// than a pair slot holds (a larger count has already failed the plot), and
// the last chunk checks the Table-2 capacity.
template <int SRC>
__global__ void __launch_bounds__(kScanCtaThreads) k_scan_counts(const Desc *__restrict__ descs,
                                                                 int nplots,
                                                                 const uint32_t *__restrict__ tile_start)
{
    constexpr int NT = kScanCtaThreads;
    constexpr uint32_t PER = kScanChunk / NT;
    __shared__ uint32_t ws[NT / 32 + 1];
    __shared__ uint32_t s_c;
    __shared__ uint64_t s_base;
    __shared__ int s_ok;
    // The slot pair hash comes onto the SMs once the sort has ended (SRC 1
    // waits for it), not onto those its CTAs leave first: at K <= 22 it has
    // too few CTAs to fill the rest (cross-bucket match, K=21: 288 us a run
    // with the CTAs let go at once, 192 so; K=22: 449 and 339, bucket match
    // 235 and 221; K=23 and above the same).
    if (SRC == 0) pdl_go();
    pdl_wait();
    if (SRC == 1) pdl_go();
    const int plot = find_plot(tile_start, nplots, blockIdx.x);
    const Desc &d = descs[plot];
    uint32_t *ticket = SRC == 0 ? d.ticket_s : d.ticket;
    uint64_t *lb = SRC == 0 ? d.lbs : d.lb;
    uint64_t *out = SRC == 0 ? d.t1off : d.t2off;
    if (threadIdx.x == 0) s_c = atomicAdd(ticket, 1u);
    __syncthreads();
    const uint32_t c = s_c;
    const uint64_t n = 1ull << d.p;
    const uint32_t nchunks = (uint32_t)((n + kScanChunk - 1) / kScanChunk);
    if (c >= nchunks) {  // only if the ticket was not reset: report, never index with it
        if (threadIdx.x == 0) atomicOr(d.status, kStBadTicket);
        return;
    }
    const uint32_t clip = SRC == 0 ? d.cap2 : d.cap2 + d.cap2 / 2u + 1u;
    const uint64_t b0 = (uint64_t)c * kScanChunk + (uint64_t)threadIdx.x * PER;
    uint32_t v[PER];
    uint32_t loc = 0;
#pragma unroll
    for (uint32_t k = 0; k < PER; ++k) {
        uint32_t x = 0;
        if (b0 + k < n) {
            if (SRC == 0) {
                x = min(d.cnt2[b0 + k], clip);
            } else {
                const uint64_t y = d.pairs[b0 + k];
                x = y < clip ? (uint32_t)y : clip;
            }
        }
        v[k] = x;
        loc += x;
    }
    uint32_t total;
    uint32_t run = block_exclusive_scan_u32<NT>(loc, ws, &total);
    if (threadIdx.x < 32) {
        uint64_t excl = 0;
        // VX_TEST_WITHHOLD_PREFIX: chunk 0 of the pair-count scan never
        // publishes, so every later chunk's bounded wait runs out.
        const bool withhold = SRC == 1 && (d.test_flags & 1u) != 0;
        const int ok = lookback_warp(lb, c, total, d.status, d.spin_limit, withhold, &excl) ? 1 : 0;
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
        if (b0 + k < n) out[b0 + k] = at;
        at += v[k];
    }
    if (c + 1 == nchunks && threadIdx.x == 0) {
        const uint64_t all = s_base + total;
        out[n] = all;
        d.totals[SRC == 0 ? 1 : 0] = all;
        if (SRC == 0) {
            // Every nonce exactly once; a window's share is random (the
            // windows of one plot add up to 2^K, checked by their caller).
            if (d.wbits == 0 && all != d.N) atomicOr(d.status, kStCountMismatch);
        } else {
            if (all > d.t2cap) atomicOr(d.status, kStT2Capacity);
        }
    }
}

cudaError_t launch_scan_counts(const Desc *descs, int nplots, const uint32_t *tile_start,
                               uint32_t total_tiles, On on)
{
    return launch_on(on, k_scan_counts<0>, total_tiles, kScanCtaThreads, 0, descs, nplots, tile_start);
}

cudaError_t launch_scan_pair_counts(const Desc *descs, int nplots, const uint32_t *tile_start,
                                    uint32_t total_tiles, On on)
{
    return launch_on(on, k_scan_counts<1>, total_tiles, kScanCtaThreads, 0, descs, nplots, tile_start);
}

// ------------------------------------------------------ pair-offset scan
// One CTA per plot: exclusive prefix of the 2^p per-partition pair counts
// -> Table-2 offsets (split vx_table1 / vx_match path), with the Table-2
// capacity check.
constexpr int kScanThreads = 1024;

__global__ void __launch_bounds__(kScanThreads) k_scan_pairs(const Desc *__restrict__ descs)
{
    constexpr int NT = kScanThreads, NW = NT / 32, PER = 4;
    __shared__ uint64_t ws[NW];
    __shared__ uint64_t s_tile;
    pdl_go();
    pdl_wait();
    const Desc &d = descs[blockIdx.x];
    const uint64_t n = 1ull << d.p;
    uint64_t *out = d.t2off;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // tiles of NT * PER consecutive counts, PER per thread (coalesced),
    // block-scanned one after the other with the running total carried
    uint64_t carry = 0;
    for (uint64_t t0 = 0; t0 < n; t0 += (uint64_t)NT * PER) {
        const uint64_t b0 = t0 + (uint64_t)threadIdx.x * PER;
        uint64_t v[PER], local = 0;
#pragma unroll
        for (int k = 0; k < PER; ++k) {
            v[k] = b0 + k < n ? d.pairs[b0 + k] : 0ull;
            local += v[k];
        }
        uint64_t incl = local;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint64_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        if (lane == 31) ws[warp] = incl;
        __syncthreads();
        if (warp == 0) {
            const uint64_t x = lane < NW ? ws[lane] : 0ull;
            uint64_t wi = x;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint64_t y = __shfl_up_sync(0xffffffffu, wi, o);
                if (lane >= o) wi += y;
            }
            if (lane < NW) ws[lane] = wi - x;  // exclusive warp prefixes
            if (lane == NW - 1) s_tile = wi;
        }
        __syncthreads();
        uint64_t at = carry + ws[warp] + incl - local;
#pragma unroll
        for (int k = 0; k < PER; ++k) {
            if (b0 + k < n) out[b0 + k] = at;
            at += v[k];
        }
        carry += s_tile;
        __syncthreads();  // ws and s_tile are reused by the next tile
    }
    if (threadIdx.x == 0) {
        out[n] = carry;
        d.totals[0] = carry;
        // A re-run of the match (e.g. after a larger Table-2 buffer was
        // bound) re-decides the capacity bit.
        if (carry > d.t2cap) atomicOr(d.status, kStT2Capacity);
        else atomicAnd(d.status, ~kStT2Capacity);
    }
}

cudaError_t launch_scan_pairs(const Desc *descs, int nplots, On on)
{
    return launch_on(on, k_scan_pairs, (uint32_t)nplots, kScanThreads, 0, descs);
}

// ----------------------------------------------- logical bucket offsets
// offsets[b] = first Table-1 record of logical bucket b, found by a binary
// search inside the physical partition that holds bucket b.  A window's
// Table 1 holds buckets [w0, w0 + 2^(24 - wbits)) only: buckets below get
// offset 0, buckets above the window's record count.
__global__ void k_bucket_offsets(const Desc *__restrict__ dp, uint64_t *__restrict__ out)
{
    const Desc &d = *dp;
    const uint32_t nb = 1u << kBucketBits;
    const uint32_t b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b > nb) return;
    const uint64_t np = 1ull << d.p;
    if (b == nb) {
        out[nb] = d.wbits ? d.t1off[np] : d.N;
        return;
    }
    const int wb = kBucketBits - (int)d.wbits;  // bucket bits inside the window
    const uint32_t w0 = d.win << wb;
    if (b < w0) {
        out[b] = 0;
        return;
    }
    if (b - w0 >= (1u << wb)) {
        out[b] = d.t1off[np];
        return;
    }
    const uint32_t f = d.p ? ((b - w0) >> (wb - d.p)) : 0u;
    uint64_t lo = d.t1off[f], hi = d.t1off[f + 1];
    const uint32_t *t1w = reinterpret_cast<const uint32_t *>(d.t1);
    while (lo < hi) {   // first record whose bucket >= b
        const uint64_t mid = (lo + hi) >> 1;
        const uint32_t hb = bswap32(t1w[3 * mid + 1]) >> 8;   // key64 >> 40
        if (hb < b) lo = mid + 1; else hi = mid;
    }
    out[b] = lo;
}

cudaError_t launch_bucket_offsets(const Desc *desc, uint64_t *out, cudaStream_t s)
{
    const uint32_t n = (1u << kBucketBits) + 1;
    k_bucket_offsets<<<(n + 255) / 256, 256, 0, s>>>(desc, out);
    return cudaGetLastError();
}

}  // namespace vx
