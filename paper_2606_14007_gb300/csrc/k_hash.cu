// k_hash.cu -- key setup, Table-1 hashing fused with the first bucketing
// scatter (also for one window of a plot: filtering every nonce's key, or
// hashing the window's listed nonces), the window-id and window-list passes
// of tiled plots, and the stand-alone hash / pair-hash kernels.
//
// Paper: Sec. III-A/III-B (one keyed BLAKE3 per nonce, little-endian nonce,
// bucket index from the hash prefix).  The paper's kernel claims one bucket
// slot per nonce with a global atomicAdd; here a CTA hashes a tile of
// nonces, histograms them by the leading hash bits in shared memory
// (warp-aggregated with __match_any_sync where bins are few), claims one
// contiguous run per (CTA, bin) with a single global atomic, and writes the
// records partition-ordered so that consecutive threads store consecutive
// addresses.  Order inside a partition is irrelevant: the partition sort
// orders records by (key64, nonce), a total order.
#include "vx_internal.cuh"

namespace vx {

// --------------------------------------------------------------- setup
// One CTA row per plot: every CTA zeroes a share of the plot's fill counters
// and look-back words, one thread the tickets and the status word.  (The
// per-key hash states come with the descriptor, so the hash may start beside
// this kernel and waits for it before its first claim.)
__global__ void k_key_setup(Desc *descs)
{
    pdl_wait();
    pdl_go();
    Desc &d = descs[blockIdx.y];
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        *d.status = 0u;
        *d.ticket = 0u;
        *d.ticket_s = 0u;
        for (int c = 0; c < kMaxPartChunks; ++c) d.ticket_i[c] = 0u;
        d.totals[0] = d.totals[1] = 0ull;
        if (d.wcount) *d.wcount = 0u;
    }
    const uint64_t n1 = d.p2 > 0 ? ((uint64_t)d.hchunks << d.p1) : 0ull;
    const uint64_t n2 = 1ull << d.p;
    const uint64_t nchunks = (n2 + kScanChunk - 1) / kScanChunk;
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    const uint64_t nz = n2 > n1 ? n2 : n1;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nz; i += stride) {
        if (i < n2) {
            d.cnt2[i] = 0u;
            d.lb[i] = 0ull;
            if (d.hcap) d.halo_cnt[i] = 0u;
        }
        if (i < n1) d.cnt1[i] = 0u;
        if (i < nchunks) d.lbs[i] = 0ull;
    }
}

cudaError_t launch_key_setup(Desc *descs, int nplots, On on)
{
    dim3 grid(64, nplots);
    k_key_setup<<<grid, 256, 0, on.s>>>(descs);
    return cudaGetLastError();
}

// --------------------------------------------- hash + first-level scatter
// Shared layout of one tile of T nonces: key64[T] in nonce order, then per
// record its bin (kNoBin: not kept), its rank inside the bin, and, once the
// bins are scanned, the record order by bin; then per bin the histogram
// (which becomes the bin's start in the tile) and the bin's place.  Bins,
// ranks and starts are kept as the byte offsets they are used at (4 * bin,
// 2 * rank, 2 * start), so that no use of them costs a shift.
// CB: the most first-level bits the instance handles.
template <int NT, int NPT, int CB>
struct HashTile {
    static constexpr uint32_t T = NT * NPT;
    uint64_t keys[T];
    uint16_t bin4[T], rank2[T], order[T];
    uint32_t start2[1 << CB];
    uint32_t place[1 << CB];
    uint32_t ws[NT / 32 + 1];
};
constexpr uint32_t kNoBin = 0xFFFFu;

template <class X>
__device__ __forceinline__ X &at_bytes(X *a, uint32_t off)
{
    return *reinterpret_cast<X *>(reinterpret_cast<unsigned char *>(a) + off);
}

// Rank of this lane's record within its bin's run of the tile.
template <bool AGG>
__device__ __forceinline__ uint32_t bin_rank(uint32_t *hist, uint32_t bin4, bool valid)
{
    if (AGG) {
        const uint32_t peers = __match_any_sync(0xffffffffu, valid ? bin4 : 0xffffffffu);
        const int leader = __ffs(peers) - 1;
        const int lane = threadIdx.x & 31;
        uint32_t base = 0;
        if (lane == leader && valid) base = atomicAdd(&at_bytes(hist, bin4), (uint32_t)__popc(peers));
        base = __shfl_sync(0xffffffffu, base, leader);
        return base + (uint32_t)__popc(peers & ((1u << lane) - 1u));
    } else {
        return valid ? atomicAdd(&at_bytes(hist, bin4), 1u) : 0u;
    }
}

// Exclusive scan of the bin counts start2[0..nbins) in place, and one global
// claim per non-empty bin; place[b] = b * cap + claim - start, so record i of
// the bin-ordered tile goes to slot index place[bin] + i (32 bits, wrapping).
// *total gets the records of the tile; true if a claim passes its slot's end.
template <int NT, int CB, class S>
__device__ __forceinline__ bool scan_and_claim(S &t, int nbins, uint32_t *cnt, uint32_t cap, uint32_t *total)
{
    constexpr int PB = ((1 << CB) + NT - 1) / NT;  // most bins a thread owns
    const int per = (nbins + NT - 1) / NT;
    const int b0 = threadIdx.x * per;
    uint32_t h[PB], local = 0;
#pragma unroll
    for (int k = 0; k < PB; ++k) {
        h[k] = k < per && b0 + k < nbins ? t.start2[b0 + k] : 0u;
        local += h[k];
    }
    uint32_t run = block_exclusive_scan_u32<NT>(local, t.ws, total);
    bool over = false;
#pragma unroll
    for (int k = 0; k < PB; ++k) {
        if (k < per && b0 + k < nbins) {
            const uint32_t b = b0 + k;
            const uint32_t c = h[k] ? atomicAdd(&cnt[b], h[k]) : 0u;
            over = over || (h[k] && (c > cap || h[k] > cap - c));
            t.start2[b] = 2u * run;
            t.place[b] = b * cap + c - run;
            run += h[k];
        }
    }
    return over;
}

// Windowed plots keep the keys whose top wbits equal win and bin them by the
// bits after those.  kWinFilter instances hash every nonce and test its key
// (a plot without a window, wbits 0, keeps every key, so one such launch may
// also carry whole plots); kWinList instances hash only the nonces listed
// for the window (Desc::wlist, from a pass that stored every nonce's window);
// kWinIds instances are kWinFilter ones that store the windows beside their
// own records.
enum { kWinNone = 0, kWinFilter = 1, kWinList = 2, kWinIds = 3 };

// Window bits plus bin bits are at most the 21 partition bits, so both tests
// read only the key's high word.
template <bool WIN>
__device__ __forceinline__ bool in_window(const Desc &d, uint64_t key)
{
    const uint32_t hi = (uint32_t)(key >> 32);
    return !WIN || ((hi >> 1) >> (31 - d.wbits)) == d.win;  // wbits 0: always
}

template <bool WIN>
__device__ __forceinline__ uint32_t key_bin(const Desc &d, uint64_t key, int bits)
{
    const uint32_t hi = (uint32_t)(key >> 32);
    // clamped funnel shift: bits 0 gives bin 0
    return __funnelshift_rc(WIN ? hi << d.wbits : hi, 0u, 32 - bits);
}

// One CTA: a tile of NT * NPT nonces.  The hash is bound by the ALU pipe
// (417 of its ~620 instructions are xors and rotations, which only that
// half-rate pipe runs), so everything around it is laid out to spend few ALU
// instructions: a rolled loop of two hashes per step (see b3_finish) that
// leaves each record's key, bin and rank in shared memory; the tile's order
// by bin as 16-bit record indices instead of moved records; slot places as
// 32-bit indices whose addresses are multiply-adds on the FMA pipe.  The
// extra shared-memory traffic is free: that path idles at 17% here.
template <int NT, int NPT, bool AGG, bool HALO, int WM, int CB>
__global__ void __launch_bounds__(NT, NPT <= 12 ? 4 : 3) k_hash_scatter(const Desc *__restrict__ descs, int nplots,
                                                     const uint32_t *__restrict__ tile_start,
                                                     int chunk)
{
    using S = HashTile<NT, NPT, CB>;
    constexpr uint32_t T = S::T;
    constexpr bool WIN = WM != kWinNone, FILTER = WM == kWinFilter || WM == kWinIds;
    static_assert(NPT % 2 == 0 && 2 * T <= 0x10000u && (4u << CB) < kNoBin, "16-bit offsets");
    extern __shared__ __align__(16) unsigned char smem_raw[];
    S &sm = *reinterpret_cast<S *>(smem_raw);

    pdl_go();
    if (WM == kWinList) pdl_wait();
    const int plot = find_plot(tile_start, nplots, blockIdx.x);
    const Desc &d = descs[plot];
    uint64_t lo, N;  // this chunk's nonces: [lo, N), or (list) list entries [0, N)
    nonce_chunk(d, chunk, lo, N);
    if (WM == kWinList) N = min(*d.wcount, d.listcap);
    const uint64_t base = lo + (uint64_t)(blockIdx.x - tile_start[plot]) * T;
    if (WM == kWinList && base >= N) return;  // the grid covers the list's capacity
    const uint32_t left = (uint32_t)(N - base < T ? N - base : T);  // nonces of the tile
    const bool two_level = d.p2 > 0;
    const int bits = two_level ? d.p1 : d.p;
    const int nbins = 1 << bits;
    const uint32_t cap = two_level ? d.cap1 : d.cap2;
    // Two levels: this chunk's own level-1 slots; one level: the final slots.
    const uint64_t slot0 = two_level ? ((uint64_t)chunk << d.p1) : 0ull;
    uint64_t *__restrict__ okeys = two_level ? d.a_keys + slot0 * cap : d.b_keys;
    uint32_t *__restrict__ ononces = two_level ? d.a_nonces + slot0 * cap : d.b_nonces;
    uint32_t *cnt = two_level ? d.cnt1 + slot0 : d.cnt2;
    const uint32_t *__restrict__ list = WM == kWinList ? d.wlist + base : nullptr;
    const uint32_t nonce0 = (uint32_t)base;

    for (int b = threadIdx.x; b < nbins; b += NT) sm.start2[b] = 0u;
    __syncthreads();
    {
        uint32_t pre[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) pre[i] = d.pre1[i];
#pragma unroll 1
        for (uint32_t i0 = threadIdx.x; i0 < T; i0 += 2 * NT) {
            uint64_t key[2];
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const uint32_t i = i0 + u * NT;
                const uint32_t nonce = WM == kWinList ? (i < left ? list[i] : 0u) : nonce0 + i;
                uint32_t h0, h1;
                b3_finish<false>(pre, nonce, 0u, h0, h1);
                key[u] = key64_of(h0, h1);
            }
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const uint32_t i = i0 + u * NT;
                const bool valid = i < left && (!FILTER || in_window<true>(d, key[u]));
                const uint32_t bin4 = 4u * key_bin<WIN>(d, key[u], bits);
                sm.keys[i] = key[u];
                if (WM == kWinIds && i < left) d.wids[base + i] = (uint8_t)(key[u] >> (64 - d.wbits));
                sm.rank2[i] = (uint16_t)(2u * bin_rank<AGG>(sm.start2, bin4, valid));
                sm.bin4[i] = (uint16_t)(!FILTER || valid ? bin4 : kNoBin);
            }
        }
    }
    if (WM != kWinList) pdl_wait();  // up to here only the descriptor was read
    __syncthreads();
    uint32_t count;  // records the tile keeps
    const bool over = scan_and_claim<NT, CB>(sm, nbins, cnt, cap, &count);
    // Every place fits 32 bits unless all slots together hold 2^32 records
    // or more (K = 32 in two levels).
    const bool slow = __syncthreads_or(over) || ((uint64_t)cap << bits) > 0xFFFFFFFFull;
#pragma unroll 4
    for (uint32_t i = threadIdx.x; i < left; i += NT) {
        const uint32_t bin4 = sm.bin4[i];
        if (!FILTER || bin4 != kNoBin)
            at_bytes(sm.order, at_bytes(sm.start2, bin4) + sm.rank2[i]) = (uint16_t)i;
    }
    __syncthreads();
    if (!slow && (!HALO || two_level)) {
#pragma unroll 4
        for (uint32_t q = threadIdx.x; q < count; q += NT) {
            const uint32_t i = sm.order[q];
            const uint32_t at = at_bytes(sm.place, sm.bin4[i]) + q;
            okeys[at] = sm.keys[i];
            ononces[at] = WM == kWinList ? list[i] : nonce0 + i;
        }
        return;
    }
    bool overflow = false, hover = false;
    for (uint32_t q = threadIdx.x; q < count; q += NT) {
        const uint32_t i = sm.order[q];
        const uint64_t k = sm.keys[i];
        const uint32_t bin = sm.bin4[i] >> 2;
        const uint32_t nonce = WM == kWinList ? list[i] : nonce0 + i;
        const uint32_t g = sm.place[bin] + q - bin * cap;
        if (g < cap) {
            const uint64_t at = (uint64_t)bin * cap + g;
            okeys[at] = k;
            ononces[at] = nonce;
        } else {
            overflow = true;
        }
        if (HALO && !two_level) halo_add(d, bin, k, nonce, hover);  // final partitions
    }
    if (overflow) atomicOr(d.status, two_level ? kStSlot1Overflow : kStSlot2Overflow);
    if (hover) atomicOr(d.status, kStHaloOverflow);
}

template <int NPT, bool AGG, bool HALO, int WM, int CB = kMaxCoarseBits>
static cudaError_t launch_hs(const Desc *descs, int nplots, const uint32_t *tile_start,
                             uint32_t total_tiles, int chunk, On on)
{
    constexpr int NT = kHashThreads;
    static SmemSeen seen;
    const size_t smem = sizeof(HashTile<NT, NPT, CB>);
    auto fn = k_hash_scatter<NT, NPT, AGG, HALO, WM, CB>;
    const cudaError_t e = allow_smem(fn, smem, seen);
    if (e != cudaSuccess) return e;
    return launch_on(on, fn, total_tiles, NT, smem, descs, nplots, tile_start, chunk);
}

// AGG (warp-aggregated ranks) pays off when a warp's 32 records fall into
// few bins; the host picks it from the smallest bin count in the launch.
// HALO instances carry the cross-bucket halo code and window instances the
// window filter or the nonce list; plain launches carry neither.  A list
// launch holds one windowed plot (never cross-bucket).
template <bool HALO, int WM, int NPT>
static cudaError_t launch_hs_npt(const Desc *descs, int nplots, const uint32_t *tile_start,
                                 uint32_t total_tiles, bool agg, int chunk, On on)
{
    return agg ? launch_hs<NPT, true, HALO, WM>(descs, nplots, tile_start, total_tiles, chunk, on)
               : launch_hs<NPT, false, HALO, WM>(descs, nplots, tile_start, total_tiles, chunk, on);
}

template <bool HALO, int WM>
static cudaError_t launch_hs_agg(const Desc *descs, int nplots, const uint32_t *tile_start,
                                 uint32_t total_tiles, bool agg, int chunk, On on, int npt, int bits)
{
    if (WM != kWinNone && npt != kHashNoncesPerThread && npt != 16) return cudaErrorInvalidValue;
    if (bits > kMaxCoarseBits) {  // 2^19 partitions and more: tiles of 4096 only
        if constexpr (WM == kWinNone || WM == kWinFilter)
            return npt == 16 ? launch_hs<16, false, HALO, WM, kMaxCoarseBitsWide>(descs, nplots, tile_start, total_tiles,
                                                                                 chunk, on)
                             : cudaErrorInvalidValue;
        return cudaErrorInvalidValue;
    }
    switch (npt) {
    case 2: return launch_hs_npt<HALO, kWinNone, 2>(descs, nplots, tile_start, total_tiles, agg, chunk, on);
    case 4: return launch_hs_npt<HALO, kWinNone, 4>(descs, nplots, tile_start, total_tiles, agg, chunk, on);
    case 8: return launch_hs_npt<HALO, WM, 8>(descs, nplots, tile_start, total_tiles, agg, chunk, on);
    case 12: return launch_hs_npt<HALO, kWinNone, 12>(descs, nplots, tile_start, total_tiles, agg, chunk, on);
    case 16: return launch_hs_npt<HALO, WM, 16>(descs, nplots, tile_start, total_tiles, agg, chunk, on);
    default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_hash_scatter(const Desc *descs, int nplots, const uint32_t *tile_start,
                                uint32_t total_tiles, HashCfg cfg, int chunk, On on)
{
    if (total_tiles == 0) return cudaSuccess;
    const int npt = cfg.npt;
    if (cfg.list)
        return cfg.halo ? cudaErrorInvalidValue
                        : launch_hs_agg<false, kWinList>(descs, nplots, tile_start, total_tiles, cfg.agg, chunk, on, npt, cfg.bits);
    if (cfg.ids)
        return cfg.halo ? cudaErrorInvalidValue
                        : launch_hs_agg<false, kWinIds>(descs, nplots, tile_start, total_tiles, cfg.agg, chunk, on, npt, cfg.bits);
    if (cfg.win)
        return cfg.halo ? launch_hs_agg<true, kWinFilter>(descs, nplots, tile_start, total_tiles, cfg.agg, chunk, on, npt, cfg.bits)
                        : launch_hs_agg<false, kWinFilter>(descs, nplots, tile_start, total_tiles, cfg.agg, chunk, on, npt, cfg.bits);
    return cfg.halo ? launch_hs_agg<true, kWinNone>(descs, nplots, tile_start, total_tiles, cfg.agg, chunk, on, npt, cfg.bits)
                    : launch_hs_agg<false, kWinNone>(descs, nplots, tile_start, total_tiles, cfg.agg, chunk, on, npt, cfg.bits);
}

// ------------------------------------------------- hash + direct scatter
// The other bucketing strategy (the paper's, Sec. III-B: an atomicAdd slot
// claim per nonce), here straight into the final partitions: every thread
// hashes NPT nonces, then claims one slot per record in its partition with
// a global atomic and stores key64 and nonce there.  No shared memory and
// no second scatter pass; the claims and scattered stores run on the LSU
// and L2 while the ALU pipe -- the kernel's bound -- keeps hashing.
template <int NT, int NPT, bool HALO, int WM>
__global__ void __launch_bounds__(NT) k_hash_direct(const Desc *__restrict__ descs, int nplots,
                                                    const uint32_t *__restrict__ tile_start,
                                                    int chunk)
{
    constexpr bool WIN = WM != kWinNone;
    pdl_go();
    pdl_wait();
    const int plot = find_plot(tile_start, nplots, blockIdx.x);
    const Desc &d = descs[plot];
    uint64_t lo, N;  // this chunk's nonces: [lo, N), or (list) list entries [0, N)
    nonce_chunk(d, chunk, lo, N);
    if (WM == kWinList) N = min(*d.wcount, d.listcap);
    const uint64_t base = lo + (uint64_t)(blockIdx.x - tile_start[plot]) * (NT * NPT);
    if (WM == kWinList && base >= N) return;  // the grid covers the list's capacity
    const int bits = d.p;
    const uint32_t cap = d.cap2;
    uint32_t pre[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) pre[i] = d.pre1[i];
    // the nonce of entry idx: the entry itself, or (list) the listed nonce
    auto nonce_of = [&](uint64_t idx) -> uint32_t {
        return WM == kWinList ? (idx < N ? d.wlist[idx] : 0u) : (uint32_t)idx;
    };
    uint64_t key[NPT];
#pragma unroll
    for (int j = 0; j < NPT; ++j) {
        uint32_t h0, h1;
        b3_finish<false>(pre, nonce_of(base + (uint64_t)j * NT + threadIdx.x), 0u, h0, h1);
        key[j] = key64_of(h0, h1);
    }
    uint32_t slot[NPT];
#pragma unroll
    for (int j = 0; j < NPT; ++j) {
        const uint64_t nonce = base + (uint64_t)j * NT + threadIdx.x;
        const uint32_t bin = WIN ? key_bin<true>(d, key[j], bits) : (bits ? (uint32_t)(key[j] >> (64 - bits)) : 0u);
        // A record outside the window claims no slot: its slot reads as "none".
        slot[j] = (nonce < N && in_window<WM == kWinFilter>(d, key[j])) ? atomicAdd(&d.cnt2[bin], 1u)
                                                                         : 0xffffffffu;
    }
    bool overflow = false, hover = false;
#pragma unroll
    for (int j = 0; j < NPT; ++j) {
        const uint64_t nonce = base + (uint64_t)j * NT + threadIdx.x;
        if (nonce >= N) continue;
        if (WIN && slot[j] == 0xffffffffu) continue;
        const uint32_t bin = WIN ? key_bin<true>(d, key[j], bits) : (bits ? (uint32_t)(key[j] >> (64 - bits)) : 0u);
        if (slot[j] < cap) {
            const uint64_t at = (uint64_t)bin * cap + slot[j];
            d.b_keys[at] = key[j];
            d.b_nonces[at] = nonce_of(nonce);
        } else {
            overflow = true;
        }
        if (HALO) halo_add(d, bin, key[j], nonce_of(nonce), hover);
    }
    if (overflow) atomicOr(d.status, kStSlot2Overflow);
    if (hover) atomicOr(d.status, kStHaloOverflow);
}

template <bool HALO, int WM>
static cudaError_t launch_hd(const Desc *descs, int nplots, const uint32_t *tile_start,
                             uint32_t total_tiles, int chunk, On on)
{
    return launch_on(on, k_hash_direct<kHashThreads, kHashNoncesPerThread, HALO, WM>, total_tiles, kHashThreads, 0,
                     descs, nplots, tile_start, chunk);
}

cudaError_t launch_hash_direct(const Desc *descs, int nplots, const uint32_t *tile_start,
                               uint32_t total_tiles, int chunk, On on, HashCfg cfg)
{
    if (total_tiles == 0) return cudaSuccess;
    if (cfg.ids) return cudaErrorInvalidValue;
    if (cfg.list)
        return cfg.halo ? cudaErrorInvalidValue
                        : launch_hd<false, kWinList>(descs, nplots, tile_start, total_tiles, chunk, on);
    if (cfg.win)
        return cfg.halo ? launch_hd<true, kWinFilter>(descs, nplots, tile_start, total_tiles, chunk, on)
                        : launch_hd<false, kWinFilter>(descs, nplots, tile_start, total_tiles, chunk, on);
    return cfg.halo ? launch_hd<true, kWinNone>(descs, nplots, tile_start, total_tiles, chunk, on)
                    : launch_hd<false, kWinNone>(descs, nplots, tile_start, total_tiles, chunk, on);
}

// ------------------------------------------------ Table-2 pair hashing
// Fills hash2 of the Table-2 records {a, b, 0, 0} the sort wrote at their
// final offsets: a streaming, barrier-free pass (one compression per
// record, all lanes busy).  One launch covers one chunk of partitions --
// the records between the look-back prefixes at the chunk's ends -- so it
// can run on a second stream while the sort works on the next chunk.  A
// plot's CTAs stride over its range.  Skips plots whose Table 2 is invalid
// (capacity exceeded, a wait timed out).
constexpr int kT2HashThreads = 256;

__global__ void __launch_bounds__(kT2HashThreads) k_t2_hash(const Desc *__restrict__ descs,
                                                            int nplots,
                                                            const uint32_t *__restrict__ tile_start,
                                                            int chunk)
{
    constexpr int NT = kT2HashThreads;
    pdl_go();
    pdl_wait();
    const int plot = find_plot(tile_start, nplots, blockIdx.x);
    const Desc &d = descs[plot];
    if (*d.status & (kStT2Capacity | kStTimeout | kStBadTicket)) return;
    // Records of this partition chunk: [prefix before its first partition,
    // inclusive prefix of its last), from the sort's look-back words.
    const uint64_t np = 1ull << d.p;
    const uint64_t fa = np * (uint64_t)chunk / (uint64_t)d.pchunks;
    const uint64_t fb = np * (uint64_t)(chunk + 1) / (uint64_t)d.pchunks;
    if (fa >= fb) return;
    const uint64_t w = ld_acquire_u64(d.lb + (fb - 1));
    if ((w & ~kLbMask) != kLbIncl) return;  // chain broken: status says why
    const uint64_t lo = fa == 0 ? 0ull : d.t2off[fa];
    uint64_t hi = w & kLbMask;
    if (hi > d.t2cap) hi = d.t2cap;
    const uint32_t me = blockIdx.x - tile_start[plot];
    const uint32_t ctas = tile_start[plot + 1] - tile_start[plot];
    uint32_t g[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) g[i] = d.pre2[i];
    uint4 *__restrict__ t2 = reinterpret_cast<uint4 *>(d.t2);
    // Two records per step, loop kept rolled (see b3_finish).
    const uint64_t stride = (uint64_t)ctas * NT;
#pragma unroll 1
    for (uint64_t q = lo + (uint64_t)me * NT + threadIdx.x; q < hi; q += 2 * stride) {
        const uint4 v = t2[q];
        uint32_t h0, h1;
        if (q + stride < hi) {
            const uint4 u = t2[q + stride];
            uint32_t h2, h3;
            b3_finish<true>(g, v.x, v.y, h0, h1);
            b3_finish<true>(g, u.x, u.y, h2, h3);
            t2[q + stride] = make_uint4(u.x, u.y, h2, h3);
        } else {
            b3_finish<true>(g, v.x, v.y, h0, h1);
        }
        t2[q] = make_uint4(v.x, v.y, h0, h1);
    }
}

cudaError_t launch_t2_hash(const Desc *descs, int nplots, const uint32_t *tile_start,
                           uint32_t total_tiles, int chunk, On on)
{
    if (total_tiles == 0) return cudaSuccess;
    return launch_on(on, k_t2_hash, total_tiles, kT2HashThreads, 0, descs, nplots, tile_start, chunk);
}

// Pair hash of the slot placement (Sec. III-A, Table 2): CTA b takes
// partitions [8b, 8b + 8) of one plot, a warp each, whose pairs the sort
// left in the partitions' level-2 slots (pair k of partition f: key array of
// slot f for k < cap2, nonce array for k >= cap2) and whose Table-2 offsets
// the pair-count scan wrote.  Bound by the ALU pipe, so a pair costs little
// but its hash: a warp reads consecutive pairs and writes consecutive
// records at 32-bit indices, with no search for the pair's partition and no
// barrier; two hashes per step (see b3_finish).
__global__ void __launch_bounds__(kT2HashThreads) k_t2_hash_slots(const Desc *__restrict__ descs,
                                                                  int nplots,
                                                                  const uint32_t *__restrict__ tile_start,
                                                                  bool split)
{
    static_assert(kT2SlotGroup == kT2HashThreads / 32, "one partition per warp");
    pdl_go();
    pdl_wait();
    const int plot = find_plot(tile_start, nplots, blockIdx.x);
    const Desc &d = descs[plot];
    // The run's result, final since the scan before this kernel, goes
    // straight to the caller's pinned words (three copies less per run).
    if (d.result && !split && blockIdx.x == tile_start[plot] && threadIdx.x == 0) {
        d.result[0] = *d.status;
        d.result[1] = d.t2off[1ull << d.p];
        d.result[2] = d.t1off[1ull << d.p];
    }
    if (*d.status & (kStT2Capacity | kStTimeout | kStBadTicket | kStPairSlot)) return;
    const uint64_t np = 1ull << d.p;
    const uint64_t f = (uint64_t)(blockIdx.x - tile_start[plot]) * kT2SlotGroup + (threadIdx.x >> 5);
    if (f >= np) return;
    // The offsets exist only if the scan's chain reached its last chunk
    // (a broken chain has set a status bit, except for a withheld chunk 0
    // in a one-chunk scan).
    const uint64_t nchunks = (np + kScanChunk - 1) / kScanChunk;
    if (!split && (ld_acquire_u64(d.lb + (nchunks - 1)) & ~kLbMask) != kLbIncl) return;
    const uint64_t off = d.t2off[f];
    const uint32_t cap = d.cap2;
    const uint64_t P64 = d.t2off[f + 1] - off;
    if (P64 > cap + cap / 2u) return;  // past the pair slot: the sort left none
    const uint32_t P = (uint32_t)P64;
    if (off + P > d.t2cap) return;  // the scan flags this; never write past Table 2
    uint32_t g[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) g[i] = d.pre2[i];
    uint4 *__restrict__ t2 = reinterpret_cast<uint4 *>(d.t2) + off;
    const uint2 *__restrict__ ab = reinterpret_cast<const uint2 *>(d.b_keys + f * cap);
    const uint32_t lane = threadIdx.x & 31u;
    for (uint32_t seg = 0; seg < P; seg += cap) {  // key array, then nonce array
        const uint32_t n = min(P - seg, cap);
        // the next step's pairs are read before this step's hashes
        uint2 x = lane < n ? ab[lane] : make_uint2(0u, 0u);
        uint2 y = lane + 32 < n ? ab[lane + 32] : make_uint2(0u, 0u);
#pragma unroll 1
        for (uint32_t k0 = 0; k0 < n; k0 += 64) {
            const uint32_t k = k0 + lane;
            const uint2 nx = k + 64 < n ? ab[k + 64] : make_uint2(0u, 0u);
            const uint2 ny = k + 96 < n ? ab[k + 96] : make_uint2(0u, 0u);
            uint32_t h0, h1;
            if (k0 + 32 < n) {  // the same for the whole warp
                uint32_t h2, h3;
                b3_finish<true>(g, x.x, x.y, h0, h1);
                b3_finish<true>(g, y.x, y.y, h2, h3);
                if (k + 32 < n) t2[k + 32] = make_uint4(y.x, y.y, h2, h3);
            } else {
                b3_finish<true>(g, x.x, x.y, h0, h1);
            }
            if (k < n) t2[k] = make_uint4(x.x, x.y, h0, h1);
            x = nx;
            y = ny;
        }
        t2 += cap;
        ab = reinterpret_cast<const uint2 *>(d.b_nonces + f * cap);
    }
}

cudaError_t launch_t2_hash_slots(const Desc *descs, int nplots, const uint32_t *tile_start,
                                 uint32_t total_tiles, On on, bool split)
{
    if (total_tiles == 0) return cudaSuccess;
    return launch_on(on, k_t2_hash_slots, total_tiles, kT2HashThreads, 0, descs, nplots, tile_start, split);
}

// ------------------------------------------------ tiled plots: windows
// The first pass of a tiled plot: the window (top c <= 8 bits of key64) of
// every nonce, one byte each; four nonces per thread and one 32-bit store.
__global__ void __launch_bounds__(256) k_window_ids(uint32_t k0, uint32_t k1, uint32_t k2,
                                                    uint32_t k3, uint32_t k4, uint32_t k5,
                                                    uint32_t k6, uint32_t k7, uint64_t N, int c,
                                                    uint32_t *__restrict__ ids4)
{
    const uint32_t key[8] = {k0, k1, k2, k3, k4, k5, k6, k7};
    uint32_t pre[16];
    b3_key_setup(key, 4u, pre);
    const uint64_t words = (N + 3) / 4;
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < words; i += stride) {
        uint32_t packed = 0;
#pragma unroll 2
        for (int j = 0; j < 4; ++j) {
            const uint64_t nonce = 4 * i + j;
            uint32_t h0, h1;
            b3_finish<false>(pre, (uint32_t)nonce, 0u, h0, h1);
            const uint32_t id = bswap32(h0) >> (32 - c);  // key64's top c bits
            packed |= (nonce < N ? id : 0u) << (8 * j);
        }
        ids4[i] = packed;
    }
}

cudaError_t launch_window_ids(const uint32_t key[8], uint64_t N, int c, uint8_t *ids, cudaStream_t s)
{
    if (N == 0 || c < 1 || c > 8) return cudaErrorInvalidValue;
    uint64_t blocks = ((N + 3) / 4 + 255) / 256;
    if (blocks > 152ull * 64) blocks = 152ull * 64;
    k_window_ids<<<(unsigned)blocks, 256, 0, s>>>(key[0], key[1], key[2], key[3], key[4], key[5],
                                                  key[6], key[7], N, c,
                                                  reinterpret_cast<uint32_t *>(ids));
    return cudaGetLastError();
}

// A window's nonces (wids[n] == win) listed into wlist in any order (the
// partition sort orders records by (key64, nonce)): each CTA reads 4096
// window ids, 16 per thread, ranks its matches with one block scan and
// claims their places with one atomic on wcount.  Entries past the list's
// capacity are dropped and reported.
constexpr int kListThreads = 256;
constexpr int kListPerThread = 16;

__global__ void __launch_bounds__(kListThreads) k_window_list(const Desc *__restrict__ dp, uint64_t N)
{
    __shared__ uint32_t ws[kListThreads / 32 + 1];
    __shared__ uint32_t s_base;
    pdl_go();
    pdl_wait();
    const Desc &d = *dp;
    const uint64_t n0 = ((uint64_t)blockIdx.x * kListThreads + threadIdx.x) * kListPerThread;
    uint4 v = make_uint4(0u, 0u, 0u, 0u);
    if (n0 < N) v = *reinterpret_cast<const uint4 *>(d.wids + n0);  // ids rounded up to 16 bytes
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
    uint32_t match = 0;  // bit b: nonce n0 + b is in the window
#pragma unroll
    for (int b = 0; b < kListPerThread; ++b) {
        const bool m = n0 + b < N && ((w[b >> 2] >> (8 * (b & 3))) & 0xffu) == d.win;
        match |= (m ? 1u : 0u) << b;
    }
    uint32_t total;
    const uint32_t r = block_exclusive_scan_u32<kListThreads>((uint32_t)__popc(match), ws, &total);
    if (threadIdx.x == 0) s_base = total ? atomicAdd(d.wcount, total) : 0u;
    __syncthreads();
    uint32_t at = s_base + r;
    bool over = false;
    for (int b = 0; b < kListPerThread; ++b) {
        if (!(match >> b & 1u)) continue;
        if (at < d.listcap) d.wlist[at] = (uint32_t)(n0 + b);
        else over = true;
        ++at;
    }
    if (over) atomicOr(d.status, kStWinList);
}

cudaError_t launch_window_list(const Desc *desc, uint64_t N, cudaStream_t s)
{
    const uint64_t per = (uint64_t)kListThreads * kListPerThread;
    const uint64_t blocks = (N + per - 1) / per;
    if (blocks == 0 || blocks > 0x7FFFFFFFull) return cudaErrorInvalidValue;
    k_window_list<<<(unsigned)blocks, kListThreads, 0, s>>>(desc, N);
    return cudaGetLastError();
}

// --------------------------------------------------- stand-alone hashing
// Records {nonce, h0, h1} of nonces nonce0 .. nonce0+count-1, nonce order.
__global__ void __launch_bounds__(256) k_hash_records(uint32_t k0, uint32_t k1, uint32_t k2,
                                                      uint32_t k3, uint32_t k4, uint32_t k5,
                                                      uint32_t k6, uint32_t k7, uint64_t nonce0,
                                                      uint64_t count, uint32_t *__restrict__ out)
{
    const uint32_t key[8] = {k0, k1, k2, k3, k4, k5, k6, k7};
    uint32_t pre[16];
    b3_key_setup(key, 4u, pre);
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += stride) {
        const uint32_t nonce = (uint32_t)(nonce0 + i);
        uint32_t h0, h1;
        b3_finish<false>(pre, nonce, 0u, h0, h1);
        out[3 * i] = nonce;
        out[3 * i + 1] = h0;
        out[3 * i + 2] = h1;
    }
}

cudaError_t launch_hash_records(const uint32_t key[8], uint64_t nonce0, uint64_t count,
                                uint32_t *out, cudaStream_t s)
{
    if (count == 0) return cudaSuccess;
    uint64_t blocks = (count + 255) / 256;
    if (blocks > 152ull * 64) blocks = 152ull * 64;
    k_hash_records<<<(unsigned)blocks, 256, 0, s>>>(key[0], key[1], key[2], key[3], key[4],
                                                      key[5], key[6], key[7], nonce0, count, out);
    return cudaGetLastError();
}

// Hash-only ceiling of the Table-1 hash: keyed BLAKE3 of nonces nonce0 ..
// nonce0 + count - 1 in the Table-1 kernel's shape (256 threads, a rolled
// loop of two nonces per thread and step, key state from the per-key setup),
// with no record stores: each thread folds its hash words into one word,
// stored once.  It measures how fast the integer pipes run this instruction
// mix with no memory work beside it.  Grid-stride over pairs of nonces.
__global__ void __launch_bounds__(256) k_hash_peak(uint32_t k0, uint32_t k1, uint32_t k2,
                                                   uint32_t k3, uint32_t k4, uint32_t k5,
                                                   uint32_t k6, uint32_t k7, uint64_t nonce0,
                                                   uint64_t count, uint32_t *__restrict__ fold)
{
    const uint32_t key[8] = {k0, k1, k2, k3, k4, k5, k6, k7};
    uint32_t pre[16];
    b3_key_setup(key, 4u, pre);
    uint32_t acc = 0;
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
#pragma unroll 1
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += 2 * stride) {
        uint32_t h0, h1, g0, g1;
        b3_finish<false>(pre, (uint32_t)(nonce0 + i), 0u, h0, h1);
        b3_finish<false>(pre, (uint32_t)(nonce0 + i + stride), 0u, g0, g1);
        acc ^= h0 ^ h1 ^ (i + stride < count ? g0 ^ g1 : 0u);
    }
    fold[(uint64_t)blockIdx.x * blockDim.x + threadIdx.x] = acc;
}

cudaError_t launch_hash_peak(const uint32_t key[8], uint64_t nonce0, uint64_t count, uint32_t *fold,
                             uint32_t blocks, cudaStream_t s)
{
    if (blocks == 0) return cudaErrorInvalidValue;
    k_hash_peak<<<blocks, kHashThreads, 0, s>>>(key[0], key[1], key[2], key[3], key[4], key[5],
                                                key[6], key[7], nonce0, count, fold);
    return cudaGetLastError();
}

// Table-2 records {a, b, g0, g1} of the pairs (a, b).
__global__ void __launch_bounds__(256) k_pair_hash(uint32_t k0, uint32_t k1, uint32_t k2,
                                                   uint32_t k3, uint32_t k4, uint32_t k5,
                                                   uint32_t k6, uint32_t k7,
                                                   const uint2 *__restrict__ pairs, uint64_t count,
                                                   uint4 *__restrict__ out)
{
    const uint32_t key[8] = {k0, k1, k2, k3, k4, k5, k6, k7};
    uint32_t pre[16];
    b3_key_setup(key, 8u, pre);
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += stride) {
        const uint2 ab = pairs[i];
        uint32_t g0, g1;
        b3_finish<true>(pre, ab.x, ab.y, g0, g1);
        out[i] = make_uint4(ab.x, ab.y, g0, g1);
    }
}

cudaError_t launch_pair_hash(const uint32_t key[8], const uint32_t *pairs, uint64_t count,
                             uint4 *out, cudaStream_t s)
{
    if (count == 0) return cudaSuccess;
    uint64_t blocks = (count + 255) / 256;
    if (blocks > 152ull * 64) blocks = 152ull * 64;
    k_pair_hash<<<(unsigned)blocks, 256, 0, s>>>(key[0], key[1], key[2], key[3], key[4], key[5],
                                                   key[6], key[7],
                                                   reinterpret_cast<const uint2 *>(pairs), count,
                                                   out);
    return cudaGetLastError();
}

}  // namespace vx
