// Dedup of a gradient batch: a stable LSD radix sort of (row id, position)
// pairs, then the runs of the sorted row ids.
//
// The sort key is the 32-bit row id, not the 64-bit key: rows are dense in
// [0, capacity), so 3 passes of 9 bits cover 10^8 rows (against 5+ passes for
// 40-bit keys), and the sorted order visits rows in memory order.  An absent
// lookup is given the all-ones digit pattern and sorts last.
//
// Each pass is a reduce-then-scan pass over tiles of 4096 elements (2048 in
// batches of fewer than kSortSmallBatch lookups, which would otherwise cover a
// fraction of the SMs): the digit counts of every tile and the pass's digit
// totals come first; then every (tile, digit) needs the output position of its
// first element (the elements of lower digits plus those of the digit in
// earlier tiles); and the scatter ranks each tile's elements stably (over
// rounds of 32, in order) and writes them out.  The positions are made by a
// kernel of their own in large batches (416 tiles of a 1.7M-lookup batch), and
// in small ones by each block of the scatter for itself: it reads the packed
// counts of the tiles before its own (200k lookups: at most 97 rows of 512 or
// 1,024 bytes) beside its elements, which costs less than the launch of a
// kernel between two passes.  (Apply + Get of 200k lookups of dim 100: 153 ->
// 140 us; apply + export of 100,003 of dim 50: 88.7 -> 78.  At 2^19 lookups the
// blocks read 33 MB of counts a pass, as long as the offsets kernel takes.)  The
// counts of the first pass are made by the probe and the miss kernel
// (FirstCounts), or by a histogram kernel where the rows come from elsewhere (a
// tiered apply); those of every later pass by the scatter before it, which
// knows the tile each element lands in and adds the element's next digit to
// that tile's count (one add per run of equal targets in a warp), so no pass
// after the first reads its input twice.  No block waits on another, so a pass
// costs the same when the sort shares the GPU with other kernels.  (A
// single-pass decoupled look-back sort was slower here: a batch is about one
// wave of tiles, and the chain of tiles that know their prefix grows one
// window per round trip.)
#include "mlkv_internal.cuh"

namespace mlkv {

namespace {

// the tiles of the dedup's output (k_seg_count, k_dedup_out), and the block of
// the histogram and offsets kernels
constexpr int kThreads = 256;
constexpr int kItems = 16;
constexpr int kTile = kThreads * kItems;  // 4096

// Exclusive scan of one value per thread over a block of THREADS threads.
template <int THREADS>
__device__ __forceinline__ uint32_t block_exclusive_scan_n(uint32_t v, uint32_t& total) {
    constexpr int kWarps = THREADS / 32;
    __shared__ uint32_t warp_sums[kWarps];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint32_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) warp_sums[w] = x;
    __syncthreads();
    if (w == 0) {
        uint32_t s = lane < kWarps ? warp_sums[lane] : 0u;
#pragma unroll
        for (int o = 1; o < kWarps; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= o) s += y;
        }
        if (lane < kWarps) warp_sums[lane] = s;
    }
    __syncthreads();
    const uint32_t wprefix = w ? warp_sums[w - 1] : 0u;
    total = warp_sums[kWarps - 1];
    __syncthreads();
    return wprefix + x - v;
}

__device__ __forceinline__ uint32_t block_exclusive_scan(uint32_t v, uint32_t& total) {
    return block_exclusive_scan_n<kThreads>(v, total);
}

// Sum of tile_sums[0..b) by the whole block.
__device__ __forceinline__ uint32_t tiles_before(const uint32_t* __restrict__ tile_sums, uint32_t b) {
    uint32_t s = 0;
    for (uint32_t i = threadIdx.x; i < b; i += kThreads) s += tile_sums[i];
    uint32_t total;
    block_exclusive_scan(s, total);
    return total;
}

// --- radix sort ---------------------------------------------------------------
// Pass 0 reads the probe's row ids (sentinels mapped to `sent`) and uses the
// lookup position as the value.
__device__ __forceinline__ uint32_t sort_key(uint32_t r, uint32_t sent, bool first) {
    return first ? (r >= ROW_ABSENT ? sent : r) : r;
}

constexpr int kMaxRadix = kSortMaxRadix;

// Lanes of the warp whose (valid, digit) equals this lane's: one ballot per
// digit bit (the warp-level multisplit of Ashkiani, Davidson, Meyer and Owens,
// "GPU Multisplit", 2016).
__device__ __forceinline__ uint32_t digit_peers(uint32_t dig, bool valid, int bits) {
    const uint32_t vm = __ballot_sync(0xffffffffu, valid);
    uint32_t peers = valid ? vm : ~vm;
    for (int b = 0; b < bits; ++b) {
        const bool one = (dig >> b) & 1u;
        const uint32_t m = __ballot_sync(0xffffffffu, one);
        peers &= one ? m : ~m;
    }
    return peers;
}

// The same from a word per digit of the warp's own in shared memory (all zero;
// the lane that counts the digit zeroes its word again).  About a quarter of the
// instructions, but an atomic in shared memory: faster where few warps share an
// SM (tiles of 2048, one or two blocks per SM: 200k lookups 136.5 -> 134.5 us,
// 65,536 of dim 512 165.9 -> 163.9), slower with 48 (1.7M lookups 546.8 -> 550.7).
__device__ __forceinline__ uint32_t digit_peers_by_mask(uint32_t* mask, uint32_t dig, bool valid, int lane) {
    if (valid) atomicOr(mask + dig, 1u << lane);
    __syncwarp();
    return valid ? mask[dig] : 0u;
}

// Digit counts of one tile, written to column `tile` of counts[d][tile], and
// added to the pass's digit totals dtot[d]: the first pass of a sort whose
// counts the probe did not make.  A thread counts consecutive elements and
// adds a run of equal digits with one atomic.
template <int TILE>
__global__ void __launch_bounds__(kThreads) k_sort_hist(const uint32_t* __restrict__ kin, uint32_t n,
                                                        uint32_t* __restrict__ counts, uint32_t* __restrict__ dtot,
                                                        uint32_t ntiles, int shift, int radix, uint32_t sent,
                                                        int first, int packed) {
    constexpr int kItems = TILE / kThreads;
    static_assert(kItems % 4 == 0, "whole 16-byte loads");
    pdl_enter();
    __shared__ uint32_t hist[kMaxRadix];
    for (int d = threadIdx.x; d < radix; d += kThreads) hist[d] = 0;
    __syncthreads();
    const uint32_t i0 = blockIdx.x * TILE + threadIdx.x * kItems;
    uint32_t key[kItems];
    if (i0 + kItems <= n) {  // consecutive keys, 16-byte aligned
        const uint4* src = reinterpret_cast<const uint4*>(kin + i0);
#pragma unroll
        for (int q = 0; q < kItems / 4; ++q) {
            const uint4 v = __ldg(src + q);
            key[4 * q] = v.x;
            key[4 * q + 1] = v.y;
            key[4 * q + 2] = v.z;
            key[4 * q + 3] = v.w;
        }
    } else {
#pragma unroll
        for (int r = 0; r < kItems; ++r) key[r] = i0 + r < n ? kin[i0 + r] : 0u;
    }
    uint32_t cur = 0xFFFFFFFFu, cnt = 0;
#pragma unroll
    for (int r = 0; r < kItems; ++r) {
        if (i0 + r >= n) break;
        const uint32_t dig = (sort_key(key[r], sent, first) >> shift) & (radix - 1);
        if (dig != cur) {
            if (cnt) atomicAdd(&hist[cur], cnt);
            cur = dig;
            cnt = 0;
        }
        ++cnt;
    }
    if (cnt) atomicAdd(&hist[cur], cnt);
    __syncthreads();
    put_counts(hist, counts, packed != 0, ntiles, radix, blockIdx.x, dtot);
}

// Output position of the first element of every (tile, digit): the elements
// of all lower digits, plus those of digit d in earlier tiles; written to
// offsets[tile][d].  Each block of OT
// threads first scans the pass's digit totals (all of them) for the elements
// of the lower digits; then a warp per digit scans the digit's counts over the
// tiles, 32 tiles a round, with the loads of 16 rounds issued together (every
// tile of a batch of up to 2M lookups in one round trip).
#ifndef MLKV_OFFSETS_THREADS
#define MLKV_OFFSETS_THREADS 256
#endif
constexpr int kOThreads = MLKV_OFFSETS_THREADS;
#ifndef MLKV_OFFSETS_PDL
#define MLKV_OFFSETS_PDL 0
#endif
__global__ void __launch_bounds__(kOThreads) k_sort_offsets(const uint32_t* __restrict__ counts,
                                                            const uint32_t* __restrict__ dtot,
                                                            uint32_t* __restrict__ offsets, uint32_t ntiles,
                                                            int radix) {
    pdl_enter();
    constexpr int kPer = kMaxRadix / kOThreads;  // digit totals per thread
    constexpr int kRounds = 16;
    __shared__ uint32_t lower[kMaxRadix];  // elements of the digits below each digit
    {
        const int i0 = kPer * threadIdx.x;
        uint32_t v[kPer], sum = 0;
#pragma unroll
        for (int k = 0; k < kPer; ++k) {
            v[k] = i0 + k < radix ? __ldg(dtot + i0 + k) : 0u;
            sum += v[k];
        }
        uint32_t total;
        uint32_t ex = block_exclusive_scan_n<kOThreads>(sum, total);
#pragma unroll
        for (int k = 0; k < kPer; ++k) {
            lower[i0 + k] = ex;
            ex += v[k];
        }
    }
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const int d = blockIdx.x * (kOThreads / 32) + (threadIdx.x >> 5);
    if (d >= radix) return;  // warp-uniform
    const uint32_t* row = counts + (size_t)d * ntiles;
    uint32_t run = lower[d];
    for (uint32_t t0 = 0; t0 < ntiles; t0 += 32 * kRounds) {
        uint32_t c[kRounds];
#pragma unroll
        for (int k = 0; k < kRounds; ++k) {
            const uint32_t t = t0 + 32 * k + lane;
            c[k] = t < ntiles ? __ldg(row + t) : 0u;
        }
#pragma unroll
        for (int k = 0; k < kRounds; ++k) {
            if (t0 + 32 * k >= ntiles) break;  // warp-uniform
            const uint32_t t = t0 + 32 * k + lane;
            uint32_t x = c[k];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
                if (lane >= o) x += y;
            }
            if (t < ntiles) offsets[(size_t)t * radix + d] = run + x - c[k];
            run += __shfl_sync(0xffffffffu, x, 31);
        }
    }
}

// Stable rank of each element of the tile among equal digits; the tile is
// then laid out in shared memory in sorted order and written out so that
// consecutive threads write consecutive addresses of a digit's run (a direct
// scatter from registers costs one L2 sector per element).  The block has
// THREADS threads; warp w owns elements w*kSItems*32 .. of the tile, in
// rounds of 32 consecutive elements (more warps a tile: fewer rounds each).
// An element of digit d goes to offsets[tile][d] plus its rank among the
// tile's elements of digit d.  With nshift >= 0 the element's digit of the
// next pass (bits nshift ..) is added to the count of the tile of the next
// pass that holds its output position (dst / TILE; ncounts, laid out as
// add_count has it, zero on entry), and to the next pass's digit totals ndtot.  The counts and totals of
// the pass before (zcounts, zdtot) are zeroed here: every block of this pass
// reads its own pass's, so the next kernel zeroes those.
// With SELF the block adds up offsets from `counts` (packed) itself.
#ifndef MLKV_SCATTER_MIN_BLOCKS
#define MLKV_SCATTER_MIN_BLOCKS 3
#endif
// dynamic shared memory with SELF (512 threads): masks and counts
constexpr size_t kScatterDyn = (size_t)16 * kMaxRadix * (4 + 2);
struct ScatterArgs {
    const uint32_t* kin;
    const uint32_t* vin;
    uint32_t* kout;
    uint32_t* vout;
    uint32_t n;
    const uint32_t* offsets;  // [tile][radix] (without SELF)
    const uint32_t* counts;   // this pass's counts and digit totals (SELF)
    const uint32_t* dtot;
    uint32_t ntiles;
    int shift, radix;
    uint32_t sent;
    int first;
    int nshift;
    uint32_t* ncounts;
    uint32_t* ndtot;
    uint32_t* zcounts;  // or null
    uint32_t* zdtot;
};

template <int TILE, int THREADS, bool SELF>
__global__ void __launch_bounds__(THREADS, SELF ? 2 : MLKV_SCATTER_MIN_BLOCKS) k_sort_scatter(ScatterArgs s) {
    constexpr int kSWarps = THREADS / 32;
    constexpr int kSItems = TILE / THREADS;
    constexpr int kTileShift = TILE == 4096 ? 12 : 11;
    static_assert(TILE == (1 << kTileShift), "tiles of 2048 or 4096");
    pdl_enter();
    const uint32_t* __restrict__ kin = s.kin;
    const uint32_t* __restrict__ vin = s.vin;
    const uint32_t n = s.n, sent = s.sent, ntiles = s.ntiles;
    const int shift = s.shift, radix = s.radix, first = s.first, nshift = s.nshift;
    const uint32_t tile0 = blockIdx.x * TILE;
    const uint32_t base = tile0 + (threadIdx.x >> 5) * (kSItems * 32);
    uint32_t key[kSItems], val[kSItems];
    // all loads together; with SELF (and its registers) beside the zeroing too
    auto load = [&]() {
#pragma unroll
        for (int r = 0; r < kSItems; ++r) {
            const uint32_t i = base + r * 32 + (threadIdx.x & 31);
            key[r] = i < n ? sort_key(kin[i], sent, first) : 0u;
            val[r] = i < n ? (first ? i : vin[i]) : 0u;
        }
    };
    if (SELF) load();
    if (s.zcounts) {
        // this tile's share of the counts of the pass before
        const uint32_t words = SELF ? radix / 2 : radix;
        for (uint32_t d = threadIdx.x; d < words; d += THREADS) {
            if (SELF) s.zcounts[(size_t)blockIdx.x * words + d] = 0u;
            else s.zcounts[(size_t)d * ntiles + blockIdx.x] = 0u;
        }
        if (blockIdx.x == 0)
            for (int d = threadIdx.x; d < radix; d += THREADS) s.zdtot[d] = 0u;
    }
    // the per-warp digit counts, then (once every position is known) the sorted tile
    constexpr int kCounts = kSWarps * kMaxRadix;
    constexpr int kPool = SELF || 2 * TILE > kCounts ? 2 * TILE : kCounts;
    __shared__ uint32_t pool[kPool];
    // SELF: [warp][digit] lane masks and 16-bit counts of their own
    extern __shared__ __align__(16) uint32_t dyn[];
    using Count = typename std::conditional<SELF, uint16_t, uint32_t>::type;
    Count* wcnts = reinterpret_cast<Count*>(SELF ? dyn + kCounts : pool);
    uint32_t* skey = pool;
    uint32_t* sval = pool + TILE;
    __shared__ uint32_t part[SELF ? 2 * THREADS : 1];  // per group of threads: counts of the tiles before this one
    __shared__ uint32_t gbase[kMaxRadix];   // output position of the tile's first element of each digit
    __shared__ uint32_t lbase[kMaxRadix];   // position in the sorted tile of its first element of each digit
    __shared__ uint32_t ntot[kMaxRadix];    // the tile's elements of each digit of the next pass
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    Count* wcnt = wcnts + w * kMaxRadix;
    uint32_t* mask = dyn + w * kMaxRadix;
    // the counts (and the masks before them)
    uint4* zero = reinterpret_cast<uint4*>(SELF ? dyn : pool);
    for (int i = threadIdx.x; i < (SELF ? kCounts + kCounts / 2 : kCounts) / 4; i += THREADS)
        zero[i] = make_uint4(0u, 0u, 0u, 0u);
    for (int d = threadIdx.x; d < radix; d += THREADS) {
        if (!SELF) gbase[d] = s.offsets[(size_t)blockIdx.x * radix + d];
        ntot[d] = 0u;
    }
    __syncthreads();
    const int digit_bits = __ffs(radix) - 1;
    const uint32_t lt = lanemask_lt();
    uint32_t rnk[kSItems];
    if (!SELF) load();
    if (SELF) {  // beside them, the counts of the tiles before: a group of radix / 2 threads per row
        const uint32_t words = radix / 2, groups = THREADS / words;
        const uint32_t grp = threadIdx.x / words, x = threadIdx.x & (words - 1);
        uint32_t lo = 0, hi = 0;
        constexpr int kRows = 16;  // in flight
        for (uint32_t t0 = grp; t0 < blockIdx.x; t0 += groups * kRows) {
            uint32_t c[kRows];
#pragma unroll
            for (int k = 0; k < kRows; ++k) {
                const uint32_t t = t0 + k * groups;
                c[k] = t < blockIdx.x ? __ldg(s.counts + (size_t)t * words + x) : 0u;
            }
#pragma unroll
            for (int k = 0; k < kRows; ++k) {
                lo += c[k] & 0xFFFFu;
                hi += c[k] >> 16;
            }
        }
        part[grp * radix + 2 * x] = lo;
        part[grp * radix + 2 * x + 1] = hi;
    }
#pragma unroll
    for (int r = 0; r < kSItems; ++r) {
        const bool valid = base + r * 32 + lane < n;
        const uint32_t dig = (key[r] >> shift) & (radix - 1);
        const uint32_t peers =
            SELF ? digit_peers_by_mask(mask, dig, valid, lane) : digit_peers(dig, valid, digit_bits);
        uint32_t before = 0;
        if (valid) before = wcnt[dig];
        __syncwarp();
        if (valid && lane == __ffs(peers) - 1) {
            wcnt[dig] = (Count)(before + __popc(peers));
            if (SELF) mask[dig] = 0u;
        }
        __syncwarp();
        rnk[r] = valid ? before + __popc(peers & lt) : 0xFFFFFFFFu;
    }
    __syncthreads();
    // per digit, a thread each: exclusive prefix over the warps; per tile: exclusive
    // prefix over the digits
    static_assert(THREADS >= kMaxRadix, "a thread per digit");
    const int d = threadIdx.x;
    uint32_t mine = 0;
    if (d < radix) {
#pragma unroll
        for (int ww = 0; ww < kSWarps; ++ww) {
            const uint32_t c = wcnts[ww * kMaxRadix + d];
            wcnts[ww * kMaxRadix + d] = (Count)mine;
            mine += c;
        }
    }
    uint32_t all;
    const uint32_t run = block_exclusive_scan_n<THREADS>(mine, all);
    if (SELF) {  // the elements of lower digits, and the digit's in the tiles before
        uint32_t total;
        uint32_t at = block_exclusive_scan_n<THREADS>(d < radix ? __ldg(s.dtot + d) : 0u, total);
        if (d < radix) {
            for (int g = 0; g < 2 * THREADS / radix; ++g) at += part[g * radix + d];
            gbase[d] = at;
        }
    }
    if (d < radix) lbase[d] = run;
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kSItems; ++r) {
        if (rnk[r] == 0xFFFFFFFFu) continue;
        const uint32_t dig = (key[r] >> shift) & (radix - 1);
        rnk[r] += lbase[dig] + wcnt[dig];  // position in the sorted tile
    }
    if (!SELF) __syncthreads();  // the counts are dead: the buffer takes the sorted tile
#pragma unroll
    for (int r = 0; r < kSItems; ++r) {
        if (rnk[r] == 0xFFFFFFFFu) continue;
        skey[rnk[r]] = key[r];
        sval[rnk[r]] = val[r];
    }
    __syncthreads();
    const uint32_t cnt = n - tile0 < (uint32_t)TILE ? n - tile0 : (uint32_t)TILE;
    if (nshift < 0) {
        for (uint32_t l = threadIdx.x; l < cnt; l += THREADS) {
            const uint32_t k = skey[l];
            const uint32_t dig = (k >> shift) & (radix - 1);
            const uint32_t dst = gbase[dig] + (l - lbase[dig]);
            s.kout[dst] = k;
            s.vout[dst] = sval[l];
        }
        return;
    }
    // every lane of the warp takes part in each round (the last may be partial)
    for (uint32_t l0 = threadIdx.x - lane; l0 < cnt; l0 += THREADS) {
        const uint32_t l = l0 + lane;
        const bool valid = l < cnt;
        uint32_t target = 0xFFFFFFFFu, e = 0;
        if (valid) {
            const uint32_t k = skey[l];
            const uint32_t dig = (k >> shift) & (radix - 1);
            const uint32_t dst = gbase[dig] + (l - lbase[dig]);
            s.kout[dst] = k;
            s.vout[dst] = sval[l];
            e = (k >> nshift) & (radix - 1);
            target = SELF ? (dst >> kTileShift) * (uint32_t)radix + e : e * ntiles + (dst >> kTileShift);
        }
        // consecutive lanes with one target (a hot row's lookups, a digit's
        // run within one tile) add their count once, from the run's first lane
        const uint32_t prev = __shfl_up_sync(0xffffffffu, target, 1);
        const bool head = valid && (lane == 0 || prev != target);
        const uint32_t heads = __ballot_sync(0xffffffffu, head);
        const uint32_t nvalid = __popc(__ballot_sync(0xffffffffu, valid));
        if (head) {
            const uint32_t later = heads & ~((2u << lane) - 1u);
            const uint32_t len = (later ? (uint32_t)(__ffs(later) - 1) : nvalid) - (uint32_t)lane;
            if (SELF) atomicAdd(s.ncounts + target / 2, len << (16 * (target & 1u)));  // packed
            else atomicAdd(s.ncounts + target, len);
            atomicAdd(&ntot[e], len);
        }
    }
    __syncthreads();
    for (int d = threadIdx.x; d < radix; d += THREADS) {
        const uint32_t c = ntot[d];
        if (c) atomicAdd(s.ndtot + d, c);
    }
}

// --- the dedup's output ----------------------------------------------------------
// The runs of the sorted row ids, as (first lookup's key, length) in order: the
// run heads of every tile of 4096 counted, then every tile finds its heads
// again, knows from the counts how many are before them, and writes its runs.
// A thread takes 16 consecutive elements (four 16-byte loads).  Bound by the
// sorted arrays' 8 bytes a lookup in L2 and the random 8-byte key of each run.
// (1.7M lookups, 0.31M runs: 44 us for three kernels that read a thread's 16
// elements one by one and kept the runs' starts in memory between them, 19 for
// these two.)

// A bit per element of this thread's 16 from position `first`: a run starts there.
__device__ __forceinline__ uint32_t head_bits(const uint32_t* __restrict__ srow, uint32_t first, uint32_t n,
                                              uint32_t sent) {
    uint32_t r[kItems];
    if (first + kItems <= n) {
        const uint4* v = reinterpret_cast<const uint4*>(srow + first);
#pragma unroll
        for (int q = 0; q < kItems / 4; ++q) {
            const uint4 x = __ldg(v + q);
            r[4 * q] = x.x;
            r[4 * q + 1] = x.y;
            r[4 * q + 2] = x.z;
            r[4 * q + 3] = x.w;
        }
    } else {
#pragma unroll
        for (int k = 0; k < kItems; ++k) r[k] = first + k < n ? __ldg(srow + first + k) : sent;
    }
    uint32_t left = first && first < n ? __ldg(srow + first - 1) : ~r[0];
    uint32_t bits = 0;
#pragma unroll
    for (int k = 0; k < kItems; ++k) {
        if (r[k] != left && r[k] != sent) bits |= 1u << k;
        left = r[k];
    }
    return bits;
}

__global__ void __launch_bounds__(kThreads) k_seg_count(const uint32_t* __restrict__ srow, uint32_t n, uint32_t sent,
                                                        uint32_t* __restrict__ tile_sums, SortTail tail) {
    pdl_enter();
    zero_tail(tail);
    const uint32_t first = blockIdx.x * kTile + threadIdx.x * kItems;
    uint32_t total;
    block_exclusive_scan((uint32_t)__popc(head_bits(srow, first, n, sent)), total);
    if (threadIdx.x == 0) tile_sums[blockIdx.x] = total;
}

// The end of the run of `row` that holds position q - 1: the first position
// from q on with another row, or n (the whole warp; the rows ascend).
__device__ __forceinline__ uint32_t end_from(const uint32_t* __restrict__ srow, uint32_t n, uint32_t q, uint32_t row,
                                             int lane) {
    uint32_t lo = q, hi = n;  // every position before lo holds row; hi is n or holds another
    while (lo < hi) {
        const uint32_t step = (hi - lo + 31) / 32;
        const unsigned long long at = (unsigned long long)lo + (unsigned long long)step * lane;
        const bool eq = at < hi && __ldg(srow + at) == row;
        const uint32_t c = __popc(__ballot_sync(0xffffffffu, eq));
        if (c == 0) return lo;
        const unsigned long long nhi = (unsigned long long)lo + (unsigned long long)step * c;
        lo += step * (c - 1) + 1;
        if (nhi < hi) hi = (uint32_t)nhi;
    }
    return hi;
}

__global__ void __launch_bounds__(kThreads) k_dedup_out(const int64_t* __restrict__ keys,
                                                        const uint32_t* __restrict__ srow,
                                                        const uint32_t* __restrict__ spos, uint32_t n, uint32_t sent,
                                                        const uint32_t* __restrict__ tile_sums,
                                                        int64_t* __restrict__ uniq, int32_t* __restrict__ counts,
                                                        int64_t* num, DevState* ds) {
    pdl_enter();
    __shared__ uint32_t at[kTile + 1];  // the tile's run heads, in order
    const uint32_t tile0 = blockIdx.x * kTile, first = tile0 + threadIdx.x * kItems;
    const uint32_t bits = head_bits(srow, first, n, sent);
    const uint32_t prefix = tiles_before(tile_sums, blockIdx.x);
    uint32_t heads;
    uint32_t r = block_exclusive_scan((uint32_t)__popc(bits), heads);
    for (uint32_t m = bits; m; m &= m - 1) at[r++] = first + (uint32_t)__ffs(m) - 1u;
    __syncthreads();
    if (heads && threadIdx.x < 32) {  // the last run may go on in later tiles
        const uint32_t s = at[heads - 1], row = __ldg(srow + s);
        const uint32_t e = end_from(srow, n, s + 1, row, (int)threadIdx.x);
        if (threadIdx.x == 0) at[heads] = e;
    }
    __syncthreads();
    for (uint32_t u = threadIdx.x; u < heads; u += kThreads) {
        const uint32_t s = at[u];
        // between two heads of a tile there is nothing but runs; lookups without a row sort last
        uniq[prefix + u] = __ldg(keys + __ldg(spos + s));
        counts[prefix + u] = (int32_t)(at[u + 1] - s);
    }
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) {
        *num = (int64_t)(prefix + heads);
        ds->last_unique = prefix + heads;
    }
}

inline unsigned tiles(int64_t n) { return (unsigned)((n + kTile - 1) / kTile); }

}  // namespace

namespace {
// Passes and digit width for ids of `bits` bits: the fewest passes of at most
// kSortMaxDigitBits bits, the bits spread evenly over them.
void sort_geometry(int bits, int& passes, int& D) {
    passes = (bits + kSortMaxDigitBits - 1) / kSortMaxDigitBits;
    D = (bits + passes - 1) / passes;
}
}  // namespace

inline unsigned sort_tiles(int64_t n) {
    const int sh = sort_tile_shift(n);
    return (unsigned)((n + (1 << sh) - 1) >> sh);
}

FirstCounts first_counts(mlkv_table* t, int64_t n) {
    int passes, D;
    sort_geometry(t->sort_bits, passes, D);
    const int shift = sort_tile_shift(n);
    return FirstCounts{t->s.sort_counts[0], t->s.sort_dtot, sort_tiles(n), 1 << D,
                       (uint32_t)((1ull << t->sort_bits) - 1), shift, shift == kSortTileSmallShift ? 1 : 0};
}

namespace {
template <int TILE, int THREADS, bool SELF>
void sort_passes(mlkv_table* t, int64_t n, cudaStream_t st, const uint32_t** srow, const uint32_t** spos,
                 bool first_counted, int passes, int D, SortTail& tail) {
    const int radix = 1 << D;
    const uint32_t sent = (uint32_t)((1ull << t->sort_bits) - 1);
    const unsigned nt = sort_tiles(n);
    // Three count buffers in turn: pass p reads counts[p % 3], counts pass p + 1
    // into counts[(p + 1) % 3] and zeroes the one pass p - 1 read; the kernel
    // after the sort zeroes the last pass's (tail).  So all are zero between
    // sorts but the first pass's, which is written whole, by the probe or the
    // histogram kernel.  The digit totals likewise, one array a pass.
    ScatterArgs a{};
    a.kin = t->s.row_of_pos;
    a.n = (uint32_t)n;
    a.offsets = t->s.sort_offsets;
    a.ntiles = nt;
    a.radix = radix;
    a.sent = sent;
    int out = 0;
    for (int p = 0; p < passes; ++p) {
        uint32_t* counts = t->s.sort_counts[p % 3];
        uint32_t* dtot = t->s.sort_dtot + p * kMaxRadix;
        if (p == 0 && !first_counted)
            MLKV_LAUNCH(t, 0, k_sort_hist<TILE>, nt, kThreads, 0, st, a.kin, (uint32_t)n, counts, dtot, nt, 0, radix,
                        sent, 1, SELF ? 1 : 0);
        // launched after the kernel before it has finished, not beside its
        // drain: placed early, its few blocks landed on the SMs the scatter
        // left room on (a tenth of them) and took twice as long
        if (!SELF)
            MLKV_LAUNCH_PDL(MLKV_OFFSETS_PDL != 0, t, 0, k_sort_offsets,
                            (unsigned)((radix + kOThreads / 32 - 1) / (kOThreads / 32)), kOThreads, 0, st, counts, dtot,
                            t->s.sort_offsets, nt, radix);
        // every pass but the last counts the next one
        a.kout = t->s.sk[out];
        a.vout = t->s.sv[out];
        a.counts = counts;
        a.dtot = dtot;
        a.shift = p * D;
        a.first = p == 0;
        a.nshift = p + 1 < passes ? (p + 1) * D : -1;
        a.ncounts = t->s.sort_counts[(p + 1) % 3];
        a.ndtot = dtot + kMaxRadix;
        a.zcounts = p ? t->s.sort_counts[(p - 1) % 3] : nullptr;
        a.zdtot = p ? dtot - kMaxRadix : nullptr;
        MLKV_LAUNCH(t, MLKV_K_SORT_SCATTER, (k_sort_scatter<TILE, THREADS, SELF>), nt, THREADS, SELF ? kScatterDyn : 0, st, a);
        tail = SortTail{counts, (uint32_t)radix * nt / (SELF ? 2u : 1u), dtot, (uint32_t)radix};
        a.kin = t->s.sk[out];
        a.vin = t->s.sv[out];
        out ^= 1;
    }
    *srow = a.kin;
    *spos = a.vin;
}
}  // namespace

cudaError_t sort_prepare() {
    return cudaFuncSetAttribute(k_sort_scatter<kSortTileSmall, 512, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)kScatterDyn);
}

cudaError_t launch_sort_rows(mlkv_table* t, int64_t n, cudaStream_t st, const uint32_t** srow,
                             const uint32_t** spos, bool first_counted, SortTail& tail) {
    int passes, D;
    sort_geometry(t->sort_bits, passes, D);
    if (sort_tile_shift(n) == 12)
        sort_passes<kSortTile, 512, false>(t, n, st, srow, spos, first_counted, passes, D, tail);
    else
        sort_passes<kSortTileSmall, 512, true>(t, n, st, srow, spos, first_counted, passes, D, tail);
    return cudaGetLastError();
}

cudaError_t launch_dedup_out(mlkv_table* t, const int64_t* keys, const uint32_t* srow, const uint32_t* spos,
                             int64_t n, int64_t* uniq, int32_t* counts, int64_t* num, cudaStream_t st,
                             const SortTail& tail) {
    const uint32_t sent = (uint32_t)((1ull << t->sort_bits) - 1);
    const unsigned nt = tiles(n);
    MLKV_LAUNCH(t, MLKV_K_SEGMENTS, k_seg_count, nt, kThreads, 0, st, srow, (uint32_t)n, sent, t->s.tile_sums, tail);
    MLKV_LAUNCH(t, MLKV_K_SEGMENTS, k_dedup_out, nt, kThreads, 0, st, keys, srow, spos, (uint32_t)n, sent,
                t->s.tile_sums, uniq, counts, num, t->dstate);
    return cudaGetLastError();
}

}  // namespace mlkv
