// Hash index kernels: probe / insert-on-miss, the fused Get (probe + row
// gather), deterministic row-id hand-out for new keys, Put, find and export.
//
// Index: open addressing with linear probing over 16-byte slots (two per
// 32-byte sector), at most half full.  A key is published by one 64-bit
// compare-and-swap on an empty slot whose row field already reads
// ROW_PENDING, so a reader never pairs a key with a stale row.
//
// New keys get dense row ids in first-occurrence order (the numbering the
// Get / Put upsert of MLKV Section 3.1 leaves open): while probing, every
// lookup of a new key lowers the slot's `aux` to its batch position with
// atomicMin; the lookup whose position survives is the first occurrence; an
// exclusive scan over first-occurrence flags gives each new key its rank, and
// row = rows handed out so far + rank.
#include <algorithm>

#include "mlkv_probe.cuh"

namespace mlkv {

namespace {

// ---------------------------------------------------------------------------
// row_of_pos[p] (and the slot) for every position.  Each thread takes
// kProbeKeys lookups spaced a block apart, so that their loads are in flight
// together (the probe is latency-bound: a key load, then a random slot load).
// With CT > 0 (the gradient apply on an HBM-resident table) a block of CT
// threads covers one tile of the sort (CT * kProbeKeys lookups: 1024 threads
// for 4096-lookup tiles, 512 for 2048) and also counts the first sort pass's
// digits of its rows (see FirstCounts).
constexpr int kProbeKeys = 4;

template <bool INSERT, int CT>
__global__ void __launch_bounds__(CT ? CT : 256) k_probe(IndexArgs ia, const int64_t* __restrict__ keys,
                                               uint32_t n, uint32_t* __restrict__ row_of_pos,
                                               uint32_t* __restrict__ slot_of_pos,
                                               uint32_t* miss_pos, uint32_t* miss_slot,
                                               CallCounters* cur, CallCounters* nxt,
                                               int report_absent, Memo memo, int memo_use, FirstCounts fc,
                                               int late_miss) {
    constexpr bool COUNT = CT > 0;
    static_assert(!COUNT || kProbeKeys * CT == kSortTile || kProbeKeys * CT == kSortTileSmall,
                  "a counting block covers one sort tile");
    if (INSERT && late_miss) pdl_enter_last();
    else pdl_enter();
    zero_counters(nxt);
    __shared__ uint32_t hist[COUNT ? kSortMaxRadix : 1];
    if (COUNT) {
        for (int d = threadIdx.x; d < fc.radix; d += blockDim.x) hist[d] = 0u;
        __syncthreads();
    }
    const uint32_t base = blockIdx.x * (blockDim.x * kProbeKeys) + threadIdx.x;
    unsigned long long k[kProbeKeys];
    uint32_t known[kProbeKeys];
#pragma unroll
    for (int j = 0; j < kProbeKeys; ++j) {
        const uint32_t p = base + j * blockDim.x;
        k[j] = p < n ? (unsigned long long)__ldg(keys + p) : 0ull;
        known[j] = ROW_PENDING;
        if (memo_use == (int)MemoUse::Read && p < n) {
            const uint32_t r = memo.row[p];  // loaded beside the key it belongs to
            if ((unsigned long long)memo.key[p] == k[j]) known[j] = r;
        }
    }
#pragma unroll
    for (int j = 0; j < kProbeKeys; ++j) {
        const uint32_t p = base + j * blockDim.x;
        if (p >= n) continue;
        uint32_t row = known[j];
        if (row >= ROW_ABSENT) {  // not the row the last Get found for this key here: probe
            uint32_t slot = 0;
            row = probe_key<INSERT>(ia, k[j], p, slot);
            if (!INSERT && report_absent && row == ROW_ABSENT) record_error(ia.err, MLKV_ERR_NOT_FOUND);
            if (slot_of_pos) slot_of_pos[p] = slot;
            if (INSERT && row == ROW_PENDING) append_miss(cur, miss_pos, miss_slot, p, slot, n);
            if (memo_use == (int)MemoUse::Save) {
                memo.key[p] = (int64_t)k[j];
                memo.row[p] = row;
            }
        }
        row_of_pos[p] = row;
        // a lookup of a new key is counted by the miss kernel, once it has its row
        if (COUNT && row != ROW_PENDING)
            atomicAdd(&hist[(row >= ROW_ABSENT ? fc.sent : row) & (uint32_t)(fc.radix - 1)], 1u);
    }
    if (COUNT) {
        __syncthreads();
        put_counts(hist, fc.counts, fc.packed != 0, fc.ntiles, fc.radix, blockIdx.x, fc.dtot);
    }
}

// The fused Get: each warp probes `lpw` consecutive lookups (one per lane), then
// its lane groups gather their rows with vector loads, streaming the output.
// Lookups of new keys are left to the miss path.  A row wider than 32 vectors
// is copied 2 or 4 vectors a lane at a time (row_vectors), whatever its dim: with
// all of them in flight (4 a lane at dim 512) the kernel spilled at the 32 registers
// that let 64 warps reside on an SM (65,536 lookups of dim 512: 49 us, 39 so;
// 48 warps of 40 registers for these rows: 64 spill again and cost 524k rows of
// 1 KiB 5 us).
// Tuning (set at build time): minimum resident blocks per SM for the Get
// kernel's register allocation.
#ifndef MLKV_GET_MIN_BLOCKS
#define MLKV_GET_MIN_BLOCKS 8
#endif
#ifndef MLKV_GET_SEG_MIN_BLOCKS
#define MLKV_GET_SEG_MIN_BLOCKS 6
#endif

// Vectors of a row that a lane copies at a time: 1 where a row has at most 32
// vectors, 2 up to 64 (and, again and again, for wider rows of 16-byte
// vectors), else 4.
template <int V>
constexpr int kMostVectors = V == 4 ? 2 : 4;
template <int V>
int row_vectors(const RowGeom& g) {
    return g.NV <= 32 ? 1 : g.NV <= 64 ? 2 : kMostVectors<V>;
}

// The rows of one warp's lookups base .. base + lpw - 1, KV vectors a lane of UNR
// rows of a lane group in flight; true where this lane's key is new.
template <int V, int KV, bool WIDE, bool INSERT, int UNR>
__device__ __forceinline__ bool get_rows(const IndexArgs& ia, const IndexRows& ra, const int64_t* __restrict__ keys,
                                         uint32_t n, float* __restrict__ out, uint32_t* miss_pos,
                                         uint32_t* miss_slot, CallCounters* cur, const Memo& memo, uint32_t base,
                                         int lpw) {
    using VT = typename Vec<V>::T;
    const int lane = threadIdx.x & 31;
    const uint32_t p = base + lane;
    uint32_t row = ROW_PENDING;  // lanes past the end skip the gather
    bool fresh = false;
    if (lane < lpw && p < n) {
        uint32_t slot = 0;
        const int64_t key = keys[p];
        row = probe_key<INSERT>(ia, (unsigned long long)key, p, slot);
        fresh = INSERT && row == ROW_PENDING;
        if (fresh) append_miss(cur, miss_pos, miss_slot, p, slot, n);
        if (!INSERT && row == ROW_ABSENT) record_error(ia.err, MLKV_ERR_NOT_FOUND);
        memo.key[p] = key;
        memo.row[p] = row;
    }
    const int G = ra.G, R = 32 / G, glane = lane & (G - 1), gid = lane / G;
    for (int q0 = 0; q0 < lpw; q0 += R * UNR) {
        // more vectors than KV a lane: in rounds (uniform; one, but for the widest rows)
        for (int j0 = glane; WIDE ? j0 - glane < ra.NV : j0 == glane; j0 += G * KV) {
            VT v[UNR][KV];
            uint32_t rr[UNR];
#pragma unroll
            for (int u = 0; u < UNR; ++u) {
                const int q = q0 + u * R + gid;
                const uint32_t r = __shfl_sync(0xffffffffu, row, q & 31);
                rr[u] = UNR == 1 || q < lpw ? r : ROW_PENDING;
                const VT* src = reinterpret_cast<const VT*>(ra.slots + (size_t)rr[u] * ra.stride) + j0;
#pragma unroll
                for (int k = 0; k < KV; ++k)
                    if (rr[u] < ROW_ABSENT && j0 + G * k < ra.NV) v[u][k] = __ldg(src + G * k);
            }
#pragma unroll
            for (int u = 0; u < UNR; ++u) {
                if (rr[u] == ROW_PENDING) continue;
                VT* dst = reinterpret_cast<VT*>(out + (size_t)(base + q0 + u * R + gid) * ra.d) + j0;
#pragma unroll
                for (int k = 0; k < KV; ++k)
                    if (j0 + G * k < ra.NV) __stcs(dst + G * k, rr[u] == ROW_ABSENT ? Vec<V>::nan() : v[u][k]);
            }
            if (!WIDE) break;
        }
    }
    return fresh;
}

template <int V, int KV, bool WIDE, bool INSERT>
__global__ void __launch_bounds__(256, V * KV >= 8 ? MLKV_GET_SEG_MIN_BLOCKS : MLKV_GET_MIN_BLOCKS) k_get(IndexArgs ia, IndexRows ra,
                                             const int64_t* __restrict__ keys, uint32_t n,
                                             float* __restrict__ out, uint32_t* miss_pos,
                                             uint32_t* miss_slot, CallCounters* cur,
                                             CallCounters* nxt, Memo memo, int lpw) {
    if (INSERT && late_miss_get(ra.NV, n)) pdl_enter_last();
    else pdl_enter();
    zero_counters(nxt);
    const uint32_t base = (blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * (uint32_t)lpw;
    if (base >= n) return;  // warp-uniform
    get_rows<V, KV, WIDE, INSERT, 1>(ia, ra, keys, n, out, miss_pos, miss_slot, cur, memo, base, lpw);
}

// The Get and its miss path in one launch (see finish_get): a warp per lpw
// lookups, in a grid that can wait for itself (its launch bounds leave room for
// the kGetBlocksPerSm blocks per SM of two tables' largest, and the launch asks).
template <int V, int KV, bool WIDE>
__global__ void __launch_bounds__(256, 2 * kGetBlocksPerSm) k_get_small(IndexArgs ia, IndexRows ra, MissArgs ma, CallCounters* nxt,
                                                                    Memo memo, int lpw, uint32_t bar_extra) {
    pdl_enter();
    zero_counters(nxt);
    const uint32_t base = (blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * (uint32_t)lpw;
    bool fresh = false;
    if (base < ma.n)
        fresh = get_rows<V, KV, WIDE, true, 4 / KV>(ia, ra, ma.keys, ma.n, ma.out, const_cast<uint32_t*>(ma.miss_pos),
                                       const_cast<uint32_t*>(ma.miss_slot), ma.cur, memo, base, lpw);
    const uint32_t lo = blockIdx.x * 8u * (uint32_t)lpw;
    finish_get<V, 256>(ia, ra, ma, fresh, min(lo, ma.n), min(lo + 8u * (uint32_t)lpw, ma.n), bar_extra);
}

// The Get with its rows moved by the SM's asynchronous copies, for calls of
// fewer than bulk_lookups lookups (rows of at most kBulkRowBytes, 16-byte
// aligned buffers).  Each warp probes kBulkRows consecutive lookups as k_get
// does, then copies their rows into its shared-memory stage with cp.async (16
// bytes a lane, L2 only; no registers hold rows in flight, so all of them are
// in flight at once), and writes the stage to the output with one bulk store:
// the output rows are contiguous.  The store runs on while the warp probes its
// next lookups; the stage is reused once the store has read it.  Rows of new
// keys are left to the miss path, which writes their output rows after this
// kernel.  Faster where a call is too small to fill the GPU with k_get's warps,
// slower above, where k_get's 64 warps a SM beat the few warps the stages leave
// room for; rows of few bytes leave little to copy at once.  (us of a Get of keys
// drawn uniformly from 4M rows, k_get / with this kernel; bulk_lookups lies where
// the two cross:
//   dim      60,000   131,000   250,000   420,000 lookups
//     4    11.7/11.3  13.4/15.2  17.0/21.0  24.1/28.6
//    16    10.7/10.9  14.9/15.4  21.4/21.9  28.5/31.3
//    64    16.0/12.6  21.7/18.7  35.5/32.1  48.4/51.9
//    96    18.0/14.9  29.5/25.0  48.5/44.1  69.1/70.6
//   128    19.0/17.2  32.4/30.5  53.9/54.3  80.1/87.5)
#ifndef MLKV_GET_BULK
#define MLKV_GET_BULK 1
#endif
// Rows that are copied to the host next leave them at this many bytes: the copy
// takes longer behind the bulk stores.  (us of a Get into host memory, k_get / with
// this kernel: 100,000 of dim 100 235/248, 180,000 414/440, 180,000 of dim 64
// 275/282; smaller ones 40,000 of dim 128 132/126, 80,000 of dim 32 82/78.)
constexpr int64_t kBulkMaxToHost = 24 << 20;
inline int64_t bulk_lookups(uint32_t rowbytes) {
    return rowbytes <= 64 ? 1 << 16 : rowbytes < 128 || rowbytes > 384 ? 200'000 : 400'000;
}
constexpr int kBulkThreads = 128;  // 4 warps
constexpr uint32_t kBulkRowBytes = 512;
#ifndef MLKV_GET_BULK_ROWS
#define MLKV_GET_BULK_ROWS 8
#endif
constexpr uint32_t kBulkRows = MLKV_GET_BULK_ROWS;  // lookups a warp takes at a time (its stage: their rows)

__device__ __forceinline__ void cp_async16(void* smem_dst, const void* gmem_src) {
    const uint32_t s = (uint32_t)__cvta_generic_to_shared(smem_dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(s), "l"(gmem_src) : "memory");
}

__device__ __forceinline__ void cp_async_wait_all() {
    asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
}

// Bulk copy of `bytes` (a multiple of 16; both addresses 16-byte aligned) from
// shared memory to global memory, as one bulk group.
__device__ __forceinline__ void bulk_store(void* gdst, const void* ssrc, uint32_t bytes) {
    const uint32_t s = (uint32_t)__cvta_generic_to_shared(ssrc);
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;\n\tcp.async.bulk.commit_group;"
                 ::"l"(gdst), "r"(s), "r"(bytes) : "memory");
}

template <bool INSERT>
__global__ void __launch_bounds__(kBulkThreads) k_get_bulk(IndexArgs ia, IndexRows ra, const int64_t* __restrict__ keys,
                                                           uint32_t n, float* __restrict__ out, uint32_t* miss_pos,
                                                           uint32_t* miss_slot, CallCounters* cur, CallCounters* nxt,
                                                           Memo memo) {
    pdl_enter();
    zero_counters(nxt);
    extern __shared__ __align__(128) unsigned char smem[];
    constexpr int kWarps = kBulkThreads / 32;
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const uint32_t nvec = (uint32_t)ra.d >> 2;  // 16-byte vectors per row
    const uint32_t rowbytes = nvec * 16u;
    float4* stage = reinterpret_cast<float4*>(smem + (size_t)wib * kBulkRows * rowbytes);
    uint32_t* srow = reinterpret_cast<uint32_t*>(smem + (size_t)kWarps * kBulkRows * rowbytes) + wib * 32;
    const float4 nan4 = Vec<4>::nan();
    const uint32_t nwarps = gridDim.x * kWarps;
    bool stored = false;  // a bulk store of this warp's stage is in flight
    for (uint32_t base = (blockIdx.x * kWarps + wib) * kBulkRows; base < n; base += nwarps * kBulkRows) {
        const uint32_t p = base + lane;
        uint32_t row = ROW_PENDING;
        if (lane < (int)kBulkRows && p < n) {
            uint32_t slot = 0;
            const int64_t key = keys[p];
            row = probe_key<INSERT>(ia, (unsigned long long)key, p, slot);
            if (INSERT && row == ROW_PENDING) append_miss(cur, miss_pos, miss_slot, p, slot, n);
            if (!INSERT && row == ROW_ABSENT) record_error(ia.err, MLKV_ERR_NOT_FOUND);
            memo.key[p] = key;
            memo.row[p] = row;
        }
        const uint32_t cnt = min(kBulkRows, n - base);
        if (stored && lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
        __syncwarp();
        srow[lane] = row;
        __syncwarp();
        for (uint32_t i = lane; i < cnt * nvec; i += 32) {
            const uint32_t q = i / nvec, c = i - q * nvec;
            const uint32_t r = srow[q];
            if (r < ROW_ABSENT)
                cp_async16(stage + i, reinterpret_cast<const float4*>(ra.slots + (size_t)r * ra.stride) + c);
            else if (r == ROW_ABSENT)
                stage[i] = nan4;  // a new key's row (ROW_PENDING) is written by the miss path later
        }
        cp_async_wait_all();
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // the stage, for the bulk store
        __syncwarp();
        if (lane == 0) bulk_store(out + (size_t)base * ra.d, stage, cnt * rowbytes);
        stored = true;
    }
    if (stored && lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
}

// The miss path in a kernel of its own, one block per SM (see miss_path).  In
// steady-state training nothing misses and every block returns at once.
constexpr int kMissThreads = 512;

template <int V>
__global__ void __launch_bounds__(kMissThreads) k_miss(IndexArgs ia, IndexRows ra, MissArgs ma, uint32_t bar_extra,
                                                       int release, FirstCounts fc) {
    // (the next kernel's blocks are placed once every block of this grid has
    // started, so they keep none of these from becoming resident)
    pdl_enter();
    CallCounters* cur = ma.cur;
    const uint32_t m = min(cur->n_miss, ma.n);  // never more misses than lookups
    if (m == 0) return;  // the call has touched no counter
    // the first sort pass's count (an apply's) of a missed lookup's digit in its tile
    auto count = [&](uint32_t p, uint32_t r) {
        if (!fc.counts) return;
        const uint32_t dig = (r >= ROW_ABSENT ? fc.sent : r) & (uint32_t)(fc.radix - 1);
        add_count(fc.counts, fc.packed != 0, fc.ntiles, fc.radix, p >> fc.tile_shift, dig, 1u);
        atomicAdd(fc.dtot + dig, 1u);
    };
    const bool done = miss_path<V, kMissThreads>(
        ia, ra, ma, m, even_share(ma.n, gridDim.x, blockIdx.x),
        [&](int i) { return grid_barrier(&cur->bar[i], gridDim.x + bar_extra, ia.err); }, count);
    if (!done) {
        // A block whose wait ran out returns at once; the first sort pass's counts
        // still get its share of the missed lookups, which keep no row (the last
        // phase's share, so that every lookup is counted once).
        for_misses<kMissThreads>(m, gridDim.x, blockIdx.x, 32u / ra.G, [&](uint32_t i, uint32_t) {
            if (i < m) count(ma.miss_pos[i], ROW_ABSENT);
        });
        return;
    }
    if (release) release_counters(cur, gridDim.x);
}

// Put 1/2: the last occurrence of each key wins: aux = min over its
// occurrences of (0xFFFFFFFE - p).  Atomics on one slot queue (about 2.7 ns
// each): with one per lookup, a Zipf(0.99) batch of 524k Puts, 6% of them of
// one key, took 89 us.  So the positions are walked from the last to the first
// by a grid of few warps, and a slot that already holds a later position is only
// read: the first round, in which a warp's lanes of one slot send one atomic,
// marks the hot keys, the others find them marked.  kMarkPerSm = 2 blocks of 256
// threads per SM: more make the first round's burst longer, fewer leave too few
// reads in flight.  Matching the lanes in every round cost 1.3M Puts of uniform
// keys of dim 4 118 us instead of 109 (one atomic per lookup, as without hot keys:
// 108), and Zipf(0.99) ones 67 instead of 61.
#ifndef MLKV_MARK_PER_SM
#define MLKV_MARK_PER_SM 2
#endif
constexpr int kMarkPerSm = MLKV_MARK_PER_SM;
__global__ void __launch_bounds__(256) k_put_mark(Slot* __restrict__ index, const uint32_t* __restrict__ row_of_pos,
                                                  const uint32_t* __restrict__ slot_of_pos, uint32_t n) {
    pdl_enter();
    const uint32_t nthreads = gridDim.x * blockDim.x;
    const int lane = threadIdx.x & 31;
    // the next round's row and slot load beside this round's slots
    uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    uint32_t row = i < n ? __ldg(row_of_pos + (n - 1 - i)) : ROW_ABSENT;
    uint32_t slot = i < n ? __ldg(slot_of_pos + (n - 1 - i)) : 0u;
    for (uint32_t base = i - lane; base < n; base += nthreads, i += nthreads) {  // warp-uniform
        const uint32_t r = row, s = slot, mark = 0xFFFFFFFEu - (n - 1 - i);
        const uint32_t j = i + nthreads;
        row = j < n ? __ldg(row_of_pos + (n - 1 - j)) : ROW_ABSENT;
        slot = j < n ? __ldg(slot_of_pos + (n - 1 - j)) : 0u;
        bool lead = r < ROW_ABSENT;
        if (i - lane < nthreads) {  // the first round: the lowest lane of a slot holds its last position
            const unsigned peers = __match_any_sync(0xffffffffu, lead ? (unsigned long long)s : ~0ull);
            lead = lead && lane == __ffs(peers) - 1;
        }
        if (lead && mark < ld_u32_relaxed(&index[s].aux)) atomicMin(&index[s].aux, mark);
    }
}

// Put 2/2: the winning occurrence writes the row and puts aux back to idle.  A
// warp finds the winners among its lpw lookups, one per lane (row and slot, then
// the slot's mark), and its lane groups copy their rows, KV * ROWS vectors a lane
// in flight.  (With a lane group walking its lookups one by one, each copy
// waited for its own mark: 75 us for 524k Puts of 1 KiB, Zipf(0.99); 70 so, 88
// with 2 vectors in flight.)
// KV vectors a lane (row_vectors) of ROWS rows are in flight, and a warp takes at
// least that many rows: with 1 or 2 a warp, 50,000 Puts of dim 64 took 27 us, 21
// so (a lane group per lookup in a loop: 20).  6 blocks per SM with one vector a
// lane: 40 registers; the 53 taken without leave fewer warps (300,000 of dim 64:
// 52 us, 49 so), 32 spill (59); 5 with more, where 40 spill.
template <int V, int KV, int ROWS>
__global__ void __launch_bounds__(256, KV == 1 ? 6 : 5) k_put_scatter(Slot* __restrict__ index, IndexRows ra,
                                                     const uint32_t* __restrict__ row_of_pos,
                                                     const uint32_t* __restrict__ slot_of_pos,
                                                     const float* __restrict__ vals,
                                                     const float* __restrict__ state, uint32_t n, int lpw) {
    pdl_enter();
    using VT = typename Vec<V>::T;
    __shared__ uint2 wins[8][32];  // (row, lookup) of the warp's winners
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int G = ra.G, R = 32 / G, glane = lane & (G - 1), gid = lane / G;
    const uint32_t p = (blockIdx.x * (blockDim.x >> 5) + wib) * (uint32_t)lpw + lane;
    bool win = false;
    uint32_t r = 0;
    if (lane < lpw && p < n) {
        r = __ldg(row_of_pos + p);
        const uint32_t s = __ldg(slot_of_pos + p);
        if (r < ROW_ABSENT && index[s].aux == 0xFFFFFFFEu - p) {
            win = true;
            index[s].aux = AUX_IDLE;  // its other lookups hold other marks
        }
    }
    const unsigned m = __ballot_sync(0xffffffffu, win);
    if (win) wins[wib][__popc(m & lanemask_lt())] = make_uint2(r, p);
    __syncwarp();
    const int nwin = __popc(m);
    auto copy = [&](const float* __restrict__ src, int off) {
        for (int w0 = 0; w0 < nwin; w0 += R * ROWS)  // uniform
            for (int j0 = glane; j0 - glane < ra.NV; j0 += G * KV) {
                VT v[ROWS][KV];
                VT* to[ROWS];
#pragma unroll
                for (int i = 0; i < ROWS; ++i) {
                    const int x = w0 + i * R + gid;
                    const uint2 rp = wins[wib][x < nwin ? x : 0];
                    const VT* from = reinterpret_cast<const VT*>(src + (size_t)rp.y * ra.d) + j0;
                    to[i] = x < nwin ? reinterpret_cast<VT*>(ra.slots + (size_t)rp.x * ra.stride + off) + j0 : nullptr;
#pragma unroll
                    for (int k = 0; k < KV; ++k)
                        if (x < nwin && j0 + G * k < ra.NV) v[i][k] = __ldcs(from + G * k);
                }
#pragma unroll
                for (int i = 0; i < ROWS; ++i)
#pragma unroll
                    for (int k = 0; k < KV; ++k)
                        if (to[i] && j0 + G * k < ra.NV) to[i][G * k] = v[i][k];
            }
    };
    copy(vals, 0);
    if (state) copy(state, ra.dpad);  // import: the state too
}

__global__ void __launch_bounds__(256) k_find(IndexArgs ia, const int64_t* __restrict__ keys,
                                              uint32_t n, int64_t* __restrict__ rows,
                                              CallCounters* nxt) {
    pdl_enter();
    zero_counters(nxt);
    const uint32_t p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n) return;
    uint32_t slot = 0;
    const uint32_t r = probe_key<false>(ia, (unsigned long long)keys[p], p, slot);
    rows[p] = r >= ROW_ABSENT ? -1 : (int64_t)r;
}

// Export: like Get without insertion, copying row and/or state.
// With a tier, a row is read from its cache line when it has one, else from
// its host slot.
struct ExportTier {
    const uint32_t* row_loc;
    const float* cache;
    const float* host;
};

template <int V, int KV>
__global__ void __launch_bounds__(256) k_export(IndexArgs ia, IndexRows ra,
                                                const int64_t* __restrict__ keys, uint32_t n,
                                                float* __restrict__ rows_out,
                                                float* __restrict__ state_out, CallCounters* nxt,
                                                ExportTier et, int lpw) {
    pdl_enter();
    using VT = typename Vec<V>::T;
    zero_counters(nxt);
    const int lane = threadIdx.x & 31;
    const uint32_t base = (blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * (uint32_t)lpw;
    if (base >= n) return;
    const uint32_t p = base + lane;
    uint32_t row = ROW_PENDING;
    if (lane < lpw && p < n) {
        uint32_t slot = 0;
        row = probe_key<false>(ia, (unsigned long long)keys[p], p, slot);
    }
    const int G = ra.G, R = 32 / G, glane = lane & (G - 1), gid = lane / G;
    for (int q0 = 0; q0 < lpw; q0 += R) {
        const int q = q0 + gid;
        const uint32_t r = __shfl_sync(0xffffffffu, row, q);
        if (r == ROW_PENDING) continue;
        const float* src = ra.slots + (size_t)(r == ROW_ABSENT ? 0 : r) * ra.stride;
        if (et.row_loc && r != ROW_ABSENT) {
            const uint32_t l = et.row_loc[r];
            src = l < LOC_HOST ? et.cache + (size_t)l * ra.stride : et.host + (size_t)(l & ~LOC_HOST) * ra.stride;
        }
        const VT* ws = reinterpret_cast<const VT*>(src);
        const VT* gs = reinterpret_cast<const VT*>(src + ra.dpad);
        constexpr int kVecs = KV;  // of the row and of the state, in flight together a lane
        const size_t o = (size_t)(base + q) * ra.d;
        for (int j0 = glane; j0 < ra.NV; j0 += G * kVecs) {
            VT w[kVecs], g[kVecs];
#pragma unroll
            for (int k = 0; k < kVecs; ++k) {
                const int j = j0 + G * k;
                if (j < ra.NV && rows_out) w[k] = __ldg(ws + j);
                if (j < ra.NV && state_out) g[k] = __ldg(gs + j);
            }
#pragma unroll
            for (int k = 0; k < kVecs; ++k) {
                const int j = j0 + G * k;
                if (j >= ra.NV) continue;
                if (rows_out) __stcs(reinterpret_cast<VT*>(rows_out + o) + j, r == ROW_ABSENT ? Vec<V>::nan() : w[k]);
                if (state_out)
                    __stcs(reinterpret_cast<VT*>(state_out + o) + j, r == ROW_ABSENT ? Vec<V>::nan() : g[k]);
            }
        }
    }
}

// Dispatch over V for the row kernels.
template <template <int> class F, typename... A>
cudaError_t dispatch_row(const RowGeom& g, A&&... a) {
    if (g.V == 4) return F<4>::run(a...);
    if (g.V == 2) return F<2>::run(a...);
    return F<1>::run(a...);
}

inline unsigned grid_for(int64_t items, int per_block) {
    return (unsigned)((items + per_block - 1) / per_block);
}

inline unsigned capped_grid(mlkv_table* t, int64_t items, int per_block, int per_sm) {
    int64_t g = (items + per_block - 1) / per_block;
    int64_t cap = (int64_t)t->num_sms * per_sm;
    if (g > cap) g = cap;
    return (unsigned)(g < 1 ? 1 : g);
}

// Blocks per SM and shared memory of k_get_bulk for rows of `rowbytes`.
template <bool INSERT>
int bulk_grid(mlkv_table* t, size_t smem, int64_t n) {
    static int configured[2] = {0, 0};
    static int per_sm_cache[kBulkRowBytes / 16 + 1] = {0};
    const int kind = INSERT ? 1 : 0;
    if (!configured[kind]) {
        cudaFuncSetAttribute(k_get_bulk<INSERT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)(4 * kBulkRows * kBulkRowBytes + 4 * 32 * 4));
        configured[kind] = 1;
    }
    const size_t idx = (smem - 4 * 32 * 4) / (4 * kBulkRows * 16);
    int per_sm = idx < sizeof(per_sm_cache) / sizeof(int) ? per_sm_cache[idx] : 0;
    if (per_sm == 0) {
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_get_bulk<INSERT>, kBulkThreads, smem) !=
                cudaSuccess || per_sm < 1)
            per_sm = 1;
        if (idx < sizeof(per_sm_cache) / sizeof(int)) per_sm_cache[idx] = per_sm;
    }
    int64_t g = (n + 4 * kBulkRows - 1) / (4 * kBulkRows);
    const int64_t cap = (int64_t)per_sm * t->num_sms;
    return (int)(g < cap ? g : cap);
}

// Lookups per warp of k_get_small: as few as a grid of kGetBlocksPerSm blocks of
// 8 warps per SM allows (two tables' waiting grids fit the GPU together; with one
// block per SM 16,384 lookups of dim 128 take 10.5 us instead of 8.0, of dim 512
// 24.9 instead of 16.1), at least the rows a warp copies at a time.
int small_get_lpw(const mlkv_table* t, int64_t n) {
    int lpw = 32 / t->geom.G;
    while (lpw < 32 && n > (int64_t)lpw * 8 * kGetBlocksPerSm * t->num_sms) lpw *= 2;
    return lpw;
}

template <int V>
struct GetRun {
    static cudaError_t run(mlkv_table* t, const int64_t* keys, int64_t n, float* out,
                           cudaStream_t st, CallCounters* cur, CallCounters* nxt, bool to_host,
                           bool& resolved) {
        const uint32_t rowbytes = (uint32_t)t->geom.d * 4;
        const int kv = row_vectors<V>(t->geom);
        constexpr int M = kMostVectors<V>;
        const bool wide = t->geom.NV > 32 * kv;
        const bool ins = t->cfg.insert_on_miss != 0;
        const auto small = kv == 1   ? k_get_small<V, 1, false>
                           : wide    ? k_get_small<V, M, true>
                           : kv == 2 ? k_get_small<V, 2, false>
                                     : k_get_small<V, M, false>;
        const int small_lpw = small_get_lpw(t, n);
        const unsigned grid = grid_for(n, 8 * small_lpw);
        // every block resident at once, with a word each for its new keys
        resolved = ins && n <= (int64_t)MLKV_SMALL_GET_MAX && miss_grid_fits(t, grid) &&
                   (int64_t)grid <= persistent_blocks(t, (const void*)small, 256);
        if (resolved) {
            const MissArgs ma = miss_args(t, keys, n, MissMode::Get, nullptr, out, cur);
            MLKV_LAUNCH(t, MLKV_K_GET_GATHER, small, grid, 256, 0, st, index_args(t), row_args(t), ma, nxt,
                        Memo{t->s.memo_key, t->s.memo_row}, small_lpw, take_injected_wait() ? 1u : 0u);
            return cudaGetLastError();
        }
        if (MLKV_GET_BULK && V == 4 && rowbytes <= kBulkRowBytes && n < bulk_lookups(rowbytes) &&
            !(to_host && n * (int64_t)rowbytes >= kBulkMaxToHost)) {
            const size_t smem = (size_t)4 * kBulkRows * rowbytes + 4 * 32 * 4;
            if (t->cfg.insert_on_miss)
                MLKV_LAUNCH(t, MLKV_K_GET_GATHER, k_get_bulk<true>, bulk_grid<true>(t, smem, n), kBulkThreads, smem,
                            st, index_args(t), row_args(t), keys, (uint32_t)n, out, t->s.miss_pos, t->s.miss_slot,
                            cur, nxt, Memo{t->s.memo_key, t->s.memo_row});
            else
                MLKV_LAUNCH(t, MLKV_K_GET_GATHER, k_get_bulk<false>, bulk_grid<false>(t, smem, n), kBulkThreads,
                            smem, st, index_args(t), row_args(t), keys, (uint32_t)n, out, t->s.miss_pos,
                            t->s.miss_slot, cur, nxt, Memo{t->s.memo_key, t->s.memo_row});
            return cudaGetLastError();
        }
        const int lpw = lookups_per_warp(t, n, 32 / t->geom.G);
        const auto kernel = kv == 1   ? (ins ? k_get<V, 1, false, true> : k_get<V, 1, false, false>)
                            : wide    ? (ins ? k_get<V, M, true, true> : k_get<V, M, true, false>)
                            : kv == 2 ? (ins ? k_get<V, 2, false, true> : k_get<V, 2, false, false>)
                                      : (ins ? k_get<V, M, false, true> : k_get<V, M, false, false>);
        MLKV_LAUNCH(t, MLKV_K_GET_GATHER, kernel, grid_for(n, 8 * lpw), 256, 0, st, index_args(t), row_args(t), keys,
                    (uint32_t)n, out, t->s.miss_pos, t->s.miss_slot, cur, nxt, Memo{t->s.memo_key, t->s.memo_row},
                    lpw);
        return cudaGetLastError();
    }
};

template <int V>
struct MissRun {
    static cudaError_t run(mlkv_table* t, const int64_t* keys, int64_t n, MissMode mode, float* out,
                           cudaStream_t st, CallCounters* cur, bool release, const FirstCounts* fc) {
        IndexRows init_ra = row_args(t);  // new rows live in the host tier when tiered
        if (t->tiered) init_ra.slots = t->tier.host_dev;
        if (!miss_grid_fits(t, t->num_sms)) return cudaErrorInvalidConfiguration;
        const MissArgs ma = miss_args(t, keys, n, mode, mode == MissMode::Get ? nullptr : t->s.row_of_pos,
                                      mode == MissMode::Get ? out : nullptr, cur);
        MLKV_LAUNCH(t, 0, (k_miss<V>), t->num_sms, kMissThreads, 0, st, index_args(t), init_ra, ma,
                    take_injected_wait() ? 1u : 0u, release ? 1 : 0, fc ? *fc : FirstCounts{});
        return cudaGetLastError();
    }
};

template <int V>
struct PutRun {
    static cudaError_t run(mlkv_table* t, const float* vals, const float* state, int64_t n, cudaStream_t st) {
        MLKV_LAUNCH(t, 0, k_put_mark, capped_grid(t, n, 256, kMarkPerSm), 256, 0, st, t->index, t->s.row_of_pos,
                    t->s.slot_of_pos, (uint32_t)n);
        const int kv = row_vectors<V>(t->geom), rows = kv == 1 ? 4 : 2;  // in flight a lane group
        const int lpw = lookups_per_warp(t, n, std::min(32, rows * (32 / t->geom.G)));
        const auto kernel = kv == 1 ? k_put_scatter<V, 1, 4> : kv == 2 ? k_put_scatter<V, 2, 2>
                                                                       : k_put_scatter<V, kMostVectors<V>, 2>;
        MLKV_LAUNCH(t, MLKV_K_PUT_SCATTER, kernel, grid_for(n, 8 * lpw), 256, 0, st, t->index, row_args(t),
                    t->s.row_of_pos, t->s.slot_of_pos, vals, state, (uint32_t)n, lpw);
        return cudaGetLastError();
    }
};

// The key of every row below n_rows, at its row: a checkpoint's keys in row
// order (rows are dense, handed out in first-occurrence order).
__global__ void __launch_bounds__(256) k_dump_keys(const Slot* __restrict__ index, unsigned long long nslots,
                                                   int64_t* __restrict__ out, uint32_t n_rows) {
    pdl_enter();
    for (unsigned long long s = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; s < nslots;
         s += (unsigned long long)gridDim.x * blockDim.x) {
        const unsigned long long key = index[s].key;
        const uint32_t row = index[s].row;
        if (key != EMPTY_KEY && row < n_rows) out[row] = (int64_t)key;
    }
}

template <int V>
struct ExportRun {
    static cudaError_t run(mlkv_table* t, const int64_t* keys, int64_t n, float* rows, float* state,
                           cudaStream_t st, CallCounters* nxt) {
        ExportTier et{nullptr, nullptr, nullptr};
        if (t->tiered) et = ExportTier{t->tier.row_loc, t->tier.cache, t->tier.host_dev};
        const int lpw = lookups_per_warp(t, n, 32 / t->geom.G);
        const int kv = row_vectors<V>(t->geom);
        const auto kernel = kv == 1 ? k_export<V, 1> : kv == 2 ? k_export<V, 2> : k_export<V, kMostVectors<V>>;
        MLKV_LAUNCH(t, 0, kernel, grid_for(n, 8 * lpw), 256, 0, st, index_args(t),
                    row_args(t), keys, (uint32_t)n, rows, state, nxt, et, lpw);
        return cudaGetLastError();
    }
};

}  // namespace

cudaError_t launch_probe(mlkv_table* t, const int64_t* keys, int64_t n, bool insert, MemoUse memo,
                         bool want_slot, bool report_absent, cudaStream_t st, CallCounters* cur,
                         CallCounters* nxt, uint32_t* rows_out, const FirstCounts* fc) {
    uint32_t* slot_of_pos = want_slot ? t->s.slot_of_pos : nullptr;
    uint32_t* rows = rows_out ? rows_out : t->s.row_of_pos;
    if (want_slot && memo == MemoUse::Read) memo = MemoUse::None;  // the memo holds no slots
    const Memo m{t->s.memo_key, t->s.memo_row};
    const int ra = report_absent ? 1 : 0, late = late_miss_probe(t->geom.NV, n) ? 1 : 0;
    if (fc) {  // one block per sort tile, counting the first pass
        const unsigned g = grid_for(n, 1 << fc->tile_shift);
        if (fc->tile_shift == 12) {
            if (insert)
                MLKV_LAUNCH(t, MLKV_K_PROBE, (k_probe<true, 1024>), g, 1024, 0, st, index_args(t), keys,
                            (uint32_t)n, rows, slot_of_pos, t->s.miss_pos, t->s.miss_slot, cur, nxt, 0, m,
                            (int)memo, *fc, late);
            else
                MLKV_LAUNCH(t, MLKV_K_PROBE, (k_probe<false, 1024>), g, 1024, 0, st, index_args(t), keys,
                            (uint32_t)n, rows, slot_of_pos, t->s.miss_pos, t->s.miss_slot, cur, nxt, ra, m,
                            (int)memo, *fc, late);
        } else {  // the small tiles: kSortTileSmall / kProbeKeys threads
            constexpr int CT = kSortTileSmall / kProbeKeys;
            if (insert)
                MLKV_LAUNCH(t, MLKV_K_PROBE, (k_probe<true, CT>), g, CT, 0, st, index_args(t), keys,
                            (uint32_t)n, rows, slot_of_pos, t->s.miss_pos, t->s.miss_slot, cur, nxt, 0, m,
                            (int)memo, *fc, late);
            else
                MLKV_LAUNCH(t, MLKV_K_PROBE, (k_probe<false, CT>), g, CT, 0, st, index_args(t), keys,
                            (uint32_t)n, rows, slot_of_pos, t->s.miss_pos, t->s.miss_slot, cur, nxt, ra, m,
                            (int)memo, *fc, late);
        }
        return cudaGetLastError();
    }
    const FirstCounts none{};
    const unsigned g = grid_for(n, 256 * kProbeKeys);
    if (insert)
        MLKV_LAUNCH(t, MLKV_K_PROBE, (k_probe<true, 0>), g, 256, 0, st, index_args(t), keys,
                    (uint32_t)n, rows, slot_of_pos, t->s.miss_pos, t->s.miss_slot, cur, nxt, 0, m, (int)memo, none, late);
    else
        MLKV_LAUNCH(t, MLKV_K_PROBE, (k_probe<false, 0>), g, 256, 0, st, index_args(t), keys,
                    (uint32_t)n, rows, slot_of_pos, t->s.miss_pos, t->s.miss_slot, cur, nxt, ra, m, (int)memo, none, late);
    return cudaGetLastError();
}

cudaError_t launch_get(mlkv_table* t, const int64_t* keys, int64_t n, float* out, cudaStream_t st,
                       CallCounters* cur, CallCounters* nxt, bool to_host, bool& resolved) {
    return dispatch_row<GetRun>(t->geom, t, keys, n, out, st, cur, nxt, to_host, resolved);
}

cudaError_t launch_resolve_misses(mlkv_table* t, const int64_t* keys, int64_t n, MissMode mode,
                                  float* out, cudaStream_t st, CallCounters* cur, bool release,
                                  const FirstCounts* fc) {
    return dispatch_row<MissRun>(t->geom, t, keys, n, mode, out, st, cur, release, fc);
}

cudaError_t launch_put_scatter(mlkv_table* t, const float* vals, const float* state, int64_t n, cudaStream_t st) {
    return dispatch_row<PutRun>(t->geom, t, vals, state, n, st);
}

// Slots of keys that never got a row (an insert cut short by a device error)
// go back to idle, so that a later call inserts them afresh.
__global__ void __launch_bounds__(256) k_reset_pending(Slot* __restrict__ index, unsigned long long nslots) {
    for (unsigned long long s = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; s < nslots;
         s += (unsigned long long)gridDim.x * blockDim.x)
        if (index[s].key != EMPTY_KEY && index[s].row == ROW_PENDING) index[s].aux = AUX_IDLE;
}

cudaError_t launch_reset_pending(mlkv_table* t, cudaStream_t st) {
    k_reset_pending<<<(unsigned)t->num_sms * 8, 256, 0, st>>>(t->index, t->index_mask + 1);
    return cudaGetLastError();
}

cudaError_t launch_dump_keys(mlkv_table* t, int64_t* out, int64_t n_rows, cudaStream_t st) {
    const unsigned long long nslots = t->index_mask + 1;
    MLKV_LAUNCH(t, 0, k_dump_keys, (unsigned)t->num_sms * 8, 256, 0, st, t->index, nslots, out, (uint32_t)n_rows);
    return cudaGetLastError();
}

cudaError_t launch_find(mlkv_table* t, const int64_t* keys, int64_t n, int64_t* rows,
                        cudaStream_t st, CallCounters* nxt) {
    MLKV_LAUNCH(t, 0, k_find, grid_for(n, 256), 256, 0, st, index_args(t), keys, (uint32_t)n, rows, nxt);
    return cudaGetLastError();
}

cudaError_t launch_export(mlkv_table* t, const int64_t* keys, int64_t n, float* rows, float* state,
                          cudaStream_t st, CallCounters* nxt) {
    return dispatch_row<ExportRun>(t->geom, t, keys, n, rows, state, st, nxt);
}

}  // namespace mlkv
