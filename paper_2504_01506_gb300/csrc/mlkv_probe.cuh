// Device code of the hash index that more than one kernel file uses: the probe,
// the miss list and the miss path.
#pragma once

#include "mlkv_internal.cuh"

namespace mlkv {

namespace {

// Device-scope relaxed loads: they see slots published by compare-and-swap in
// the same kernel and still hit in L2 (the coherence point of GPU accesses);
// a volatile load would be a system-scope access.
__device__ __forceinline__ ulonglong2 ld_slot_relaxed(const Slot* s) {
    ulonglong2 v;
    asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(v.x), "=l"(v.y) : "l"(s) : "memory");
    return v;
}

__device__ __forceinline__ uint32_t ld_u32_relaxed(const uint32_t* p) {
    uint32_t v;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// Probes `key`.  Returns its row, ROW_ABSENT, or (INSERT only) ROW_PENDING
// with `slot_out` = the slot that now holds the key and the slot's aux
// lowered to `pos`.
template <bool INSERT>
__device__ __forceinline__ uint32_t probe_key(const IndexArgs& ia, unsigned long long key,
                                              uint32_t pos, uint32_t& slot_out) {
    if (key == EMPTY_KEY) {
        record_error(ia.err, MLKV_ERR_INVALID);
        return ROW_ABSENT;
    }
    unsigned long long s = (ia.identity_hash ? key : hash_key(key)) & ia.mask;
    for (int i = 0; i < PROBE_LIMIT; ++i) {
        ulonglong2 v = INSERT ? ld_slot_relaxed(ia.index + s)
                              : __ldg(reinterpret_cast<const ulonglong2*>(ia.index + s));
        if (v.x == key) {
            uint32_t row = (uint32_t)v.y;
            slot_out = (uint32_t)s;
            if (row != ROW_PENDING || !INSERT) return row == ROW_PENDING ? ROW_ABSENT : row;
            atomicMin(&ia.index[s].aux, pos);
            return ROW_PENDING;
        }
        if (v.x == EMPTY_KEY) {
            if (!INSERT) return ROW_ABSENT;
            unsigned long long old = atomicCAS(&ia.index[s].key, EMPTY_KEY, key);
            if (old == EMPTY_KEY || old == key) {
                slot_out = (uint32_t)s;
                uint32_t row = ld_u32_relaxed(&ia.index[s].row);
                if (row != ROW_PENDING) return row;
                atomicMin(&ia.index[s].aux, pos);
                return ROW_PENDING;
            }
            // another key took this slot first: keep probing
        }
        s = (s + 1) & ia.mask;
    }
    record_error(ia.err, MLKV_ERR_PROBE_LIMIT);
    return ROW_ABSENT;
}

// Appends (pos, slot) to the miss list with one atomic per converged group of
// lanes.  The list holds at most one entry per lookup (n): an entry past that
// could only come from a counter left set, and is not written.
__device__ __forceinline__ void append_miss(CallCounters* cur, uint32_t* miss_pos,
                                            uint32_t* miss_slot, uint32_t pos, uint32_t slot, uint32_t n) {
    const unsigned m = __activemask();
    const int lane = threadIdx.x & 31;
    const int leader = __ffs(m) - 1;
    uint32_t base = 0;
    if (lane == leader) base = atomicAdd(&cur->n_miss, (uint32_t)__popc(m));
    base = __shfl_sync(m, base, leader);
    const uint32_t i = base + __popc(m & lanemask_lt());
    if (i < n) {
        miss_pos[i] = pos;
        miss_slot[i] = slot;
    }
}

__device__ __forceinline__ void zero_counters(CallCounters* nxt) {
    if (nxt && blockIdx.x == 0 && threadIdx.x < sizeof(CallCounters) / 4)
        reinterpret_cast<uint32_t*>(nxt)[threadIdx.x] = 0u;
}

constexpr uint32_t kBarrierSpins = 1u << 21;  // with its L2 load and 100 ns sleep, 1-2 s a barrier

__device__ __forceinline__ uint32_t ld_acquire_u32(const uint32_t* p) {
    uint32_t v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// Waits (one thread) until the count ctr & mask reaches `want`.  The wait is
// bounded: a spin that runs out records MLKV_ERR_TIMEOUT and returns false.
__device__ __forceinline__ bool wait_count(const uint32_t* ctr, uint32_t mask, uint32_t want, const ErrSink& err) {
    uint32_t spins = 0;
    while ((ld_acquire_u32(ctr) & mask) < want) {
        if (++spins > kBarrierSpins) {
            record_error(err, MLKV_ERR_TIMEOUT);
            return false;
        }
        __nanosleep(100);
    }
    return true;
}

// `want` blocks arrive at `ctr` (zero at the call's start) and wait until all
// have, or until one's wait has run out (false).  Only blocks of this one grid
// wait here, and a grid that does is small enough for all its blocks to be
// resident.  (mlkv_debug_fail's wait injection asks for one arrival more than
// there are, so that the wait runs out.)
__device__ __forceinline__ bool grid_barrier(uint32_t* ctr, uint32_t want, const ErrSink& err) {
    __shared__ int ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(ctr, 1u);
        ok = wait_count(ctr, 0xFFFFFFFFu, want, err);
        __threadfence();
    }
    __syncthreads();
    return ok != 0;
}

// The slot array as the index kernels use it.
struct IndexRows {
    float* slots;
    int stride;
    int dpad;
    int d;
    int NV;
    int G;
};

inline IndexRows row_args(mlkv_table* t) {
    return IndexRows{t->slots, t->geom.stride, t->geom.dpad, t->geom.d, t->geom.NV, t->geom.G};
}

inline IndexArgs index_args(mlkv_table* t) {
    return IndexArgs{t->index, t->index_mask, (t->cfg.flags & MLKV_IDENTITY_HASH) ? 1u : 0u,
                     ErrSink{&t->dstate->status, t->status_dev_alias, t->dstate->chk}};
}

// ---------------------------------------------------------------------------
// The miss path: new keys of a call get rows, in four phases separated by
// barriers of all its blocks (`barrier`; MissShare says which blocks they are):
//   1. flag the first occurrence of each new key (the lookup whose position
//      survived in the slot's aux);
//   2. rank the flags: an exclusive scan over the call's positions, every block
//      over a range of them of its own;
//   3. each first occurrence takes row = rows handed out so far + rank and
//      writes its init row (not for Put) and state_init (or, with new_keys, its
//      key alone: the apply's plan, whose few SMs would be long about the rows);
//   4. every missed lookup reads its key's row (a Get gathers it into its
//      output), flags and the slot's aux go back to idle, the row counter
//      advances.
// `on_row` is told every missed lookup's row in phase 4.  Data written by other
// blocks within the kernel is read from L2 (ld.cg).
// Phases 3 and 4 take the miss list's entries as for_misses deals them out: a
// warp loads up to 32 entries, one a lane, and its lane groups then write or copy
// their rows one after another.  (With a lane group loading the entry of each
// row it wrote, every row waited for three dependent loads: a Get of 16,384
// lookups of dim 128 whose last 64 keys are new took 64 us, 25 so.)
struct MissArgs {
    const int64_t* keys;
    uint32_t n;
    const uint32_t* miss_pos;
    const uint32_t* miss_slot;
    uint32_t* flag;
    uint32_t* rank;
    uint32_t* block_sums;  // [max_blocks]
    uint32_t max_blocks;
    uint32_t* row_of_pos;
    float* out;
    CallCounters* cur;
    DevState* ds;
    unsigned long long capacity;
    int init_row;
    int64_t* new_keys;  // or null
    unsigned long long seed;
    float lo, span, state_init;
};

inline MissArgs miss_args(mlkv_table* t, const int64_t* keys, int64_t n, MissMode mode, uint32_t* row_of_pos,
                          float* out, CallCounters* cur) {
    return MissArgs{keys, (uint32_t)n, t->s.miss_pos, t->s.miss_slot, t->s.first_flag, t->s.rank, t->s.miss_sums,
                    (uint32_t)t->s.max_miss_blocks, row_of_pos, out, cur, t->dstate, (unsigned long long)t->cfg.capacity,
                    mode == MissMode::Put ? 0 : 1, nullptr, (unsigned long long)t->cfg.seed, t->cfg.init_lo,
                    t->cfg.init_hi - t->cfg.init_lo, t->cfg.state_init};
}

// Whether the miss path may run in this many blocks.
inline bool miss_grid_fits(const mlkv_table* t, int64_t blocks) { return blocks <= t->s.max_miss_blocks; }

// Sum over the block of one value per thread.
template <int THREADS>
__device__ __forceinline__ uint32_t miss_block_sum(uint32_t v) {
    __shared__ uint32_t part[(THREADS / 32)];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    __syncthreads();
    if (lane == 0) part[w] = v;
    __syncthreads();
    uint32_t t = 0;
#pragma unroll
    for (int k = 0; k < (THREADS / 32); ++k) t += part[k];
    return t;
}

// Exclusive scan over the block of one value per thread; *total = the sum.
template <int THREADS>
__device__ __forceinline__ uint32_t miss_block_scan(uint32_t v, uint32_t& total) {
    __shared__ uint32_t part[(THREADS / 32)];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint32_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    __syncthreads();
    if (lane == 31) part[w] = x;
    __syncthreads();
    uint32_t before = 0;
    total = 0;
#pragma unroll
    for (int k = 0; k < (THREADS / 32); ++k) {
        if (k < w) before += part[k];
        total += part[k];
    }
    return before + x - v;
}

// The blocks of a miss path, and the positions this one ranks.  A block's
// place in the order of positions is `order` of the `nsums` that blocks (not all
// of them blocks of the miss path) have in MissArgs::block_sums.
struct MissShare {
    uint32_t nblocks, block;  // blocks of the miss path (the host keeps them within MissArgs::max_blocks), this one
    uint32_t nsums, order;
    uint32_t p_lo, p_hi;
};

// Every block of the grid, the positions in equal shares.
__device__ __forceinline__ MissShare even_share(uint32_t n, uint32_t nblocks, uint32_t block) {
    const uint32_t per = (n + nblocks - 1) / nblocks, lo = min(n, block * per);
    return MissShare{nblocks, block, nblocks, block, lo, min(n, lo + per)};
}

// f(i, at_once) for this lane's entry i (or a value >= m) of every round of the
// warp over the m entries of the miss list (the whole warp; at_once entries a
// round, whole groups of R = 32 / G and at most 32: every warp gets about as many).
template <int THREADS, class F>
__device__ __forceinline__ void for_misses(uint32_t m, uint32_t nblocks, uint32_t block, uint32_t R, F f) {
    const uint32_t warps = nblocks * (THREADS / 32), lane = threadIdx.x & 31;
    const uint32_t rounds = (m + warps * 32 - 1) / (warps * 32);
    const uint32_t at_once = ((m + warps * rounds - 1) / (warps * rounds) + R - 1) / R * R;
    for (uint32_t i0 = (block * (THREADS / 32) + (threadIdx.x >> 5)) * at_once; i0 < m; i0 += warps * at_once)
        f(lane < at_once ? i0 + lane : 0xFFFFFFFFu, at_once);
}

template <int V, int THREADS, class Barrier, class OnRow>
__device__ __forceinline__ bool miss_path(const IndexArgs& ia, const IndexRows& ra, const MissArgs& ma, uint32_t m,
                                          const MissShare& sh, Barrier barrier, OnRow on_row) {
    using VT = typename Vec<V>::T;
    const uint32_t nthreads = sh.nblocks * THREADS;
    const int lane = threadIdx.x & 31, G = ra.G, glane = lane & (G - 1), gid = lane / G;
    const uint32_t R = 32u / G;
    // 1. first occurrences
    for (uint32_t i = sh.block * THREADS + threadIdx.x; i < m; i += nthreads) {
        const uint32_t p = __ldcg(ma.miss_pos + i);
        if (ld_u32_relaxed(&ia.index[__ldcg(ma.miss_slot + i)].aux) == p) ma.flag[p] = 1u;
    }
    if (!barrier(0)) return false;
    // 2. ranks: the first occurrences at earlier positions
    uint32_t cnt = 0;
    for (uint32_t p = sh.p_lo + threadIdx.x; p < sh.p_hi; p += THREADS) cnt += __ldcg(ma.flag + p);
    const uint32_t mine = miss_block_sum<THREADS>(cnt);
    if (threadIdx.x == 0 && in_bounds(ia.err, kChkMissBlock, sh.order, ma.max_blocks)) ma.block_sums[sh.order] = mine;
    if (!barrier(1)) return false;
    uint32_t b_before = 0, b_all = 0;
    for (uint32_t b = threadIdx.x; b < sh.nsums; b += THREADS) {
        const uint32_t c = __ldcg(ma.block_sums + b);
        b_all += c;
        if (b < sh.order) b_before += c;
    }
    uint32_t run = miss_block_sum<THREADS>(b_before);
    if (sh.block == 0) {  // every first occurrence
        const uint32_t all = miss_block_sum<THREADS>(b_all);
        if (threadIdx.x == 0) ma.cur->n_new = all;
    }
    for (uint32_t p0 = sh.p_lo; p0 < sh.p_hi; p0 += THREADS) {  // uniform
        const uint32_t p = p0 + threadIdx.x;
        const uint32_t f = p < sh.p_hi ? __ldcg(ma.flag + p) : 0u;
        uint32_t tot;
        const uint32_t ex = miss_block_scan<THREADS>(f, tot);
        if (f) ma.rank[p] = run + ex;
        run += tot;
    }
    if (!barrier(2)) return false;
    // 3. rows of the first occurrences
    const unsigned long long next = ma.ds->next_row;
    for_misses<THREADS>(m, sh.nblocks, sh.block, R, [&](uint32_t i, uint32_t at_once) {
        uint32_t row = ROW_ABSENT;
        unsigned long long key = 0ull;
        if (i < m) {
            const uint32_t p = __ldcg(ma.miss_pos + i), s = __ldcg(ma.miss_slot + i);
            if (ld_u32_relaxed(&ia.index[s].aux) == p) {
                const unsigned long long r = next + __ldcg(ma.rank + p);
                key = (unsigned long long)ma.keys[p];
                if (r >= ma.capacity) record_error(ia.err, MLKV_ERR_FULL);
                else {
                    ia.index[s].row = row = (uint32_t)r;
                    if (ma.new_keys) ma.new_keys[r - next] = (int64_t)key;
                }
            }
        }
        if (ma.new_keys) return;
        for (uint32_t q = 0; q < at_once; q += R) {
            const uint32_t r = __shfl_sync(0xffffffffu, row, (int)q + gid);
            const unsigned long long key_q = __shfl_sync(0xffffffffu, key, (int)q + gid);
            if (r == ROW_ABSENT) continue;
            float* w = ra.slots + (size_t)r * ra.stride;
            VT* wv = reinterpret_cast<VT*>(w);
            VT* gv = reinterpret_cast<VT*>(w + ra.dpad);
            for (int j = glane; j < ra.NV; j += G) {
                if (ma.init_row) wv[j] = init_vec<V>(ma.seed, key_q, j, ma.lo, ma.span);
                gv[j] = Vec<V>::splat(ma.state_init);
            }
        }
    });
    if (!barrier(3)) return false;
    // 4. every missed lookup takes its key's row
    if (sh.block == 0 && threadIdx.x == 0) {
        const unsigned long long nr = next + __ldcg(&ma.cur->n_new);
        ma.ds->next_row = nr < ma.capacity ? nr : ma.capacity;
        if (ma.new_keys) ma.cur->new_base = (uint32_t)next + 1u;
    }
    for_misses<THREADS>(m, sh.nblocks, sh.block, R, [&](uint32_t i, uint32_t at_once) {
        uint32_t p = 0, row = ROW_PENDING;  // lanes without an entry copy nothing
        if (i < m) {
            const uint32_t s = __ldcg(ma.miss_slot + i);
            p = __ldcg(ma.miss_pos + i);
            row = ld_u32_relaxed(&ia.index[s].row);
            if (row == ROW_PENDING) row = ROW_ABSENT;
            if (ma.row_of_pos) ma.row_of_pos[p] = row;
            ma.flag[p] = 0u;
            ia.index[s].aux = AUX_IDLE;
            on_row(p, row);
        }
        if (!ma.out) return;
        for (uint32_t q = 0; q < at_once; q += R) {
            const uint32_t r = __shfl_sync(0xffffffffu, row, (int)q + gid);
            const uint32_t x = __shfl_sync(0xffffffffu, p, (int)q + gid);
            if (r == ROW_PENDING) continue;
            // (written by other blocks of this kernel)
            const VT* src = reinterpret_cast<const VT*>(ra.slots + (size_t)(r == ROW_ABSENT ? 0 : r) * ra.stride);
            VT* dst = reinterpret_cast<VT*>(ma.out + (size_t)x * ra.d);
#pragma unroll 2
            for (int j = glane; j < ra.NV; j += G) __stcs(dst + j, r == ROW_ABSENT ? Vec<V>::nan() : __ldcg(src + j));
        }
    });
    return true;
}

// The end of a Get whose grid is small enough to wait for itself: new keys get
// their rows, and the call's counters are released, in the same launch.  Every
// block arrives once it has copied its rows, with a mark where it met a new
// key.  Where no block did, the last to arrive zeroes the counters and nothing
// waits; else the marked blocks, alone, wait for the others and run the miss
// path.  (A miss kernel of its own that finds nothing to do cost a Get of 416
// lookups 4 of its 15 us, and the step of 4,096 lookups 2.5 of 36.)  The whole
// block, whose lookups start at position p_lo and end before p_hi, calls it: it
// ranks those positions, since a new key's are all in marked blocks.  (With the
// marked blocks sharing all of the call's positions, a Get of 16,384 lookups
// that met one new key had a single block scan them all: 52 us of dim 128 where
// one without new keys takes 13; 21 so.)  (mlkv_debug_fail's wait injection, bar_extra, makes the first
// marked block wait for one arrival too many; the other marked blocks then wait
// for that one in the miss path, in vain too.)
template <int V, int THREADS>
__device__ __forceinline__ void finish_get(const IndexArgs& ia, const IndexRows& ra, const MissArgs& ma,
                                           bool new_key, uint32_t p_lo, uint32_t p_hi, uint32_t bar_extra) {
    __shared__ uint32_t share[2];  // marked blocks, this block among them
    CallCounters* cur = ma.cur;
    const uint32_t grid = gridDim.x;
    const int marked = __syncthreads_or(new_key);
    if (threadIdx.x == 0) {
        if (!marked && in_bounds(ia.err, kChkMissBlock, blockIdx.x, ma.max_blocks)) ma.block_sums[blockIdx.x] = 0u;
        __threadfence();
        const uint32_t old = atomicAdd(&cur->bar[0], marked ? 0x10001u : 1u);
        share[1] = old >> 16;
        if (!marked) {
            if (old == grid - 1) {  // the last, and no block is marked
                uint32_t* w = reinterpret_cast<uint32_t*>(cur);
                for (unsigned i = 0; i < sizeof(CallCounters) / 4; ++i) w[i] = 0u;
            }
        } else {
            const uint32_t want = grid + (share[1] ? 0u : bar_extra);
            share[0] = wait_count(&cur->bar[0], 0xFFFFu, want, ia.err) ? ld_acquire_u32(&cur->bar[0]) >> 16 : 0u;
            __threadfence();
        }
    }
    if (!marked) return;
    __syncthreads();
    const uint32_t blocks = share[0];
    if (!blocks) return;  // the wait ran out
    const uint32_t m = min(ld_u32_relaxed(&cur->n_miss), ma.n);
    if (!miss_path<V, THREADS>(
            ia, ra, ma, m, MissShare{blocks, share[1], grid, blockIdx.x, p_lo, p_hi},
            [&](int i) { return grid_barrier(&cur->bar[i + 1], blocks, ia.err); },
            [](uint32_t, uint32_t) {}))
        return;
    release_counters(cur, blocks);
}

}  // namespace

}  // namespace mlkv
