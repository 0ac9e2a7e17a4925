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

// Group-cooperative copy of one row (or NaN) into dst.  The row was written by
// another block of this kernel: read from L2.
template <int V>
__device__ __forceinline__ void copy_row(const float* src, float* __restrict__ dst,
                                         int NV, int G, int glane, bool absent) {
    using VT = typename Vec<V>::T;
    const VT* s = reinterpret_cast<const VT*>(src);
    VT* o = reinterpret_cast<VT*>(dst);
#pragma unroll 2
    for (int j = glane; j < NV; j += G) __stcs(o + j, absent ? Vec<V>::nan() : __ldcg(s + j));
}

// ---------------------------------------------------------------------------
// The miss path: new keys of a call get rows, in four phases separated by
// barriers of all its blocks (`barrier`; `nblocks` blocks, this one `block`):
//   1. flag the first occurrence of each new key (the lookup whose position
//      survived in the slot's aux);
//   2. rank the flags: an exclusive scan over the call's positions, block b
//      owning positions [b * per, (b + 1) * per);
//   3. each first occurrence takes row = rows handed out so far + rank and
//      writes its init row (not for Put) and state_init;
//   4. every missed lookup reads its key's row (a Get gathers it into its
//      output), flags and the slot's aux go back to idle, the row counter
//      advances.
// The host keeps nblocks within MissArgs::max_blocks (miss_grid_fits).
// `on_row` is told every missed lookup's row in phase 4.  Data written by other
// blocks within the kernel is read from L2 (ld.cg).
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
    unsigned long long seed;
    float lo, span, state_init;
};

inline MissArgs miss_args(mlkv_table* t, const int64_t* keys, int64_t n, MissMode mode, uint32_t* row_of_pos,
                          float* out, CallCounters* cur) {
    return MissArgs{keys, (uint32_t)n, t->s.miss_pos, t->s.miss_slot, t->s.first_flag, t->s.rank, t->s.miss_sums,
                    (uint32_t)t->s.max_miss_blocks, row_of_pos, out, cur, t->dstate, (unsigned long long)t->cfg.capacity,
                    mode == MissMode::Put ? 0 : 1, (unsigned long long)t->cfg.seed, t->cfg.init_lo,
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

template <int V, int THREADS, class Barrier, class OnRow>
__device__ __forceinline__ bool miss_path(const IndexArgs& ia, const IndexRows& ra, const MissArgs& ma, uint32_t m,
                                          uint32_t nblocks, uint32_t block, Barrier barrier, OnRow on_row) {
    using VT = typename Vec<V>::T;
    const uint32_t nthreads = nblocks * blockDim.x;
    const uint32_t tid = block * blockDim.x + threadIdx.x;
    const int G = ra.G, glane = threadIdx.x & (G - 1);
    const uint32_t group = tid / G, ngroups = nthreads / G;
    // 1. first occurrences
    for (uint32_t i = tid; i < m; i += nthreads) {
        const uint32_t p = __ldcg(ma.miss_pos + i);
        if (ld_u32_relaxed(&ia.index[__ldcg(ma.miss_slot + i)].aux) == p) ma.flag[p] = 1u;
    }
    if (!barrier(0)) return false;
    // 2. ranks: the first occurrences at earlier positions
    const uint32_t per = (ma.n + nblocks - 1) / nblocks;
    const uint32_t p_lo = min(ma.n, block * per), p_hi = min(ma.n, p_lo + per);
    uint32_t cnt = 0;
    for (uint32_t p = p_lo + threadIdx.x; p < p_hi; p += blockDim.x) cnt += __ldcg(ma.flag + p);
    const uint32_t mine = miss_block_sum<THREADS>(cnt);
    if (threadIdx.x == 0 && in_bounds(ia.err, kChkMissBlock, block, ma.max_blocks)) ma.block_sums[block] = mine;
    if (!barrier(1)) return false;
    uint32_t b_before = 0;
    for (uint32_t b = threadIdx.x; b < block; b += blockDim.x) b_before += __ldcg(ma.block_sums + b);
    uint32_t run = miss_block_sum<THREADS>(b_before);
    for (uint32_t p0 = p_lo; p0 < p_hi; p0 += blockDim.x) {  // uniform
        const uint32_t p = p0 + threadIdx.x;
        const uint32_t f = p < p_hi ? __ldcg(ma.flag + p) : 0u;
        uint32_t tot;
        const uint32_t ex = miss_block_scan<THREADS>(f, tot);
        if (f) ma.rank[p] = run + ex;
        run += tot;
    }
    if (block == nblocks - 1 && threadIdx.x == 0) ma.cur->n_new = run;  // every first occurrence
    if (!barrier(2)) return false;
    // 3. rows of the first occurrences
    const unsigned long long next = ma.ds->next_row;
    for (uint32_t i = group; i < m; i += ngroups) {
        const uint32_t p = __ldcg(ma.miss_pos + i), s = __ldcg(ma.miss_slot + i);
        if (ld_u32_relaxed(&ia.index[s].aux) != p) continue;
        const unsigned long long r = next + __ldcg(ma.rank + p);
        if (r >= ma.capacity) {
            if (glane == 0) record_error(ia.err, MLKV_ERR_FULL);
            continue;
        }
        const unsigned long long key = (unsigned long long)ma.keys[p];
        float* w = ra.slots + (size_t)r * ra.stride;
        VT* wv = reinterpret_cast<VT*>(w);
        VT* gv = reinterpret_cast<VT*>(w + ra.dpad);
        for (int j = glane; j < ra.NV; j += G) {
            if (ma.init_row) {
                float e[V];
#pragma unroll
                for (int c = 0; c < V; ++c) e[c] = init_element(ma.seed, key, (uint32_t)(j * V + c), ma.lo, ma.span);
                wv[j] = Vec<V>::from(e);
            }
            gv[j] = Vec<V>::splat(ma.state_init);
        }
        if (glane == 0) ia.index[s].row = (uint32_t)r;
    }
    if (!barrier(3)) return false;
    // 4. every missed lookup takes its key's row
    if (block == 0 && threadIdx.x == 0) {
        const unsigned long long nr = next + __ldcg(&ma.cur->n_new);
        ma.ds->next_row = nr < ma.capacity ? nr : ma.capacity;
    }
    for (uint32_t i = group; i < m; i += ngroups) {
        const uint32_t p = __ldcg(ma.miss_pos + i), s = __ldcg(ma.miss_slot + i);
        const uint32_t r0 = ld_u32_relaxed(&ia.index[s].row);
        const uint32_t r = r0 == ROW_PENDING ? ROW_ABSENT : r0;
        if (glane == 0) {
            if (ma.row_of_pos) ma.row_of_pos[p] = r;
            ma.flag[p] = 0u;
            ia.index[s].aux = AUX_IDLE;
            on_row(p, r);
        }
        if (ma.out)
            copy_row<V>(ra.slots + (size_t)(r == ROW_ABSENT ? 0 : r) * ra.stride,
                        ma.out + (size_t)p * ra.d, ra.NV, G, glane, r == ROW_ABSENT);
    }
    return true;
}

// The end of a Get whose grid is small enough to wait for itself: new keys get
// their rows, and the call's counters are released, in the same launch.  Every
// block arrives once it has copied its rows, with a mark where it met a new
// key.  Where no block did, the last to arrive zeroes the counters and nothing
// waits; else the marked blocks, alone, wait for the others and run the miss
// path.  (A miss kernel of its own that finds nothing to do cost a Get of 416
// lookups 4 of its 15 us, and the step of 4,096 lookups 2.5 of 36.)  The whole
// block calls it.  (mlkv_debug_fail's wait injection, bar_extra, makes the first
// marked block wait for one arrival too many; the other marked blocks then wait
// for that one in the miss path, in vain too.)
template <int V, int THREADS>
__device__ __forceinline__ void finish_get(const IndexArgs& ia, const IndexRows& ra, const MissArgs& ma,
                                           bool new_key, uint32_t bar_extra) {
    __shared__ uint32_t share[2];  // marked blocks, this block among them
    CallCounters* cur = ma.cur;
    const uint32_t grid = gridDim.x;
    const int marked = __syncthreads_or(new_key);
    if (threadIdx.x == 0) {
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
            ia, ra, ma, m, blocks, share[1],
            [&](int i) { return grid_barrier(&cur->bar[i + 1], blocks, ia.err); },
            [](uint32_t, uint32_t) {}))
        return;
    release_counters(cur, blocks);
}

}  // namespace

}  // namespace mlkv
