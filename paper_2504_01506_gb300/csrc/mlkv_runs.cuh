// The records of a gradient apply's runs: what the kernels that find the runs
// write, and the reduce kernels read.
#pragma once

#include "mlkv_internal.cuh"

namespace mlkv {

namespace {

// Long runs are summed in chunks: of kChunkLarge lookups in calls of at least
// MLKV_SMALL_BATCH lookups, of kChunkSmall in smaller ones (few long runs: more
// chunks to sum in parallel; also in the runs of thousands of lookups, whose
// chunks the combine takes 256 a block: 64-lookup chunks there cost 100,003
// lookups of dim 50 78 us instead of 74).  Set at build time.
#ifndef MLKV_SMALL_BATCH
#define MLKV_SMALL_BATCH (1u << 19)
#endif
#ifndef MLKV_CHUNK_SMALL
#define MLKV_CHUNK_SMALL 16
#endif
constexpr uint32_t kChunkLarge = 64, kChunkSmall = MLKV_CHUNK_SMALL, kSmallBatch = MLKV_SMALL_BATCH;
#ifndef MLKV_GROUP_CHUNKS
#define MLKV_GROUP_CHUNKS 8
#endif
#ifndef MLKV_NODE
#define MLKV_NODE 256
#endif
constexpr uint32_t NONE = 0xFFFFFFFFu;  // no position (a small run's record past its end)
// k_combine: a lane group adds up the chunk sums of a run of at most
// kGroupChunks chunks; of longer runs, a block takes kNode chunks at a time.
constexpr uint32_t kGroupChunks = MLKV_GROUP_CHUNKS, kNode = MLKV_NODE;

constexpr uint32_t kItemLenBits = 7;  // a chunk holds at most 64 lookups; a run at most 2^24 chunks of 64
static_assert(kChunkLarge < (1u << kItemLenBits) && kChunkSmall < (1u << kItemLenBits), "chunk lengths fit their bits");

struct RunArgs {
    const float* grads;
    const uint32_t* srow;  // sorted row ids; lookups without a row hold `sent` and come last
    const uint32_t* spos;  // their lookup positions
    uint32_t n;
    uint32_t sent;
    CallCounters* cur;
    uint4* runs;           // [max_batch] short runs of 2 or more lookups: (first sorted position, one
                           //   past the last, row, first lookup position)
    uint2* singles;        // [max_batch] runs of one lookup: (row, lookup position)
    uint4* smalls;         // [max_batch] runs of 2 .. kSmallRun lookups: (row, p0, p1, p2), positions in
                           //   occurrence order, NONE past the run's end
    uint32_t* small_p3;    // [max_batch] their fourth position (or NONE)
    uint4* long_runs;      // [max_long] long runs of at most kGroupChunks chunks: (first chunk, chunks, row, -)
    uint4* nodes;          // [max_nodes] kNode chunks each of the longer runs: (the run's first chunk, its chunks,
                           //   row, node of the run)
    uint4* items;          // [max_items] chunks of the long runs: (first sorted position, lookups |
                           //   chunks of the run << kItemLenBits, row, the run's first chunk)
    float* partial;        // [max_items][2][dpad] sums of chunks, and of nodes in their first chunk's place
    uint32_t* node_cnt;    // [max_items][nseg] nodes of a run done (k_combine, at the run's first chunk's entry), or
                           //   arrivals at the lowest nodes of k_reduce's trees; behind them the higher levels',
                           //   [levels - 1][kTreeEntries]; zero at rest
    uint32_t max_long;
    uint32_t max_nodes;
    uint32_t max_items;
    uint32_t chunk;        // lookups per chunk of a long run (kChunkLarge or kChunkSmall)
    ErrSink err;
    float lr, eps;
    struct {               // what the new rows of a plan's apply start with (make_new)
        const int64_t* keys;  // [new rows] their keys
        unsigned long long seed;
        float lo, span, state_init;
    } new_rows;
    uint32_t release;      // non-zero in the apply's last kernels: the blocks of all of them (release_counters)
};

inline RunArgs run_args(mlkv_table* t, const float* grads, const uint32_t* srow, const uint32_t* spos, int64_t n,
                        uint32_t sent, CallCounters* cur) {
    return RunArgs{grads, srow, spos, (uint32_t)n, sent, cur, t->s.short_runs, t->s.single_runs, t->s.small_runs,
                   t->s.small_p3, t->s.long_runs, t->s.nodes, t->s.items, t->s.partial, t->s.node_cnt,
                   (uint32_t)t->s.max_long, (uint32_t)t->s.max_nodes, (uint32_t)t->s.max_items,
                   n >= kSmallBatch ? kChunkLarge : kChunkSmall,
                   ErrSink{&t->dstate->status, t->status_dev_alias, t->dstate->chk}, t->cfg.lr, t->cfg.eps,
                   {t->s.new_keys, (unsigned long long)t->cfg.seed, t->cfg.init_lo, t->cfg.init_hi - t->cfg.init_lo,
                    t->cfg.state_init}, 0u};
}

// What the long runs qs[k] .. qe[k] (k < nq) add to the lists: chunks, runs
// combined by a lane group, and nodes.
struct LongCounts {
    uint32_t items, runs, nodes;
};

__device__ __forceinline__ uint32_t warp_inclusive(uint32_t x, int lane) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    return x;
}

// This lane's run's counts, their exclusive prefix over the lanes, and the sums
// (the whole warp).
__device__ __forceinline__ LongCounts long_counts(const uint32_t* qs, const uint32_t* qe, int nq, int lane,
                                                  uint32_t chunk, LongCounts& mine, LongCounts& excl) {
    const uint32_t len = lane < nq ? qe[lane] - qs[lane] : 0u;
    mine.items = (len + chunk - 1) / chunk;
    mine.runs = lane < nq && mine.items <= kGroupChunks;
    mine.nodes = mine.items > kGroupChunks ? (mine.items + kNode - 1) / kNode : 0u;
    const LongCounts in = {warp_inclusive(mine.items, lane), warp_inclusive(mine.runs, lane),
                           warp_inclusive(mine.nodes, lane)};
    excl = {in.items - mine.items, in.runs - mine.runs, in.nodes - mine.nodes};
    return {__shfl_sync(0xffffffffu, in.items, 31), __shfl_sync(0xffffffffu, in.runs, 31),
            __shfl_sync(0xffffffffu, in.nodes, 31)};
}

// Writes the chunks of the long runs qs[k], qe[k], qr[k] (k < nq: start, end,
// row) and their runs or nodes at list entries base.. (the whole warp).
__device__ __forceinline__ void write_long_runs(const RunArgs& a, const uint32_t* qs, const uint32_t* qe,
                                                const uint32_t* qr, int nq, const LongCounts& base, int lane) {
    LongCounts mine, excl;
    long_counts(qs, qe, nq, lane, a.chunk, mine, excl);
    if (mine.runs) a.long_runs[base.runs + excl.runs] = make_uint4(base.items + excl.items, mine.items, qr[lane], 0u);
    for (int k = 0; k < nq; ++k) {
        const uint32_t s = qs[k], e = qe[k], row = qr[k], chunk = a.chunk;
        const uint32_t m = __shfl_sync(0xffffffffu, mine.items, k);
        const uint32_t ib = base.items + __shfl_sync(0xffffffffu, excl.items, k);
        const uint32_t nodes = __shfl_sync(0xffffffffu, mine.nodes, k);
        const uint32_t nb = base.nodes + __shfl_sync(0xffffffffu, excl.nodes, k);
        for (uint32_t c = lane; c < m; c += 32) {
            const uint32_t cs = s + c * chunk;
            a.items[ib + c] = make_uint4(cs, min(chunk, e - cs) | m << kItemLenBits, row, ib);
        }
        for (uint32_t c = lane; c < nodes; c += 32) a.nodes[nb + c] = make_uint4(ib, m, row, c);
    }
}

// Room for what base + tot would reach in the lists.
__device__ __forceinline__ bool long_room(const RunArgs& a, const LongCounts& base, const LongCounts& tot) {
    return base.items + tot.items <= a.max_items && base.runs + tot.runs <= a.max_long &&
           base.nodes + tot.nodes <= a.max_nodes;
}

}  // namespace

}  // namespace mlkv
