// The plan of a small gradient apply in one launch: probe (and the miss path),
// sort and run lists, by one thread-block cluster.
//
// A batch of up to kPlanMax lookups is a fraction of a wave for the general
// kernels (probe, miss, then an offsets and a scatter kernel a sort pass, then
// k_heads): each waits for the one before it, and 3-6 us go by in each for a
// few hundred KB.  Here up to 16 blocks of 1024 threads, on 16 SMs of one GPU
// processing cluster, hold the whole batch in their shared memory: a sort pass
// ranks each block's elements, the blocks read one another's digit counts
// through distributed shared memory, and every element is stored straight into
// the shared memory of the block that owns its sorted position.  The blocks
// meet at the cluster's hardware barrier (all of a cluster's blocks are
// resident together, so it needs no bound).
//
// Bound by latency: of the 16 us of 4,096 lookups (4 blocks, 17-bit row ids) 2
// go to the rows, 5 to each of two sort passes, 4-5 to the run lists.  With one
// lookup a thread on as many blocks as the batch fills a pass is a single round
// of 32 per warp; 4 lookups a thread on a quarter of the blocks took 4 us more
// at 4,096 lookups and 13 at 13,312.  Apply + Get, before -> with the plan and
// the one-kernel reduce: 2,048 lookups of dim 128 55 -> 34 us, 8,192 58 -> 39,
// 16,384 61 -> 48, 32,768 70 -> 62.  At 65,536 (4 lookups a thread) the 16 SMs
// take as long as the general kernels take on all of them (dim 16: 77 -> 75,
// dim 512: 156 -> 161), so kPlanMax = 32,768.
//
// A block takes an SM's whole register file (1,024 threads of 64 registers), and
// all blocks start at once: beside a grid that keeps its blocks on many SMs for
// long (another stream's) the plan waits until enough SMs of one processing
// cluster are free, where the general kernels would run in what room there is.  An
// apply beside the table's own look-ahead avoids that (plan_beside_fetch).
#include <cooperative_groups.h>

#include <mutex>
#include <unordered_map>

#include "mlkv_probe.cuh"
#include "mlkv_runs.cuh"

namespace mlkv {

namespace {

namespace cg = cooperative_groups;

constexpr int kPlanThreads = 1024;
constexpr int kPlanWarps = kPlanThreads / 32;
constexpr int kPlanDigitBits = 10;  // one digit per thread
constexpr int kPlanRadix = 1 << kPlanDigitBits;
constexpr int kPlanItems = 2;       // most lookups per thread
constexpr int kLongBatch = 8;       // long runs a warp writes at a time

// A tile of T = 1024 * items lookups per block.
struct __align__(16) PlanShared {
    uint16_t wcnt[kPlanWarps * kPlanRadix];     // [warp][radix] elements of each digit, then their exclusive prefix
    uint16_t ctot[kPlanRadix];                  // the block's elements of each digit (read by the other blocks)
    uint16_t all[kPlanCluster * kPlanRadix];    // [block][radix] every block's
    uint32_t gbase[kPlanRadix];                 // sorted position of the block's first element of each digit
    uint32_t bits[kPlanThreads * kPlanItems / 32];  // a bit per sorted element: another row than its left neighbour's
    uint32_t words[kPlanItems];             // a bit per word of `bits`: not zero
    uint32_t firsts[kPlanCluster];          // sorted position of every block's first set bit, or NONE
    uint32_t halo[kSmallRun];               // the next block's first sorted positions' lookups
    uint32_t nlong;
    uint32_t cnt[3], base[3];               // runs of one, of 2 .. kSmallRun, of more lookups: count, list entry
    uint32_t warp_sums[kPlanWarps];
    uint32_t ls[kPlanThreads * kPlanItems / (MLKV_SEQ_SEGMENT_MAX + 1) + 2];  // long runs: start, end, row
    uint32_t le[kPlanThreads * kPlanItems / (MLKV_SEQ_SEGMENT_MAX + 1) + 2];
    uint32_t lr[kPlanThreads * kPlanItems / (MLKV_SEQ_SEGMENT_MAX + 1) + 2];
};

// Flags of PlanArgs::how
constexpr int kPlanInsert = 1;   // absent keys get rows (else they are skipped and reported)
constexpr int kPlanMemo = 2;     // a lookup may take the row the last Get found for its key
constexpr int kPlanRows = 4;     // the rows are in row_of_pos already

struct PlanArgs {
    const int64_t* keys;
    uint32_t n;
    int how;
    int passes, digit_bits;
    uint32_t* row_of_pos;
    uint32_t* miss_pos;
    uint32_t* miss_slot;
    uint32_t* spos;  // [n] out: the sorted lookup positions
    CallCounters* nxt;
    Memo memo;
};

__device__ __forceinline__ uint32_t block_exclusive(uint32_t v, uint32_t* warp_sums) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const uint32_t x = warp_inclusive(v, lane);
    if (lane == 31) warp_sums[w] = x;
    __syncthreads();
    if (w == 0) warp_sums[lane] = warp_inclusive(warp_sums[lane], lane);
    __syncthreads();
    return (w ? warp_sums[w - 1] : 0u) + x - v;
}

// The list of a run of len lookups: 0 one, 1 of 2 .. kSmallRun, 2 of up to
// MLKV_SEQ_SEGMENT_MAX, -1 none of these.
__device__ __forceinline__ int list_of(uint32_t len) {
    return len == 0 || len > MLKV_SEQ_SEGMENT_MAX ? -1 : len == 1 ? 0 : len <= kSmallRun ? 1 : 2;
}

template <int V, int ITEMS>
__global__ void __launch_bounds__(kPlanThreads, 1) k_plan(IndexArgs ia, IndexRows ra, MissArgs ma, PlanArgs pa,
                                                          RunArgs a) {
    pdl_enter();
    constexpr int kItemsShift = ITEMS == 1 ? 0 : 1;
    constexpr int kTileShift = 10 + kItemsShift;
    constexpr uint32_t T = 1u << kTileShift;
    static_assert(ITEMS == (1 << kItemsShift) && ITEMS <= kPlanItems, "1 or 2 lookups a thread");
    extern __shared__ __align__(16) unsigned char smem[];
    PlanShared& sh = *reinterpret_cast<PlanShared*>(smem);
    // [T] sorted (row id, lookup position)
    uint2* skv = reinterpret_cast<uint2*>(smem + sizeof(PlanShared));
    cg::cluster_group cluster = cg::this_cluster();
    const uint32_t nblocks = gridDim.x, me = blockIdx.x;  // the grid is one cluster
    auto meet = [&]() {
        if (nblocks > 1) cluster.sync();
        else __syncthreads();
    };
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const uint32_t lt = lanemask_lt();
    const uint32_t n = pa.n, sent = a.sent;
    const uint32_t tile0 = me << kTileShift;
    // element r of this thread: a warp holds 32 * ITEMS consecutive elements, in rounds of 32
    auto elem = [&](int r) { return (uint32_t)(w * 32 * ITEMS + r * 32 + lane); };
    zero_counters(pa.nxt);

    // 1. rows
    uint32_t key[ITEMS], val[ITEMS];
    {
        unsigned long long k[ITEMS];
        uint32_t row[ITEMS];
#pragma unroll
        for (int r = 0; r < ITEMS; ++r) {
            const uint32_t p = tile0 + elem(r);
            val[r] = p;
            row[r] = ROW_PENDING;
            k[r] = 0ull;
            if (p >= n) continue;
            if (pa.how & kPlanRows) {
                row[r] = __ldg(pa.row_of_pos + p);
                continue;
            }
            k[r] = (unsigned long long)__ldg(pa.keys + p);
            if (pa.how & kPlanMemo) {
                const uint32_t mr = pa.memo.row[p];
                if ((unsigned long long)pa.memo.key[p] == k[r]) row[r] = mr;
            }
        }
        if (!(pa.how & kPlanRows)) {
#pragma unroll
            for (int r = 0; r < ITEMS; ++r) {
                const uint32_t p = tile0 + elem(r);
                if (p >= n || row[r] < ROW_ABSENT) continue;
                uint32_t slot = 0;
                if (pa.how & kPlanInsert) {
                    row[r] = probe_key<true>(ia, k[r], p, slot);
                    if (row[r] == ROW_PENDING) append_miss(ma.cur, pa.miss_pos, pa.miss_slot, p, slot, n);
                } else {
                    row[r] = probe_key<false>(ia, k[r], p, slot);
                    if (row[r] == ROW_ABSENT) record_error(ia.err, MLKV_ERR_NOT_FOUND);
                }
            }
            if (pa.how & kPlanInsert) {
                __threadfence();
                meet();
                const uint32_t m = min(ld_u32_relaxed(&ma.cur->n_miss), n);
                if (m) {  // the same for every block
                    auto none = [](uint32_t, uint32_t) {};
                    miss_path<V, kPlanThreads>(
                        ia, ra, ma, m, even_share(ma.n, nblocks, me),
                        [&](int) {
                            __threadfence();
                            meet();
                            return true;
                        },
                        none);
                    __threadfence();
                    meet();
#pragma unroll
                    for (int r = 0; r < ITEMS; ++r) {
                        const uint32_t p = tile0 + elem(r);
                        if (p < n && row[r] == ROW_PENDING) row[r] = __ldcg(pa.row_of_pos + p);
                    }
                }
            }
        }
#pragma unroll
        for (int r = 0; r < ITEMS; ++r) key[r] = row[r] >= ROW_ABSENT ? sent : row[r];
    }

    // 2. stable radix sort of (row, position), least significant digit first
    const int D = pa.digit_bits, radix = 1 << D;
    for (int pass = 0; pass < pa.passes; ++pass) {
        const int shift = pass * D;
        for (int i = threadIdx.x; i < (kPlanWarps << D) / 8; i += kPlanThreads)
            reinterpret_cast<uint4*>(sh.wcnt)[i] = make_uint4(0u, 0u, 0u, 0u);
        uint16_t* wc = sh.wcnt + (w << D);
        if (pass) {
#pragma unroll
            for (int r = 0; r < ITEMS; ++r) {
                const uint2 kv = skv[elem(r)];
                key[r] = kv.x;
                val[r] = kv.y;
            }
        }
        __syncthreads();
        uint32_t rnk[ITEMS];
#pragma unroll
        for (int r = 0; r < ITEMS; ++r) {
            const bool valid = tile0 + elem(r) < n;
            const uint32_t dig = (key[r] >> shift) & (uint32_t)(radix - 1);
            const uint32_t vm = __ballot_sync(0xffffffffu, valid);
            uint32_t peers = valid ? vm : ~vm;
            for (int b = 0; b < D; ++b) {
                const bool one = (dig >> b) & 1u;
                const uint32_t m = __ballot_sync(0xffffffffu, one);
                peers &= one ? m : ~m;
            }
            uint32_t before = 0;
            if (valid) before = wc[dig];
            __syncwarp();
            if (valid && lane == __ffs(peers) - 1) wc[dig] = (uint16_t)(before + __popc(peers));
            __syncwarp();
            rnk[r] = before + __popc(peers & lt);
        }
        __syncthreads();
        const int d = threadIdx.x;
        if (d < radix) {
            uint32_t tot = 0;
#pragma unroll 8
            for (int ww = 0; ww < kPlanWarps; ++ww) {
                const uint32_t c = sh.wcnt[(ww << D) + d];
                sh.wcnt[(ww << D) + d] = (uint16_t)tot;
                tot += c;
            }
            sh.ctot[d] = (uint16_t)tot;
        }
        meet();  // every block's counts are there, and its elements in registers
        // the blocks' counts, 8 digits a load (thread per digit and block: 16
        // remote loads each at 16 blocks, 3 us a pass instead of 1)
        if (nblocks > 1) {
            const uint32_t per = (uint32_t)radix / 8, loads = per * nblocks;
            for (uint32_t i = threadIdx.x; i < loads; i += kPlanThreads) {
                const uint32_t c = i / per, x = i - c * per;
                reinterpret_cast<uint4*>(sh.all)[i] =
                    reinterpret_cast<const uint4*>(cluster.map_shared_rank(sh.ctot, c))[x];
            }
            __syncthreads();
        }
        uint32_t all = 0, before = 0;
        if (d < radix) {
            const uint16_t* from = nblocks > 1 ? sh.all : sh.ctot;
            for (uint32_t c = 0; c < nblocks; ++c) {
                const uint32_t x = from[(c << D) + d];
                all += x;
                before += c < me ? x : 0u;
            }
        }
        const uint32_t ex = block_exclusive(all, sh.warp_sums);
        sh.gbase[d] = ex + before;
        __syncthreads();
#pragma unroll
        for (int r = 0; r < ITEMS; ++r) {
            if (tile0 + elem(r) >= n) continue;
            const uint32_t dig = (key[r] >> shift) & (uint32_t)(radix - 1);
            const uint32_t dst = sh.gbase[dig] + wc[dig] + rnk[r];
            uint2* to = nblocks > 1 ? cluster.map_shared_rank(skv, dst >> kTileShift) : skv;
            to[dst & (T - 1)] = make_uint2(key[r], val[r]);
        }
        meet();
    }

    // 3. run heads: a bit per sorted element whose left neighbour has another row
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) {
        const uint32_t e = elem(r), g = tile0 + e;
        const uint2 kv = skv[e];
        key[r] = kv.x;
        val[r] = kv.y;
        bool head = false;
        if (g < n) {
            pa.spos[g] = val[r];
            const uint32_t left = e ? skv[e - 1].x : g ? cluster.map_shared_rank(skv, me - 1)[T - 1].x : ~key[r];
            head = key[r] != left;
        }
        const uint32_t b = __ballot_sync(0xffffffffu, head);
        if (lane == 0) sh.bits[e >> 5] = b;
    }
    if (threadIdx.x < 3) sh.cnt[threadIdx.x] = 0u;
    if (threadIdx.x == 3) sh.nlong = 0u;
    __syncthreads();
    if (w == 0) {
        uint32_t f = NONE;
#pragma unroll
        for (int k = 0; k < ITEMS; ++k) {
            const uint32_t b = sh.bits[k * 32 + lane];
            const uint32_t nz = __ballot_sync(0xffffffffu, b != 0u);
            if (lane == 0) sh.words[k] = nz;
            if (f == NONE && nz) {
                const int l = __ffs(nz) - 1;
                f = tile0 + (uint32_t)(k * 32 + l) * 32u + (uint32_t)__ffs(__shfl_sync(0xffffffffu, b, l)) - 1u;
            }
        }
        // ... which the other blocks are told (a run may end in a later block)
        if ((uint32_t)lane < nblocks) {
            uint32_t* to = nblocks > 1 ? cluster.map_shared_rank(sh.firsts, lane) : sh.firsts;
            to[me] = f;
        }
    }
    // the next block's first positions, for a run of 2 .. kSmallRun that goes on there
    if (me + 1 < nblocks && threadIdx.x >= 32 && threadIdx.x < 32 + kSmallRun)
        sh.halo[threadIdx.x - 32] = cluster.map_shared_rank(skv, me + 1)[threadIdx.x - 32].y;
    meet();  // the last: nothing of another block is read after it
    // the end of a run that starts at element e: the next set bit, here or in a later block
    auto run_end = [&](uint32_t e) {
        uint32_t wd = e >> 5;
        uint32_t b = (e & 31u) == 31u ? 0u : sh.bits[wd] & (0xFFFFFFFEu << (e & 31u));
        if (b) return tile0 + (wd << 5) + (uint32_t)__ffs(b) - 1u;
        ++wd;
        for (uint32_t k = wd >> 5; k < (uint32_t)ITEMS; ++k) {
            uint32_t nz = sh.words[k];
            if (k == wd >> 5) nz &= 0xFFFFFFFFu << (wd & 31u);
            if (nz) {
                const uint32_t x = k * 32 + (uint32_t)__ffs(nz) - 1u;
                return tile0 + (x << 5) + (uint32_t)__ffs(sh.bits[x]) - 1u;
            }
        }
        for (uint32_t c = me + 1; c < nblocks; ++c) {
            if (sh.firsts[c] != NONE) return sh.firsts[c];
        }
        return n;
    };
    // 4. the runs to their lists: a place within the block, then one atomic per block and list
    uint32_t place[ITEMS], len[ITEMS];
    {
        uint32_t tot[3] = {0u, 0u, 0u};  // the warp's runs of each list
#pragma unroll
        for (int r = 0; r < ITEMS; ++r) {
            const uint32_t e = elem(r), g = tile0 + e;
            const bool head = g < n && ((sh.bits[e >> 5] >> (e & 31u)) & 1u) && key[r] != sent;
            len[r] = head ? run_end(e) - g : 0u;
            place[r] = 0;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const bool in = list_of(len[r]) == c;
                const uint32_t m = __ballot_sync(0xffffffffu, in);
                if (in) place[r] = tot[c] + __popc(m & lt);
                tot[c] += __popc(m);
            }
            if (len[r] > MLKV_SEQ_SEGMENT_MAX) {
                const uint32_t q = atomicAdd(&sh.nlong, 1u);
                sh.ls[q] = g;
                sh.le[q] = g + len[r];
                sh.lr[q] = key[r];
            }
        }
        uint32_t b = 0;
        if (lane < 3) b = atomicAdd(&sh.cnt[lane], lane == 0 ? tot[0] : lane == 1 ? tot[1] : tot[2]);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const uint32_t at = __shfl_sync(0xffffffffu, b, c);
#pragma unroll
            for (int r = 0; r < ITEMS; ++r)
                if (list_of(len[r]) == c) place[r] += at;
        }
    }
    __syncthreads();
    if (threadIdx.x < 3) {
        const uint32_t c = sh.cnt[threadIdx.x];
        uint32_t* to = threadIdx.x == 0 ? &a.cur->n_single : threadIdx.x == 1 ? &a.cur->n_small : &a.cur->n_short;
        sh.base[threadIdx.x] = c ? atomicAdd(to, c) : 0u;
    }
    // the long runs, a warp per kLongBatch of them (warp 0 has the counts above)
    for (uint32_t q0 = (uint32_t)((w + kPlanWarps - 1) % kPlanWarps) * kLongBatch; q0 < sh.nlong;
         q0 += kPlanWarps * kLongBatch) {
        const int nq = (int)min((uint32_t)kLongBatch, sh.nlong - q0);
        LongCounts mine, excl, base = {0u, 0u, 0u};
        const LongCounts tot = long_counts(sh.ls + q0, sh.le + q0, nq, lane, a.chunk, mine, excl);
        uint32_t b = 0;  // the four counters at once
        if (lane == 0) b = atomicAdd(&a.cur->n_items, tot.items);
        if (lane == 1) b = atomicAdd(&a.cur->n_group, tot.runs);
        if (lane == 2) b = atomicAdd(&a.cur->n_nodes, tot.nodes);
        if (lane == 3) atomicAdd(&a.cur->n_long, (uint32_t)nq);
        base.items = __shfl_sync(0xffffffffu, b, 0);
        base.runs = __shfl_sync(0xffffffffu, b, 1);
        base.nodes = __shfl_sync(0xffffffffu, b, 2);
        if (!long_room(a, base, tot)) {
            if (lane == 0) record_error(a.err, MLKV_ERR_FULL);
        } else {
            write_long_runs(a, sh.ls + q0, sh.le + q0, sh.lr + q0, nq, base, lane);
        }
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) {
        if (len[r] == 0 || len[r] > MLKV_SEQ_SEGMENT_MAX) continue;
        const uint32_t e = elem(r), g = tile0 + e;
        if (len[r] == 1) {
            a.singles[sh.base[0] + place[r]] = make_uint2(key[r], val[r]);
        } else if (len[r] <= kSmallRun) {
            auto pos = [&](uint32_t k) -> uint32_t {
                if (k >= len[r]) return NONE;
                return e + k < T ? skv[e + k].y : sh.halo[e + k - T];
            };
            const uint32_t i = sh.base[1] + place[r];
            a.smalls[i] = make_uint4(key[r], val[r], pos(1), pos(2));
            a.small_p3[i] = pos(3);
        } else {
            a.runs[sh.base[2] + place[r]] = make_uint4(g, g + len[r], key[r], val[r]);
        }
    }
}

template <int V, int ITEMS>
cudaError_t run_plan(mlkv_table* t, int blocks, const MissArgs& ma, const PlanArgs& pa, const RunArgs& a,
                     cudaStream_t st) {
    const size_t smem = sizeof(PlanShared) + (size_t)kPlanThreads * ITEMS * 8;
    const auto kernel = k_plan<V, ITEMS>;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = (unsigned)blocks;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3(kPlanThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = MLKV_PDL ? attr : attr + 1;
    cfg.numAttrs = MLKV_PDL ? 2 : 1;
    timer_before(t, MLKV_K_PLAN, st);
    cudaLaunchKernelEx(&cfg, kernel, index_args(t), row_args(t), ma, pa, a);  // an error stays in cudaGetLastError()
    timer_after(t, MLKV_K_PLAN, st);
    t->launches++;
    return cudaGetLastError();
}

template <int ITEMS>
bool prepare_items(int& largest) {
    const int smem = (int)(sizeof(PlanShared) + (size_t)kPlanThreads * ITEMS * 8);
    const void* kernels[3] = {(const void*)k_plan<4, ITEMS>, (const void*)k_plan<2, ITEMS>,
                              (const void*)k_plan<1, ITEMS>};
    for (const void* k : kernels) {
        if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess ||
            cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)
            return false;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
        cudaLaunchConfig_t cfg = {};
        cfg.blockDim = dim3(kPlanThreads);
        cfg.dynamicSmemBytes = (size_t)smem;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        for (; largest > 1; largest /= 2) {  // the largest cluster the GPU can place
            attr[0].val.clusterDim.x = (unsigned)largest;
            cfg.gridDim = dim3((unsigned)largest);
            int clusters = 0;
            if (cudaOccupancyMaxActiveClusters(&clusters, k, &cfg) == cudaSuccess && clusters > 0) break;
            cudaGetLastError();
        }
    }
    return true;
}

}  // namespace

// A device's answer is kept: the attributes and occupancy queries take 0.1 ms.
int plan_prepare(int device) try {
    static std::mutex mu;
    static std::unordered_map<int, int> known;
    std::lock_guard<std::mutex> lock(mu);
    const auto it = known.find(device);
    if (it != known.end()) return it->second;
    int largest = kPlanCluster;
    if (!prepare_items<1>(largest) || !prepare_items<kPlanItems>(largest)) {
        cudaGetLastError();
        largest = 0;
    }
    return known[device] = largest;
} catch (...) {  // no memory for the entry, under a C entry: the general kernels
    return 0;
}

bool plan_fits(const mlkv_table* t, int64_t n) {
    return n <= (int64_t)t->plan_cluster * kPlanThreads * kPlanItems && n <= (int64_t)kPlanMax;
}

cudaError_t launch_plan(mlkv_table* t, const int64_t* keys, int64_t n, bool insert, bool memo, bool rows,
                        cudaStream_t st, CallCounters* cur, CallCounters* nxt, const uint32_t** spos) {
    // few lookups a thread where the cluster's blocks allow it: a pass's time is
    // its rounds of 32 lookups a warp
    int items = 1;
    while (items < kPlanItems && n > (int64_t)t->plan_cluster * kPlanThreads * items) items *= 2;
    const int64_t tile = (int64_t)kPlanThreads * items;
    int blocks = 1;
    while (blocks * tile < n) blocks *= 2;
    if (!miss_grid_fits(t, blocks)) return cudaErrorInvalidConfiguration;
    const int passes = (t->sort_bits + kPlanDigitBits - 1) / kPlanDigitBits;
    PlanArgs pa{};
    pa.keys = keys;
    pa.n = (uint32_t)n;
    pa.how = (insert ? kPlanInsert : 0) | (memo ? kPlanMemo : 0) | (rows ? kPlanRows : 0);
    pa.passes = passes;
    pa.digit_bits = (t->sort_bits + passes - 1) / passes;
    if (pa.digit_bits < 3) pa.digit_bits = 3;  // whole 16-byte loads of the counts
    pa.row_of_pos = t->s.row_of_pos;
    pa.miss_pos = t->s.miss_pos;
    pa.miss_slot = t->s.miss_slot;
    pa.nxt = nxt;
    pa.memo = Memo{t->s.memo_key, t->s.memo_row};
    *spos = pa.spos = t->s.sv[0];
    const uint32_t sent = (uint32_t)((1ull << t->sort_bits) - 1);
    const RunArgs a = run_args(t, nullptr, nullptr, *spos, n, sent, cur);
    MissArgs ma = miss_args(t, keys, n, MissMode::Init, t->s.row_of_pos, nullptr, cur);
    ma.new_keys = t->s.new_keys;
    auto go = [&](auto v) {
        constexpr int V = decltype(v)::value;
        if (items == 1) return run_plan<V, 1>(t, blocks, ma, pa, a, st);
        return run_plan<V, kPlanItems>(t, blocks, ma, pa, a, st);
    };
    if (t->geom.V == 4) return go(std::integral_constant<int, 4>());
    if (t->geom.V == 2) return go(std::integral_constant<int, 2>());
    return go(std::integral_constant<int, 1>());
}

}  // namespace mlkv
