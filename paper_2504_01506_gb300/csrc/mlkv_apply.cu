// Segmented gradient reduction fused with the sparse Adagrad read-modify-write.
//
// After the sort, the lookups of one row form a run (segment) of consecutive
// sorted positions, in occurrence order (the sort is stable).  For every run
// the sum g of its gradient rows is formed and one Adagrad step is applied to
// the row and its state, each read once and written once:
//     G += g*g ;  w -= lr * g / (sqrt(G) + eps)          (element-wise)
// This is the per-key Rmw of MLKV Section 3.2 step 8, with the gradient of the
// embedding map E (Section 2.1) summed over the key's lookups.
//
//  k_heads        a warp per window of 32 sorted positions finds the runs
//                 that start there (a row id unlike its left neighbour) and
//                 their lengths; runs of one lookup, of 2 .. kSmallRun lookups
//                 (with their positions) and the other runs of <=
//                 MLKV_SEQ_SEGMENT_MAX lookups go to three lists (one atomic
//                 per block and list; any order: every run is summed on its
//                 own), longer ones are measured (a warp-wide search for their
//                 end) and listed for k_long.
//  k_single       runs of one lookup: row, state and the gradient row loaded
//                 together, then the Adagrad step.
//  k_small        runs of 2 .. kSmallRun lookups, whose positions k_heads wrote
//                 into the run's record: row, state and every gradient row in
//                 one round trip, the occurrence-order sum, the Adagrad step.
//  k_short        runs of kSmallRun + 1 .. MLKV_SEQ_SEGMENT_MAX lookups: row,
//                 state, first gradient row and the run's other positions
//                 loaded together, the rest summed in occurrence order, then
//                 the Adagrad step.
//  k_long         chunks of 64 lookups (16 in calls of fewer than 2^19 lookups)
//                 of a long run (Zipf-hot keys reach 10^4-10^5 lookups): the
//                 chunk's sum, compensated, to scratch as a (sum, compensation)
//                 pair.
//  k_combine      per long run: the chunk pairs added in a fixed order with
//                 compensation, the sum rounded once, and the row updated.
//  k_reduce       all of these in one launch, for small calls (whose run lists
//                 the plan of mlkv_plan.cu makes in place of k_heads).
//
// The row kernels' unit of work is one segment of a run: a lane group (G
// lanes, the power of two that holds a row of up to 32 vectors) reduces G
// vectors of the row at a time, and a wider row is nseg units.  Every operation
// is element-wise, so the segments are independent, and a segment takes the
// registers of a narrow row.  (With a wide row's vectors all held by one lane
// group, 4 a lane at dim 512, k_single spilled at its 40 registers and took
// 172 us for 65,536 lookups, Zipf(0.8), of dim 512; by segments it takes 67,
// and the apply + Get 190 us instead of 319.)
//
// Long runs are summed with compensation because the Adagrad step is
// ill-conditioned where a summed gradient element lands near eps (with zero
// state, u = lr * g / (|g| + eps) changes fast in g there): a plain fp32 sum
// of 10^2-10^4 terms can then move the update by more than 1e-5, while the
// compensated sum stays within about one rounding of the exact sum.
// Each kernel is tuned for requests in flight (resident warps against rows in
// flight per warp): the access pattern is random 512-byte rows, which HBM
// serves near its copy bandwidth only with many requests in flight.  Results do
// not depend on scheduling.
#include <algorithm>

#include "mlkv_runs.cuh"

namespace mlkv {

namespace {

// Tuning (set at build time): gradient rows in flight per lane group in a long
// chunk and in a run of 5-32 lookups, and the resident blocks per SM the
// register allocations must allow.
#ifndef MLKV_LONG_ROWS
#define MLKV_LONG_ROWS 8
#endif
#ifndef MLKV_SHORT_ROWS
#define MLKV_SHORT_ROWS 8
#endif
#ifndef MLKV_LONG_MIN_BLOCKS
#define MLKV_LONG_MIN_BLOCKS 2
#endif
#ifndef MLKV_SHORT_MIN_BLOCKS
#define MLKV_SHORT_MIN_BLOCKS 2
#endif
#ifndef MLKV_SMALL_MIN_BLOCKS
#define MLKV_SMALL_MIN_BLOCKS 4
#endif
#ifndef MLKV_SINGLE_MIN_BLOCKS
#define MLKV_SINGLE_MIN_BLOCKS 6
#endif
// k_short: runs a lane group claims at a time.
#ifndef MLKV_SHORT_GRAB
#define MLKV_SHORT_GRAB 4
#endif

struct RowArgs {
    float* slots;
    int stride;
    int dpad;
    int NV;
    int G;
    int gshift;      // log2 of G
    int d;
    uint32_t nseg;   // segments of G vectors per row: a lane group reduces one segment of a run at a time
    uint32_t nrows;  // rows of the slot array (bounds-checked build)
};

__device__ __forceinline__ unsigned group_mask(int G, int gid) {
    return G == 32 ? 0xffffffffu : (((1u << G) - 1u) << (gid * G));
}

// acc += the gradient vectors (this lane's column j, live when j < NV) of
// sorted positions s .. s+len-1, in that order, ROWS in flight.  The group
// loads up to G positions at a time (one per lane) and hands them round with
// group shuffles.  With PRE the first G positions were loaded by the caller
// (pl_first, one per lane).  With COMP every addition is compensated
// (comp_add): acc + cmp is then the sum to about twice fp32's precision;
// without it cmp is not touched.
template <int V, int ROWS, bool PRE, bool COMP>
__device__ __forceinline__ void sum_rows(typename Vec<V>::T& acc, typename Vec<V>::T& cmp,
                                         const float* __restrict__ grads, const uint32_t* __restrict__ spos,
                                         uint32_t s, uint32_t len, int d, int j, bool act, int G, int glane,
                                         unsigned gmask, const ErrSink& err, uint32_t site, uint32_t n,
                                         uint32_t pl_first = 0u) {
    using VT = typename Vec<V>::T;
    for (uint32_t base = 0; base < len; base += G) {
        const uint32_t cnt = min((uint32_t)G, len - base);
        if (MLKV_CHECK && !in_bounds(err, site, s + base + cnt - 1, n)) return;
        const uint32_t pl = (PRE && base == 0) ? pl_first
                            : (uint32_t)glane < cnt ? __ldg(spos + s + base + glane) : 0u;
        for (uint32_t x = 0; x < cnt; x += ROWS) {
            VT g[ROWS];
#pragma unroll
            for (int u = 0; u < ROWS; ++u) {
                uint32_t p = __shfl_sync(gmask, pl, (int)(x + u) & (G - 1), G);
                if (MLKV_CHECK && x + u < cnt && !in_bounds(err, site, p, n)) p = 0;
                if (x + u < cnt && act) g[u] = __ldcs(reinterpret_cast<const VT*>(grads + (size_t)p * d) + j);
            }
#pragma unroll
            for (int u = 0; u < ROWS; ++u)
                if (x + u < cnt && act) {
                    if (COMP) Vec<V>::cadd(acc, cmp, g[u]);
                    else Vec<V>::add(acc, g[u]);
                }
        }
    }
}

// This lane's vectors (column j) of a row and of its state.
template <int V>
__device__ __forceinline__ typename Vec<V>::T* row_vec(const RowArgs& ra, uint32_t row, int j) {
    return reinterpret_cast<typename Vec<V>::T*>(ra.slots + (size_t)row * ra.stride) + j;
}

// The state's (or a pair's compensation's) vector beside p.
template <class VT>
__device__ __forceinline__ VT* beside(const RowArgs& ra, VT* p) {
    return reinterpret_cast<VT*>(reinterpret_cast<float*>(p) + ra.dpad);
}
template <class VT>
__device__ __forceinline__ const VT* beside(const RowArgs& ra, const VT* p) {
    return reinterpret_cast<const VT*>(reinterpret_cast<const float*>(p) + ra.dpad);
}

// The Adagrad step on loaded row and state vectors, and their stores.
template <int V>
__device__ __forceinline__ void adagrad_store(const RowArgs& ra, uint32_t row, int j, typename Vec<V>::T w,
                                              typename Vec<V>::T G, const typename Vec<V>::T& g, float lr,
                                              float eps) {
    typename Vec<V>::T* p = row_vec<V>(ra, row, j);
    Vec<V>::adagrad(w, G, g, lr, eps);
    *p = w;
    *beside(ra, p) = G;
}

// The rows that an apply's plan gave new keys, from row first_new on, hold nothing
// yet: the lanes that reduce a row's run write its init values and its state
// before they load them.  (The plan's 16 SMs at most took longer for the rows than
// all the rest of an apply: 4,096 new keys of dim 128 111 us, 46 so, of dim 512 224
// and 58; an apply without new keys pays one load and a comparison a unit.)
__device__ __forceinline__ uint32_t first_new(const RunArgs& a) { return a.cur->new_base - 1u; }  // or NONE

template <int V>
__device__ __forceinline__ void make_new(const RowArgs& ra, const RunArgs& a, uint32_t row, uint32_t from, int j) {
    if (row < from || j >= ra.NV) return;
    typename Vec<V>::T* p = row_vec<V>(ra, row, j);
    *p = init_vec<V>(a.new_rows.seed, (unsigned long long)__ldg(a.new_rows.keys + (row - from)), j, a.new_rows.lo,
                     a.new_rows.span);
    *beside(ra, p) = Vec<V>::splat(a.new_rows.state_init);
}

// Where the run of `row` that starts at sorted position s ends: the first
// later position holding another row, or n.  The whole warp searches: 32
// probes at doubling distances, then rounds of 32 evenly spaced probes, each
// round narrowing [lo, hi) (srow[lo] == row; hi == n or srow[hi] != row) 32-fold.
__device__ __forceinline__ uint32_t run_end(const uint32_t* __restrict__ srow, uint32_t n, uint32_t s,
                                            uint32_t row, int lane) {
    uint32_t lo = s, hi = n;
    {
        const unsigned long long q = (unsigned long long)s + (64ull << lane);
        const bool eq = q < hi && __ldg(srow + q) == row;
        const int k = __popc(__ballot_sync(0xffffffffu, eq));  // the equal probes are the first k lanes
        if (k) lo = (uint32_t)((unsigned long long)s + (64ull << (k - 1)));
        const unsigned long long qh = (unsigned long long)s + (64ull << k);
        if (qh < hi) hi = (uint32_t)qh;
    }
    while (hi - lo > 1) {
        const uint32_t step = (hi - lo + 31) / 32;
        const unsigned long long q = (unsigned long long)lo + (unsigned long long)step * (lane + 1);
        const bool eq = q < hi && __ldg(srow + q) == row;
        const uint32_t c = __popc(__ballot_sync(0xffffffffu, eq));
        const unsigned long long nhi = (unsigned long long)lo + (unsigned long long)step * (c + 1);
        lo += step * c;
        if (nhi < hi) hi = (uint32_t)nhi;
    }
    return hi;
}

// The same, for a run of `row` that covers position q0 - 1 (q0 a multiple of
// 32): first the next 1024 positions in one round (32 consecutive per lane,
// 16-byte loads), which ends most runs; beyond that, run_end.
__device__ __forceinline__ uint32_t scan_end(const uint32_t* __restrict__ srow, uint32_t n, uint32_t q0,
                                             uint32_t row, int lane) {
    if (q0 >= n) return n;
    const uint32_t b = q0 + 32u * lane;
    int first = 32;  // first position of this lane's 32 with another row
    if (b + 32 <= n) {
        const uint4* v = reinterpret_cast<const uint4*>(srow + b);
#pragma unroll
        for (int k = 7; k >= 0; --k) {
            const uint4 x = __ldg(v + k);
            if (x.w != row) first = 4 * k + 3;
            if (x.z != row) first = 4 * k + 2;
            if (x.y != row) first = 4 * k + 1;
            if (x.x != row) first = 4 * k;
        }
    } else {
        for (int k = 31; k >= 0; --k)
            if (b + k >= n || __ldg(srow + b + k) != row) first = k;
    }
    const unsigned m = __ballot_sync(0xffffffffu, first < 32);
    if (m) {
        const int l = __ffs(m) - 1;
        return q0 + 32u * l + (uint32_t)__shfl_sync(0xffffffffu, first, l);
    }
    return run_end(srow, n, q0 + 1023u, row, lane);
}

// A warp per window of 32 sorted positions (windows dealt out grid-stride).
// A run starts where a row id differs from its left neighbour; it ends at the
// next change of value in the window (the next run, or the absent lookups
// that sort last) or, for the window's last run, where the next window's row
// ids first differ (past that, it is long and its end is searched for after
// the windows).  Runs of one lookup and the other runs of <=
// MLKV_SEQ_SEGMENT_MAX lookups are staged in the warp's shared-memory lists,
// long ones in its queue; at the end the block reserves room in the run lists
// and the chunk list with one atomic each and the warps copy their runs out.  (Counters that every warp bumps queue up at
// the end of the kernel.)
#ifndef MLKV_HEADS_MIN_BLOCKS
#define MLKV_HEADS_MIN_BLOCKS 4
#endif
__global__ void __launch_bounds__(256, MLKV_HEADS_MIN_BLOCKS) k_heads(RunArgs a, SortTail tail) {
    pdl_enter();
    zero_tail(tail);
    constexpr int kList = 128, kListS = 64, kQueue = 16;
    __shared__ uint4 lst[8][kListS];  // (start, end, row, first lookup) of short runs
    __shared__ uint2 sgl[8][kList];   // (row, lookup) of runs of one lookup
    __shared__ uint4 sml[8][kListS];  // (row, p0, p1, p2) of small runs
    __shared__ uint32_t sp3[8][kListS];  // ... and their p3
    __shared__ uint32_t qs[8][kQueue], qr[8][kQueue], qe[8][kQueue];  // long runs: start, row, end (0: unknown)
    __shared__ LongCounts wlc[8];  // per warp: what its long runs add to the lists; then their bases
    __shared__ uint32_t wsh[8], wlg[8], ws1[8], ws2[8];  // per warp: short runs, long runs,
                                                                 // runs of one lookup, small runs; then
                                                                 // their bases
    const uint32_t n = a.n, sent = a.sent;
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const uint32_t lt = lanemask_lt();
    const uint32_t warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint32_t nwarps = (gridDim.x * blockDim.x) >> 5;
    const uint32_t nwin = (n + 31) >> 5;
    int cnt = 0, cnt1 = 0, cnt2 = 0, nq = 0;  // warp-uniform
    // full lists or a full queue go out at once (only batches far above a few
    // runs per window and warp get here)
    auto flush = [&]() {
        __syncwarp();
        uint32_t base = 0, base1 = 0, base2 = 0;
        if (lane == 0 && cnt) base = atomicAdd(&a.cur->n_short, (uint32_t)cnt);
        if (lane == 0 && cnt1) base1 = atomicAdd(&a.cur->n_single, (uint32_t)cnt1);
        if (lane == 0 && cnt2) base2 = atomicAdd(&a.cur->n_small, (uint32_t)cnt2);
        base = __shfl_sync(0xffffffffu, base, 0);
        base1 = __shfl_sync(0xffffffffu, base1, 0);
        base2 = __shfl_sync(0xffffffffu, base2, 0);
        for (int k = lane; k < cnt; k += 32) a.runs[base + k] = lst[wib][k];
        for (int k = lane; k < cnt1; k += 32) a.singles[base1 + k] = sgl[wib][k];
        for (int k = lane; k < cnt2; k += 32) {
            a.smalls[base2 + k] = sml[wib][k];
            a.small_p3[base2 + k] = sp3[wib][k];
        }
        cnt = 0;
        cnt1 = 0;
        cnt2 = 0;
        __syncwarp();
    };
    auto measure = [&]() {  // fills in the unknown ends of the queued long runs
        __syncwarp();
        for (int k = 0; k < nq; ++k) {
            // an unknown end lies past the window after the run's first one
            if (qe[wib][k] == 0u) {
                const uint32_t e = scan_end(a.srow, n, (qs[wib][k] & ~31u) + 64u, qr[wib][k], lane);
                __syncwarp();
                if (lane == 0) qe[wib][k] = e;
                __syncwarp();
            }
        }
    };
    auto emit_long = [&](const LongCounts& base) {
        if (nq) write_long_runs(a, qs[wib], qe[wib], qr[wib], nq, base, lane);
        nq = 0;
        __syncwarp();
    };
    // a window's row ids, the next window's, the left neighbour and the
    // positions, loaded one window ahead
    auto load = [&](uint32_t w, uint32_t& r, uint32_t& nr, uint32_t& l0, uint32_t& pos) {
        const uint32_t p = (w << 5) + lane;
        r = p < n ? __ldg(a.srow + p) : sent;
        nr = p + 32 < n ? __ldg(a.srow + p + 32) : sent;
        pos = p < n ? __ldg(a.spos + p) : 0u;
        l0 = lane == 0 && p > 0 && p <= n ? __ldg(a.srow + p - 1) : ~r;
    };
    uint32_t xr = sent, xnr = sent, xl0 = 0u, xpos = 0u;
    if (warp < nwin) load(warp, xr, xnr, xl0, xpos);
    for (uint32_t w = warp; w < nwin; w += nwarps) {  // warp-uniform
        const uint32_t p = (w << 5) + lane;
        const uint32_t r = xr, nr = xnr, pos = xpos;
        uint32_t left = __shfl_up_sync(0xffffffffu, r, 1);
        if (lane == 0) left = xl0;
        if (w + nwarps < nwin) load(w + nwarps, xr, xnr, xl0, xpos);
        const unsigned em = __ballot_sync(0xffffffffu, r != left);  // a run, or the absent tail, starts here
        const bool head = r != sent && r != left;
        const unsigned hm = __ballot_sync(0xffffffffu, head);
        if (!hm) continue;
        const uint32_t lrow = __shfl_sync(0xffffffffu, r, 31 - __clz(hm));
        const unsigned diff = __ballot_sync(0xffffffffu, nr != lrow);  // for the window's last run
        const unsigned after = lane == 31 ? 0u : em & (0xFFFFFFFEu << lane);
        uint32_t len = 0;
        bool lng = false;
        if (head) {
            if (after) len = (uint32_t)(__ffs(after) - 1 - lane);
            else if (diff) len = 32 - lane + (__ffs(diff) - 1);
            else lng = true;
            lng = lng || len > MLKV_SEQ_SEGMENT_MAX;
        }
        const bool shrt = head && !lng;  // len >= 1
        const bool smll = shrt && len > 1 && len <= kSmallRun;
        const unsigned sm = __ballot_sync(0xffffffffu, shrt && len > kSmallRun);
        const unsigned s1 = __ballot_sync(0xffffffffu, shrt && len == 1);
        const unsigned s2 = __ballot_sync(0xffffffffu, smll);
        // a small run's other positions: from the lanes after its head, or, where
        // the run goes on into the next window, from the sorted positions
        const uint32_t q1 = __shfl_down_sync(0xffffffffu, pos, 1);
        const uint32_t q2 = __shfl_down_sync(0xffffffffu, pos, 2);
        const uint32_t q3 = __shfl_down_sync(0xffffffffu, pos, 3);
        if (cnt + __popc(sm) > kListS || cnt1 + __popc(s1) > kList || cnt2 + __popc(s2) > kListS) flush();
        if (shrt && len > kSmallRun) lst[wib][cnt + __popc(sm & lt)] = make_uint4(p, p + len, r, pos);
        if (shrt && len == 1) sgl[wib][cnt1 + __popc(s1 & lt)] = make_uint2(r, pos);
        if (smll && MLKV_CHECK && !in_bounds(a.err, kChkHeadsPos, p + len - 1, n)) len = 2;
        if (smll && (!MLKV_CHECK || in_bounds(a.err, kChkHeadsPos, p + len - 1, n))) {
            const uint32_t p1 = lane + 1 < 32 ? q1 : __ldg(a.spos + p + 1);
            const uint32_t p2 = len < 3 ? NONE : lane + 2 < 32 ? q2 : __ldg(a.spos + p + 2);
            const uint32_t p3 = len < 4 ? NONE : lane + 3 < 32 ? q3 : __ldg(a.spos + p + 3);
            const int k = cnt2 + __popc(s2 & lt);
            sml[wib][k] = make_uint4(r, pos, p1, p2);
            sp3[wib][k] = p3;
        }
        cnt += __popc(sm);
        cnt1 += __popc(s1);
        cnt2 += __popc(s2);
        for (unsigned lm = __ballot_sync(0xffffffffu, head && lng); lm; lm &= lm - 1) {
            const int i = __ffs(lm) - 1;
            if (nq == kQueue) {
                measure();
                LongCounts mine, excl, base = {0u, 0u, 0u};
                const LongCounts tot = long_counts(qs[wib], qe[wib], nq, lane, a.chunk, mine, excl);
                if (lane == 0) {
                    atomicAdd(&a.cur->n_long, (uint32_t)nq);
                    base.items = atomicAdd(&a.cur->n_items, tot.items);
                    base.runs = atomicAdd(&a.cur->n_group, tot.runs);
                    base.nodes = atomicAdd(&a.cur->n_nodes, tot.nodes);
                }
                base.items = __shfl_sync(0xffffffffu, base.items, 0);
                base.runs = __shfl_sync(0xffffffffu, base.runs, 0);
                base.nodes = __shfl_sync(0xffffffffu, base.nodes, 0);
                if (!long_room(a, base, tot)) {
                    if (lane == 0) record_error(a.err, MLKV_ERR_FULL);
                    nq = 0;
                } else {
                    emit_long(base);
                }
            }
            const uint32_t row = __shfl_sync(0xffffffffu, r, i);
            const uint32_t ln = __shfl_sync(0xffffffffu, len, i);  // 0 when the end is past the next window
            if (lane == 0) {
                qs[wib][nq] = (w << 5) + i;
                qr[wib][nq] = row;
                qe[wib][nq] = ln ? (w << 5) + i + ln : 0u;
            }
            ++nq;
        }
    }
    measure();
    LongCounts mine, excl;
    const LongCounts tot = long_counts(qs[wib], qe[wib], nq, lane, a.chunk, mine, excl);
    if (lane == 0) {
        wsh[wib] = (uint32_t)cnt;
        wlg[wib] = (uint32_t)nq;
        wlc[wib] = tot;
        ws1[wib] = (uint32_t)cnt1;
        ws2[wib] = (uint32_t)cnt2;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t ts = 0, tl = 0, t1 = 0, t2 = 0;
        LongCounts t = {0u, 0u, 0u};
        for (int k = 0; k < 8; ++k) {
            ts += wsh[k];
            tl += wlg[k];
            t = {t.items + wlc[k].items, t.runs + wlc[k].runs, t.nodes + wlc[k].nodes};
            t1 += ws1[k];
            t2 += ws2[k];
        }
        uint32_t bs = ts ? atomicAdd(&a.cur->n_short, ts) : 0u;
        if (tl) atomicAdd(&a.cur->n_long, tl);
        LongCounts b = {t.items ? atomicAdd(&a.cur->n_items, t.items) : 0u,
                        t.runs ? atomicAdd(&a.cur->n_group, t.runs) : 0u,
                        t.nodes ? atomicAdd(&a.cur->n_nodes, t.nodes) : 0u};
        uint32_t b1 = t1 ? atomicAdd(&a.cur->n_single, t1) : 0u;
        uint32_t b2 = t2 ? atomicAdd(&a.cur->n_small, t2) : 0u;
        for (int k = 0; k < 8; ++k) {
            const uint32_t c0 = wsh[k], c3 = ws1[k], c4 = ws2[k];
            const LongCounts c = wlc[k];
            wsh[k] = bs;
            wlc[k] = b;
            ws1[k] = b1;
            ws2[k] = b2;
            bs += c0;
            b = {b.items + c.items, b.runs + c.runs, b.nodes + c.nodes};
            b1 += c3;
            b2 += c4;
        }
    }
    __syncthreads();
    for (int k = lane; k < cnt; k += 32) a.runs[wsh[wib] + k] = lst[wib][k];
    for (int k = lane; k < cnt1; k += 32) a.singles[ws1[wib] + k] = sgl[wib][k];
    for (int k = lane; k < cnt2; k += 32) {
        a.smalls[ws2[wib] + k] = sml[wib][k];
        a.small_p3[ws2[wib] + k] = sp3[wib][k];
    }
    const LongCounts base = wlc[wib];
    if (!long_room(a, base, tot)) {
        if (lane == 0 && nq) record_error(a.err, MLKV_ERR_FULL);
        return;
    }
    emit_long(base);
}

// (acc, cmp) = the pairs of tree entries slot0, slot0 + stride, ... (cnt of
// them, in that order): each entry's sum added with compensation, then its own
// compensation added to cmp.
template <int V>
__device__ __forceinline__ void sum_pairs(typename Vec<V>::T& acc, typename Vec<V>::T& cmp, const RowArgs& ra,
                                          const float* partial, uint32_t slot0, uint32_t stride, uint32_t cnt, int j,
                                          bool act) {
    using VT = typename Vec<V>::T;
    constexpr int UNR = 4;
    acc = Vec<V>::zero();
    cmp = Vec<V>::zero();
    if (!act) return;
    for (uint32_t x = 0; x < cnt; x += UNR) {
        VT g[UNR], c[UNR];
#pragma unroll
        for (int u = 0; u < UNR; ++u)
            if (x + u < cnt) {
                const VT* src =
                    reinterpret_cast<const VT*>(partial + (size_t)(slot0 + (x + u) * stride) * 2 * ra.dpad) + j;
                g[u] = __ldcg(src);
                c[u] = __ldcg(beside(ra, src));
            }
#pragma unroll
        for (int u = 0; u < UNR; ++u)
            if (x + u < cnt) {
                Vec<V>::cadd(acc, cmp, g[u]);
                Vec<V>::add(cmp, c[u]);
            }
    }
}

// The compensated sum of one segment of chunk rec of a long run, by one lane group.
template <int V>
__device__ __forceinline__ bool chunk_sum(typename Vec<V>::T& acc, typename Vec<V>::T& cmp, const RowArgs& ra,
                                          const RunArgs& a, const uint4& rec, int j, int G, int glane,
                                          unsigned gmask) {
    const uint32_t len = rec.y & ((1u << kItemLenBits) - 1);
    if (MLKV_CHECK && !(in_bounds(a.err, kChkLongItem, rec.x + len, (unsigned long long)a.n + 1) &&
                        in_bounds(a.err, kChkLongItem, rec.w + (rec.y >> kItemLenBits),
                                  (unsigned long long)a.max_items + 1) &&
                        in_bounds(a.err, kChkLongRow, rec.z, ra.nrows)))
        return false;
    acc = Vec<V>::zero();
    cmp = Vec<V>::zero();
    sum_rows<V, MLKV_LONG_ROWS, false, true>(acc, cmp, a.grads, a.spos, rec.x, len, ra.d, j, j < ra.NV, G, glane,
                                             gmask, a.err, kChkLongPos, a.n);
    return true;
}

// Tree entry `slot`'s (sum, compensation) pair: this lane's vectors.
template <int V>
__device__ __forceinline__ void store_pair(const RowArgs& ra, const RunArgs& a, uint32_t slot, int j,
                                           const typename Vec<V>::T& acc, const typename Vec<V>::T& cmp) {
    typename Vec<V>::T* part = reinterpret_cast<typename Vec<V>::T*>(a.partial + (size_t)slot * 2 * ra.dpad) + j;
    __stcg(part, acc);
    __stcg(beside(ra, part), cmp);
}

// The sum acc + cmp rounded once, and the Adagrad step of `row` with it.
template <int V>
__device__ __forceinline__ void finish_long(const RowArgs& ra, const RunArgs& a, uint32_t row, int j,
                                            typename Vec<V>::T acc, const typename Vec<V>::T& cmp) {
    Vec<V>::add(acc, cmp);
    const typename Vec<V>::T* p = row_vec<V>(ra, row, j);
    adagrad_store<V>(ra, row, j, *p, *beside(ra, p), acc, a.lr, a.eps);
}

// One segment of a run of kSmallRun + 1 .. MLKV_SEQ_SEGMENT_MAX lookups (sorted
// positions s .. e-1, first lookup p0), by one lane group: the row, the state,
// the first gradient row and the other lookups' positions load together, the
// rest of the gradient rows are added in occurrence order, then the Adagrad
// step.
template <int V, int ROWS>
__device__ __forceinline__ void short_run(const RowArgs& ra, const RunArgs& a, uint32_t s, uint32_t e, uint32_t row,
                                          uint32_t p0, int j, int G, int glane, unsigned gmask) {
    using VT = typename Vec<V>::T;
    if (MLKV_CHECK && !(in_bounds(a.err, kChkShortRun, e, (unsigned long long)a.n + 1) &&
                        in_bounds(a.err, kChkShortRun, s, e) && in_bounds(a.err, kChkShortRow, row, ra.nrows) &&
                        in_bounds(a.err, kChkShortPos, p0, a.n)))
        return;
    const bool act = j < ra.NV;
    const uint32_t rest = e - s - 1;
    const uint32_t pl0 = (uint32_t)glane < min(rest, (uint32_t)G) ? __ldg(a.spos + s + 1 + glane) : 0u;
    VT w, Gs, acc = Vec<V>::zero();
    if (act) {
        const VT* p = row_vec<V>(ra, row, j);
        w = p[0];
        Gs = *beside(ra, p);
        Vec<V>::add(acc, __ldcs(reinterpret_cast<const VT*>(a.grads + (size_t)p0 * ra.d) + j));  // 0 + g: in order
    }
    sum_rows<V, ROWS, true, false>(acc, acc, a.grads, a.spos, s + 1, rest, ra.d, j, act, G, glane, gmask, a.err,
                                   kChkShortPos, a.n, pl0);
    if (act) adagrad_store<V>(ra, row, j, w, Gs, acc, a.lr, a.eps);
}

// One segment of a run of 2 .. kSmallRun lookups, whose positions are in its
// record: the row, the state and every gradient row load together, then the
// sum 0 + g0 + g1 + ... in occurrence order and the Adagrad step.
template <int V>
__device__ __forceinline__ void small_run(const RowArgs& ra, const RunArgs& a, const uint4& m, uint32_t p3, int j) {
    using VT = typename Vec<V>::T;
    if (j >= ra.NV) return;
    const uint32_t ps[kSmallRun] = {m.y, m.z, m.w, p3};
    if (MLKV_CHECK && !(in_bounds(a.err, kChkSmallRow, m.x, ra.nrows) && in_bounds(a.err, kChkSmallPos, m.y, a.n) &&
                        in_bounds(a.err, kChkSmallPos, m.z, a.n) &&
                        (m.w == NONE || in_bounds(a.err, kChkSmallPos, m.w, a.n)) &&
                        (p3 == NONE || in_bounds(a.err, kChkSmallPos, p3, a.n))))
        return;
    const VT* p = row_vec<V>(ra, m.x, j);
    const VT w = p[0], Gs = *beside(ra, p);
    VT g[kSmallRun];
#pragma unroll
    for (int i = 0; i < kSmallRun; ++i)
        if (ps[i] != NONE) g[i] = __ldcs(reinterpret_cast<const VT*>(a.grads + (size_t)ps[i] * ra.d) + j);
    VT acc = Vec<V>::zero();
#pragma unroll
    for (int i = 0; i < kSmallRun; ++i)
        if (ps[i] != NONE) Vec<V>::add(acc, g[i]);
    adagrad_store<V>(ra, m.x, j, w, Gs, acc, a.lr, a.eps);
}

// --- a kernel per run length, on three streams ---------------------------------
// Work items are run segments: v = run * nseg + segment (SEG; without it a row is
// one segment).

// The chunks of the long runs: their sums, compensated, to scratch.  (Combining
// them here too, by the last chunk of a run to arrive, cost a fence a chunk: a
// recommendation step of 1.7M lookups took 600 us instead of 556.)
template <int V, bool SEG>
__global__ void __launch_bounds__(256, MLKV_LONG_MIN_BLOCKS) k_long(RowArgs ra, RunArgs a) {
    pdl_enter();
    using VT = typename Vec<V>::T;
    const uint32_t nseg = SEG ? ra.nseg : 1u, N = min(a.cur->n_items, a.max_items) * nseg;
    const int lane = threadIdx.x & 31, G = ra.G, glane = lane & (G - 1), gid = lane >> ra.gshift;
    const unsigned gmask = group_mask(G, gid);
    const uint32_t group = (blockIdx.x * blockDim.x + threadIdx.x) >> ra.gshift;
    const uint32_t ngroups = (gridDim.x * blockDim.x) >> ra.gshift;
    for (uint32_t v = group; v < N; v += ngroups) {
        const uint32_t it = SEG ? v / nseg : v;
        const int j = glane + G * (int)(v - it * nseg);
        VT acc, cmp;
        if (chunk_sum<V>(acc, cmp, ra, a, __ldg(a.items + it), j, G, glane, gmask) && j < ra.NV)
            store_pair<V>(ra, a, it, j, acc, cmp);
    }
}

// The long runs' chunk sums combined, always in chunk order, and their rows
// updated.  A node of up to kNode chunks of a run takes a block (one segment of
// its rows): the lane groups split its chunk sums in a fixed way and group 0
// adds the groups' results up; where the run has more nodes, the pair goes to
// scratch and the block that finishes the run's last node adds the nodes' pairs
// up the same way (nodes counted by an atomic: no block waits for another).
// Every run of at most kGroupChunks chunks takes one lane group.  (With one
// block for all chunks of a run, 8 lane groups each added up to a hundred chunks
// one after another: 100,003 lookups, Zipf(1.0), dim 50, took 119 us for apply +
// export, 113 with nodes.)  kGroupChunks = 8: 4, 16 and 32 cost the 1.7M- and
// 200k-lookup steps about 1 us.
// 256 threads fit the slots that retiring blocks of the other reduce kernels
// free, where a 1024-thread block waits for a whole SM to drain.
constexpr int kCombineThreads = 256;

// acc, cmp of group 0: entries slot0, slot0 + stride, ... (cnt of them) added
// up by the block's lane groups.  sh: the groups' pairs, G vectors each.
template <int V>
__device__ __forceinline__ void block_pairs(typename Vec<V>::T& acc, typename Vec<V>::T& cmp, const RowArgs& ra,
                                            const float* partial, uint32_t slot0, uint32_t stride, uint32_t cnt,
                                            int j, int group, int ngroups, typename Vec<V>::T* sh) {
    const int G = ra.G, glane = threadIdx.x & (G - 1);
    const bool act = j < ra.NV;
    const uint32_t per = (cnt + ngroups - 1) / ngroups;
    const uint32_t k0 = min(cnt, group * per), k1 = min(cnt, k0 + per);
    sum_pairs<V>(acc, cmp, ra, partial, slot0 + k0 * stride, stride, k1 - k0, j, act);
    sh[(group * 2) * G + glane] = acc;
    sh[(group * 2 + 1) * G + glane] = cmp;
    __syncthreads();
    if (group == 0) {
        acc = Vec<V>::zero();
        cmp = Vec<V>::zero();
        for (int x = 0; x < ngroups; ++x) {
            Vec<V>::cadd(acc, cmp, sh[(x * 2) * G + glane]);
            Vec<V>::add(cmp, sh[(x * 2 + 1) * G + glane]);
        }
    }
    __syncthreads();
}

template <int V, bool NEW>
__global__ void __launch_bounds__(kCombineThreads, 3) k_combine(RowArgs ra, RunArgs a, DevState* ds) {
    pdl_enter();
    using VT = typename Vec<V>::T;
    __shared__ VT sh[2 * kCombineThreads];
    __shared__ int last_node;
    const uint32_t nseg = ra.nseg;
    const uint32_t from = NEW ? first_new(a) : NONE;
    const uint32_t NR = min(a.cur->n_group, a.max_long) * nseg, NN = min(a.cur->n_nodes, a.max_nodes) * nseg;
    if (blockIdx.x == 0 && threadIdx.x == 0)
        ds->last_unique = a.cur->n_single + a.cur->n_small + a.cur->n_short + a.cur->n_long;  // one run per row
    const int G = ra.G, glane = threadIdx.x & (G - 1), group = threadIdx.x >> ra.gshift;
    const int ngroups = kCombineThreads >> ra.gshift;
    for (uint32_t v = blockIdx.x; v < NN; v += gridDim.x) {  // block-uniform
        const uint32_t x = v / nseg, seg = v - x * nseg;
        const uint4 nd = __ldg(a.nodes + x);  // (the run's first chunk, its chunks, row, node)
        const uint32_t first = nd.w * kNode, nodes = (nd.y + kNode - 1) / kNode;
        const int j = glane + G * (int)seg;
        if (MLKV_CHECK && !(in_bounds(a.err, kChkLongItem, nd.x + nd.y, (unsigned long long)a.max_items + 1) &&
                            in_bounds(a.err, kChkLongRow, nd.z, ra.nrows)))
            continue;
        VT acc, cmp;
        bool done = nodes == 1;
        uint32_t slot0 = nd.x + first, stride = 1, cnt = min(kNode, nd.y - first);
        while (true) {  // the node's chunks, then, in the run's last block, its nodes
            block_pairs<V>(acc, cmp, ra, a.partial, slot0, stride, cnt, j, group, ngroups, sh);
            if (done) break;
            if (group == 0) {
                if (j < ra.NV) store_pair<V>(ra, a, nd.x + first, j, acc, cmp);
                __threadfence();
            }
            __syncthreads();
            if (threadIdx.x == 0) {
                uint32_t* ctr = a.node_cnt + (size_t)nd.x * nseg + seg;
                last_node = atomicAdd(ctr, 1u) == nodes - 1;
                if (last_node) *ctr = 0u;  // zero again for the next call
                __threadfence();
            }
            __syncthreads();
            if (!last_node) break;
            done = true;
            slot0 = nd.x;
            stride = kNode;
            cnt = nodes;
        }
        if (!done) continue;
        if (group == 0 && j < ra.NV) {
            if (NEW) make_new<V>(ra, a, nd.z, from, j);
            finish_long<V>(ra, a, nd.z, j, acc, cmp);
        }
    }
    // the other long runs: on the blocks that took no node (all blocks when the
    // nodes outnumber them)
    const uint32_t b0 = NN < gridDim.x ? NN : 0u;
    const uint32_t gg = (blockIdx.x - b0) * ngroups + group, ngg = (gridDim.x - b0) * ngroups;
    for (uint32_t v = blockIdx.x < b0 ? NR : gg; v < NR; v += ngg) {  // uniform within the group
        const uint32_t x = v / nseg;
        const uint4 r = __ldg(a.long_runs + x);  // (first chunk, chunks, row, -)
        const int j = glane + G * (int)(v - x * nseg);
        if (MLKV_CHECK && !(in_bounds(a.err, kChkLongItem, r.x + r.y, (unsigned long long)a.max_items + 1) &&
                            in_bounds(a.err, kChkLongRow, r.z, ra.nrows)))
            continue;
        if (j >= ra.NV) continue;
        if (NEW) make_new<V>(ra, a, r.z, from, j);
        const VT* p = row_vec<V>(ra, r.z, j);
        const VT w = p[0], Gs = *beside(ra, p);  // beside the chunk sums
        VT acc, cmp;
        sum_pairs<V>(acc, cmp, ra, a.partial, r.x, 1, r.y, j, true);
        Vec<V>::add(acc, cmp);  // the sum, rounded once
        adagrad_store<V>(ra, r.z, j, w, Gs, acc, a.lr, a.eps);
    }
    if (a.release) release_counters(a.cur, a.release);
}

// Runs of 5 .. 32 lookups, records loaded one run ahead.  Fixed shares would
// leave the kernel to the group with the most lookups: each group claims
// `grab` run segments at a time, its first ones by its index, the rest from a
// counter; one at a time when they are few, so that every run starts at once.
template <int V, bool SEG, int ROWS, bool NEW>
__global__ void __launch_bounds__(256, ROWS >= 8 ? MLKV_SHORT_MIN_BLOCKS : 3) k_short(RowArgs ra, RunArgs a) {
    pdl_enter();
    if (MLKV_CHECK && !in_bounds(a.err, kChkListEntry, a.cur->n_short, (unsigned long long)a.n + 1)) return;
    const uint32_t nseg = SEG ? ra.nseg : 1u, N = min(a.cur->n_short, a.n) * nseg;  // a list never holds more runs than lookups
    const int lane = threadIdx.x & 31, G = ra.G, glane = lane & (G - 1), gid = lane >> ra.gshift;
    const unsigned gmask = group_mask(G, gid);
    const uint32_t group = (blockIdx.x * blockDim.x + threadIdx.x) >> ra.gshift;
    const uint32_t ngroups = (gridDim.x * blockDim.x) >> ra.gshift;
    const uint32_t grab = N >= ngroups * (uint32_t)MLKV_SHORT_GRAB ? (uint32_t)MLKV_SHORT_GRAB : 1u;
    auto run_of = [&](uint32_t v) { return SEG ? v / nseg : v; };
    const uint32_t from = NEW ? first_new(a) : NONE;
    uint32_t base = group * grab;
    while (base < N) {  // uniform within the group
        const uint32_t end = min(N, base + grab);
        uint4 next = __ldg(a.runs + run_of(base));
        for (uint32_t v = base; v < end; ++v) {
            const uint4 m = next;  // (start, end, row, first lookup)
            if (v + 1 < end) next = __ldg(a.runs + run_of(v + 1));
            const int j = glane + G * (int)(v - run_of(v) * nseg);
            if (NEW) make_new<V>(ra, a, m.z, from, j);
            short_run<V, ROWS>(ra, a, m.x, m.y, m.z, m.w, j, G, glane, gmask);
        }
        uint32_t c = 0;
        if (glane == 0) c = atomicAdd(&a.cur->short_next, grab);
        base = ngroups * grab + __shfl_sync(gmask, c, 0, G);
    }
    if (a.release) release_counters(a.cur, a.release);
}

// Runs of 2 .. kSmallRun lookups, records loaded one run ahead.
template <int V, bool SEG, bool NEW>
__global__ void __launch_bounds__(256, MLKV_SMALL_MIN_BLOCKS) k_small(RowArgs ra, RunArgs a) {
    pdl_enter();
    if (MLKV_CHECK && !in_bounds(a.err, kChkListEntry, a.cur->n_small, (unsigned long long)a.n + 1)) return;
    const uint32_t nseg = SEG ? ra.nseg : 1u, N = min(a.cur->n_small, a.n) * nseg;
    const int lane = threadIdx.x & 31, G = ra.G, glane = lane & (G - 1);
    const uint32_t group = (blockIdx.x * blockDim.x + threadIdx.x) >> ra.gshift;
    const uint32_t ngroups = (gridDim.x * blockDim.x) >> ra.gshift;
    auto run_of = [&](uint32_t v) { return SEG ? v / nseg : v; };
    const uint32_t from = NEW ? first_new(a) : NONE;
    if (NEW && from != NONE)
        for (uint32_t v = group; v < N; v += ngroups)
            make_new<V>(ra, a, __ldg(a.smalls + run_of(v)).x, from, glane + G * (int)(v - run_of(v) * nseg));
    uint4 next = group < N ? __ldg(a.smalls + run_of(group)) : make_uint4(0u, 0u, 0u, 0u);
    uint32_t next3 = group < N ? __ldg(a.small_p3 + run_of(group)) : NONE;
    for (uint32_t v = group; v < N; v += ngroups) {  // uniform within the group
        const uint4 m = next;
        const uint32_t p3 = next3, x = v + ngroups;
        if (x < N) {
            next = __ldg(a.smalls + run_of(x));
            next3 = __ldg(a.small_p3 + run_of(x));
        }
        small_run<V>(ra, a, m, p3, glane + G * (int)(v - run_of(v) * nseg));
    }
    if (a.release) release_counters(a.cur, a.release);
}

// Runs of one lookup (most runs of a Zipf batch): row, state and gradient row
// loaded together, SG runs at a time, records loaded one round ahead.  With no
// loop over positions it needs few registers, so many warps (and rows) are in
// flight.
template <int V, bool SEG, int SG, bool NEW>
__global__ void __launch_bounds__(256, SG == 1 ? MLKV_SINGLE_MIN_BLOCKS : 4) k_single(RowArgs ra, RunArgs a) {
    pdl_enter();
    using VT = typename Vec<V>::T;
    if (MLKV_CHECK && !in_bounds(a.err, kChkListEntry, a.cur->n_single, (unsigned long long)a.n + 1)) return;
    const uint32_t nseg = SEG ? ra.nseg : 1u, N = min(a.cur->n_single, a.n) * nseg;
    const int lane = threadIdx.x & 31, G = ra.G, glane = lane & (G - 1);
    const uint32_t group = (blockIdx.x * blockDim.x + threadIdx.x) >> ra.gshift;
    const uint32_t ngroups = (gridDim.x * blockDim.x) >> ra.gshift;
    const uint2 none = make_uint2(0xFFFFFFFFu, 0u);
    auto run_of = [&](uint32_t v) { return SEG ? v / nseg : v; };
    const uint32_t from = NEW ? first_new(a) : NONE;
    if (NEW && from != NONE)
        for (uint32_t x = group * SG; x < N; x += ngroups * SG)
            for (uint32_t v = x; v < min(x + SG, N); ++v)
                make_new<V>(ra, a, __ldg(a.singles + run_of(v)).x, from, glane + G * (int)(v - run_of(v) * nseg));
    uint2 next[SG];
#pragma unroll
    for (int i = 0; i < SG; ++i) next[i] = group * SG + i < N ? __ldg(a.singles + run_of(group * SG + i)) : none;
    for (uint32_t v = group * SG; v < N; v += ngroups * SG) {  // uniform within the group
        uint2 m[SG];
        VT w[SG], Gs[SG], g[SG];
#pragma unroll
        for (int i = 0; i < SG; ++i) {
            m[i] = next[i];
            const uint32_t x = v + ngroups * SG + i;
            next[i] = x < N ? __ldg(a.singles + run_of(x)) : none;
        }
#pragma unroll
        for (int i = 0; i < SG; ++i) {
            const int j = glane + G * (int)(v + i - run_of(v + i) * nseg);
            if (m[i].x == none.x || j >= ra.NV) {
                m[i].x = none.x;
                continue;
            }
            if (MLKV_CHECK && !(in_bounds(a.err, kChkSingleRow, m[i].x, ra.nrows) &&
                                in_bounds(a.err, kChkSinglePos, m[i].y, a.n))) {
                m[i].x = none.x;
                continue;
            }
            const VT* p = row_vec<V>(ra, m[i].x, j);
            w[i] = p[0];
            Gs[i] = *beside(ra, p);
            g[i] = __ldcs(reinterpret_cast<const VT*>(a.grads + (size_t)m[i].y * ra.d) + j);
        }
#pragma unroll
        for (int i = 0; i < SG; ++i) {
            if (m[i].x == none.x) continue;
            VT acc = Vec<V>::zero();
            Vec<V>::add(acc, g[i]);  // 0 + g, as in a longer run
            adagrad_store<V>(ra, m[i].x, glane + G * (int)(v + i - run_of(v + i) * nseg), w[i], Gs[i], acc, a.lr,
                             a.eps);
        }
    }
    if (a.release) release_counters(a.cur, a.release);
}

// Calls of at most this many run segments reduce all their runs in k_reduce.
#ifndef MLKV_FUSED_MAX
#define MLKV_FUSED_MAX (1 << 15)
#endif
constexpr uint32_t kFusedMax = MLKV_FUSED_MAX;
static_assert(kPlanMax <= kFusedMax, "a plan's narrow rows go to k_reduce, which makes new ones (run_kernels)");

// --- calls of few lookups: one kernel ------------------------------------------

constexpr uint32_t kFanShift = 5, kFan = 1u << kFanShift;  // fan-in of the combine tree
// ... its levels, and the counters of one level above the lowest: run segments'
// chunks (of kChunkSmall lookups, one more a run) in a call of kFusedMax segments.
constexpr int tree_levels() {
    int levels = 1;
    for (uint32_t m = kFusedMax / kChunkSmall + 1; m > kFan; m = (m + kFan - 1) / kFan) ++levels;
    return levels;
}
constexpr int kMostSegs = 8;  // dim 256 in 4-byte vectors, dim 1,024 in 16-byte ones
constexpr uint32_t kTreeEntries = kFusedMax / kChunkSmall + kFusedMax / (MLKV_SEQ_SEGMENT_MAX + 1) + 2 * kMostSegs;
static_assert(MLKV_MAX_DIM <= kMostSegs * 128, "segments of the widest row");

// One segment of a chunk of a long run, by one lane group.  The chunk sums of a
// run are combined in a tree of fan-in kFan, always in chunk order: the group
// whose entry is the last of a node to arrive (an atomic count per node) adds
// the node's entries up and goes on to the next level; at the root the sum is
// rounded once and the row updated.  No group waits for another.
template <int V>
__device__ __forceinline__ void long_chunk(const RowArgs& ra, const RunArgs& a, uint32_t it, uint32_t seg, uint32_t from,
                                           int G, int glane, unsigned gmask) {
    using VT = typename Vec<V>::T;
    const uint4 rec = __ldg(a.items + it);
    const uint32_t m = rec.y >> kItemLenBits, ib = rec.w;
    const int j = glane + G * (int)seg;
    const bool act = j < ra.NV;
    VT acc, cmp;
    if (!chunk_sum<V>(acc, cmp, ra, a, rec, j, G, glane, gmask)) return;
    uint32_t idx = it - ib, count = m, stride = 1;
    for (int level = 0; count > 1; ++level) {
        if (act) store_pair<V>(ra, a, ib + idx * stride, j, acc, cmp);
        const uint32_t node = idx >> kFanShift, first = node << kFanShift;
        const uint32_t width = min(kFan, count - first);
        __threadfence();
        __syncwarp(gmask);
        uint32_t arrived = 0;
        if (glane == 0) {
            const uint32_t at = (ib + first * stride) * ra.nseg + seg;
            uint32_t* ctr = a.node_cnt + at;
            if (level) ctr += (size_t)a.max_items * ra.nseg + (size_t)(level - 1) * kTreeEntries;
            arrived = atomicAdd(ctr, 1u);
            if (arrived == width - 1) *ctr = 0u;  // zero again for the next call
        }
        arrived = __shfl_sync(gmask, arrived, 0, G);
        if (arrived != width - 1) return;
        __threadfence();
        sum_pairs<V>(acc, cmp, ra, a.partial, ib + first * stride, stride, width, j, act);
        idx = node;
        count = (count + kFan - 1) >> kFanShift;
        stride <<= kFanShift;
    }
    if (!act) return;
    make_new<V>(ra, a, rec.z, from, j);
    finish_long<V>(ra, a, rec.z, j, acc, cmp);
}

// k_reduce's units of runs: [0, us) of 5 .. 32 lookups, [us, um) of 2 ..
// kSmallRun, [um, uc) and [uc, units) of one; ls, lm, lc, lf run segments each.
struct Units {
    uint32_t NS, NM, NC, N1;  // run segments of each kind (NC: those of one lookup in coarse units)
    uint32_t ls, lm, lc, lf;
    uint32_t us, um, uc, units;
    uint32_t new_from;  // first row that holds nothing yet, or NONE
};

__device__ __forceinline__ Units make_units(const RunArgs& a, uint32_t R, uint32_t nwarps, uint32_t nseg) {
    Units q;
    q.NS = min(a.cur->n_short, a.n) * nseg;
    q.NM = min(a.cur->n_small, a.n) * nseg;
    q.N1 = min(a.cur->n_single, a.n) * nseg;
    q.NC = q.N1 - q.N1 / 4;
    // segments per lane group so that each warp gets some `rounds` units, at most 32 a unit
    auto unit = [&](uint32_t work, uint32_t rounds, uint32_t most) {
        return R * max(1u, min(min(work / (R * nwarps * rounds), most), 32u / R));
    };
    q.ls = unit(q.NS, 2, 4);
    q.lm = unit(q.NM, 2, 8);
    q.lc = unit(q.N1, 4, 24);
    q.lf = R * max(1u, q.lc / R / 4);
    q.us = (q.NS + q.ls - 1) / q.ls;
    q.um = q.us + (q.NM + q.lm - 1) / q.lm;
    q.uc = q.um + (q.NC + q.lc - 1) / q.lc;
    q.units = q.uc + (q.N1 - q.NC + q.lf - 1) / q.lf;
    return q;
}

// Every run's sum and its row's Adagrad step, in one launch, for calls of at
// most kFusedMax run segments: latency is all that counts there, and the
// kernels per run length cost five launches, three event records and four
// waits.  (Apply + Get of 4,096 lookups: 41 us with those, 36 with this; 13,312:
// 48 and 42; 32,768 segments: equal.  In large calls those are faster: this
// kernel's 128 registers leave 16 warps a SM, too few for the square roots and
// divisions between a run's loads: 1.7M lookups 556 us, 637 with this.)
//   1. The chunks of the long runs, in fixed shares (a lane group each).
//   2. Everything else as units of up to 32 runs, claimed from one counter by
//      the warps as they get free: runs of 5-32 lookups, of 2-4, of one in
//      coarse units and the last quarter of those in fine ones, so that the
//      warps end together.  A unit's run records are loaded by one coalesced
//      load and handed round with shuffles; the next unit is claimed before
//      this one is worked on.
template <int V>
__global__ void __launch_bounds__(256, 2) k_reduce(RowArgs ra, RunArgs a, DevState* ds) {
    pdl_enter();
    using VT = typename Vec<V>::T;
    const uint32_t nseg = ra.nseg;
    const uint32_t NI = min(a.cur->n_items, a.max_items), from = first_new(a);
    // a list never holds more runs than lookups
    if (MLKV_CHECK && !(in_bounds(a.err, kChkListEntry, a.cur->n_short, (unsigned long long)a.n + 1) &&
                        in_bounds(a.err, kChkListEntry, a.cur->n_small, (unsigned long long)a.n + 1) &&
                        in_bounds(a.err, kChkListEntry, a.cur->n_single, (unsigned long long)a.n + 1)))
        return;
    const int lane = threadIdx.x & 31, G = ra.G, glane = lane & (G - 1), gid = lane >> ra.gshift;
    const uint32_t R = 32u >> ra.gshift;  // lane groups per warp
    const unsigned gmask = group_mask(G, gid);
    // neighbouring warps of the order are on different SMs: a batch with little work spreads
    const uint32_t nwarps = gridDim.x * (blockDim.x >> 5);
    const uint32_t warp = (threadIdx.x >> 5) * gridDim.x + blockIdx.x;
    // the units' layout, in shared memory: read once a unit, it would only hold registers
    __shared__ Units q;
    if (threadIdx.x == 0) {
        q = make_units(a, R, nwarps, nseg);
        q.new_from = from;
        if (blockIdx.x == 0)
            ds->last_unique = a.cur->n_single + a.cur->n_small + a.cur->n_short + a.cur->n_long;  // one run per row
    }
    for (uint32_t v = warp * R + gid; v < NI * nseg; v += nwarps * R) {
        const uint32_t it = nseg == 1 ? v : v / nseg;
        long_chunk<V>(ra, a, it, v - it * nseg, from, G, glane, gmask);
    }
    __syncthreads();
    // the new rows among a unit's cnt (row, segment) pairs, one a lane; a lane writes the vectors it loads next
    auto new_rows = [&](uint32_t mrow, uint32_t mseg, uint32_t cnt) {
        if (!__any_sync(0xffffffffu, mrow >= q.new_from)) return;
        for (uint32_t k = 0; k < cnt; k += R) {
            const int src = (int)min(k + gid, cnt - 1);
            const uint32_t row = __shfl_sync(0xffffffffu, mrow, src);
            const int j = glane + G * (int)__shfl_sync(0xffffffffu, mseg, src);
            if (k + gid < cnt) make_new<V>(ra, a, row, q.new_from, j);
        }
    };
    // first units from the other end: the warps that had a chunk get one last (4
    // of the 14 us of 4,096 lookups went by with both on the same warps)
    uint32_t u = nwarps - 1 - warp;
    while (u < q.units) {  // warp-uniform
        uint32_t claim = 0;
        if (lane == 0) claim = atomicAdd(&a.cur->short_next, 1u);
        if (u < q.us) {  // runs of 5 .. 32 lookups
            const uint32_t v0 = u * q.ls, cnt = min(q.ls, q.NS - v0);
            const uint32_t mine = v0 + min((uint32_t)lane, cnt - 1);
            const uint32_t mrun = nseg == 1 ? mine : mine / nseg;
            const uint4 mrec = __ldg(a.runs + mrun);  // (start, end, row, first lookup)
            const uint32_t mseg = mine - mrun * nseg;
            new_rows(mrec.z, mseg, cnt);
            for (uint32_t k = 0; k < cnt; k += R) {
                const int src = (int)min(k + gid, cnt - 1);
                const uint32_t s = __shfl_sync(0xffffffffu, mrec.x, src), e = __shfl_sync(0xffffffffu, mrec.y, src);
                const uint32_t row = __shfl_sync(0xffffffffu, mrec.z, src), p0 = __shfl_sync(0xffffffffu, mrec.w, src);
                const int j = glane + G * (int)__shfl_sync(0xffffffffu, mseg, src);
                if (k + gid < cnt)
                    short_run<V, MLKV_SHORT_ROWS>(ra, a, s, e, row, p0, j, G, glane, gmask);
                __syncwarp();
            }
        } else if (u < q.um) {  // runs of 2 .. kSmallRun lookups, their positions in the record
            const uint32_t v0 = (u - q.us) * q.lm, cnt = min(q.lm, q.NM - v0);
            const uint32_t mine = v0 + min((uint32_t)lane, cnt - 1);
            const uint32_t mrun = nseg == 1 ? mine : mine / nseg;
            const uint4 mrec = __ldg(a.smalls + mrun);  // (row, p0, p1, p2)
            const uint32_t mp3 = __ldg(a.small_p3 + mrun), mseg = mine - mrun * nseg;
            new_rows(mrec.x, mseg, cnt);
            for (uint32_t k = 0; k < cnt; k += R) {
                const int src = (int)min(k + gid, cnt - 1);
                const uint4 m = make_uint4(__shfl_sync(0xffffffffu, mrec.x, src), __shfl_sync(0xffffffffu, mrec.y, src),
                                           __shfl_sync(0xffffffffu, mrec.z, src), __shfl_sync(0xffffffffu, mrec.w, src));
                const uint32_t p3 = __shfl_sync(0xffffffffu, mp3, src);
                const int j = glane + G * (int)__shfl_sync(0xffffffffu, mseg, src);
                if (k + gid < cnt) small_run<V>(ra, a, m, p3, j);
                __syncwarp();
            }
        } else {  // runs of one lookup
            const bool coarse = u < q.uc;
            const uint32_t v0 = coarse ? (u - q.um) * q.lc : q.NC + (u - q.uc) * q.lf;
            const uint32_t cnt = coarse ? min(q.lc, q.NC - v0) : min(q.lf, q.N1 - v0);
            const uint32_t mine = v0 + min((uint32_t)lane, cnt - 1);
            const uint32_t mrun = nseg == 1 ? mine : mine / nseg;
            const uint2 mrec = __ldg(a.singles + mrun);  // (row, lookup)
            const uint32_t mseg = mine - mrun * nseg;
            new_rows(mrec.x, mseg, cnt);
            for (uint32_t k = 0; k < cnt; k += R) {
                const int src = (int)min(k + gid, cnt - 1);
                const uint32_t row = __shfl_sync(0xffffffffu, mrec.x, src), p = __shfl_sync(0xffffffffu, mrec.y, src);
                const int j = glane + G * (int)__shfl_sync(0xffffffffu, mseg, src);
                if (k + gid < cnt && j < ra.NV && in_bounds(a.err, kChkSingleRow, row, ra.nrows) &&
                    in_bounds(a.err, kChkSinglePos, p, a.n)) {
                    const VT* src_row = row_vec<V>(ra, row, j);
                    const VT w = src_row[0], Gs = *beside(ra, src_row);
                    const VT g = __ldcs(reinterpret_cast<const VT*>(a.grads + (size_t)p * ra.d) + j);
                    VT acc = Vec<V>::zero();
                    Vec<V>::add(acc, g);  // 0 + g, as in a longer run
                    adagrad_store<V>(ra, row, j, w, Gs, acc, a.lr, a.eps);
                }
                __syncwarp();
            }
        }
        u = nwarps + __shfl_sync(0xffffffffu, claim, 0);
    }
    release_counters(a.cur, gridDim.x);  // the apply's last kernel
}

using RunKernel = void (*)(RowArgs, RunArgs);

// Narrow rows (on at most 16 lanes: dim <= 64): runs of one lookup two at a
// time per lane group on at most 3 blocks per SM, runs of 5-32 lookups with 4
// gradient rows in flight at 3 blocks per SM (more warps).
struct RunKernels {
    RunKernel longs, shorts, smalls, singles;
    void (*combine)(RowArgs, RunArgs, DevState*);
};

// new_rows (make_new): after a plan, whose narrow rows' runs (seg not set) all go
// to k_reduce.  Kernels of their own, since k_short's 8-byte vectors would pay for
// the comparison with 7 registers and a block per SM (1.3M lookups of dim 50,
// Zipf(1.1): 282 -> 292 us).
template <int V>
RunKernels run_kernels(bool seg, bool narrow, bool new_rows) {
    constexpr int R = MLKV_SHORT_ROWS;
    if (seg && new_rows)
        return {k_long<V, true>, k_short<V, true, R, true>, k_small<V, true, true>, k_single<V, true, 1, true>,
                k_combine<V, true>};
    if (seg)
        return {k_long<V, true>, k_short<V, true, R, false>, k_small<V, true, false>, k_single<V, true, 1, false>,
                k_combine<V, false>};
    if (narrow)
        return {k_long<V, false>, k_short<V, false, 4, false>, k_small<V, false, false>, k_single<V, false, 2, false>,
                k_combine<V, false>};
    return {k_long<V, false>, k_short<V, false, R, false>, k_small<V, false, false>, k_single<V, false, 1, false>,
            k_combine<V, false>};
}

template <int V>
cudaError_t run_reduce(mlkv_table* t, const float* grads, const uint32_t* spos, int64_t n, cudaStream_t st,
                       CallCounters* cur, bool new_rows) {
    const uint32_t nseg = (uint32_t)((t->geom.NV + t->geom.G - 1) / t->geom.G);
    RowArgs ra{t->slots, t->geom.stride, t->geom.dpad, t->geom.NV, t->geom.G, __builtin_ctz((unsigned)t->geom.G),
               t->geom.d, nseg,
               (uint32_t)(t->tiered ? t->cfg.hbm_cache_rows : t->cfg.capacity)};
    const RunArgs a = run_args(t, grads, nullptr, spos, n, 0u, cur);
    const int64_t segs = n * (int64_t)nseg;
    if (segs <= (int64_t)kFusedMax) {
        // one wave, or as many blocks as give every lane group a segment of a lookup
        int64_t gr = (segs * t->geom.G + 255) / 256;
        const int64_t wave = persistent_blocks(t, (const void*)k_reduce<V>, 256);
        if (gr > wave) gr = wave;
        MLKV_LAUNCH_PERSISTENT(t, MLKV_K_REDUCE, (k_reduce<V>), (unsigned)gr, 256, 0, st, ra, a, t->dstate);
        return cudaGetLastError();
    }
    // The runs of one lookup, of 2 .. kSmallRun and of up to
    // MLKV_SEQ_SEGMENT_MAX lookups, and the long runs touch disjoint rows and
    // scratch: they run on three streams at once, each filling the others'
    // tails, and join at the end of the call; the last kernel of each stream
    // releases the counters they read.  While a kernel class is being timed
    // (mlkv_time_kernel) they run one after another: on three streams a
    // kernel's events would also span the time it waits for the SMs the others
    // hold.
    cudaStream_t s1 = st, s2 = st;
    const bool branches = t->timer.kernel_id == 0;
    if (branches) {
        cudaError_t e;
        if ((e = cudaEventRecord(t->ev_fork, st)) != cudaSuccess ||
            (e = cudaStreamWaitEvent(t->branch[0], t->ev_fork, 0)) != cudaSuccess ||
            (e = cudaStreamWaitEvent(t->branch[1], t->ev_fork, 0)) != cudaSuccess)
            return e;
        s1 = t->branch[0];
        s2 = t->branch[1];
    }
    const bool narrow = t->geom.G <= 16;
    const RunKernels k = run_kernels<V>(nseg > 1, narrow, new_rows);
    const int gl = persistent_blocks(t, (const void*)k.longs, 256);
    const int g2 = persistent_blocks(t, (const void*)k.smalls, 256);
    const int gs = persistent_blocks(t, (const void*)k.shorts, 256);
    int g1 = persistent_blocks(t, (const void*)k.singles, 256);
    if (narrow && g1 > 3 * t->num_sms) g1 = 3 * t->num_sms;
    // In a call of fewer than kSmallBatch lookups the runs of 5-32 (the longest
    // per run of the three) go before those of 2-4: they would otherwise be last
    // to start, after the runs of one had filled the SMs.
    const bool short_first = n < (int64_t)kSmallBatch;
    RunArgs last = a;
    const int gc = t->num_sms * 4;  // 1024 threads per SM
    last.release = branches ? (uint32_t)(gc + g1 + (short_first ? g2 : gs)) : (uint32_t)g1;
    const RunArgs& tail = branches ? last : a;
    MLKV_LAUNCH_PERSISTENT(t, MLKV_K_REDUCE_LONG, k.longs, gl, 256, 0, s2, ra, a);
    MLKV_LAUNCH_PERSISTENT(t, MLKV_K_LONG_COMBINE, k.combine, gc, kCombineThreads, 0, s2, ra, tail, t->dstate);
    if (short_first) {
        MLKV_LAUNCH_PERSISTENT(t, MLKV_K_REDUCE_SHORT, k.shorts, gs, 256, 0, s1, ra, a);
        MLKV_LAUNCH_PERSISTENT(t, MLKV_K_REDUCE_SMALL, k.smalls, g2, 256, 0, s1, ra, tail);
    } else {
        MLKV_LAUNCH_PERSISTENT(t, MLKV_K_REDUCE_SMALL, k.smalls, g2, 256, 0, s1, ra, a);
        MLKV_LAUNCH_PERSISTENT(t, MLKV_K_REDUCE_SHORT, k.shorts, gs, 256, 0, s1, ra, tail);
    }
    MLKV_LAUNCH_PERSISTENT(t, MLKV_K_REDUCE_SINGLE, k.singles, g1, 256, 0, st, ra, last);
    if (branches) {
        cudaError_t e;
        if ((e = cudaEventRecord(t->ev_join[0], s1)) != cudaSuccess ||
            (e = cudaEventRecord(t->ev_join[1], s2)) != cudaSuccess ||
            (e = cudaStreamWaitEvent(st, t->ev_join[0], 0)) != cudaSuccess ||
            (e = cudaStreamWaitEvent(st, t->ev_join[1], 0)) != cudaSuccess)
            return e;
    }
    return cudaGetLastError();
}

}  // namespace

void long_bounds(int64_t max_batch, int64_t& runs, int64_t& nodes, int64_t& items) {
    // chunks of kChunkLarge lookups in calls of at least kSmallBatch lookups, of
    // kChunkSmall (or kChunkLarge) below, and one partial chunk per long run
    const int64_t small = std::min<int64_t>(max_batch, (int64_t)kSmallBatch - 1) / kChunkSmall;
    runs = max_batch / (MLKV_SEQ_SEGMENT_MAX + 1) + 1;
    items = std::max<int64_t>(max_batch / kChunkLarge, small) + runs + 1;
    // a run cut into nodes has more than kGroupChunks chunks, one partial node
    nodes = items / kNode + items / (kGroupChunks + 1) + 2;
}

int64_t node_counters(int64_t max_items, int dim) {
    // segments per row of the widest split: the scalar kernels' (dim <= 256) or the float4 kernels'
    const int64_t nseg = std::max<int64_t>((std::min(dim, 256) + 31) / 32, (dim + 127) / 128);
    return max_items * nseg + (tree_levels() - 1) * (int64_t)kTreeEntries;
}

cudaError_t launch_heads(mlkv_table* t, const uint32_t* srow, const uint32_t* spos, int64_t n, uint32_t sent,
                         cudaStream_t st, CallCounters* cur, const SortTail& tail) {
    const RunArgs a = run_args(t, nullptr, srow, spos, n, sent, cur);
    // a warp per 32 positions, the windows dealt out grid-stride over at most
    // one wave of blocks
    const int64_t cap = persistent_blocks(t, (const void*)k_heads, 256);
    int64_t gh = (n + 255) / 256;
    if (gh > cap) gh = cap;
    if (gh < 1) gh = 1;
    MLKV_LAUNCH(t, MLKV_K_SEGMENTS, k_heads, (unsigned)gh, 256, 0, st, a, tail);
    return cudaGetLastError();
}

cudaError_t launch_reduce_apply(mlkv_table* t, const float* grads, const uint32_t* spos, int64_t n,
                                cudaStream_t st, CallCounters* cur, bool new_rows) {
    if (t->geom.V == 4) return run_reduce<4>(t, grads, spos, n, st, cur, new_rows);
    if (t->geom.V == 2) return run_reduce<2>(t, grads, spos, n, st, cur, new_rows);
    return run_reduce<1>(t, grads, spos, n, st, cur, new_rows);
}

}  // namespace mlkv
