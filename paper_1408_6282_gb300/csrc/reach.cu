// reach.cu -- level-by-level forward searches, one thread block per instance.
//
// The residual search of a new seed (Algorithm 1) is, in every instance, a
// walk of tens of levels with at most a few thousand pairs per level, so it is
// bound by the latency of a level and not by throughput.  Instances never
// meet (a covered pair belongs to one instance), so each gets a block of its
// own that keeps its frontier in shared memory: a level is one round of row
// reads, one round of covering ORs (the new pair's row bounds and index length
// are requested together with the OR), and a block barrier.  No item passes
// through a queue in global memory, no cursor is shared between blocks, and
// nothing polls.  A frontier wider than the shared buffer continues in the
// instance's part of a global scratch array; what does not fit there is parked
// in pend_trav and resumed by the global-queue search (k_traverse).
//
// Bound: two dependent random reads a level (the row, then the OR with the row
// bounds), about 2.2 us with the barrier.  Measured against the global queue
// with block rings (searches of 50 seeds, l = 64): R-MAT 18 wc 7.6 -> 3.9 ms,
// R-MAT 20 p = 0.01 3.4 -> 1.2 ms; 30 seeds of R-MAT 20 wc 9.8 -> 5.3 ms.  An
// index segment erased by one warp (a rank that hit a giant component lists
// 160 K nodes) cost R-MAT 20 p = 0.05 2.5 ms a search: the block erases such a
// segment together.  One barrier per level instead of five: 5.6 -> 5.3 ms.  A level
// waits for the warp with the longest row, so rows of 128 entries and more are swept
// by the block (50 seeds of R-MAT 18 wc: from 512 entries 4.24 ms, 256 4.0, 128 3.94, 64
// 3.86, but R-MAT 20 p = 0.01 1.27, 1.26, 1.28, 1.33).  Two to four entries of a lane in
// flight: 4.7 to 5.2 ms (registers; most rounds have one).
#include "internal.cuh"

namespace skim {

namespace {

constexpr int kReachThreads = 1024;
constexpr uint32_t kReachWarps = kReachThreads / 32;
constexpr uint32_t kFrontCap = 1024;  // frontier rows kept in shared memory, per level parity
constexpr uint32_t kEraseCap = 1024;  // index segments kept for erasing
constexpr uint32_t kLongCap = 64;     // rows swept by the whole block, per level
constexpr uint32_t kLongRow = 128;    // entries from which a row is swept by the block
// A walk from the pivots of more levels than this, of fewer rows each on average, is
// given up and counts as reaching nothing: a component of that shape is not
// worth a level-by-level walk (a cycle of 20000 nodes, p = 1: sketches 97 ms with
// the walk, 71 without; a chain of 60000: 292 and 223 ms; wide ones have tens of levels,
// a 400 x 400 grid at p = 0.5 about a thousand of a hundred rows).
constexpr uint32_t kNarrowLevels = 512, kNarrowRows = 32;
constexpr uint32_t kSeen = 4096;      // nodes remembered as reached (direct-mapped)

struct ReachShared {
    uint2 front[2][kFrontCap];        // {first row entry, entries}
    uint2 erase[kEraseCap];           // {pair, index entries}
    uint2 longs[kLongCap];
    uint32_t seen[kSeen];
    uint32_t n_rows[3], n_erase, n_long, parked;
    unsigned long long visits, edges;
};

template <bool RES>
struct Reach {
    const ReachArgs &A;
    ReachShared &sh;
    const uint32_t *off, *rows;
    uint64_t *mask, *pend;
    uint32_t inst;
    uint64_t bit;
    uint32_t par;                     // parity the new rows are written to
    uint32_t *n_next;                 // and their number
    uint64_t visits = 0, edges = 0;   // per lane

    SKIM_DEV uint2 *spill_list(uint32_t p) const {
        return A.list + (static_cast<uint64_t>(blockIdx.x) * 2 + p) * A.cap;
    }

    // Warp-collective: lanes with `has` reach node x.
    SKIM_DEV void visit(bool has, uint32_t x) {
        uint32_t b = 0, len = 0, sl = 0;
        bool fresh = false;
        const uint64_t r = static_cast<uint64_t>(x) * A.l + inst;
        if (has) {
            // a hub is an entry of thousands of rows: the node last seen at
            // its place needs no second OR on a word that every instance uses
            uint32_t *s = &sh.seen[(x * 0x9E3779B1u) / (0xFFFFFFFFu / kSeen + 1)];
            if (*s == x) has = false;
            else *s = x;
        }
        if (has) {
            // independent requests, in flight together; an index is erased
            // only by the lane whose OR newly covers its pair, so reading its
            // length first is safe
            const uint64_t old = atomicOr(reinterpret_cast<unsigned long long *>(&mask[x]), bit);
            b = off[r];
            len = off[r + 1] - b;
            if (RES) sl = A.seg_len[r];
            fresh = !(old & bit);
        }
        visits += fresh ? 1 : 0;
        const bool row = fresh && len != 0;
        const unsigned rb = __ballot_sync(kFull, row);
        if (rb) {
            uint32_t base = 0;
            if ((threadIdx.x & 31) == 0) base = atomicAdd(n_next, __popc(rb));
            base = __shfl_sync(kFull, base, 0);
            if (row) {
                const uint32_t at = base + __popc(rb & lanemask_lt());
                if (at < kFrontCap) {
                    sh.front[par][at] = make_uint2(b, len);
                } else if (at - kFrontCap < A.cap) {
                    spill_list(par)[at - kFrontCap] = make_uint2(b, len);
                } else if (!RES) {  // parked: taken up when the frontier runs dry
                    atomicOr(reinterpret_cast<unsigned long long *>(&pend[x]), bit);
                    sh.parked = 1;
                } else {  // parked: re-queued by the host
                    atomicOr(reinterpret_cast<unsigned long long *>(&A.pend_trav[x]), bit);
                    A.ctl->spill = 1;
                }
            }
        }
        if (RES && fresh && sl == kLeafSegment) {  // only x has this rank
            atomicSub(&A.size[x], 1u);
            A.seg_len[r] = 0;
        } else if (RES && fresh && sl) {
            const uint32_t at = atomicAdd(&sh.n_erase, 1u);
            if (at < kEraseCap)
                sh.erase[at] = make_uint2(static_cast<uint32_t>(r), sl);
            else
                erase_segment(r, sl, 0, 1);
        }
    }

    // Entries t, t + step, .. of the index segment of pair r: each listed
    // node's partial sketch loses the pair's rank.
    SKIM_DEV void erase_segment(uint64_t r, uint32_t len, uint32_t t, uint32_t step) {
        const uint64_t st = A.seg_start[r];
#pragma unroll 4
        for (uint32_t e = t; e < len; e += step) atomicSub(&A.size[A.idx_nodes[st + e]], 1u);
        if (t == 0) A.seg_len[r] = 0;
    }

    // Warp-collective: the rows held by the lanes (len 0: none).  A row of 32
    // or more entries is swept by the warp, the entries of the others are
    // spread over the lanes, 32 per round.
    SKIM_DEV void expand(uint32_t begin, uint32_t len) {
        const uint32_t lane = threadIdx.x & 31;
        edges += len;
        unsigned big = __ballot_sync(kFull, len >= 32);
        while (big) {
            const int src = __ffs(big) - 1;
            big &= big - 1;
            const uint32_t bb = __shfl_sync(kFull, begin, src), bc = __shfl_sync(kFull, len, src);
            uint32_t q = 0;
            if (bc >= kLongRow) {
                if (lane == 0) {
                    q = atomicAdd(&sh.n_long, 1u);
                    if (q < kLongCap) sh.longs[q] = make_uint2(bb, bc);
                }
                q = __shfl_sync(kFull, q, 0);
                if (q < kLongCap) continue;
            }
            sweep(bb, bc, lane, 32);
        }
        const uint32_t c = len < 32 ? len : 0;
        uint32_t incl = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(kFull, incl, o);
            if (lane >= static_cast<uint32_t>(o)) incl += y;
        }
        const uint32_t total = __shfl_sync(kFull, incl, 31);
        const uint32_t first = begin - (incl - c);  // entry g of the warp is begin + (g - its row's first)
        for (uint32_t g = 0; g < total; g += 32) {
            const uint32_t o = g + lane;
            uint32_t sl = 0;  // owner: the first lane whose inclusive count exceeds o
#pragma unroll
            for (uint32_t step = 16; step > 0; step >>= 1) {
                const uint32_t v = __shfl_sync(kFull, incl, sl + step - 1);
                if (v <= o) sl += step;
            }
            const uint32_t sb = __shfl_sync(kFull, first, sl);
            const bool has = o < total;
            visit(has, has ? rows[sb + o] : 0);
        }
    }

    // Warp-collective: entries t, t + step, .. of a row (t of lane 0 the same
    // for the whole warp up to the lane).
    SKIM_DEV void sweep(uint32_t b, uint32_t len, uint32_t t, uint32_t step) {
        uint32_t x = t < len ? rows[b + t] : 0;
        for (uint32_t k0 = t - (threadIdx.x & 31); k0 < len; k0 += step) {
            const uint32_t k = k0 + (threadIdx.x & 31);
            const uint32_t xn = k + step < len ? rows[b + k + step] : 0;
            visit(k < len, x);
            x = xn;
        }
    }

    // Block-collective: rows parked for want of room become the frontier of
    // level t, as many as it holds; returns how many.
    SKIM_DEV uint32_t unpark(uint32_t t) {
        __syncthreads();
        if (threadIdx.x == 0) sh.parked = 0;
        par = t & 1;
        n_next = &sh.n_rows[t % 3];
        __syncthreads();
        for (uint32_t v0 = 0; v0 < A.n; v0 += kReachThreads) {
            const uint32_t v = v0 + threadIdx.x;
            const bool mine = v < A.n && (*reinterpret_cast<volatile uint64_t *>(&pend[v]) & bit);
            if (!mine) continue;
            const uint32_t at = atomicAdd(n_next, 1u);
            if (at >= kFrontCap + A.cap) {
                sh.parked = 1;
                continue;
            }
            atomicAnd(reinterpret_cast<unsigned long long *>(&pend[v]), ~bit);
            const uint64_t r = static_cast<uint64_t>(v) * A.l + inst;
            const uint2 it = make_uint2(off[r], off[r + 1] - off[r]);
            if (at < kFrontCap) sh.front[par][at] = it;
            else spill_list(par)[at - kFrontCap] = it;
        }
        __syncthreads();
        return min(sh.n_rows[t % 3], kFrontCap + A.cap);
    }

    // Block-collective: erase the kept index segments, a warp per segment (a
    // rank that hit a giant component has a segment of its whole upstream:
    // the block takes such a one together).
    SKIM_DEV void erase_all() {
        const uint32_t n = min(sh.n_erase, kEraseCap);
        for (uint32_t q = threadIdx.x >> 5; q < n; q += kReachWarps)
            if (sh.erase[q].y < kLongRow) erase_segment(sh.erase[q].x, sh.erase[q].y, threadIdx.x & 31, 32);
        for (uint32_t q = 0; q < n; q++)
            if (sh.erase[q].y >= kLongRow) erase_segment(sh.erase[q].x, sh.erase[q].y, threadIdx.x, kReachThreads);
        __syncthreads();
        if (threadIdx.x == 0) sh.n_erase = 0;
        __syncthreads();
    }
};

// Block i searches instance i, from node x (RES: the residual search of seed
// x, or of the seed the step before it found, if any) or from the pivots of instance i
// (blocks from l on: against the edges).  A level that makes no progress ends the search
// with the error flag: each of its rows may take the wait limit (phase_limit; what the
// block sweeps and erases together always ends).
template <bool RES>
__global__ void __launch_bounds__(kReachThreads, 1) k_reach(ReachArgs A, uint32_t x, const uint32_t *pivot,
                                                            uint32_t starts, uint32_t *count) {
    extern __shared__ char s_raw[];
    ReachShared &sh = *reinterpret_cast<ReachShared *>(s_raw);
    if (RES && x == kSeedOfStep) {
        if (A.ctl->step.best == ~0ull) return;
        x = static_cast<uint32_t>(A.ctl->step.best);
    }
    const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const bool back = !RES && blockIdx.x >= A.l;
    const uint32_t inst = back ? blockIdx.x - A.l : blockIdx.x;
    Reach<RES> R{A, sh, back ? A.back_off : A.off, back ? A.back_rows : A.rows, back ? A.back_mask : A.mask,
                 back ? A.back_pend : A.pend_trav, inst, 1ull << inst, 0, &sh.n_rows[0]};
    for (uint32_t q = threadIdx.x; q < kSeen; q += kReachThreads) sh.seen[q] = 0xFFFFFFFFu;
    if (threadIdx.x == 0) {
        sh.n_rows[0] = sh.n_rows[1] = sh.n_rows[2] = sh.n_erase = sh.n_long = sh.parked = 0;
        sh.visits = sh.edges = 0;
        if (RES && blockIdx.x == 0) A.chosen[x] = 1;
    }
    __syncthreads();
    if (RES) {
        if (warp == 0) R.visit(lane == 0, x);
    } else {
        for (uint32_t q0 = warp * 32; q0 < starts; q0 += kReachThreads) {
            const bool in = q0 + lane < starts;
            R.visit(in, in ? pivot[(q0 + lane) * 64 + inst] : 0);
        }
    }
    __syncthreads();
    // Level t reads its rows from parity t & 1 and their number from
    // n_rows[t % 3], adds the next level's to n_rows[(t + 1) % 3] and empties
    // n_rows[(t + 2) % 3], last read a barrier ago: one barrier per level.
    // What the barrier's vote finds (rows for the block, a fuller erase list,
    // the wait limit) is handled behind it.
    uint64_t t_level = globaltimer(), walked = 0;
    bool narrow = false;
    for (uint32_t t = 0;; t++) {
        uint32_t m = min(sh.n_rows[t % 3], kFrontCap + A.cap);
        if (!RES && m == 0 && sh.parked) {
            m = R.unpark(t);
            t_level = globaltimer();
        }
        if (m == 0) break;
        if (!RES) {
            walked += m;
            narrow = t >= kNarrowLevels && walked < kNarrowRows * t;
            if (narrow) break;
        }
        R.par = (t + 1) & 1;
        R.n_next = &sh.n_rows[(t + 1) % 3];
        if (threadIdx.x == 0) sh.n_rows[(t + 2) % 3] = 0;
        // row q goes to warp q % kReachWarps, so that a narrow level uses every warp
        for (uint32_t q0 = 0; q0 + warp < m; q0 += kReachThreads) {
            const uint32_t q = q0 + lane * kReachWarps + warp;
            uint2 it = make_uint2(0, 0);
            if (q < m) it = q < kFrontCap ? sh.front[t & 1][q] : R.spill_list(t & 1)[q - kFrontCap];
            R.expand(it.x, it.y);
        }
        int late = 0;
        if (threadIdx.x == 0) {
            const uint64_t now = globaltimer();
            late = now - t_level > phase_limit(A.timeout_ns, m);
            if (late) atomicOr(&A.ctl->err, kErrTimeout);
            t_level = now;
        }
        if (__syncthreads_or(late | (sh.n_long != 0) | (sh.n_erase > kEraseCap / 2))) {
            if (__syncthreads_or(late)) break;
            const uint32_t nl = min(sh.n_long, kLongCap);
            for (uint32_t q = 0; q < nl; q++) R.sweep(sh.longs[q].x, sh.longs[q].y, threadIdx.x, kReachThreads);
            __syncthreads();
            if (threadIdx.x == 0) sh.n_long = 0;
            R.erase_all();
            if (threadIdx.x == 0) t_level = globaltimer();
        }
    }
    __syncthreads();
    R.erase_all();
    // counters
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        R.visits += __shfl_down_sync(kFull, R.visits, o);
        R.edges += __shfl_down_sync(kFull, R.edges, o);
    }
    if (lane == 0) {
        if (R.visits) atomicAdd(&sh.visits, R.visits);
        if (R.edges) atomicAdd(&sh.edges, R.edges);
    }
    __syncthreads();
    if (!RES) {
        if (threadIdx.x == 0) count[(back ? 64 : 0) + inst] = narrow ? 0 : static_cast<uint32_t>(sh.visits);
        return;
    }
    if (threadIdx.x == 0) {
        if (sh.visits) {
            atomicAdd(&A.ctl->stats[kStFwdVisits], sh.visits);
            atomicAdd(&A.ctl->ix_cov, sh.visits);
        }
        if (sh.edges) atomicAdd(&A.ctl->stats[kStFwdEdges], sh.edges);
    }
}

}  // namespace

cudaError_t launch_reach(const ReachArgs &a, uint32_t x, cudaStream_t s) {
    cudaError_t e = cudaFuncSetAttribute(k_reach<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         static_cast<int>(sizeof(ReachShared)));
    if (e != cudaSuccess) return e;
    note_launch();
    k_reach<true><<<a.l, kReachThreads, sizeof(ReachShared), s>>>(a, x, nullptr, 1, nullptr);
    return cudaGetLastError();
}

cudaError_t launch_reach_from(const ReachArgs &a, const uint32_t *pivot, uint32_t starts, uint32_t *count,
                              cudaStream_t s) {
    cudaError_t e = cudaFuncSetAttribute(k_reach<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         static_cast<int>(sizeof(ReachShared)));
    if (e != cudaSuccess) return e;
    note_launch();
    k_reach<false><<<2 * a.l, kReachThreads, sizeof(ReachShared), s>>>(a, 0, pivot, starts, count);
    return cudaGetLastError();
}

}  // namespace skim
