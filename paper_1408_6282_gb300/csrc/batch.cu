// batch.cu -- per-batch steps after a reverse search has marked, for every
// visited (node, lane word), the lanes that reached the node.  Visit records
// (node << tbits | word, table slot) arrive sorted by key, so each node's
// words form one run in increasing rank order.
//
// Algorithm 2 acceptance (Section 5.2): for node v and instance i the first
// k - lcnt[v][i] lanes of instance i (in rank order) join v's local sketch;
// the ranks that join also enter the global sketch X_v while it holds fewer
// than k ranks.  Batches advance in increasing rank order, so X_v is filled
// in increasing order and needs no merge: appending is the bottom-k merge of
// Algorithm 2.  Pruning in the search used the counts at the start of the
// batch, so every lane whose rank belongs in a local sketch did reach it.
//
// SKIM (Algorithm 1): size[v] counts the processed, uncovered ranks that reach
// v.  The batch's stop lane is the earliest lane at which some node's size
// reaches k (smallest node id on ties); lanes up to it are committed (sizes
// and the inverted index), the rest stay valid for the next step because a
// search from an uncovered pair never meets a covered node.
#include "internal.cuh"

namespace skim {

namespace {

inline unsigned grid_for(size_t n, int threads, unsigned cap = 152 * 32) {
    size_t g = (n + threads - 1) / threads;
    if (g > cap) g = cap;
    return static_cast<unsigned>(g ? g : 1);
}

// Instance and coin-stream offset of every lane: instance i = pair % l, or in
// the IC model (lane_rank given) a fresh instance numbered by the position.
__global__ void k_lane_inst(const uint32_t *lane_pair, const uint64_t *lane_rank, uint32_t B, uint32_t l,
                            uint8_t *lane_inst, uint64_t *lane_g) {
    for (uint32_t j = blockIdx.x * blockDim.x + threadIdx.x; j < B; j += gridDim.x * blockDim.x) {
        if (lane_rank) {
            lane_inst[j] = 0;
            lane_g[j] = kGolden * (lane_rank[j] + 1);
            continue;
        }
        const uint32_t i = lane_pair[j] % l;
        lane_inst[j] = static_cast<uint8_t>(i);
        lane_g[j] = kGolden * static_cast<uint64_t>(i + 1);
    }
}

SKIM_DEV bool run_start(const uint64_t *rec_key, uint64_t r, uint32_t tbits) {
    return r == 0 || (rec_key[r] >> tbits) != (rec_key[r - 1] >> tbits);
}

// Algorithm 2's acceptance for the records of one batch, sorted by key so that
// a node's records are adjacent and in word (= rank) order.  Per (node v,
// instance i) the first k - lcnt[v,i] offers are accepted (the instance-local
// sketch), and accepted ranks are appended to X_v while it holds fewer than k.
//
// Records are split into windows of 32; a warp owns the nodes whose runs start
// in its window and walks their records 32 at a time, past the window's end
// for the last one.  The offers (record, lane bit) are taken 32 per step in
// rank order.  An offer of (v, i) with rank rho among the step's offers of
// (v, i) is accepted iff lcnt[v,i] + rho < k, which is the sequential rule;
// its place in X_v is xlen[v] plus the accepted offers of v before it in the
// step.  Counts, lengths and full bits are written back after every step, so
// the next step reads them current.

// One step: offer `has` of node v at batch lane ln (one per warp lane).
SKIM_DEV void accept_step(bool has, uint32_t v, uint64_t ln, const uint8_t *__restrict__ lane_inst,
                          const uint64_t *__restrict__ lane_rank, uint32_t l, uint32_t k, uint8_t *lcnt,
                          uint64_t *full, uint64_t *X, uint32_t *xlen, unsigned long long &ins) {
    const uint32_t lane = threadIdx.x & 31;
    uint32_t i = 0, lc0 = 0, len0 = 0;
    if (has) {
        i = lane_inst[ln];
        lc0 = lcnt[static_cast<uint64_t>(v) * l + i];
        len0 = xlen[v];
    }
    // peers in (v, i) and in v; idle lanes get keys no offer has
    const unsigned pvi = __match_any_sync(kFull, has ? (static_cast<uint64_t>(v) << 6 | i) : ~0ull - lane);
    const unsigned pv = __match_any_sync(kFull, has ? static_cast<uint64_t>(v) : (1ull << 32 | lane));
    const uint32_t rho = __popc(pvi & lanemask_lt());
    const bool acc = has && lc0 + rho < k;
    const unsigned ab = __ballot_sync(kFull, acc);
    if (acc) {
        const uint32_t pos = len0 + __popc(ab & pv & lanemask_lt());
        if (pos < k) X[static_cast<uint64_t>(v) * k + pos] = lane_rank[ln];
        ins++;
    }
    __syncwarp();
    if (has && rho == 0 && lc0 < k) {  // one lane per (v, i)
        const uint32_t c = min(k, lc0 + __popc(pvi));
        lcnt[static_cast<uint64_t>(v) * l + i] = static_cast<uint8_t>(c);
        if (c == k) atomicOr(reinterpret_cast<unsigned long long *>(&full[v]), 1ull << i);
    }
    if (has && (pv & lanemask_lt()) == 0) {  // one lane per v
        const uint32_t len = min(k, len0 + __popc(ab & pv));
        if (len != len0) xlen[v] = len;
    }
    __syncwarp();
}

// Record r's lane bits are those of its table slot, hvals[2 * rec_val[r]].
__global__ void __launch_bounds__(256)
    k_accept(const uint64_t *__restrict__ rec_key, const uint32_t *__restrict__ rec_val,
             const uint64_t *__restrict__ hvals, uint64_t R, uint32_t tbits,
             const uint8_t *__restrict__ lane_inst, const uint64_t *__restrict__ lane_rank, uint32_t l, uint32_t k,
             uint8_t *lcnt, uint64_t *full, uint64_t *X, uint32_t *xlen, DevCtl *ctl) {
    const uint32_t lane = threadIdx.x & 31;
    const uint64_t tmask = (1ull << tbits) - 1;
    unsigned long long ins = 0;
    const uint64_t warps = (static_cast<uint64_t>(gridDim.x) * blockDim.x) >> 5;
    const uint64_t nwin = (R + 31) / 32;
    for (uint64_t w = (blockIdx.x * static_cast<uint64_t>(blockDim.x) + threadIdx.x) >> 5; w < nwin; w += warps) {
        const uint64_t W0 = w * 32, W1 = min(R, W0 + 32);
        bool st = false;
        if (W0 + lane < W1) st = run_start(rec_key, W0 + lane, tbits);
        const unsigned sb = __ballot_sync(kFull, st);
        if (!sb) continue;  // the window lies inside a run owned by an earlier warp
        const uint64_t s0 = W0 + __ffs(sb) - 1;
        const uint64_t last = rec_key[W1 - 1] >> tbits;
        for (uint64_t c0 = s0;; c0 += 32) {
            // the warp's records form one stretch [s0, end of last's run)
            const uint64_t rr = c0 + lane;
            uint64_t key = 0, m = 0;
            bool act = false;
            if (rr < R) {
                key = rec_key[rr];
                act = rr < W1 || (key >> tbits) == last;
            }
            const unsigned actb = __ballot_sync(kFull, act);
            if (!actb) break;
            if (act) m = hvals[2ull * rec_val[rr]];
            const uint32_t vr = static_cast<uint32_t>(key >> tbits);
            const uint64_t tr = key & tmask;
            if (!__any_sync(kFull, __popcll(m) > 1)) {
                // one offer per record (the common case)
                const bool has = m != 0;
                accept_step(has, vr, tr * 64 + (has ? __ffsll(m) - 1 : 0), lane_inst, lane_rank, l, k, lcnt, full,
                            X, xlen, ins);
            } else {
                // offer o is bit (o - pre_s) of record s with pre_s <= o < pre_s + cnt_s
                const uint32_t cnt = __popcll(m);
                uint32_t incl = cnt;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t y = __shfl_up_sync(kFull, incl, o);
                    if (lane >= static_cast<unsigned>(o)) incl += y;
                }
                const uint32_t pre = incl - cnt, total = __shfl_sync(kFull, incl, 31);
                for (uint32_t g = 0; g < total; g += 32) {
                    const uint32_t o = g + lane;
                    const bool has = o < total;
                    uint32_t src = 0;
#pragma unroll
                    for (int step = 16; step > 0; step >>= 1) {
                        const uint32_t cand = src + step;
                        const uint32_t pc = __shfl_sync(kFull, pre, cand);
                        if (has && pc <= o) src = cand;
                    }
                    const uint64_t ms = __shfl_sync(kFull, m, src), ts = __shfl_sync(kFull, tr, src);
                    const uint32_t ps = __shfl_sync(kFull, pre, src), vs = __shfl_sync(kFull, vr, src);
                    uint64_t ln = 0;
                    if (has) {
                        uint64_t x = ms;
                        for (uint32_t skip = o - ps; skip; skip--) x &= x - 1;
                        ln = ts * 64 + (__ffsll(x) - 1);
                    }
                    accept_step(has, vs, ln, lane_inst, lane_rank, l, k, lcnt, full, X, xlen, ins);
                }
            }
            if (actb != kFull) break;
        }
    }
    warp_add(&ctl->stats[kStInsert], ins);
}

// lanes of word t inside [lo, hi] (inclusive), lo <= hi
SKIM_DEV uint64_t range_mask(uint64_t t, uint32_t lo, uint32_t hi) {
    const uint64_t w0 = t * 64, w1 = w0 + 63;
    if (w1 < lo || w0 > hi) return 0;
    uint64_t m = ~0ull;
    if (lo > w0) m &= ~0ull << (lo - w0);
    if (hi < w1) m &= ~0ull >> (w1 - hi);
    return m;
}

// SKIM batches read a record's lane bits in every candidate scan and in both
// commit passes: they are gathered once from the visited table, next to the
// records, after the records are put in order.
__global__ void k_gather_bits(const uint32_t *__restrict__ rec_val, const uint64_t *__restrict__ hvals, uint64_t R,
                              uint64_t *__restrict__ rbits) {
    for (uint64_t r = blockIdx.x * static_cast<uint64_t>(blockDim.x) + threadIdx.x; r < R;
         r += static_cast<uint64_t>(gridDim.x) * blockDim.x)
        rbits[r] = hvals[2ull * rec_val[r]];
}

// ---- a SKIM step ------------------------------------------------------------------
//
// Everything between two residual searches: lanes whose source the last search
// covered leave the batch, the scan for the next stop, the commit of the lanes up
// to it.  One launch with four grid barriers (one block of 1024 threads per SM: a
// barrier costs 2-3 us) instead of ten kernels and clears; with few records the
// launches were the cost.  The residual search takes the seed from ctl->step, so it
// is queued behind the step at once and the host's wait runs beside it.  50 seeds,
// l = 64: R-MAT 18 wc 11.0 -> 9.6 ms (steps 2.0 -> 1.4 ms), R-MAT 20 p = 0.01, whose
// batches have up to 2 M records, 30 -> 27 ms (12 -> 10 ms).  Two blocks of 512 or
// 1024 threads per SM and other back-offs are within 1 %, one of 512 is 20 % slower
// there.
constexpr int kStepThreads = 1024;

// Grid barrier number i of the launch: false once the wait limit has passed.  Its
// counter is zero again when the next barrier has been passed.
SKIM_DEV bool step_barrier(DevCtl *ctl, int i, uint64_t timeout_ns) {
    __shared__ int s_ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(&ctl->step.bar[i], 1u);
        const uint64_t t0 = globaltimer();
        int ok = 1;
        while (*reinterpret_cast<volatile unsigned *>(&ctl->step.bar[i]) < gridDim.x) {
            if (globaltimer() - t0 > timeout_ns) {
                atomicOr(&ctl->err, kErrTimeout);
                ok = 0;
                break;
            }
            __nanosleep(40);
        }
        __threadfence();
        if (blockIdx.x == 0) ctl->step.bar[(i + 3) & 3] = 0;
        s_ok = ok;
    }
    __syncthreads();
    return s_ok != 0;
}

// Lanes from lo on whose source was covered are no longer alive.  (Leaf lanes are
// looked at when they are committed.)
SKIM_DEV void step_refilter(const StepArgs &a) {
    for (uint32_t j = a.lo + blockIdx.x * blockDim.x + threadIdx.x; j < a.B; j += gridDim.x * blockDim.x) {
        const uint64_t bit = 1ull << (j & 63);
        if (!(a.alive[j >> 6] & ~a.leaf[j >> 6] & bit)) continue;
        const uint32_t pr = a.lane_pair[j], u = pr / a.l, i = pr % a.l;
        if ((a.covered[u] >> i) & 1ull) atomicAnd(reinterpret_cast<unsigned long long *>(&a.alive[j >> 6]), ~bit);
    }
}

// SKIM's stop: per node v the lane at which size[v] reaches k, i.e. the
// need = k - size[v]-th uncovered lane bit (from lane lo on) of v's records in
// rank order (a node already at k stops at its first record).  Warps own the
// runs that start in 32-record windows, as in the acceptance; a segmented
// scan over the lanes counts each node's bits in order.
SKIM_DEV void step_candidates(const StepArgs &a) {
    const uint32_t lane = threadIdx.x & 31;
    const uint64_t tmask = (1ull << a.tbits) - 1;
    const uint64_t warps = (static_cast<uint64_t>(gridDim.x) * blockDim.x) >> 5;
    const uint64_t nwin = (a.R + 31) / 32;
    for (uint64_t w = (blockIdx.x * static_cast<uint64_t>(blockDim.x) + threadIdx.x) >> 5; w < nwin; w += warps) {
        const uint64_t W0 = w * 32, W1 = min(a.R, W0 + 32);
        bool st = false;
        if (W0 + lane < W1) st = run_start(a.rec_key, W0 + lane, a.tbits);
        const unsigned sb = __ballot_sync(kFull, st);
        if (!sb) continue;
        const uint64_t s0 = W0 + __ffs(sb) - 1;
        const uint64_t last = a.rec_key[W1 - 1] >> a.tbits;
        uint64_t cv = ~0ull;  // node that continues from the previous chunk, and its count so far
        uint32_t ccum = 0;
        for (uint64_t c0 = s0;; c0 += 32) {
            const uint64_t rr = c0 + lane;
            uint64_t key = 0, m = 0;
            bool act = false;
            if (rr < a.R) {
                key = a.rec_key[rr];
                act = rr < W1 || (key >> a.tbits) == last;
            }
            const unsigned actb = __ballot_sync(kFull, act);
            if (!actb) break;
            const uint64_t v = key >> a.tbits, t = key & tmask;
            // lanes of the record's word from lo on; its lane bits only when
            // some are left
            if (act) {
                m = range_mask(t, a.lo, 0xffffffffu);
                if (m) m &= a.rbits[rr] & __ldcg(&a.alive[t]);
            }
            const uint32_t c = __popcll(m);
            // inclusive count of v's bits up to this record (runs are contiguous)
            uint32_t incl = c;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(kFull, incl, o);
                const uint64_t vo = __shfl_up_sync(kFull, v, o);
                if (lane >= static_cast<unsigned>(o) && vo == v) incl += y;
            }
            if (v == cv) incl += ccum;
            if (act) {
                const uint32_t excl = incl - c, need = a.k - a.size[v];
                const bool hit = need == 0 ? run_start(a.rec_key, rr, a.tbits) : (excl < need && incl >= need);
                if (hit) {
                    const uint64_t p = t * 64 + nth_set_bit(m, static_cast<int>(need - excl - 1));
                    atomicMin(&a.ctl->step.best, (p << 32) | v);
                }
            }
            const int ll = 31 - __clz(actb);
            cv = __shfl_sync(kFull, v, ll);
            ccum = __shfl_sync(kFull, incl, ll);
            if (actb != kFull) break;
        }
    }
}

// Calls f(node, lane bits, word) for the records with uncovered lanes in [lo, hi].
template <class F>
SKIM_DEV void step_records(const StepArgs &a, uint32_t hi, const F &f) {
    const uint64_t tmask = (1ull << a.tbits) - 1;
    for (uint64_t r = blockIdx.x * static_cast<uint64_t>(blockDim.x) + threadIdx.x; r < a.R;
         r += static_cast<uint64_t>(gridDim.x) * blockDim.x) {
        const uint64_t key = a.rec_key[r], t = key & tmask;
        uint64_t m = range_mask(t, a.lo, hi);
        if (m) m &= a.rbits[r] & __ldcg(&a.alive[t]);
        if (m) f(static_cast<uint32_t>(key >> a.tbits), m, t);
    }
}

// Index space for the lanes [lo, hi] from their counts, which are zero again
// after; lane_pos = where the next entry of a lane goes.
SKIM_DEV void step_segments(const StepArgs &a, uint32_t hi) {
    __shared__ unsigned long long s_warp[kStepThreads / 32], s_base;
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (uint64_t j0 = a.lo + static_cast<uint64_t>(blockIdx.x) * kStepThreads; j0 <= hi;
         j0 += static_cast<uint64_t>(gridDim.x) * kStepThreads) {
        const uint64_t j = j0 + threadIdx.x;
        uint32_t c = 0;
        if (j <= hi) c = __ldcg(&a.lane_cnt[j]);
        unsigned long long tot;
        const unsigned long long ex = warp_excl_scan(c, &tot);
        if (lane == 0) s_warp[warp] = tot;
        __syncthreads();
        if (warp == 0) {
            const unsigned long long w = warp_excl_scan(s_warp[lane], &tot);
            s_warp[lane] = w;
            if (lane == 0) s_base = tot ? atomicAdd(reinterpret_cast<unsigned long long *>(a.idx_ctr), tot) : 0;
        }
        __syncthreads();
        if (c) {
            const uint64_t at = s_base + s_warp[warp] + ex;
            const uint32_t pr = a.lane_pair[j];
            a.lane_pos[j] = at;
            a.lane_cnt[j] = 0;
            a.seg_start[pr] = at;
            a.seg_len[pr] = c;
        }
        __syncthreads();
    }
}

// The leaf lanes of [lo, hi]; returns their number.
SKIM_DEV uint32_t step_leafs(const StepArgs &a, uint32_t hi) {
    uint32_t n = 0;
    for (uint64_t j = a.lo + blockIdx.x * blockDim.x + threadIdx.x; j <= hi; j += gridDim.x * blockDim.x) {
        if (!((a.leaf[j >> 6] & __ldcg(&a.alive[j >> 6])) >> (j & 63) & 1u)) continue;
        const uint32_t pr = a.lane_pair[j], u = pr / a.l;
        if (a.covered[u] >> (pr - u * a.l) & 1u) continue;
        atomicAdd(&a.size[u], 1u);
        a.seg_len[pr] = kLeafSegment;
        n++;
    }
    return n;
}

// k' of Section 4.3.2: the largest size among the nodes other than x.
SKIM_DEV void step_second(const StepArgs &a, uint32_t x) {
    uint32_t best = 0;
    for (uint32_t v = blockIdx.x * blockDim.x + threadIdx.x; v < a.n; v += gridDim.x * blockDim.x)
        if (v != x) best = max(best, __ldcg(&a.size[v]));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) best = max(best, __shfl_down_sync(kFull, best, o));
    if ((threadIdx.x & 31) == 0 && best) atomicMax(a.kprime, best);
}

// Lanes of a commit up to which a block counts them in shared memory, and takes its
// places in their segments at once: the first batches have few lanes that reach up to
// every node, and their records' atomics would meet on as few counters (50 seeds of R-MAT
// 18 trivalency: steps 10.1 -> 9.4 ms; R-MAT 20 p = 0.01: 5.6 -> 4.6 ms).
constexpr uint32_t kDenseLanes = 3072;

__global__ void __launch_bounds__(kStepThreads, 1) k_step(const __grid_constant__ StepArgs a) {
    __shared__ uint32_t s_cnt[kDenseLanes];
    __shared__ unsigned long long s_pos[kDenseLanes];
    DevCtl *C = a.ctl;
    const bool first = blockIdx.x == 0 && threadIdx.x == 0;
    // the last search is not finished: the host ends it and launches the step again
    // (a block that gives up at a barrier sets err: one decision for the block)
    if (__syncthreads_or(*reinterpret_cast<volatile unsigned *>(&C->spill) |
                         *reinterpret_cast<volatile unsigned *>(&C->err))) {
        if (first) {
            C->step.best = ~0ull;
            C->step.stalled = 1;
        }
        return;
    }
    if (first) C->step.best = ~0ull;
    if (a.refilter) step_refilter(a);
    if (!step_barrier(C, 0, a.timeout_ns)) return;
    step_candidates(a);
    if (!step_barrier(C, 1, a.timeout_ns)) return;
    const uint64_t best = ld_volatile(&C->step.best);
    const uint32_t hi = best == ~0ull ? a.B - 1 : static_cast<uint32_t>(best >> 32);
    // Additive, so a thread per record.  The stop lane's own part of the sizes
    // follows in the last phase: k' is counted without it.
    const uint64_t stop = best == ~0ull ? ~0ull : hi;
    const uint32_t range = hi >= a.lo && a.lo < a.B ? hi - a.lo + 1 : 0;
    const bool dense = range <= kDenseLanes;
    for (uint32_t i = threadIdx.x; dense && i < range; i += kStepThreads) s_cnt[i] = 0;
    __syncthreads();
    unsigned long long ins = step_leafs(a, hi);
    step_records(a, hi, [&](uint32_t v, uint64_t m, uint64_t t) {
        const uint32_t c = __popcll(m), d = t == stop >> 6 ? static_cast<uint32_t>(m >> (stop & 63)) & 1u : 0;
        if (c > d) atomicAdd(&a.size[v], c - d);
        ins += c;
        for (; m; m &= m - 1) {
            const uint64_t j = t * 64 + __ffsll(m) - 1;
            atomicAdd(dense ? &s_cnt[j - a.lo] : &a.lane_cnt[j], 1u);
        }
    });
    __syncthreads();
    for (uint32_t i = threadIdx.x; dense && i < range; i += kStepThreads)
        if (s_cnt[i]) atomicAdd(&a.lane_cnt[a.lo + i], s_cnt[i]);
    warp_add(&C->stats[kStInsert], ins);
    if (!step_barrier(C, 2, a.timeout_ns)) return;
    step_segments(a, hi);
    if (a.kprime && best != ~0ull) {
        step_second(a, static_cast<uint32_t>(best));
        if (first) *a.tau = a.lane_rank[hi];
    }
    if (!step_barrier(C, 3, a.timeout_ns)) return;
    // (the block's records are those it counted)
    for (uint32_t i = threadIdx.x; dense && i < range; i += kStepThreads)
        if (s_cnt[i]) s_pos[i] = atomicAdd(reinterpret_cast<unsigned long long *>(&a.lane_pos[a.lo + i]), s_cnt[i]);
    __syncthreads();
    step_records(a, hi, [&](uint32_t v, uint64_t m, uint64_t t) {
        if (t == stop >> 6 && (m >> (stop & 63) & 1u)) atomicAdd(&a.size[v], 1u);
        for (; m; m &= m - 1) {
            const uint64_t j = t * 64 + __ffsll(m) - 1;
            const uint64_t at =
                dense ? s_pos[j - a.lo] + atomicSub(&s_cnt[j - a.lo], 1u) - 1
                      : atomicAdd(reinterpret_cast<unsigned long long *>(&a.lane_pos[j]), 1ull);
            a.idx_nodes[at] = v;
        }
    });
    if (first) {  // what the host takes, and the count of the next search from zero
        C->step.cov = C->ix_cov;
        C->ix_cov = 0;
        C->step.stalled = 0;
    }
}

__global__ void k_argmax_size(const uint32_t *size, uint32_t n, DevCtl *ctl) {
    unsigned long long best = 0;
    for (uint32_t v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x) {
        unsigned long long key = (static_cast<unsigned long long>(size[v]) << 32) | (0xffffffffu - v);
        best = max(best, key);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) best = max(best, __shfl_down_sync(kFull, best, o));
    if ((threadIdx.x & 31) == 0) atomicMax(&ctl->argmax, best);
}

__global__ void k_min_unchosen(const uint8_t *chosen, uint32_t n, DevCtl *ctl) {
    unsigned long long best = ~0ull;
    for (uint32_t v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x)
        if (!chosen[v]) best = min(best, static_cast<unsigned long long>(v));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) best = min(best, __shfl_down_sync(kFull, best, o));
    if ((threadIdx.x & 31) == 0) atomicMin(&ctl->best, best);
}

}  // namespace

cudaError_t launch_lane_inst(const uint32_t *lane_pair, const uint64_t *lane_rank, uint32_t B, uint32_t l,
                             uint8_t *lane_inst, uint64_t *lane_g, cudaStream_t s) {
    note_launch();
    k_lane_inst<<<grid_for(B, 256), 256, 0, s>>>(lane_pair, lane_rank, B, l, lane_inst, lane_g);
    return cudaGetLastError();
}
cudaError_t launch_accept(const uint64_t *rec_key, const uint32_t *rec_val, const uint64_t *hvals, uint64_t R,
                          uint32_t tbits, const uint8_t *lane_inst, const uint64_t *lane_rank, uint32_t l, uint32_t k,
                          uint8_t *lcnt, uint64_t *full, uint64_t *X, uint32_t *xlen, DevCtl *ctl,
                          cudaStream_t s) {
    if (R == 0) return cudaSuccess;
    note_launch();
    k_accept<<<grid_for(R, 256), 256, 0, s>>>(rec_key, rec_val, hvals, R, tbits, lane_inst, lane_rank, l, k,
                                               lcnt, full, X, xlen, ctl);
    return cudaGetLastError();
}
cudaError_t launch_gather_bits(const uint32_t *rec_val, const uint64_t *hvals, uint64_t R, uint64_t *rbits,
                               cudaStream_t s) {
    if (R == 0) return cudaSuccess;
    note_launch();
    k_gather_bits<<<grid_for(R, 256), 256, 0, s>>>(rec_val, hvals, R, rbits);
    return cudaGetLastError();
}
cudaError_t launch_step(const StepArgs &a, cudaStream_t s) {
    int dev = 0, sms = 0, per = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_step, kStepThreads, 0);
    if (e != cudaSuccess) return e;
    const uint64_t work = std::max<uint64_t>(a.R, a.B - std::min(a.lo, a.B));
    const unsigned grid = std::min<unsigned>(grid_for(work, kStepThreads), static_cast<unsigned>(sms) * std::min(per, 1));
    note_launch();
    // between two barriers a warp walks a node's records 32 at a time, a thread the lanes in steps of the grid
    StepArgs b = a;
    b.timeout_ns = phase_limit(a.timeout_ns, 1 + a.R / 32 + work / kStepThreads);
    void *args[] = {&b};
    return cudaLaunchCooperativeKernel(reinterpret_cast<void *>(k_step), dim3(grid), dim3(kStepThreads), args, 0, s);
}
cudaError_t launch_argmax_size(const uint32_t *size, uint32_t n, DevCtl *ctl, cudaStream_t s) {
    note_launch();
    k_argmax_size<<<grid_for(n, 256), 256, 0, s>>>(size, n, ctl);
    return cudaGetLastError();
}
cudaError_t launch_min_unchosen(const uint8_t *chosen, uint32_t n, DevCtl *ctl, cudaStream_t s) {
    note_launch();
    k_min_unchosen<<<grid_for(n, 256), 256, 0, s>>>(chosen, n, ctl);
    return cudaGetLastError();
}

}  // namespace skim
