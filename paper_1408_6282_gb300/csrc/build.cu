// build.cu -- Algorithm 2 (Section 5.2) over materialised instances: the
// kernels that turn a batch of ranks into sketch entries.
//
// What a node's combined sketch X_v needs is only the k smallest ranks of all
// its instances together, so a reverse search is cut where no node can still
// use its rank, which is far earlier than where a pair (v, i) has seen k ranks
// of its own instance:
//
//   need    need[v] bit i: some node that reaches v in instance i (v itself
//           included) holds fewer than k ranks.  A search skips a pair whose
//           bit is clear.  Recomputed between batches as a least fixed point
//           over the live rows of the full nodes; a stale mask only has more
//           bits, so the result does not depend on when that is done.  It
//           subsumes the per-instance count: k ranks of instance i at (v, i)
//           have also reached every node that reaches (v, i).
//   own     A node reaches itself in every instance, so its own l ranks are
//           merged at the end (k_merge) instead of being searched for: most
//           source lanes have an empty row and cost a look at the row bounds.
//   full    A visit to a node that holds k ranks leaves no record.
//   giant   Where the searches are large (supercritical live graphs), each
//           instance's largest strongly connected component is contracted: all
//           its members have the same upstream, so the first k ranks of the
//           instance that hit it are all that anything upstream can use of
//           them.  They go to a list of the instance that k_merge merges into
//           every node reaching the component, and the search stops there.
//
// Measured against the search of every rank with per-instance counts, a sort of
// its visit records and an acceptance pass (whole builds, l = k = 64): R-MAT 20
// wc 33.7 -> 13.5 ms (150 M visits -> 62 M, most of them looks at a source with
// an empty row), R-MAT 22 p = 0.01 316 -> 17.4 ms (1.1 G -> 4 M), 24 trivalency
// graphs 21.5 -> 2.2 ms, Erdos-Renyi 50021 with positions 4.1 -> 3.1 ms.
//
// Order inside a batch does not matter: records are appended to X_v as they
// come (k_append) and a row that would exceed k keeps its k smallest ranks
// (k_over_*); rows are sorted once, by k_merge.
#include <algorithm>

#include "internal.cuh"

namespace skim {

namespace {

inline unsigned grid_for(size_t n, int threads, unsigned cap = 152 * 32) {
    size_t g = (n + threads - 1) / threads;
    if (g > cap) g = cap;
    return static_cast<unsigned>(g ? g : 1);
}

// ---- searches of small rank lanes, one warp's lanes at a time ----------------
//
// Most lanes reach a handful of nodes.  A warp takes kIds lanes at a time and
// walks them from a stack of rows in shared memory; which (node, lane) pairs
// they have reached is a hash set in shared memory, so a visit costs one random
// row-bounds read, the need word of the node and its share of a row, and no
// atomic in global memory.  A lane whose search does not fit (stack or set)
// is deferred to the searches with a global visited table (traverse.cu), which
// run it again from its source; its records from here are dropped.
#ifndef SKIM_ID_BITS
#define SKIM_ID_BITS 8
#endif
#ifndef SKIM_TAB_BITS
#define SKIM_TAB_BITS 10
#endif
constexpr int kSearchThreads = 256;
constexpr uint32_t kIdBits = SKIM_ID_BITS, kIds = 1u << kIdBits;  // lanes of a warp's epoch
constexpr uint32_t kTabBits = SKIM_TAB_BITS, kTab = 1u << kTabBits;  // slots of the reached set
constexpr uint32_t kTabStop = kTab * 11 / 16;          // entries from which nothing is added
constexpr uint32_t kTabStart = kTab * 7 / 16;          // entries from which no lanes are started
constexpr uint32_t kStack = 192;                       // rows
constexpr uint32_t kStage = 96;                        // staged records

template <class KT>
struct WarpMem {
    KT tab[kTab];
    uint2 stack[kStack];  // {first entry, entries << kIdBits | lane id}
    uint64_t stage[kStage];
    uint32_t pair[kIds];  // source pairs v * l + i
    uint32_t base[kIds / 32];
    uint32_t defer[kIds / 32], hit[kIds / 32];
};

template <class KT, bool SCC>
struct WarpSearch {
    const BuildArgs &A;
    WarpMem<KT> &W;
    uint32_t sp = 0, cnt = 0, nst = 0;  // warp-uniform: stack, set and stage fill
    uint64_t visits = 0, edges = 0;     // per lane

    SKIM_DEV bool deferred(uint32_t id) const {
        return (*reinterpret_cast<const volatile uint32_t *>(&W.defer[id >> 5]) >> (id & 31)) & 1u;
    }
    SKIM_DEV void defer(uint32_t id) { atomicOr(&W.defer[id >> 5], 1u << (id & 31)); }

    SKIM_DEV void flush() {
        __syncwarp();
        if (!nst) return;
        const uint32_t lane = threadIdx.x & 31;
        unsigned long long b = 0;
        if (lane == 0) b = atomicAdd(&A.ctl->rec_count.v, static_cast<unsigned long long>(nst));
        b = __shfl_sync(kFull, b, 0);
        for (uint32_t q = lane; q < nst; q += 32) {
            if (b + q < A.rcap) A.rec[b + q] = W.stage[q];
            else atomicOr(&A.ctl->err, kErrRecords);
        }
        __syncwarp();
        nst = 0;
    }
    SKIM_DEV void record(bool rec, uint32_t v, uint32_t ln) {
        const unsigned b = __ballot_sync(kFull, rec);
        if (!b) return;
        if (rec) W.stage[nst + __popc(b & lanemask_lt())] = static_cast<uint64_t>(v) << A.lbits | ln;
        nst += __popc(b);
        if (nst > kStage - 32) flush();
    }

    // Warp-collective: lanes with `row` push a row of search id.
    SKIM_DEV void push(bool row, uint32_t b, uint32_t len, uint32_t id) {
        if (row && len >> (32 - kIdBits)) {
            defer(id);
            row = false;
        }
        const unsigned pb = __ballot_sync(kFull, row);
        if (row) {
            const uint32_t at = sp + __popc(pb & lanemask_lt());
            if (at < kStack) W.stack[at] = make_uint2(b, len << kIdBits | id);
            else defer(id);
        }
        sp = min(sp + __popc(pb), kStack);
        __syncwarp();
    }

    // Warp-collective: lanes with `act` reach node x in search id.
    SKIM_DEV void visit(bool act, uint32_t x, uint32_t id) {
        uint32_t i = 0, w0 = 0, w1 = 0;
        uint64_t nd = 0;
        if (act) {
            const uint32_t pr = W.pair[id], u = pr / A.l;
            i = pr - u * A.l;
            act = x != u && !deferred(id);  // (a source's row is walked already)
        }
        if (act) {
            const uint64_t r = static_cast<uint64_t>(x) * A.l + i;
            nd = A.need[x];
            w0 = A.loff[r];
            w1 = A.loff[r + 1];
            if (!((nd >> i) & 1ull)) act = false;
            if (SCC && ((A.scc[x] >> i) & 1ull)) {
                if (act) {  // the instance's hit list is open
                    const uint32_t bit = 1u << (id & 31);
                    if (!(atomicOr(&W.hit[id >> 5], bit) & bit)) atomicOr(&A.hit[W.base[id >> 5] >> 5], bit);
                }
                act = false;
            }
        }
        bool fresh = false;
        if (cnt >= kTabStop) {
            if (act) defer(id);
        } else if (act) {
            const KT key = static_cast<KT>(x) << kIdBits | id;
            uint32_t h = (static_cast<uint32_t>(key ^ (static_cast<uint64_t>(key) >> 25)) * 0x9E3779B1u) >> (32 - kTabBits);
            for (;;) {
                const KT o = atomicCAS(&W.tab[h], static_cast<KT>(~static_cast<KT>(0)), key);
                if (o == static_cast<KT>(~static_cast<KT>(0))) {
                    fresh = true;
                    break;
                }
                if (o == key) break;
                h = (h + 1) & (kTab - 1);
            }
        }
        cnt += __popc(__ballot_sync(kFull, fresh));
        visits += fresh ? 1 : 0;
        record(fresh && nd == A.lmask, x, W.base[id >> 5] + (id & 31));
        push(fresh && w1 > w0, w0, w1 - w0, id);
    }

    // Warp-collective: start source lanes j0 .. j0 + 31 as group g.  Most rows
    // are empty, which one word per node tells (a member of a component has a
    // row that is not).
    SKIM_DEV void start(uint32_t j0, uint32_t g) {
        const uint32_t lane = threadIdx.x & 31, j = j0 + lane;
        const bool in = j < A.B;
        const uint32_t pr = in ? A.pair[j] : 0;
        const uint32_t u = pr / A.l, i = pr - u * A.l;
        const bool row = in && ((A.nonempty[u] >> i) & 1ull);
        bool act = row || (in && A.own), hit = false;
        uint32_t w0 = 0, w1 = 0;
        uint64_t nd = 0;
        if (act) {
            nd = A.need[u];
            if (row) {
                w0 = A.loff[pr];
                w1 = A.loff[pr + 1ull];
            }
            if (!((nd >> i) & 1ull)) act = false;
            if (SCC && row && ((A.scc[u] >> i) & 1ull)) {
                hit = act;
                act = false;
            }
        }
        W.pair[g * 32 + lane] = pr;
        const unsigned hb = __ballot_sync(kFull, hit);
        if (lane == 0) {
            W.base[g] = j0;
            if (hb) atomicOr(&A.hit[j0 >> 5], hb);
        }
        __syncwarp();
        visits += act ? 1 : 0;
        if (A.own) record(act && nd == A.lmask, u, j);
        push(act && w1 > w0, w0, w1 - w0, g * 32 + lane);
    }

    // Warp-collective: take up to 32 rows off the stack and visit their entries.
    SKIM_DEV void expand() {
        const uint32_t lane = threadIdx.x & 31;
        const uint32_t n = min(sp, 32u);
        sp -= n;
        uint32_t begin = 0, len = 0, id = 0;
        if (lane < n) {
            const uint2 it = W.stack[sp + lane];
            id = it.y & (kIds - 1);
            begin = it.x;
            len = deferred(id) ? 0 : it.y >> kIdBits;
        }
        __syncwarp();
        edges += len;
        unsigned big = __ballot_sync(kFull, len >= 32);
        while (big) {
            const int s = __ffs(big) - 1;
            big &= big - 1;
            const uint32_t bb = __shfl_sync(kFull, begin, s), bc = __shfl_sync(kFull, len, s);
            const uint32_t bi = __shfl_sync(kFull, id, s);
            uint32_t x = A.rlive[bb + lane];
            for (uint32_t k0 = 0; k0 < bc; k0 += 32) {
                const uint32_t k = k0 + lane;
                const uint32_t xn = k + 32 < bc ? A.rlive[bb + k + 32] : 0;
                visit(k < bc, x, bi);
                // one decision for the warp: the next visit may defer the search
                // before every lane has looked
                if (__any_sync(kFull, deferred(bi))) break;
                x = xn;
            }
        }
        const uint32_t c = len < 32 ? len : 0;
        uint32_t incl = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(kFull, incl, o);
            if (lane >= static_cast<uint32_t>(o)) incl += y;
        }
        const uint32_t total = __shfl_sync(kFull, incl, 31);
        const uint32_t first = begin - (incl - c);  // entry g of the warp is first of its row + g
        for (uint32_t g = 0; g < total; g += 32) {
            const uint32_t o = g + lane;
            uint32_t sl = 0;  // owner: the first lane whose inclusive count exceeds o
#pragma unroll
            for (uint32_t step = 16; step > 0; step >>= 1) {
                const uint32_t v = __shfl_sync(kFull, incl, sl + step - 1);
                if (v <= o) sl += step;
            }
            const uint32_t sb = __shfl_sync(kFull, first, sl), si = __shfl_sync(kFull, id, sl);
            const bool has = o < total;
            visit(has, has ? A.rlive[sb + o] : 0, si);
        }
    }

    // Warp-collective: end an epoch of `groups` groups: hand over the deferred
    // lanes, empty the set.
    SKIM_DEV void finish(uint32_t groups) {
        const uint32_t lane = threadIdx.x & 31;
        __syncwarp();
        for (uint32_t g = 0; g < groups; g++) {
            const uint32_t d = W.defer[g];
            if (!d) continue;
            uint32_t at = 0;
            if (lane == 0) {
                at = atomicAdd(&A.ctl->b.n_def, static_cast<unsigned>(__popc(d)));
                A.defbits[W.base[g] >> 5] = d;
            }
            at = __shfl_sync(kFull, at, 0);
            if ((d >> lane) & 1u) A.deflist[at + __popc(d & lanemask_lt())] = W.base[g] + lane;
        }
        __syncwarp();
        if (lane < kIds / 32) W.defer[lane] = W.hit[lane] = 0;
        if (cnt) {
            uint4 *t = reinterpret_cast<uint4 *>(W.tab);
            const uint4 e = make_uint4(~0u, ~0u, ~0u, ~0u);
            for (uint32_t q = lane; q < kTab * sizeof(KT) / 16; q += 32) t[q] = e;
        }
        cnt = 0;
        __syncwarp();
    }
};

template <class KT, bool SCC>
__global__ void __launch_bounds__(kSearchThreads) k_build_search(BuildArgs A) {
    extern __shared__ uint4 s_mem[];
    if (A.ctl->b.n_full == A.n) return;  // every node has its k ranks
    const uint32_t lane = threadIdx.x & 31;
    WarpMem<KT> &W = reinterpret_cast<WarpMem<KT> *>(s_mem)[threadIdx.x >> 5];
    WarpSearch<KT, SCC> S{A, W};
    S.cnt = 1;
    S.finish(0);
    uint32_t cur = 0, end = 0, groups = 0;
    bool more = true;
    for (;;) {
        if (cur == end && more && groups == 0) {  // the next lanes of the batch
            unsigned long long j = 0;
            unsigned e = 0;
            if (lane == 0) {
                j = atomicAdd(&A.ctl->src_next.v, static_cast<unsigned long long>(kIds));
                e = *reinterpret_cast<volatile unsigned *>(&A.ctl->err);
            }
            j = __shfl_sync(kFull, j, 0);
            // a batch that overflowed its record table is run again smaller
            if (j >= A.B || __shfl_sync(kFull, e, 0)) more = false;
            else {
                cur = static_cast<uint32_t>(j);
                end = min(A.B - cur, kIds) + cur;
            }
        }
        // rows of full warps first: lanes are started while the stack holds
        // less than a warp's worth and the set has room for them
        if (cur < end && groups < kIds / 32 && S.sp < 32 && S.cnt < kTabStart) {
            S.start(cur, groups++);
            cur = min(cur + 32, end);
            continue;
        }
        if (S.sp) {
            S.expand();
            continue;
        }
        if (!groups) break;
        S.finish(groups);
        groups = 0;
    }
    S.flush();
    warp_add(&A.ctl->stats[kStRevVisits], S.visits);
    warp_add(&A.ctl->stats[kStRevEdges], S.edges);
}

// (all: every lane of the batch, which the list is filled with)
__global__ void k_deferred_lanes(uint32_t *deflist, uint32_t D, bool all, const uint32_t *pair, uint32_t l,
                                 uint32_t *defpair, uint8_t *lane_inst) {
    for (uint32_t q = blockIdx.x * blockDim.x + threadIdx.x; q < D; q += gridDim.x * blockDim.x) {
        if (all) deflist[q] = q;
        const uint32_t pr = pair[deflist[q]];
        defpair[q] = pr;
        lane_inst[q] = static_cast<uint8_t>(pr % l);
    }
}

// ---- records into sketch rows ------------------------------------------------

// Record (node, lane) of the batch appends the lane's rank to the node's row.
// Ranks past the k-th place of a row go to an overflow list {record, place - k};
// the node is listed once.  Rows flagged full (all ranks of this batch are
// larger) take nothing.  Records [r0, r1); those of deferred lanes are dropped
// (defbits, null: none).
__global__ void k_append(const uint64_t *__restrict__ rec, uint64_t r0, uint64_t r1, uint32_t lbits,
                         const uint32_t *__restrict__ defbits, const uint64_t *__restrict__ lane_rank, uint32_t k,
                         uint32_t *len, uint64_t *X, uint64_t *over_key, uint32_t *over_pos, uint32_t *list,
                         DevCtl *ctl, const unsigned *count) {
    const uint64_t lm = (1ull << lbits) - 1;
    if (count) r1 = *count;
    for (uint64_t r = r0 + blockIdx.x * static_cast<uint64_t>(blockDim.x) + threadIdx.x; r < r1;
         r += static_cast<uint64_t>(gridDim.x) * blockDim.x) {
        const uint64_t key = rec[r];
        const uint32_t v = static_cast<uint32_t>(key >> lbits), ln = static_cast<uint32_t>(key & lm);
        if (defbits && ((defbits[ln >> 5] >> (ln & 31)) & 1u)) continue;
        if (len[v] & kRowDone) continue;
        const uint32_t at = atomicAdd(&len[v], 1u);
        if (at < k) {
            X[static_cast<uint64_t>(v) * k + at] = lane_rank[ln];
        } else {
            const unsigned o = atomicAdd(&ctl->b.n_over, 1u);
            over_key[o] = key;
            over_pos[o] = at - k;
            if (at == k) list[atomicAdd(&ctl->b.n_list, 1u)] = v;
        }
    }
}

// The same for records per table entry (node, lane word): a record's lanes are
// the bits of its table slot, in rank order, so only the first k of them can
// matter.  The node's own ranks are left out unless `own` (they are merged).
// For a first batch, whose visits may be far more than the record table holds, and for
// dense ones behind it (R-MAT 20 wc with every batch of the first 400 K lanes in this
// form: 14.8 ms instead of 13.2, for the look at every lane's source).
__global__ void k_append_words(const uint64_t *__restrict__ rec, const uint32_t *__restrict__ rec_val, uint64_t R,
                               uint32_t tbits, const uint64_t *__restrict__ hvals, const uint32_t *__restrict__ pair,
                               uint32_t l, int own, uint32_t lbits,
                               const uint64_t *__restrict__ lane_rank, uint32_t k, uint32_t *len, uint64_t *X,
                               uint64_t *over_key, uint32_t *over_pos, uint32_t *list, DevCtl *ctl) {
    const uint64_t tm = (1ull << tbits) - 1;
    for (uint64_t r = blockIdx.x * static_cast<uint64_t>(blockDim.x) + threadIdx.x; r < R;
         r += static_cast<uint64_t>(gridDim.x) * blockDim.x) {
        const uint64_t key = rec[r];
        const uint32_t v = static_cast<uint32_t>(key >> tbits);
        const uint32_t ln0 = static_cast<uint32_t>(key & tm) * 64;
        uint64_t bits = hvals[2ull * rec_val[r]];
        if (len[v] & kRowDone) continue;
        if (!own)
            for (uint64_t m = bits; m; m &= m - 1)
                if (pair[ln0 + __ffsll(m) - 1] / l == v) bits &= ~(m & (~m + 1));
        const uint32_t n = min(static_cast<uint32_t>(__popcll(bits)), k);
        if (!n) continue;
        uint32_t at = atomicAdd(&len[v], n);
        unsigned o = 0;
        if (at + n > k) o = atomicAdd(&ctl->b.n_over, at + n - max(at, k));
        if (at <= k && at + n > k) list[atomicAdd(&ctl->b.n_list, 1u)] = v;
        for (uint32_t q = 0; q < n; q++, at++, bits &= bits - 1) {
            const uint32_t ln = ln0 + __ffsll(bits) - 1;
            if (at < k) {
                X[static_cast<uint64_t>(v) * k + at] = lane_rank[ln];
            } else {
                over_key[o] = static_cast<uint64_t>(v) << lbits | ln;
                over_pos[o++] = at - k;
            }
        }
    }
}

// Lanes of the records of each chunk.
__global__ void __launch_bounds__(kWordChunk) k_count_words(const uint32_t *__restrict__ rec_val, uint64_t R,
                                                            const uint64_t *__restrict__ hvals, uint32_t *cnt) {
    __shared__ uint32_t s_n;
    for (uint64_t q = blockIdx.x; q * kWordChunk < R; q += gridDim.x) {
        if (threadIdx.x == 0) s_n = 0;
        __syncthreads();
        const uint64_t r = q * kWordChunk + threadIdx.x;
        const uint32_t n = __reduce_add_sync(kFull, r < R ? __popcll(hvals[2ull * rec_val[r]]) : 0);
        if ((threadIdx.x & 31) == 0) atomicAdd(&s_n, n);
        __syncthreads();
        if (threadIdx.x == 0) cnt[q] = s_n;
    }
}

// space of each listed node's overflow
__global__ void k_over_alloc(const uint32_t *list, const uint32_t *len, uint32_t k, uint32_t *seg, DevCtl *ctl) {
    const uint32_t n = ctl->b.n_list;
    for (uint32_t q = blockIdx.x * blockDim.x + threadIdx.x; q < n; q += gridDim.x * blockDim.x) {
        const uint32_t v = list[q];
        seg[v] = atomicAdd(&ctl->b.over_total, len[v] - k);
    }
}

__global__ void k_over_scatter(const uint64_t *over_key, const uint32_t *over_pos, uint32_t lbits,
                               const uint64_t *__restrict__ lane_rank, const uint32_t *seg, uint64_t *buf,
                               const DevCtl *ctl) {
    const uint64_t lm = (1ull << lbits) - 1;
    const uint32_t n = ctl->b.n_over;
    for (uint32_t o = blockIdx.x * blockDim.x + threadIdx.x; o < n; o += gridDim.x * blockDim.x)
        buf[seg[over_key[o] >> lbits] + over_pos[o]] = lane_rank[over_key[o] & lm];
}

// Warp-collective ascending bitonic sort of a[0 .. P), P a power of two of at least 64.
SKIM_DEV void warp_sort(uint64_t *a, uint32_t P) {
    const uint32_t lane = threadIdx.x & 31;
    for (uint32_t kk = 2; kk <= P; kk <<= 1)
        for (uint32_t j = kk >> 1; j > 0; j >>= 1) {
            __syncwarp();
            for (uint32_t q = lane; q < P / 2; q += 32) {
                const uint32_t lo = ((q & ~(j - 1)) << 1) | (q & (j - 1)), hi = lo | j;
                const uint64_t x = a[lo], y = a[hi];
                if ((x > y) == ((lo & kk) == 0)) {
                    a[lo] = y;
                    a[hi] = x;
                }
            }
        }
    __syncwarp();
}

SKIM_DEV uint32_t pow2_from64(uint32_t x) { return x <= 64 ? 64 : 1u << (32 - __clz(x - 1)); }

// A warp per listed node: the k smallest of its row and its overflow become
// the row (any order).  done: every smaller rank has been seen, so the row takes
// no more.
constexpr uint32_t kSelWarps = 4, kSelCap = 512;
__global__ void __launch_bounds__(kSelWarps * 32) k_over_select(const uint32_t *list, uint32_t k, uint32_t *len,
                                                                const uint32_t *seg, const uint64_t *buf,
                                                                uint64_t *X, uint32_t done, const DevCtl *ctl) {
    __shared__ uint64_t s_a[kSelWarps][kSelCap];
    const uint32_t lane = threadIdx.x & 31;
    uint64_t *a = s_a[threadIdx.x >> 5];
    const uint32_t n = ctl->b.n_list;
    const uint32_t cap = pow2_from64(k + 64);  // at most 512 (k <= 255)
    for (uint32_t q = blockIdx.x * kSelWarps + (threadIdx.x >> 5); q < n; q += gridDim.x * kSelWarps) {
        const uint32_t v = list[q], s = len[v] - k;
        uint64_t *row = X + static_cast<uint64_t>(v) * k;
        const uint64_t *b = buf + seg[v];
        __syncwarp();
        for (uint32_t j = lane; j < k; j += 32) a[j] = row[j];
        uint32_t fill = k, at = 0;
        uint64_t top = ~0ull;  // the k-th smallest so far
        bool first = true;
        while (at < s) {
            // smaller candidates join the array until it has no room for 32 more
            while (at < s && fill + 32 <= cap) {
                const uint64_t x = at + lane < s ? b[at + lane] : ~0ull;
                const bool in = at + lane < s && (first || x < top);
                const unsigned ib = __ballot_sync(kFull, in);
                if (in) a[fill + __popc(ib & lanemask_lt())] = x;
                fill += __popc(ib);
                at += 32;
            }
            if (fill > k) {
                const uint32_t P = pow2_from64(fill);
                for (uint32_t j = fill + lane; j < P; j += 32) a[j] = ~0ull;
                warp_sort(a, P);
                fill = k;
                top = a[k - 1];
                first = false;
            }
        }
        __syncwarp();
        for (uint32_t j = lane; j < k; j += 32) row[j] = a[j];
        if (lane == 0) len[v] = k | done;
    }
}

// ---- what is still needed ------------------------------------------------------

struct OwnRanks {  // own ranks of a node (rank_of in graph.cu's order); l == 0: recorded by the searches
    uint64_t rank_key;
    const uint64_t *rbase;
    uint32_t l;
    SKIM_DEV uint64_t rank(uint32_t v, uint32_t i) const {
        return rbase ? fmix(rbase[v] + kGolden * i) : pair_rank(rank_key, static_cast<uint64_t>(v) * l + i);
    }
};

__global__ void k_fill_u64(uint64_t *p, uint32_t n, uint64_t x) {
    for (uint32_t v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x) p[v] = x;
}

SKIM_DEV uint32_t graph_of(const uint32_t *node_off, uint32_t graphs, uint32_t v) {
    if (graphs == 1) return 0;
    uint32_t lo = 0, hi = graphs;  // last graph whose first node is at most v
    while (hi - lo > 1) {
        const uint32_t mid = (lo + hi) >> 1;
        if (node_off[mid] <= v) lo = mid;
        else hi = mid;
    }
    return lo;
}

// The nodes that have become full, flagged (kRowDone) and added to the list of
// full nodes.  A node's ranks so far: its row and the own ranks below *next
// (they are disjoint), or the entries of the hit lists of the components that
// it reaches.  Own ranks are counted only where chance lets the count matter
// (about x l of them are below *next = x 2^64): a full node taken for one that
// is not only costs time.
__global__ void k_need_full(BuildNode g, const uint64_t *next, uint32_t *list, DevCtl *ctl) {
    const uint32_t lane = threadIdx.x & 31;
    const uint64_t thr = *next;
    const OwnRanks own{g.rank_key, g.rbase, g.own ? g.l : 0};
    const float mean = static_cast<float>(thr >> 40) * (1.0f / 16777216.0f) * own.l;
    const float most = mean + 6.0f * sqrtf(mean) + 4.0f;
    for (uint32_t v0 = blockIdx.x * blockDim.x; v0 < g.n; v0 += gridDim.x * blockDim.x) {
        const uint32_t v = v0 + threadIdx.x;
        bool full = false;
        if (v < g.n) {
            const uint32_t f = g.len[v], c = f & ~kRowDone;
            if (!(f & kRowListed)) {
                full = c >= g.k;
                if (!full && own.l && g.k - c <= own.l && static_cast<float>(g.k - c) <= most) {
                    uint32_t have = c;
                    for (uint32_t i = 0; i < own.l && have < g.k; i++) have += own.rank(v, i) < thr;
                    full = have >= g.k;
                }
                if (!full && g.up && g.up[v]) {
                    const uint32_t *tl = g.tlen + graph_of(g.node_off, g.graphs, v) * 64ull;
                    uint32_t t = 0;
                    for (uint64_t m = g.up[v]; m && t < g.k; m &= m - 1) t += tl[__ffsll(m) - 1] & ~kRowDone;
                    full = t >= g.k;
                }
                if (full) g.len[v] = min(c, g.k) | kRowDone | kRowListed;
            }
        }
        const unsigned fb = __ballot_sync(kFull, full);
        if (fb) {
            unsigned at = 0;
            if (lane == 0) at = atomicAdd(&ctl->b.n_full, static_cast<unsigned>(__popc(fb)));
            at = __shfl_sync(kFull, at, 0);
            if (full) list[at + __popc(fb & lanemask_lt())] = v;
        }
    }
}

// need of the listed nodes as far as their own live in-neighbours tell: a bit
// is set where one of them is not full; of the component only the bit that
// says whether its hit list is open.  A row whose in-neighbours are all full
// becomes a task {node, row (or its only entry), entries << 6 | instance} for
// the sweeps, one of more than kTaskRow entries a task at the other end of the
// space; one that finds no room sets its bit (searched for longer, same result).
// Nothing to do while the full nodes and the open lists are those of the last pass.
constexpr uint32_t kTaskLook = 16;  // entries a lane looks at by itself
constexpr uint32_t kTaskRow = 96;   // and the longest row of a short task
__global__ void __launch_bounds__(256) k_need_tasks(BuildNode g, uint64_t *need, const uint32_t *__restrict__ list,
                                                    uint4 *tasks, uint32_t cap, DevCtl *ctl) {
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t nf = ctl->b.n_full;
    if (nf == ctl->b.n_full_last && ctl->b.n_open == ctl->b.n_open_last) return;
    const uint32_t warps = gridDim.x * (blockDim.x / 32);
    for (uint32_t q = blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5); q < nf; q += warps) {
        const uint32_t v = list[q];
        const uint64_t sc = g.scc ? g.scc[v] : 0;
        const uint64_t todo = g.nonempty[v] & ~sc;
        uint64_t got = sc ? sc & g.topen[graph_of(g.node_off, g.graphs, v)] : 0;
#pragma unroll
        for (uint32_t h = 0; h < 2; h++) {
            const uint32_t i = lane + 32 * h;
            uint32_t a = 0, e = 0;
            if ((todo >> i) & 1ull) {
                const uint64_t r = static_cast<uint64_t>(v) * g.l + i;
                a = g.loff[r];
                e = g.loff[r + 1];
            }
            bool found = false;
            uint32_t x = 0;
            const uint32_t stop = min(e, a + kTaskLook);
            for (uint32_t z = a; z < stop && !found; z++) {
                x = g.rlive[z];
                found = !(g.len[x] & kRowListed);
            }
            unsigned lb = __ballot_sync(kFull, !found && e > stop && e - a <= kTaskRow);
            while (lb) {  // longer rows: the warp together, 32 entries at a time
                const int s = __ffs(lb) - 1;
                lb &= lb - 1;
                const uint32_t za = __shfl_sync(kFull, stop, s), ze = __shfl_sync(kFull, e, s);
                for (uint32_t z = za; z < ze; z += 32) {
                    const bool f = z + lane < ze && !(g.len[g.rlive[z + lane]] & kRowListed);
                    if (__any_sync(kFull, f)) {
                        if (lane == static_cast<uint32_t>(s)) found = true;
                        break;
                    }
                }
            }
            const bool task = !found && e > a, longer = task && e - a > kTaskRow;
            const unsigned tb = __ballot_sync(kFull, task && !longer);
            unsigned at = 0;
            if (tb && lane == 0) at = atomicAdd(&ctl->b.n_task, static_cast<unsigned>(__popc(tb)));
            at = __shfl_sync(kFull, at, 0) + __popc(tb & lanemask_lt());
            if (longer) at = atomicAdd(&ctl->b.n_long, 1u);
            if (task) {
                if (at >= (longer ? cap / 16 : cap - cap / 16)) found = true;  // (the two ends cannot meet)
                else if (longer) tasks[cap - 1 - at] = make_uint4(v, a, e - a, i);
                else tasks[at] = make_uint4(v, e - a == 1 ? x : a, (e - a) << 6 | i, 0);
            }
            got |= static_cast<uint64_t>(__ballot_sync(kFull, found)) << (32 * h);
        }
        if (lane == 0) need[v] = got;
    }
}

// All blocks of a cooperative launch meet; false when the wait limit ran out.
SKIM_DEV bool grid_meet(DevCtl *ctl, unsigned round, uint64_t timeout_ns) {
    __shared__ int s_ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(&ctl->b.bar, 1u);
        const unsigned want = (round + 1) * gridDim.x;
        const uint64_t t0 = globaltimer();
        int ok = 1;
        while (*reinterpret_cast<volatile unsigned *>(&ctl->b.bar) < want) {
            if (globaltimer() - t0 > timeout_ns) {
                ctl->b.failed = 1;  // (err is cleared before the next search)
                ok = 0;
                break;
            }
            __nanosleep(100);
        }
        __threadfence();
        s_ok = ok;
    }
    __syncthreads();
    return s_ok != 0;
}

// Least fixed point of need over the tasks: a task's bit is set once one of
// its row's nodes has it.  Two sweeps over the tasks, a thread each, find most
// (long rows: a warp each, in the second); chains are up to 75 pairs long, so
// what the second sweep sets is followed along the rows of live out-neighbours,
// a level at a time, instead of looking at every task again.  One block per SM:
// with eight a barrier took 50 us.  A word that another thread is adding bits to only changes who sees
// them first.
constexpr unsigned kNeedPulls = 2;
constexpr int kSweepThreads = 1024;
constexpr uint32_t kSweepLong = 256;  // entries from which a row is swept by the block, and rows it keeps
__global__ void __launch_bounds__(kSweepThreads) k_need_sweep(BuildNode g, uint64_t *need, uint4 *tasks, uint32_t *wl0,
                                                    uint32_t *wl1, uint32_t cap, DevCtl *ctl, uint64_t timeout_ns) {
    __shared__ uint4 s_long[kSweepLong];
    __shared__ uint32_t s_n;
    const uint32_t nt = min(ctl->b.n_task, cap - cap / 16), nlong = min(ctl->b.n_long, cap / 16);
    const uint32_t lane = threadIdx.x & 31;
    if (threadIdx.x == 0) s_n = 0;
    if (blockIdx.x == 0 && threadIdx.x == 0) {  // what this pass has seen
        ctl->b.n_full_last = ctl->b.n_full;
        ctl->b.n_open_last = ctl->b.n_open;
    }
    if (nt + nlong == 0) return;
    const uint32_t step = gridDim.x * blockDim.x;
    unsigned round = 0;
    for (; round < kNeedPulls; round++) {
        const bool last = round + 1 == kNeedPulls;
        bool any = false;
        for (uint32_t q0 = blockIdx.x * blockDim.x; q0 < nt; q0 += step) {
            const uint32_t q = q0 + threadIdx.x;
            const uint4 t = q < nt ? tasks[q] : make_uint4(0, 0, 0, 0);
            const uint32_t i = t.z & 63u, n = t.z >> 6;
            bool found = false;
            if (n == 1) found = (__ldcg(&need[t.y]) >> i) & 1ull;
            else
                for (uint32_t z = 0; z < n && !found; z++) found = (__ldcg(&need[g.rlive[t.y + z]]) >> i) & 1ull;
            if (found) {
                atomicOr(reinterpret_cast<unsigned long long *>(&need[t.x]), 1ull << i);
                tasks[q].z = 0;
                any = true;
            }
            if (last) {
                const unsigned fb = __ballot_sync(kFull, found);
                unsigned at = 0;
                if (fb && lane == 0) at = atomicAdd(&ctl->b.wl[0], static_cast<unsigned>(__popc(fb)));
                at = __shfl_sync(kFull, at, 0);
                if (found) wl0[at + __popc(fb & lanemask_lt())] = t.x * g.l + i;
            }
        }
        if (last)
            for (uint32_t q = (blockIdx.x * blockDim.x + threadIdx.x) / 32; q < nlong; q += step / 32) {
                const uint4 t = tasks[cap - 1 - q];
                bool found = false;
                for (uint32_t z = 0; z < t.z && !found; z += 32) {
                    const bool f = z + lane < t.z && ((__ldcg(&need[g.rlive[t.y + z + lane]]) >> t.w) & 1ull);
                    found = __any_sync(kFull, f);
                }
                if (!found) continue;
                if (lane == 0) {
                    atomicOr(reinterpret_cast<unsigned long long *>(&need[t.x]), 1ull << t.w);
                    wl0[atomicAdd(&ctl->b.wl[0], 1u)] = t.x * g.l + t.w;
                }
                any = true;
            }
        if (any) *reinterpret_cast<volatile unsigned *>(&ctl->b.changed[round]) = 1;
        if (!grid_meet(ctl, round, timeout_ns)) return;
        if ((last || nlong == 0) && !*reinterpret_cast<volatile unsigned *>(&ctl->b.changed[round])) return;
    }
    for (unsigned level = 0;; level++, round++) {
        const uint32_t np = *reinterpret_cast<volatile unsigned *>(&ctl->b.wl[level % 3]);
        if (np == 0) return;
        const uint32_t *from = level & 1 ? wl1 : wl0;
        uint32_t *to = level & 1 ? wl0 : wl1;
        unsigned *n_to = &ctl->b.wl[(level + 1) % 3];
        if (blockIdx.x == 0 && threadIdx.x == 0) ctl->b.wl[(level + 2) % 3] = 0;
        const auto reach = [&](bool in, uint32_t w, uint32_t i) {
            bool fresh = false;
            if (in) {
                const uint64_t nd = __ldcg(&need[w]), sc = g.scc ? g.scc[w] : 0;
                if (!(((nd | sc) >> i) & 1ull))
                    fresh = !((atomicOr(reinterpret_cast<unsigned long long *>(&need[w]), 1ull << i) >> i) & 1ull);
            }
            const unsigned fb = __ballot_sync(kFull, fresh);
            if (!fb) return;
            unsigned at = 0;
            if (lane == 0) at = atomicAdd(n_to, static_cast<unsigned>(__popc(fb)));
            at = __shfl_sync(kFull, at, 0);
            if (fresh) to[at + __popc(fb & lanemask_lt())] = w * g.l + i;
        };
        // few pairs: one or a few per warp, so that their rows are walked at once
        const uint32_t warps = step / 32, per = min(32u, (np + warps - 1) / warps);
        for (uint32_t q0 = (blockIdx.x * blockDim.x + threadIdx.x) / 32 * per; q0 < np; q0 += warps * per) {
            uint32_t a = 0, len = 0, i = 0;
            if (lane < per && q0 + lane < np) {
                const uint32_t p = __ldcg(&from[q0 + lane]);
                a = g.foff[p];
                len = g.foff[p + 1ull] - a;
                i = p % g.l;
            }
            unsigned big = __ballot_sync(kFull, len >= 32);
            while (big) {
                const int s = __ffs(big) - 1;
                big &= big - 1;
                const uint32_t ba = __shfl_sync(kFull, a, s), bn = __shfl_sync(kFull, len, s);
                const uint32_t bi = __shfl_sync(kFull, i, s);
                uint32_t q = kSweepLong;
                if (bn >= kSweepLong) {  // the block together, below
                    if (lane == 0) q = atomicAdd(&s_n, 1u);
                    q = __shfl_sync(kFull, q, 0);
                    if (q < kSweepLong && lane == 0) s_long[q] = make_uint4(ba, bn, bi, 0);
                }
                if (q >= kSweepLong)
                    for (uint32_t z = lane; z < bn + lane; z += 32) reach(z < bn, z < bn ? g.flive[ba + z] : 0, bi);
            }
            const uint32_t c = len < 32 ? len : 0;
            uint32_t incl = c;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(kFull, incl, o);
                if (lane >= static_cast<uint32_t>(o)) incl += y;
            }
            const uint32_t total = __shfl_sync(kFull, incl, 31), first = a - (incl - c);
            for (uint32_t x = 0; x < total; x += 32) {
                const uint32_t o = x + lane;
                uint32_t sl = 0;  // owner: the first lane whose inclusive count exceeds o
#pragma unroll
                for (uint32_t st = 16; st > 0; st >>= 1) {
                    const uint32_t v = __shfl_sync(kFull, incl, sl + st - 1);
                    if (v <= o) sl += st;
                }
                const uint32_t sb = __shfl_sync(kFull, first, sl), si = __shfl_sync(kFull, i, sl);
                reach(o < total, o < total ? g.flive[sb + o] : 0, si);
            }
        }
        __syncthreads();
        const uint32_t nl = min(s_n, kSweepLong);
        for (uint32_t q = 0; q < nl; q++)
            for (uint32_t z = threadIdx.x - lane; z < s_long[q].y; z += kSweepThreads)
                reach(z + lane < s_long[q].y, z + lane < s_long[q].y ? g.flive[s_long[q].x + z + lane] : 0, s_long[q].z);
        __syncthreads();
        if (threadIdx.x == 0) s_n = 0;
        if (!grid_meet(ctl, round, timeout_ns)) return;
    }
}

// Open hit lists: closed ones are flagged, the masks per graph and their
// number written.  One block.
__global__ void k_need_open(uint32_t k, uint32_t graphs, uint32_t *tlen, uint64_t *topen, DevCtl *ctl) {
    if (threadIdx.x == 0) ctl->b.n_open = 0;
    __syncthreads();
    for (uint32_t g = threadIdx.x; g < graphs; g += blockDim.x) {
        uint64_t o = topen[g];
        for (uint64_t m = o; m; m &= m - 1) {
            const uint32_t i = __ffsll(m) - 1;
            if ((tlen[g * 64 + i] & ~kRowDone) >= k) {
                tlen[g * 64 + i] = k | kRowDone;
                o &= ~(1ull << i);
            }
        }
        topen[g] = o;
        if (o) atomicAdd(&ctl->b.n_open, static_cast<unsigned>(__popcll(o)));
    }
}

// ---- contracted components -----------------------------------------------------

// Per graph and instance the node with the largest product of live in- and
// out-degree (a member of the largest component where there is a large one).
// `per` blocks a graph, the graphs in steps of the grid (a batch may have more than
// any grid dimension holds).
__global__ void __launch_bounds__(256) k_pivots(BuildNode g, uint32_t per, unsigned long long *best) {
    const uint32_t lane = threadIdx.x & 31, part = blockIdx.x % per;
    for (uint32_t q = blockIdx.x / per; q < g.graphs; q += gridDim.x / per) {
        const uint32_t v0 = g.graphs == 1 ? 0 : g.node_off[q], v1 = g.graphs == 1 ? g.n : g.node_off[q + 1];
        unsigned long long b[2] = {0, 0};
        for (uint32_t v = v0 + ((part * blockDim.x + threadIdx.x) >> 5); v < v1; v += (per * blockDim.x) >> 5) {
            const uint64_t ne = g.nonempty[v];
#pragma unroll
            for (uint32_t h = 0; h < 2; h++) {
                const uint32_t i = lane + 32 * h;
                uint64_t d = 0;
                if ((ne >> i) & 1ull) {
                    const uint64_t r = static_cast<uint64_t>(v) * g.l + i;
                    d = static_cast<uint64_t>(g.loff[r + 1] - g.loff[r]) * (g.foff[r + 1] - g.foff[r]);
                }
                const unsigned long long x =
                    static_cast<unsigned long long>(d < 0xFFFFFFFFu ? d : 0xFFFFFFFFu) << 32 | (0xFFFFFFFFu - v);
                b[h] = max(b[h], x);
            }
        }
#pragma unroll
        for (uint32_t h = 0; h < 2; h++)
            if (lane + 32 * h < g.l && b[h]) atomicMax(&best[q * 64ull + lane + 32 * h], b[h]);
    }
}

__global__ void k_pivot_nodes(const unsigned long long *best, uint32_t count, uint32_t *pivot) {
    for (uint32_t q = blockIdx.x * blockDim.x + threadIdx.x; q < count; q += gridDim.x * blockDim.x)
        pivot[q] = 0xFFFFFFFFu - static_cast<uint32_t>(best[q]);
}

// The component of the pivot in instance i is what it reaches and is reached
// by.  Instances where a rank saves fewer than kGiantVisits visits on average
// (down / n of the ranks hit the component, each would visit `up` nodes; graphs
// of a batch taken as equal) keep plain searches.
constexpr uint64_t kGiantVisits = 8;
__global__ void k_components(uint32_t n, uint32_t l, uint32_t graphs, uint64_t *down, uint64_t *up,
                             const uint32_t *ndown, const uint32_t *nup, uint64_t *topen, DevCtl *ctl) {
    __shared__ uint64_t s_ok;
    if (threadIdx.x == 0) {
        uint64_t ok = 0;
        for (uint32_t i = 0; i < l; i++)
            if (static_cast<uint64_t>(ndown[i]) * nup[i] >= kGiantVisits * n * graphs) ok |= 1ull << i;
        s_ok = ok;
        if (blockIdx.x == 0) ctl->b.n_open = static_cast<unsigned>(__popcll(s_ok)) * graphs;
    }
    __syncthreads();
    for (uint32_t q = blockIdx.x * blockDim.x + threadIdx.x; q < graphs; q += gridDim.x * blockDim.x) topen[q] = s_ok;
    for (uint32_t v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x) {
        const uint64_t u = up[v] & s_ok;
        up[v] = u;
        down[v] &= u;  // now the component itself
    }
}

// The lanes that hit a component whose list is open leave a record of the
// list: (graph * 64 + instance) << lbits | lane.
__global__ void k_hit_records(BuildNode g, const uint32_t *hit, const uint32_t *pair, uint32_t B, uint32_t lbits,
                              uint64_t *rec, DevCtl *ctl) {
    const uint32_t words = (B + 31) / 32;
    for (uint32_t w = blockIdx.x * blockDim.x + threadIdx.x; w < words; w += gridDim.x * blockDim.x)
        for (uint32_t x = hit[w]; x; x &= x - 1) {
            const uint32_t ln = w * 32 + __ffs(x) - 1, pr = pair[ln], u = pr / g.l;
            const uint32_t q = graph_of(g.node_off, g.graphs, u) * 64 + (pr - u * g.l);
            if (g.tlen[q] & kRowDone) continue;
            rec[atomicAdd(&ctl->b.n_hit, 1u)] = static_cast<uint64_t>(q) << lbits | ln;
        }
}

// A warp per hit list: ascending.
__global__ void __launch_bounds__(128) k_hit_rows(uint32_t lists, uint32_t l, uint32_t k, const uint32_t *tlen,
                                                  uint64_t *hits) {
    __shared__ uint64_t s_a[4][256];
    uint64_t *a = s_a[threadIdx.x >> 5];
    const uint32_t lane = threadIdx.x & 31;
    for (uint32_t q = blockIdx.x * 4 + (threadIdx.x >> 5); q < lists; q += gridDim.x * 4) {
        const uint32_t n = (q & 63) < l ? min(tlen[q] & ~kRowDone, k) : 0;
        if (n < 2) continue;
        uint64_t *row = hits + static_cast<uint64_t>(q) * k;
        const uint32_t P = pow2_from64(n);
        __syncwarp();
        for (uint32_t j = lane; j < P; j += 32) a[j] = j < n ? row[j] : ~0ull;
        warp_sort(a, P);
        for (uint32_t j = lane; j < n; j += 32) row[j] = a[j];
    }
}

// A block per list i of a graph, in steps of the grid: places of the list's entries in
// the graph's rank order of all hits, out[graph][place], and per instance the bitmap
// of its places.
__global__ void k_hits_sort(const uint64_t *hits, const uint32_t *tlen, uint32_t graphs, uint32_t l, uint32_t k,
                            uint64_t *out, uint64_t *places, uint32_t *total) {
    __shared__ uint32_t s_cnt[64];
    const uint32_t words = (l * k + 63) / 64;
    for (uint64_t b = blockIdx.x; b < static_cast<uint64_t>(graphs) * l; b += gridDim.x) {
        const uint64_t g = b / l;
        const uint32_t i = static_cast<uint32_t>(b - g * l);
        __syncthreads();  // (the counts of the list before have been used)
        if (threadIdx.x < 64) s_cnt[threadIdx.x] = threadIdx.x < l ? min(tlen[g * 64 + threadIdx.x] & ~kRowDone, k) : 0;
        const uint64_t *h = hits + g * 64 * k;
        uint64_t *bits = places + (g * 64 + i) * words;
        for (uint32_t w = threadIdx.x; w < words; w += blockDim.x) bits[w] = 0;
        __syncthreads();
        for (uint32_t q = threadIdx.x; q < s_cnt[i]; q += blockDim.x) {
            const uint64_t x = h[static_cast<uint64_t>(i) * k + q];
            uint32_t at = q;
            for (uint32_t o = 0; o < l; o++) {  // entries of the other (ascending) lists below x
                if (o == i) continue;
                uint32_t lo = 0, hi = s_cnt[o];
                while (lo < hi) {
                    const uint32_t mid = (lo + hi) >> 1;
                    if (h[static_cast<uint64_t>(o) * k + mid] < x) lo = mid + 1;
                    else hi = mid;
                }
                at += lo;
            }
            out[g * l * k + at] = x;
            atomicOr(reinterpret_cast<unsigned long long *>(&bits[at >> 6]), 1ull << (at & 63));
        }
        if (i == 0 && threadIdx.x == 0) {
            uint32_t t = 0;
            for (uint32_t o = 0; o < l; o++) t += s_cnt[o];
            total[g] = t;
        }
    }
}

// ---- the sketches ----------------------------------------------------------------

SKIM_DEV void sort_regs(uint64_t &x0, uint64_t &x1, bool two) {
    const uint32_t lane = threadIdx.x & 31;
#pragma unroll
    for (uint32_t kk = 2; kk <= 64; kk <<= 1) {
        if (kk == 64 && !two) break;
#pragma unroll
        for (uint32_t j = kk >> 1; j > 0; j >>= 1) {
            if (j == 32) {
                const uint64_t lo = min(x0, x1), hi = max(x0, x1);
                x0 = lo;
                x1 = hi;
            } else {
                const uint64_t y0 = __shfl_xor_sync(kFull, x0, j);
                const bool lower = (lane & j) == 0;
                const bool up0 = (lane & kk) == 0 || kk == 64 || (!two && kk == 32);
                x0 = (lower == up0) ? min(x0, y0) : max(x0, y0);
                if (two) {
                    const uint64_t y1 = __shfl_xor_sync(kFull, x1, j);
                    const bool up1 = kk == 64 || (kk < 32 && (lane & kk) == 0);
                    x1 = (lower == up1) ? min(x1, y1) : max(x1, y1);
                }
            }
        }
    }
}

SKIM_DEV uint32_t count_below(const uint64_t *a, uint32_t n, uint64_t x) {
    uint32_t lo = 0, hi = n;
    while (lo < hi) {
        const uint32_t mid = (lo + hi) >> 1;
        if (a[mid] < x) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

// Warp-collective: the `most` smallest of two ascending arrays without common
// elements, in order, to out; returns how many.
SKIM_DEV uint32_t merge_two(const uint64_t *a, uint32_t na, const uint64_t *b, uint32_t nb, uint64_t *out,
                            uint32_t most) {
    const uint32_t lane = threadIdx.x & 31;
    for (uint32_t j = lane; j < na; j += 32) {
        const uint32_t at = j + count_below(b, nb, a[j]);
        if (at < most) out[at] = a[j];
    }
    for (uint32_t j = lane; j < nb; j += 32) {
        const uint32_t at = j + count_below(a, na, b[j]);
        if (at < most) out[at] = b[j];
    }
    __syncwarp();
    return min(na + nb, most);
}

// A warp per node: X_v = the k smallest of its row (found by the searches), its
// own ranks and the hit lists of the components that it reaches, ascending,
// zeros behind; rows of up to 64 ranks and the own ranks are sorted in
// registers.
constexpr uint32_t kMergeWarps = 8;
template <uint32_t CAP>  // at least k and 64
struct MergeMem {
    uint64_t own[64], row[CAP], hits[CAP], out[CAP];
    uint32_t off[65];
};

// Warp-collective: those of the node's own ranks that are below `bound` (or
// all), in order, to M.own; returns how many.  They are uniform hashes, so where many
// are below it their top six bits put about one in each of 64 buckets, and
// inside a bucket each counts the smaller ones; a few count among themselves.
template <class MM>
SKIM_DEV uint32_t sort_own(MM &M, const OwnRanks &own, uint32_t v, bool all, uint64_t bound) {
    const uint32_t lane = threadIdx.x & 31;
    const uint64_t x0 = lane < own.l ? own.rank(v, lane) : 0, x1 = lane + 32 < own.l ? own.rank(v, lane + 32) : 0;
    const bool in0 = lane < own.l && (all || x0 < bound), in1 = lane + 32 < own.l && (all || x1 < bound);
    const unsigned ib0 = __ballot_sync(kFull, in0), ib1 = __ballot_sync(kFull, in1);
    const uint32_t n0 = __popc(ib0), n = n0 + __popc(ib1);
    if (n == 0) return 0;
    uint64_t *st = M.hits;  // free until the hits are gathered
    __syncwarp();
    if (n <= 16) {
        if (in0) st[__popc(ib0 & lanemask_lt())] = x0;
        if (in1) st[n0 + __popc(ib1 & lanemask_lt())] = x1;
        __syncwarp();
        if (lane < n) {
            const uint64_t x = st[lane];
            uint32_t at = 0;
            for (uint32_t q = 0; q < n; q++) at += st[q] < x;
            M.own[at] = x;
        }
        __syncwarp();
        return n;
    }
    const uint32_t b0 = static_cast<uint32_t>(x0 >> 58), b1 = static_cast<uint32_t>(x1 >> 58);
    M.off[lane] = M.off[lane + 32] = 0;
    __syncwarp();
    uint32_t p0 = 0, p1 = 0;
    if (in0) p0 = atomicAdd(&M.off[b0], 1u);
    if (in1) p1 = atomicAdd(&M.off[b1], 1u);
    __syncwarp();
    const uint32_t c0 = M.off[2 * lane], c1 = M.off[2 * lane + 1];
    uint32_t incl = c0 + c1;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(kFull, incl, o);
        if (lane >= static_cast<uint32_t>(o)) incl += y;
    }
    M.off[2 * lane] = incl - c0 - c1;
    M.off[2 * lane + 1] = incl - c1;
    if (lane == 31) M.off[64] = incl;
    __syncwarp();
    const uint32_t s0 = M.off[b0], s1 = M.off[b1];
    if (in0) st[s0 + p0] = x0;
    if (in1) st[s1 + p1] = x1;
    __syncwarp();
    if (in0) {
        uint32_t at = s0;
        for (uint32_t q = s0; q < M.off[b0 + 1]; q++) at += st[q] < x0;
        M.own[at] = x0;
    }
    if (in1) {
        uint32_t at = s1;
        for (uint32_t q = s1; q < M.off[b1 + 1]; q++) at += st[q] < x1;
        M.own[at] = x1;
    }
    __syncwarp();
    return n;
}

template <uint32_t CAP>
__global__ void __launch_bounds__(kMergeWarps * 32) k_merge(BuildNode g, const uint64_t *hits, const uint64_t *places,
                                                            const uint32_t *total, uint64_t *X, DevCtl *ctl) {
    extern __shared__ uint4 s_mem[];
    MergeMem<CAP> &M = reinterpret_cast<MergeMem<CAP> *>(s_mem)[threadIdx.x >> 5];
    const uint32_t lane = threadIdx.x & 31, k = g.k;
    const OwnRanks own{g.rank_key, g.rbase, g.own ? g.l : 0};
    unsigned long long ins = 0;
    for (uint32_t v = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; v < g.n; v += (gridDim.x * blockDim.x) >> 5) {
        uint64_t *row = X + static_cast<uint64_t>(v) * k;
        const uint32_t nr = min(g.len[v] & ~(kRowDone | kRowListed), k);
        const uint64_t reach = g.up ? g.up[v] : 0;
        __syncwarp();
        if (nr) {
            if (nr <= 64) {
                uint64_t x0 = lane < nr ? row[lane] : ~0ull, x1 = lane + 32 < nr ? row[lane + 32] : ~0ull;
                sort_regs(x0, x1, nr > 32);
                M.row[lane] = x0;
                M.row[lane + 32] = x1;
            } else {
                const uint32_t P = pow2_from64(nr);
                for (uint32_t j = lane; j < P; j += 32) M.row[j] = j < nr ? row[j] : ~0ull;
                warp_sort(M.row, P);
            }
        }
        __syncwarp();
        const uint64_t *res = M.row;
        uint32_t m = nr;
        uint64_t *spare = M.out;
        if (reach) {
            // the first k hits of the node's components: the union of their
            // bitmaps of places, 32 words at a time
            const uint32_t gr = graph_of(g.node_off, g.graphs, v), words = (g.l * k + 63) / 64;
            const uint64_t *p = places + static_cast<uint64_t>(gr) * 64 * words;
            const uint64_t *h = hits + static_cast<uint64_t>(gr) * g.l * k;
            const uint32_t used = (total[gr] + 63) / 64;
            uint32_t nh = 0;
            for (uint32_t w0 = 0; w0 < used && nh < k; w0 += 32) {
                const uint32_t w = w0 + lane;
                uint64_t u = 0;
                if (w < used)
                    for (uint64_t x = reach; x; x &= x - 1) u |= p[(__ffsll(x) - 1) * words + w];
                uint32_t incl = __popcll(u);
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t y = __shfl_up_sync(kFull, incl, o);
                    if (lane >= static_cast<uint32_t>(o)) incl += y;
                }
                uint32_t at = nh + incl - __popcll(u);
                for (; u && at < k; u &= u - 1, at++) M.hits[at] = h[w * 64 + (__ffsll(u) - 1)];
                nh = min(k, nh + __shfl_sync(kFull, incl, 31));
            }
            __syncwarp();
            // without those that the node holds already
            uint32_t kept = 0;
            for (uint32_t j0 = 0; j0 < nh; j0 += 32) {
                const uint64_t x = j0 + lane < nh ? M.hits[j0 + lane] : 0;
                bool take = j0 + lane < nh;
                if (take) {
                    const uint32_t at = count_below(res, m, x);
                    take = at < m ? res[at] != x : m < k;
                }
                const unsigned tb = __ballot_sync(kFull, take);
                if (take) M.hits[kept + __popc(tb & lanemask_lt())] = x;
                kept += __popc(tb);
                __syncwarp();
            }
            if (kept && m) {
                m = merge_two(res, m, M.hits, kept, spare, k);
                res = spare;
                spare = M.row;
            } else if (kept) {
                m = kept;
                res = M.hits;
                spare = M.row;
            }
        }
        // own ranks (a hit may be one of them)
        if (own.l) {
            if (res == M.hits) {  // sort_own's scratch
                for (uint32_t j = lane; j < m; j += 32) M.out[j] = M.hits[j];
                __syncwarp();
                res = M.out;
            }
            uint32_t no = sort_own(M, own, v, m < k, m < k ? 0 : res[k - 1]);
            if (reach && no) {
                uint32_t kept = 0;
                for (uint32_t j0 = 0; j0 < no; j0 += 32) {
                    const uint64_t x = j0 + lane < no ? M.own[j0 + lane] : 0;
                    bool take = j0 + lane < no;
                    if (take) {
                        const uint32_t at = count_below(res, m, x);
                        take = !(at < m && res[at] == x);
                    }
                    const unsigned tb = __ballot_sync(kFull, take);
                    if (take) M.own[kept + __popc(tb & lanemask_lt())] = x;
                    kept += __popc(tb);
                    __syncwarp();
                }
                no = kept;
            }
            if (no && m) {
                m = merge_two(res, m, M.own, no, spare, k);
                res = spare;
            } else if (no) {
                m = min(no, k);
                res = M.own;
            }
        }
        for (uint32_t j = lane; j < k; j += 32) row[j] = j < m ? res[j] : 0;
        if (lane == 0) {
            g.len[v] = m;
            ins += m;
        }
    }
    warp_add(&ctl->stats[kStInsert], ins);
}

template <class KT, bool SCC>
cudaError_t search_launch(const BuildArgs &a, cudaStream_t s) {
    const size_t smem = sizeof(WarpMem<KT>) * (kSearchThreads / 32);
    cudaError_t e = cudaFuncSetAttribute(k_build_search<KT, SCC>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         static_cast<int>(smem));
    if (e != cudaSuccess) return e;
    int per = 0, dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_build_search<KT, SCC>, kSearchThreads, smem);
    if (e != cudaSuccess) return e;
    const uint64_t want = (static_cast<uint64_t>(a.B) + kIds * 8 - 1) / (kIds * 8);
    note_launch();
    k_build_search<KT, SCC><<<static_cast<unsigned>(std::min<uint64_t>(want, static_cast<uint64_t>(sms) * per)),
                              kSearchThreads, smem, s>>>(a);
    return cudaGetLastError();
}

}  // namespace

// A (node, lane id) key has 32 bits while node ids leave kIdBits of them.
cudaError_t launch_build_search(const BuildArgs &a, cudaStream_t s) {
    if (a.n < (1u << (32 - kIdBits)))
        return a.scc ? search_launch<uint32_t, true>(a, s) : search_launch<uint32_t, false>(a, s);
    return a.scc ? search_launch<unsigned long long, true>(a, s) : search_launch<unsigned long long, false>(a, s);
}

cudaError_t launch_deferred_lanes(uint32_t *deflist, uint32_t D, bool all, const uint32_t *pair, uint32_t l,
                                  uint32_t *defpair, uint8_t *lane_inst, cudaStream_t s) {
    note_launch();
    k_deferred_lanes<<<grid_for(D, 256), 256, 0, s>>>(deflist, D, all, pair, l, defpair, lane_inst);
    return cudaGetLastError();
}

cudaError_t launch_append(const uint64_t *rec, uint64_t r0, uint64_t r1, uint32_t lbits, const uint32_t *defbits,
                          const uint64_t *lane_rank, uint32_t k, uint32_t *len, uint64_t *X, const BuildScratch &b,
                          DevCtl *ctl, cudaStream_t s) {
    if (r0 >= r1) return cudaSuccess;
    note_launch();
    k_append<<<grid_for(r1 - r0, 256), 256, 0, s>>>(rec, r0, r1, lbits, defbits, lane_rank, k, len, X, b.over_key,
                                                    b.over_pos, b.list, ctl, nullptr);
    return cudaGetLastError();
}

cudaError_t launch_count_words(const uint32_t *rec_val, uint64_t R, const uint64_t *hvals, uint32_t *cnt,
                               cudaStream_t s) {
    note_launch();
    k_count_words<<<grid_for(R, kWordChunk, 152 * 4), kWordChunk, 0, s>>>(rec_val, R, hvals, cnt);
    return cudaGetLastError();
}

cudaError_t launch_append_words(const uint64_t *rec, const uint32_t *rec_val, uint64_t R, uint32_t tbits,
                                const uint64_t *hvals, const uint32_t *pair, uint32_t l, int own, uint32_t lbits,
                                const uint64_t *lane_rank, uint32_t k, uint32_t *len, uint64_t *X,
                                const BuildScratch &b, DevCtl *ctl, cudaStream_t s) {
    if (R == 0) return cudaSuccess;
    note_launch();
    k_append_words<<<grid_for(R, 128), 128, 0, s>>>(rec, rec_val, R, tbits, hvals, pair, l, own, lbits,
                                                    lane_rank, k, len, X, b.over_key, b.over_pos, b.list, ctl);
    return cudaGetLastError();
}

cudaError_t launch_overflow(uint64_t R, uint32_t lbits, const uint64_t *lane_rank, uint32_t k, uint32_t *len,
                            uint64_t *X, bool done, const BuildScratch &b, DevCtl *ctl, cudaStream_t s) {
    if (R == 0) return cudaSuccess;
    note_launch();
    k_over_alloc<<<grid_for(R, 256, 152 * 2), 256, 0, s>>>(b.list, len, k, b.seg, ctl);
    note_launch();
    k_over_scatter<<<grid_for(R, 256, 152 * 8), 256, 0, s>>>(b.over_key, b.over_pos, lbits, lane_rank, b.seg, b.buf,
                                                             ctl);
    note_launch();
    k_over_select<<<grid_for(R, kSelWarps, 152 * 12), kSelWarps * 32, 0, s>>>(b.list, k, len, b.seg, b.buf, X,
                                                                               done ? kRowDone : 0, ctl);
    return cudaGetLastError();
}

cudaError_t launch_need_start(uint64_t *need, uint32_t n, uint64_t lmask, cudaStream_t s) {
    note_launch();
    k_fill_u64<<<grid_for(n, 256), 256, 0, s>>>(need, n, lmask);
    return cudaGetLastError();
}

cudaError_t launch_need(const BuildNode &g, const uint64_t *next, uint64_t *need, uint32_t *full_list, void *scratch,
                        uint64_t scratch_bytes, DevCtl *ctl, uint64_t timeout_ns, cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(&ctl->b.n_task, 0, 9 * sizeof(unsigned), s);  // n_task .. wl
    if (e != cudaSuccess) return e;
    uint32_t task_cap = static_cast<uint32_t>(std::min<uint64_t>(scratch_bytes / 24, 0xFFFFFFFFu));
    uint4 *tasks = static_cast<uint4 *>(scratch);
    uint32_t *wl0 = reinterpret_cast<uint32_t *>(tasks + task_cap), *wl1 = wl0 + task_cap;
    note_launch();
    k_need_full<<<grid_for(g.n, 256), 256, 0, s>>>(g, next, full_list, ctl);
    note_launch();
    k_need_tasks<<<grid_for(static_cast<size_t>(g.n) * 32, 256, 152 * 8), 256, 0, s>>>(g, need, full_list, tasks,
                                                                                       task_cap, ctl);
    int dev = 0, sms = 0, per = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_need_sweep, kSweepThreads, 0);  // all blocks resident at once
    if (e != cudaSuccess) return e;
    const unsigned grid = std::min<unsigned>(grid_for(g.n, 64), static_cast<unsigned>(sms) * std::min(per, 1));
    // between two barriers a warp walks a row 32 entries at a time, a thread the tasks in steps of the grid
    timeout_ns = phase_limit(timeout_ns, 1 + g.n / 32 + static_cast<uint64_t>(g.n) * g.l / kSweepThreads);
    note_launch();
    void *args[] = {const_cast<BuildNode *>(&g), &need, &tasks, &wl0, &wl1, &task_cap, &ctl, &timeout_ns};
    return cudaLaunchCooperativeKernel(reinterpret_cast<void *>(k_need_sweep), dim3(grid), dim3(kSweepThreads), args, 0, s);
}

cudaError_t launch_pivots(const BuildNode &g, unsigned long long *best, uint32_t *pivot, cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(best, 0, g.graphs * 64ull * sizeof(unsigned long long), s);
    if (e != cudaSuccess) return e;
    const unsigned per = grid_for(static_cast<size_t>(g.n) * 32 / g.graphs + 1, 256, std::max(1u, 152 * 8 / g.graphs));
    note_launch();
    k_pivots<<<per * std::min(g.graphs, 152u * 32), 256, 0, s>>>(g, per, best);
    note_launch();
    k_pivot_nodes<<<grid_for(g.graphs * 64, 256), 256, 0, s>>>(best, g.graphs * 64, pivot);
    return cudaGetLastError();
}

cudaError_t launch_components(const BuildNode &g, uint64_t *down, uint64_t *up, const uint32_t *ndown,
                              const uint32_t *nup, DevCtl *ctl, cudaStream_t s) {
    note_launch();
    k_components<<<grid_for(g.n, 256), 256, 0, s>>>(g.n, g.l, g.graphs, down, up, ndown, nup, g.topen, ctl);
    return cudaGetLastError();
}

cudaError_t launch_hits(const BuildNode &g, const uint32_t *hit, const uint32_t *pair, const uint64_t *lane_rank,
                        uint32_t B, uint32_t lbits, uint64_t *rec, uint64_t *hits, const BuildScratch &b, DevCtl *ctl,
                        cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(&ctl->b.n_over, 0, 4 * sizeof(unsigned), s);  // n_over, n_list, over_total, n_hit
    if (e != cudaSuccess) return e;
    note_launch();
    k_hit_records<<<grid_for(B / 32 + 1, 128), 128, 0, s>>>(g, hit, pair, B, lbits, rec, ctl);
    note_launch();
    k_append<<<grid_for(B, 256, 152 * 4), 256, 0, s>>>(rec, 0, 0, lbits, nullptr, lane_rank, g.k, g.tlen, hits,
                                                       b.over_key, b.over_pos, b.list, ctl, &ctl->b.n_hit);
    e = launch_overflow(B, lbits, lane_rank, g.k, g.tlen, hits, true, b, ctl, s);
    if (e != cudaSuccess) return e;
    note_launch();
    k_need_open<<<1, 256, 0, s>>>(g.k, g.graphs, g.tlen, g.topen, ctl);
    return cudaGetLastError();
}

cudaError_t launch_merge(const BuildNode &g, uint64_t *X, uint64_t *hits, uint64_t *hits_sorted, uint64_t *places,
                         uint32_t *total, DevCtl *ctl, cudaStream_t s) {
    if (g.up) {
        note_launch();
        k_hit_rows<<<grid_for(g.graphs * 64, 4), 128, 0, s>>>(g.graphs * 64, g.l, g.k, g.tlen, hits);
        note_launch();
        k_hits_sort<<<grid_for(static_cast<size_t>(g.l) * g.graphs, 1), 256, 0, s>>>(hits, g.tlen, g.graphs, g.l, g.k,
                                                                                     hits_sorted, places, total);
    }
    const unsigned grid = grid_for(static_cast<size_t>(g.n) * 32, kMergeWarps * 32, 152 * 64);
    note_launch();
    if (g.k <= 64) {
        k_merge<64><<<grid, kMergeWarps * 32, sizeof(MergeMem<64>) * kMergeWarps, s>>>(g, hits_sorted, places, total, X,
                                                                                       ctl);
        return cudaGetLastError();
    }
    const size_t smem = sizeof(MergeMem<256>) * kMergeWarps;
    cudaError_t e = cudaFuncSetAttribute(k_merge<256>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         static_cast<int>(smem));
    if (e != cudaSuccess) return e;
    k_merge<256><<<grid, kMergeWarps * 32, smem, s>>>(g, hits_sorted, places, total, X, ctl);
    return cudaGetLastError();
}

}  // namespace skim
