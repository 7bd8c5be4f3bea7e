// query.cu -- influence oracle queries (Section 5.1, Eq. unionest).
//
// For a seed set S, every rank z of X_u minus {tau_u} (u in S) is charged
// 1/max{tau_u : z in X_u minus {tau_u}}; the sum estimates |union of R_u| and
// is divided by l.  tau_u is the k-th smallest rank of a full sketch and 1 for
// a sketch with fewer than k ranks (Eq. combinedthresh).
//
// A hash table per query keeps, per distinct z, the
// largest tau (as a 64-bit integer; the integer order equals the order of
// the reals h/2^64 and the rounding to double is monotone).  Each term 1/tau is
// formed in double exactly as h -> double -> scale by 2^-64 -> 1/x, then added
// exactly in 192-bit fixed point (64 fraction bits suffice: every term is >= 1
// with a 53-bit significand) and the total is rounded to double once, to
// nearest-even.  The result therefore does not depend on the order in which
// ranks are visited, and a query gives the same bits alone or in a batch.
// With permutation ranks (Sections 3.1, 3.2) a sketch holds positions and a
// threshold q becomes the term (n*l - 1)/q, or n/q in the IC model, each
// formed as one double division (terms are at least 1/k >= 2^-8, so 64
// fraction bits still hold them exactly).
#include <algorithm>
#include <cooperative_groups.h>

#include "internal.cuh"

namespace skim {

namespace {

constexpr int kQThreads = 512;

struct U192 {
    uint64_t w[3];
};

SKIM_DEV void add192(U192 &a, const U192 &b) {
    uint64_t s0 = a.w[0] + b.w[0];
    uint64_t c0 = s0 < a.w[0];
    uint64_t s1 = a.w[1] + b.w[1];
    uint64_t c1 = s1 < a.w[1];
    s1 += c0;
    c1 |= (s1 < c0);
    a.w[0] = s0;
    a.w[1] = s1;
    a.w[2] = a.w[2] + b.w[2] + c1;
}

// term 1/tau for the integer threshold h (h = ~0 stands for tau = 1)
SKIM_DEV double inv_tau(uint64_t h) {
    double tau = ldexp(__ull2double_rn(h), -64);
    return 1.0 / tau;
}

// term of a threshold h under the context's rank reading (QueryTerms)
SKIM_DEV double term_of(const QueryTerms &t, uint64_t h) {
    if (t.mode == 0) return inv_tau(h);
    if (h == ~0ull) return t.mode == 2 ? 0.0 : 1.0;
    return t.num / __ull2double_rn(h);
}

// exact fixed-point image (value * 2^64) of a double in [2^-12, 2^64]
SKIM_DEV U192 to_fixed(double v) {
    const uint64_t bits = static_cast<uint64_t>(__double_as_longlong(v));
    const int e = static_cast<int>((bits >> 52) & 0x7ff) - 1023;
    const uint64_t mant = (bits & ((1ull << 52) - 1)) | (1ull << 52);
    const int sh = e + 12;  // value * 2^64 = mant * 2^(e - 52 + 64)
    const int q = sh >> 6, rb = sh & 63;
    const uint64_t lo = mant << rb, hi = rb ? mant >> (64 - rb) : 0;
    return U192{{q == 0 ? lo : 0, q == 0 ? hi : q == 1 ? lo : 0, q == 1 ? hi : q == 2 ? lo : 0}};
}

SKIM_DEV int top_bit(const U192 &a) {
    for (int i = 2; i >= 0; i--)
        if (a.w[i]) return i * 64 + 63 - __clzll(static_cast<long long>(a.w[i]));
    return -1;
}

SKIM_DEV uint64_t bit_at(const U192 &a, int p) { return (a.w[p >> 6] >> (p & 63)) & 1ull; }

SKIM_DEV bool any_below(const U192 &a, int p) {  // any bit set strictly below position p
    for (int i = 0; i < 3; i++) {
        int lo = i * 64;
        if (p <= lo) break;
        uint64_t m = (p - lo >= 64) ? ~0ull : ((1ull << (p - lo)) - 1);
        if (a.w[i] & m) return true;
    }
    return false;
}

// round (a * 2^-64) to the nearest double, ties to even
SKIM_DEV double fixed_to_double(const U192 &a) {
    int p = top_bit(a);
    if (p < 0) return 0.0;
    if (p <= 52) return ldexp(static_cast<double>(a.w[0]), -64);
    int sh = p - 52;
    const int w = sh >> 6, b = sh & 63;
    uint64_t mant = a.w[w] >> b;
    if (b && w + 1 < 3) mant |= a.w[w + 1] << (64 - b);
    mant &= (1ull << 53) - 1;
    bool rnd = bit_at(a, sh - 1);
    bool sticky = any_below(a, sh - 1);
    if (rnd && (sticky || (mant & 1ull))) {
        mant++;
        if (mant == (1ull << 53)) {
            mant >>= 1;
            sh++;
        }
    }
    return ldexp(static_cast<double>(mant), sh - 64);
}

// ---- hash tables of rank -> term -------------------------------------------------
//
// A slot holds a rank and the term of the threshold it is charged to, as the
// double's bits (all ones: empty).  Terms fall as thresholds rise, in every
// rank reading, so the largest threshold of equal ranks is the smallest term, and
// the order of non-negative doubles is that of their bits.  So the one division
// is made per seed, 32 at a time (FP64 runs at a thirty-second of the integer
// rate), and not per rank.
//
// The table is in shared memory.  A query of up to kSmallEntries ranks takes one
// block; a larger one is cut by the hash of the rank into parts of about
// kPartEntries, a block each: every block reads all of the query's sketches (from
// L2 after the first) and keeps the ranks of its part, so nothing is scattered
// through global memory, and the last block of a query adds the parts.  A part that
// does not fit its table is cut finer and read again.
//
// Measured: 1000 queries of 1 to 1000 seeds (145 K sketches of 64 ranks, R-MAT 20),
// kernels: 1.03 ms with a table per query in global memory (two arrays, two
// atomics per rank, a pass to clear and one to sum), 0.66 ms with 16-byte slots and
// terms per seed there (0.54 ms of it the atomics: 15 G/s, also where the tables
// stay in L2), 0.44 ms so (0.58 ms before a warp collected 32 ranks of its part).
//
// A single query is one kernel that has the seeds as arguments and writes the
// estimate to host memory (host to host: 48 -> 19 us for 10 seeds; before, four
// kernels, two uploads and two downloads).  Reading every sketch in every block is
// what it would wait for, so a larger one takes a cluster of 16 blocks whose
// warps share the seeds and put a rank into the table of the block that has its
// hash, through distributed shared memory: 64 ranks per sketch, 445 seeds 61 -> 32
// us, 1000 seeds 66 -> 40 us (clusters of 8: 66 us, of 4: 118 us; parts: 85 us).  So do the
// larger ones of a call with few of them, the small ones beside them in the same launch; a
// cluster of 4 does where it holds the whole query, and the chip has room for more of
// those.  Calls of 10, 32, 64, 128 queries of 1 to 1000 seeds, 16 ranks per sketch: parts
// 100, 110, 125, 130 us, clusters 55, 70, 74, 92 us (a table in global memory, four launches:
// 67, 75, 85, 102 us); 64 ranks, 10, 16, 32, 64 queries: parts 75, 84, 90, 95 us, clusters of 16 59, 69,
// then parts (four launches: 76, 86, 96, 126 us).  A batch fills the chip with parts and is
// slower with clusters (1000 queries, with copies: 0.52 ms; clusters of 4, 8, 16: 0.63,
// 0.76, 1.07 ms).  Both read a query once per part or round of clusters, so the
// largest have their table in global memory (in_memory; 9000 seeds of 64 ranks, clusters:
// 107 us).  One block is as fast as the cluster up to kOneEntries (100 seeds of 16 ranks:
// 28 us both; 43 seeds of 64: 30 and 29 us).

constexpr uint32_t kSmallEntries = 2700, kSmallSlots = 4095;  // 64 KB: three blocks per SM
// Threads of a small query's block: many while a call leaves room for them (host to host,
// 64 ranks per sketch, 1 to 42 seeds; 256, 512, 1024 threads: 10 queries 66, 57, 53 us, 152
// 69, 68, 62, 304 71, 71, 82, 608 91, 97, 114, 2000 174, 196, 273).
constexpr uint32_t kSmsUsual = 152;
constexpr int small_threads(uint32_t queries) {
    return queries <= kSmsUsual ? 1024 : queries <= 3 * kSmsUsual ? 512 : 256;
}
// Small queries go in one launch with the clusters of a few larger ones, in a block of
// 1024 threads each and one per SM, while they are few: with clusters of 4 up to
// kFewSmall, with clusters of 16, of which kClusterParts are resident at once, where all
// take one round more at most.  Else they take a launch of their own (as above, beside one
// larger query 152, 304, 608, 2000 small ones: 81, 108, 174, 438 us together, 96, 111, 116, 208 us
// apart; beside 7 150, 250 132, 158 and 127, 139 us, beside 10 60, 150 113, 135 and 139, 148).
constexpr uint32_t kFewSmall = 2 * kSmsUsual;
constexpr uint32_t kPartEntries = 8000, kPartSlots = 12287;  // 192 KB
constexpr int kPartThreads = 1024;
constexpr uint32_t kStage = 64;  // pairs a warp collects
constexpr uint32_t kOneEntries = 1500;
constexpr uint32_t kCluster = 16, kClusterSlots = kPartSlots, kBlockEntries = 7800;
constexpr uint32_t kClusterEntries = kCluster * kBlockEntries;
constexpr uint32_t kClusterFour = 4;
// larger queries of a call that take clusters of 16, the same if some do not fit four
// blocks, and those that take clusters of 4 if all do
constexpr uint32_t kFewLarge = 8, kFewLargest = 16, kMoreLarge = 64;
// Clusters of 16 that are resident at once (an eighth waits for another to end: 60000 seeds
// of 16 ranks 243 us with 8, 147 us with 7), and ranks per block that they take in a round,
// all distinct (0.8 of the slots).
constexpr uint32_t kClusterParts = 7, kBlockFill = 9800;
// Ranks above which the table is in global memory: what the resident clusters take in a
// round, or with long rows a little more, whose ranks meet on as few slots (20000 seeds of 64
// ranks, table 418 us, two rounds 329; 100000 of 16 191 and 398; 60000 of 32 265 and 497).
constexpr uint64_t kBlockMost = kClusterParts * kCluster * kBlockFill, kBlockMostLong = 1500000;
constexpr uint32_t kLongRanks = 64;
// Seeds above which a query alone has its table there too, with short rows and others:
// reading them is what a cluster waits for, and each reads all (k = 2, 100000 seeds 138 and
// 104 us, k = 4, 60000 122 and 105, k = 16, 60000 209 and 178).
constexpr uint32_t kTableSeedsShort = 25000, kTableSeeds = 50000, kShortRanks = 8;
constexpr uint32_t kTableBlocks = 152 * 2;

// (alone: the only query of its call)
bool in_memory(uint64_t seeds, uint32_t k, bool alone) {
    return seeds * (k - 1) > (k >= kLongRanks ? kBlockMostLong : kBlockMost) ||
           (alone && seeds > (k <= kShortRanks ? kTableSeedsShort : kTableSeeds));
}

SKIM_DEV uint32_t upper_bound_u64(const uint64_t *a, uint32_t n, uint64_t x) {  // first i with a[i] > x
    uint32_t lo = 0, hi = n;
    while (lo < hi) {
        const uint32_t mid = (lo + hi) >> 1;
        if (a[mid] <= x) lo = mid + 1;
        else hi = mid;
    }
    return lo;
}

// Rank z (hash h) with stored term t into a table of H slots: the smallest term
// of equal ranks stays.  False if the table is full.
SKIM_DEV uint32_t rank_hash(uint64_t z) {
    uint32_t h = static_cast<uint32_t>(z ^ (z >> 32)) * 0x9E3779B1u;
    h = (h ^ (h >> 15)) * 0x85EBCA77u;
    return h ^ (h >> 13);
}
// GLOBAL: a table in global memory, looked at through the first-level cache (a key
// stays once it is there and a term only falls, so an old value costs a trip more).
template <bool GLOBAL = false>
SKIM_DEV bool table_put(uint64_t *keys, uint64_t *terms, uint32_t H, uint32_t at, uint64_t z, uint64_t t) {
    if (z == kEmptyKey) at = H;  // a place of its own
    for (uint32_t p = 0; p < H; p++) {
        uint64_t k = GLOBAL ? __ldca(&keys[at]) : *reinterpret_cast<volatile uint64_t *>(&keys[at]);
        if (k == kEmptyKey && at != H)
            k = atomicCAS(reinterpret_cast<unsigned long long *>(&keys[at]), kEmptyKey, z);
        if (k == kEmptyKey || k == z) {
            if ((GLOBAL ? __ldca(&terms[at]) : *reinterpret_cast<volatile uint64_t *>(&terms[at])) > t)
                atomicMin(reinterpret_cast<unsigned long long *>(&terms[at]), t);
            return true;
        }
        if (++at == H) at = 0;
    }
    return false;
}

// The same from any block of the cluster.  Every access is a trip to the other
// block, so an exchange is tried without looking first; and the minimum is a loop over the
// 64-bit exchange, the one 64-bit operation that shared memory makes atomic
// for local and remote callers alike (an atomicMin of 64 bits lost updates here).
SKIM_DEV bool table_put_remote(uint64_t *keys, uint64_t *terms, uint32_t H, uint32_t at, uint64_t z, uint64_t t) {
    if (z == kEmptyKey) at = H;
    for (uint32_t p = 0; p < H; p++) {
        const uint64_t k =
            at == H ? z : atomicCAS(reinterpret_cast<unsigned long long *>(&keys[at]), kEmptyKey, z);
        if (k == kEmptyKey || k == z) {
            for (uint64_t v = kEmptyKey; v > t;) {
                const uint64_t o = atomicCAS(reinterpret_cast<unsigned long long *>(&terms[at]), v, t);
                if (o == v) break;
                v = o;
            }
            return true;
        }
        if (++at == H) at = 0;
    }
    return false;
}

// What a lane has of its seed: the row, its ranks below the threshold, the
// stored term.
struct SeedRow {
    uint32_t u, body;
    uint64_t term;
};
SKIM_DEV SeedRow seed_row(const uint64_t *X, const uint32_t *xlen, uint32_t k, const QueryTerms &terms, uint32_t u) {
    const uint32_t ln = xlen[u];
    const uint64_t tau = ln == k ? X[static_cast<uint64_t>(u) * k + k - 1] : ~0ull;
    return SeedRow{u, ln == k ? k - 1 : ln, static_cast<uint64_t>(__double_as_longlong(term_of(terms, tau)))};
}

// How a warp reads rows of up to `most` ranks: `rows` of them at a step, lane's share
// is rank `pos` (and every 32nd after it) of row `row`.  (One row at a step left 31 lanes
// idle with k = 2: 100000 seeds in 396 us.)
struct RowShare {
    uint32_t rows, row, pos;
};
SKIM_DEV RowShare row_share(uint32_t most) {
    const uint32_t lane = threadIdx.x & 31, w = most > 16 ? 32 : most <= 1 ? 1 : 1u << (32 - __clz(most - 1));
    return RowShare{32 / w, lane / w, lane & (w - 1)};
}

SKIM_DEV U192 warp_sum192(U192 a) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        U192 other;
        for (int w = 0; w < 3; w++) other.w[w] = __shfl_down_sync(kFull, a.w[w], o);
        add192(a, other);
    }
    return a;
}

SKIM_DEV void add_term(U192 &acc, uint64_t stored) {
    if (stored != kEmptyKey && stored) add192(acc, to_fixed(__longlong_as_double(static_cast<long long>(stored))));
}

SKIM_DEV U192 block_sum192(U192 acc) {  // valid in thread 0
    __shared__ U192 wsum[32];
    acc = warp_sum192(acc);
    if ((threadIdx.x & 31) == 0) wsum[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x < 32) {
        U192 t{{0, 0, 0}};
        if (threadIdx.x < (blockDim.x >> 5)) t = wsum[threadIdx.x];
        acc = warp_sum192(t);
    }
    return acc;
}

// Block-collective: the exact sum over the ranks of a query whose hash lies in
// part `part` of `parts` (thread 0's return value), table of H + 1 slots in tab.
// PART: a row has few ranks of the part, so a warp collects 32 before it goes to
// the table (kStage pairs per warp behind it).  LONG: rows are not shared (row_share; a
// batch is bound by what it issues, 1000 queries of 64 ranks 504 and 520 us).
template <bool PART, bool LONG = false>
SKIM_DEV U192 query_block(const uint64_t *X, const uint32_t *xlen, uint32_t n, uint32_t k, const QueryTerms &terms,
                          const uint32_t *seeds, uint32_t s, uint64_t part, uint64_t parts, uint64_t *tab, uint32_t H,
                          unsigned *err) {
    const uint32_t warp = threadIdx.x >> 5, warps = blockDim.x >> 5, lane = threadIdx.x & 31;
    uint64_t *keys = tab, *val = tab + H + 1;
    ulonglong2 *st = reinterpret_cast<ulonglong2 *>(val + H + 1) + warp * kStage;
    const RowShare sh = LONG ? RowShare{1, 0, lane} : row_share(k - 1);
    U192 acc{{0, 0, 0}};
    for (uint64_t cut = 1, c = 0; c < cut;) {  // one piece, unless the table overflows
        const uint64_t pieces = parts * cut, piece = part * cut + c;
        const uint64_t lo = (piece << 32) / pieces, hi = ((piece + 1) << 32) / pieces;  // of the 32-bit hash
        const uint32_t lo32 = static_cast<uint32_t>(lo), last = static_cast<uint32_t>(hi - lo - 1);
        const uint64_t scale = (static_cast<uint64_t>(H) << 32) / (hi - lo);           // hash - lo -> slot
        for (uint32_t i = threadIdx.x; i <= H; i += blockDim.x) keys[i] = val[i] = kEmptyKey;
        __syncthreads();
        bool full = false;
        uint32_t nst = 0;
        const auto slot_of = [&](uint32_t h) { return min(H - 1, static_cast<uint32_t>(((h - lo32) * scale) >> 32)); };
        for (uint32_t j0 = 0; j0 + warp < s; j0 += warps * 32) {  // lane i: seed j0 + i warps + warp
            const uint32_t j = j0 + lane * warps + warp;
            SeedRow r{0, 0, 0};
            if (j < s) {
                const uint32_t u = seeds[j];
                if (u < n) r = seed_row(X, xlen, k, terms, u);
                else atomicOr(err, 1u);
            }
            const uint32_t cnt = min(32u, (s - j0 - warp + warps - 1) / warps);
            for (uint32_t i = 0; i < cnt; i += sh.rows) {  // (rows past cnt have no ranks)
                const uint32_t u = __shfl_sync(kFull, r.u, i + sh.row), body = __shfl_sync(kFull, r.body, i + sh.row);
                const uint64_t t = __shfl_sync(kFull, r.term, i + sh.row);
                const uint64_t *row = X + static_cast<uint64_t>(u) * k;
                const uint32_t end = sh.rows > 1 ? 1 : body;  // (the same for the warp)
                for (uint32_t p0 = 0; p0 < end; p0 += 32) {
                    const bool in = p0 + sh.pos < body;
                    const uint64_t z = in ? row[p0 + sh.pos] : 0;
                    const uint32_t h = rank_hash(z);
                    const bool mine = in && h - lo32 <= last;
                    if (!PART) {
                        if (mine) full |= !table_put(keys, val, H, slot_of(h), z, t);
                        continue;
                    }
                    const unsigned mb = __ballot_sync(kFull, mine);
                    if (mine) st[nst + __popc(mb & lanemask_lt())] = make_ulonglong2(z, t);
                    nst += __popc(mb);
                    __syncwarp();
                    if (nst < 32) continue;
                    const ulonglong2 e = st[lane];
                    full |= !table_put(keys, val, H, slot_of(rank_hash(e.x)), e.x, e.y);
                    __syncwarp();
                    if (lane < nst - 32) st[lane] = st[lane + 32];
                    nst -= 32;
                    __syncwarp();
                }
            }
        }
        if (PART && lane < nst) full |= !table_put(keys, val, H, slot_of(rank_hash(st[lane].x)), st[lane].x, st[lane].y);
        if (__syncthreads_or(full)) {
            if (hi - lo < 2) {  // (thousands of ranks of one hash)
                if (threadIdx.x == 0 && err) atomicOr(err, 2u);
                break;
            }
            cut *= 2;  // the pieces done so far stay done
            c *= 2;
            continue;
        }
        for (uint32_t i = threadIdx.x; i <= H; i += blockDim.x) add_term(acc, val[i]);
        c++;
        if (c < cut) __syncthreads();
    }
    return block_sum192(acc);
}

// Cluster-collective: the exact sum over the ranks of a query whose hash lies in
// part `part` of `parts`, in the tables of the cluster's blocks (H + 1 slots each; a
// block has a range of the hashes), in `cut` pieces or more.  Thread 0 of block 0
// has the total; *bad: the ranks of some hash are more than fit.
template <uint32_t CL>
SKIM_DEV U192 query_cluster(const uint64_t *X, const uint32_t *xlen, uint32_t n, uint32_t k, const QueryTerms &terms,
                            const uint32_t *seeds, uint32_t s, uint64_t part, uint64_t parts, uint64_t cut,
                            uint64_t *tab, uint32_t H, unsigned *err, bool *bad) {
    __shared__ U192 sums[CL];
    __shared__ int s_full;
    namespace cg = cooperative_groups;
    const cg::cluster_group cl = cg::this_cluster();
    const uint32_t rank = cl.block_rank(), lane = threadIdx.x & 31;
    const uint32_t w = rank * (blockDim.x >> 5) + (threadIdx.x >> 5), ways = CL * (blockDim.x >> 5);
    uint64_t *keys = tab, *val = tab + H + 1;
    const RowShare sh = row_share(k - 1);
    U192 acc{{0, 0, 0}};
    *bad = false;
    for (uint64_t c = 0; c < cut;) {
        const uint64_t pieces = parts * cut, piece = part * cut + c;
        const uint64_t lo = (piece << 32) / pieces, hi = ((piece + 1) << 32) / pieces;  // of the 32-bit hash
        const uint32_t lo32 = static_cast<uint32_t>(lo), last = static_cast<uint32_t>(hi - lo - 1);
        const uint64_t scale = (static_cast<uint64_t>(CL * H) << 32) / (hi - lo);
        for (uint32_t i = threadIdx.x; i <= H; i += blockDim.x) keys[i] = val[i] = kEmptyKey;
        if (threadIdx.x == 0) s_full = 0;
        cl.sync();
        bool over = false;
        for (uint32_t j0 = w; j0 < s; j0 += ways * 32) {  // lane i: seed j0 + i ways
            const uint32_t j = j0 + lane * ways;
            SeedRow r{0, 0, 0};
            if (j < s) {
                const uint32_t u = seeds[j];
                if (u < n) r = seed_row(X, xlen, k, terms, u);
                else atomicOr(err, 1u);
            }
            const uint32_t cnt = min(32u, (s - j0 + ways - 1) / ways);
            for (uint32_t i = 0; i < cnt; i += sh.rows) {  // (rows past cnt have no ranks)
                const uint32_t u = __shfl_sync(kFull, r.u, i + sh.row), body = __shfl_sync(kFull, r.body, i + sh.row);
                const uint64_t t = __shfl_sync(kFull, r.term, i + sh.row);
                const uint64_t *row = X + static_cast<uint64_t>(u) * k;
                for (uint32_t p = sh.pos; p < body; p += 32) {
                    const uint64_t z = row[p];
                    const uint32_t h = rank_hash(z) - lo32;
                    if (h > last) continue;
                    const uint32_t at = static_cast<uint32_t>(__umul64hi(static_cast<uint64_t>(h) << 32, scale));
                    const uint32_t g = min(CL * H - 1, at), b = g / H;
                    over |= !table_put_remote(cl.map_shared_rank(keys, b), cl.map_shared_rank(val, b), H, g - b * H, z, t);
                }
            }
        }
        if (over) *cl.map_shared_rank(&s_full, 0) = 1;
        cl.sync();
        const bool again = *cl.map_shared_rank(&s_full, 0) != 0;
        if (!again)
            for (uint32_t i = threadIdx.x; i <= H; i += blockDim.x) add_term(acc, val[i]);
        cl.sync();  // all have read the flag
        if (!again) {
            c++;
        } else if (hi - lo < 2) {
            *bad = true;
            break;
        } else {
            cut *= 2;  // the pieces done so far stay done
            c *= 2;
        }
    }
    acc = block_sum192(acc);
    if (threadIdx.x == 0) *cl.map_shared_rank(&sums[rank], 0) = acc;
    cl.sync();  // (a block leaves when nobody needs its memory any more)
    if (rank == 0 && threadIdx.x == 0)
        for (uint32_t r = 1; r < CL; r++) add192(acc, sums[r]);
    return acc;
}

// slots of each block of a cluster
template <uint32_t CL>
SKIM_HD uint32_t cluster_slots(uint64_t entries) {
    const uint64_t h = entries * 2 / CL + 64;
    return h < kClusterSlots ? static_cast<uint32_t>(h) : kClusterSlots;
}
constexpr SKIM_HD uint32_t small_slots(uint64_t entries) { return static_cast<uint32_t>(entries + entries / 2 + 32); }

// One query whose seeds are kernel arguments; the estimate goes to host memory.
template <uint32_t CAP>
struct SeedArgs {
    uint32_t s;
    uint32_t seeds[CAP];
};
template <uint32_t CAP>
__global__ void __launch_bounds__(1024) k_q_one(const uint64_t *X, const uint32_t *xlen, uint32_t n, uint32_t k,
                                                QueryTerms terms, const __grid_constant__ SeedArgs<CAP> a, double *out) {
    extern __shared__ ulonglong2 s_tab[];
    const U192 e = query_block<false>(X, xlen, n, k, terms, a.seeds, a.s, 0, 1, reinterpret_cast<uint64_t *>(s_tab),
                               small_slots(static_cast<uint64_t>(a.s) * (k - 1)), nullptr);
    if (threadIdx.x == 0) *out = fixed_to_double(e) / terms.div;
}
// (an estimate is never negative: -1 tells the host to take the batch path)
template <uint32_t CAP>
__global__ void __launch_bounds__(1024)
    k_q_one_cluster(const uint64_t *X, const uint32_t *xlen, uint32_t n, uint32_t k, QueryTerms terms,
                    const __grid_constant__ SeedArgs<CAP> a, uint32_t H, double *out) {
    extern __shared__ ulonglong2 s_tab[];
    bool full;
    const U192 e = query_cluster<kCluster>(X, xlen, n, k, terms, a.seeds, a.s, 0, 1, 1,
                                           reinterpret_cast<uint64_t *>(s_tab), H, nullptr, &full);
    if (blockIdx.x == 0 && threadIdx.x == 0) *out = full ? -1.0 : fixed_to_double(e) / terms.div;
}

// Block q: query q, if it is small.
template <bool LONG>
__global__ void __launch_bounds__(1024) k_q_small(const uint64_t *X, const uint32_t *xlen, uint32_t n, uint32_t k,
                                                  QueryTerms terms, const uint32_t *seeds, const uint64_t *offsets,
                                                  double *out, unsigned *err) {
    extern __shared__ ulonglong2 s_tab[];
    const uint32_t q = blockIdx.x;
    const uint64_t s0 = offsets[q];
    const uint32_t s = static_cast<uint32_t>(offsets[q + 1] - s0);
    if (static_cast<uint64_t>(s) * (k - 1) > kSmallEntries) return;
    const U192 e = query_block<false, LONG>(X, xlen, n, k, terms, seeds + s0, s, 0, 1, reinterpret_cast<uint64_t *>(s_tab),
                               small_slots(static_cast<uint64_t>(s) * (k - 1)), err);
    if (threadIdx.x == 0) out[q] = fixed_to_double(e) / terms.div;
}

// Block-collective: part c (of first .. end) of a query has the sum e in thread 0;
// the last one to come adds them up (*done counts, zero again after).
SKIM_DEV void add_parts(const U192 &e, uint64_t c, uint64_t first, uint64_t end, U192 *partial, unsigned *done,
                        double *out, double div) {
    __shared__ int s_last;
    if (threadIdx.x == 0) {
        partial[c] = e;
        __threadfence();
        s_last = atomicAdd(done, 1u) + 1 == static_cast<unsigned>(end - first);
    }
    __syncthreads();
    if (!s_last || threadIdx.x >= 32) return;
    __threadfence();
    U192 tot{{0, 0, 0}};
    for (uint64_t p = first + threadIdx.x; p < end; p += 32) {
        U192 x;
        for (int w = 0; w < 3; w++) x.w[w] = __ldcg(&partial[p].w[w]);
        add192(tot, x);
    }
    tot = warp_sum192(tot);
    if (threadIdx.x == 0) {
        *out = fixed_to_double(tot) / div;
        *done = 0;
    }
}

// A query for in_memory: into a table of H + 1 slots in global
// memory, then the sum over it.
__global__ void __launch_bounds__(512) k_q_table(const uint64_t *X, const uint32_t *xlen, uint32_t n, uint32_t k,
                                                 QueryTerms terms, const uint32_t *seeds, uint64_t s, uint64_t *tab,
                                                 uint32_t H, unsigned *err) {
    const uint32_t lane = threadIdx.x & 31, ways = gridDim.x * (blockDim.x >> 5);
    const uint32_t w = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const RowShare sh = row_share(k - 1);
    for (uint64_t j0 = static_cast<uint64_t>(w) * 32; j0 < s; j0 += static_cast<uint64_t>(ways) * 32) {
        SeedRow r{0, 0, 0};
        if (j0 + lane < s) {
            const uint32_t u = seeds[j0 + lane];
            if (u < n) r = seed_row(X, xlen, k, terms, u);
            else atomicOr(err, 1u);
        }
        for (uint32_t i = 0; i < 32; i += sh.rows) {
            const uint32_t u = __shfl_sync(kFull, r.u, i + sh.row), body = __shfl_sync(kFull, r.body, i + sh.row);
            const uint64_t t = __shfl_sync(kFull, r.term, i + sh.row);
            for (uint32_t p = sh.pos; p < body; p += 32) {
                const uint64_t z = X[static_cast<uint64_t>(u) * k + p];
                if (!table_put<true>(tab, tab + H + 1, H, __umulhi(rank_hash(z), H), z, t)) atomicOr(err, 2u);
            }
        }
    }
}
__global__ void __launch_bounds__(512) k_q_table_sum(const uint64_t *val, uint32_t H, U192 *partial, unsigned *done,
                                                     double *out, double div) {
    U192 acc{{0, 0, 0}};
    for (uint64_t i = blockIdx.x * blockDim.x + threadIdx.x; i <= H; i += gridDim.x * blockDim.x) add_term(acc, val[i]);
    add_parts(block_sum192(acc), blockIdx.x, 0, gridDim.x, partial, done, out, div);
}

// One block per part of the larger queries.
template <bool LONG>
__global__ void __launch_bounds__(kPartThreads) k_q_part(const uint64_t *X, const uint32_t *xlen, uint32_t n,
                                                         uint32_t k, QueryTerms terms, const uint32_t *seeds,
                                                         const uint64_t *offsets, const uint64_t *block_off,
                                                         uint32_t q, U192 *partial, unsigned *done, double *out,
                                                         unsigned *err) {
    extern __shared__ ulonglong2 s_tab[];
    const uint32_t c = blockIdx.x;
    const uint32_t qi = upper_bound_u64(block_off + 1, q, c);
    const uint64_t first = block_off[qi], end = block_off[qi + 1], s0 = offsets[qi];
    const uint32_t s = static_cast<uint32_t>(offsets[qi + 1] - s0);
    const U192 e = query_block<true, LONG>(X, xlen, n, k, terms, seeds + s0, s, c - first, end - first, reinterpret_cast<uint64_t *>(s_tab), kPartSlots, err);
    add_parts(e, c, first, end, partial, &done[qi], &out[qi], terms.div);
}

// A few queries: `ways` clusters for each of the larger ones, then a block for each
// of the small ones.
struct FewArgs {
    uint32_t q, n_large, ways, large[kMoreLarge];
};
template <uint32_t CL>
__global__ void __launch_bounds__(kPartThreads) k_q_few(const uint64_t *X, const uint32_t *xlen, uint32_t n, uint32_t k,
                                                        QueryTerms terms, const uint32_t *seeds,
                                                        const uint64_t *offsets, const FewArgs f, U192 *partial,
                                                        unsigned *done, double *out, unsigned *err) {
    extern __shared__ ulonglong2 s_tab[];
    uint64_t *tab = reinterpret_cast<uint64_t *>(s_tab);
    const uint32_t c = blockIdx.x / CL, ways = f.ways;
    const uint32_t qi = c < f.n_large * ways ? f.large[c / ways] : blockIdx.x - f.n_large * ways * CL;
    if (qi >= f.q) return;
    const uint64_t s0 = offsets[qi], s = offsets[qi + 1] - s0, entries = s * (k - 1);
    if (c >= f.n_large * ways) {
        if (entries > kSmallEntries) return;
        const U192 e = query_block<false>(X, xlen, n, k, terms, seeds + s0, static_cast<uint32_t>(s), 0, 1, tab,
                                          small_slots(entries), err);
        if (threadIdx.x == 0) out[qi] = fixed_to_double(e) / terms.div;
        return;
    }
    const uint64_t room = static_cast<uint64_t>(CL * (CL == kCluster ? kBlockFill : kBlockEntries)) * ways;
    const uint64_t cut = (entries + room - 1) / room;
    bool bad;
    const U192 e = query_cluster<CL>(X, xlen, n, k, terms, seeds + s0, static_cast<uint32_t>(s), c % ways, ways, cut, tab,
                                 cluster_slots<CL>(entries / (ways * cut)), err, &bad);
    if (blockIdx.x % CL) return;
    if (bad && threadIdx.x == 0) atomicOr(err, 2u);
    add_parts(e, c, c / ways * ways, (c / ways + 1) * ways, partial, &done[qi], &out[qi], terms.div);
}

// Single-node influence estimates from each node's own sketch: the bottom-k
// estimator (k-1)/tau of Section 3 (mode 0), the permutation estimator
// 1 + (k-1)(D-1)/(T-1) of Section 3.1 (mode 1) and n(k-1)/(T-1) of Section 3.2
// (mode 2); |X_v| (mode 0, 1) or 0 (mode 2) for a sketch that is not full.
__global__ void k_node_estimates(const uint64_t *X, const uint32_t *xlen, uint32_t n, uint32_t k, uint32_t l,
                                 int mode, double *out) {
    const double dl = static_cast<double>(l), k1 = static_cast<double>(k - 1);
    const double d1 = static_cast<double>(static_cast<uint64_t>(n) * l - 1);
    for (uint32_t v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += gridDim.x * blockDim.x) {
        const uint32_t lv = xlen[v];
        double e;
        if (lv < k) {
            e = mode == 2 ? 0.0 : static_cast<double>(lv) / dl;
        } else {
            const double q = __ull2double_rn(X[static_cast<uint64_t>(v) * k + k - 1]);
            if (mode == 0) e = k1 / ldexp(q, -64) / dl;
            else if (mode == 1) e = (1.0 + k1 * d1 / q) / dl;
            else e = static_cast<double>(n) * k1 / q;
        }
        out[v] = e;
    }
}

}  // namespace

uint32_t query_blocks(uint64_t seeds, uint32_t k, bool alone) {
    const uint64_t e = seeds * (k - 1);
    if (e <= kSmallEntries) return 0;
    return in_memory(seeds, k, alone) ? 0 : static_cast<uint32_t>((e + kPartEntries - 1) / kPartEntries);
}

uint64_t query_table_slots(uint64_t seeds, uint32_t k, bool alone) {
    const uint64_t e = seeds * (k - 1);
    return e <= kSmallEntries || !in_memory(seeds, k, alone) ? 0 : std::min<uint64_t>(e + e / 2, 0xfffffffeu) + 1;
}

size_t query_partial_bytes() { return sizeof(U192); }

cudaError_t launch_node_estimates(const uint64_t *X, const uint32_t *xlen, uint32_t n, uint32_t k, uint32_t l,
                                  int mode, double *out, cudaStream_t s) {
    note_launch();
    const unsigned g = static_cast<unsigned>(std::min<uint64_t>((n + 255) / 256, 152 * 16));
    k_node_estimates<<<g ? g : 1, 256, 0, s>>>(X, xlen, n, k, l, mode, out);
    return cudaGetLastError();
}

// 960 and 8000 seeds are 4 and 32 KB of arguments, the usual and the largest size.
bool query_fits_args(uint64_t seeds, uint32_t k) {
    return seeds <= kQueryArgSeeds && seeds * (k - 1) <= kClusterEntries;
}

namespace {

// An error: the device would not take clusters of this size (another program's
// partition of it, for instance); nothing has been launched.
template <uint32_t CL, class K, class... Args>
cudaError_t cluster_launch(bool allowed, K kernel, unsigned clusters, uint32_t H, cudaStream_t st, const Args &...args) {
    if (!allowed) return cudaErrorInvalidClusterSize;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (kClusterSlots + 1) * sizeof(ulonglong2));
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    cudaLaunchAttribute at = {};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = CL;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(clusters * CL);
    cfg.blockDim = dim3(kPartThreads);
    cfg.dynamicSmemBytes = (H + 1) * sizeof(ulonglong2);
    cfg.stream = st;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    e = cudaLaunchKernelEx(&cfg, kernel, args...);
    if (e == cudaSuccess) note_launch();
    else cudaGetLastError();
    return e;
}

template <uint32_t CAP>
cudaError_t one_launch(const uint64_t *X, const uint32_t *xlen, uint32_t n, uint32_t k, const QueryTerms &terms,
                       const uint32_t *seeds, uint32_t s, double *out_host, bool clusters, cudaStream_t st) {
    SeedArgs<CAP> a;
    a.s = s;
    std::copy(seeds, seeds + s, a.seeds);
    const uint64_t entries = static_cast<uint64_t>(s) * (k - 1);
    if (entries <= kOneEntries) {
        static_assert((small_slots(kOneEntries) + 1) * sizeof(ulonglong2) < 40 * 1024, "needs no asking");
        const uint32_t threads = std::min<uint32_t>(1024, std::max<uint32_t>(128, s * 32));
        note_launch();
        k_q_one<CAP><<<1, threads, (small_slots(entries) + 1) * sizeof(ulonglong2), st>>>(X, xlen, n, k, terms, a, out_host);
        return cudaGetLastError();
    }
    if constexpr (CAP > 60) {
        const uint32_t H = cluster_slots<kCluster>(entries);
        return cluster_launch<kCluster>(clusters, k_q_one_cluster<CAP>, 1, H, st, X, xlen, n, k, terms, a, H, out_host);
    }
    return cudaErrorInvalidValue;
}
}  // namespace

cudaError_t launch_query_one(const uint64_t *X, const uint32_t *xlen, uint32_t n, uint32_t k, const QueryTerms &terms,
                             const uint32_t *seeds, uint32_t s, double *out_host, bool clusters, cudaStream_t st) {
    if (s <= 60 && s * (k - 1) <= kOneEntries)
        return one_launch<60>(X, xlen, n, k, terms, seeds, s, out_host, clusters, st);
    return s <= 960 ? one_launch<960>(X, xlen, n, k, terms, seeds, s, out_host, clusters, st)
                    : one_launch<kQueryArgSeeds>(X, xlen, n, k, terms, seeds, s, out_host, clusters, st);
}

cudaError_t launch_query_multi(const uint64_t *X, const uint32_t *xlen, uint32_t n, uint32_t k, const QueryTerms &terms,
                               const uint32_t *seeds, const uint64_t *offsets, const uint64_t *block_off, uint32_t q,
                               const uint64_t *h_offsets, uint32_t blocks, bool alone, const QueryScratch &qs,
                               double *out, cudaStream_t s) {
    if (q == 0) return cudaSuccess;
    static_assert(kSmallSlots >= kSmallEntries + kSmallEntries / 2 + 32, "a small query's table");
    U192 *partial = static_cast<U192 *>(qs.partial);
    cudaError_t e = cudaSuccess;
    uint32_t tables = 0;
    if (in_memory(h_offsets[q], k, alone)) {  // some query may be one of those
        for (uint32_t i = 0; i < q && e == cudaSuccess; i++) {
            const uint64_t cnt = h_offsets[i + 1] - h_offsets[i], slots = query_table_slots(cnt, k, alone);
            if (!slots) continue;
            if (slots > qs.table_slots) return cudaErrorInvalidValue;
            tables++;
            e = cudaMemsetAsync(qs.table, 0xff, slots * sizeof(ulonglong2), s);
            if (e != cudaSuccess) return e;
            uint64_t *tab = static_cast<uint64_t *>(qs.table);
            const uint32_t H = static_cast<uint32_t>(slots - 1);
            note_launch();
            note_launch();
            k_q_table<<<kTableBlocks * 2, 512, 0, s>>>(X, xlen, n, k, terms, seeds + h_offsets[i], cnt, tab, H, qs.err);
            k_q_table_sum<<<kTableBlocks, 512, 0, s>>>(tab + slots, H, partial + blocks, qs.done + i, out + i, terms.div);
            e = cudaGetLastError();
        }
    }
    FewArgs f{q, 0, 0, {}};
    uint64_t most = 0;
    for (uint32_t i = 0; blocks && i < q && f.n_large <= kMoreLarge; i++) {
        const uint64_t cnt = h_offsets[i + 1] - h_offsets[i];
        if (!query_blocks(cnt, k, alone)) continue;
        if (f.n_large < kMoreLarge) f.large[f.n_large] = i;
        f.n_large++;
        most = std::max(most, cnt * (k - 1));
    }
    const bool fits_four = most <= kClusterFour * kBlockEntries;
    if (e == cudaSuccess && f.n_large && f.n_large <= (fits_four ? kMoreLarge : kFewLargest)) {
        const bool few = f.n_large <= kFewLarge || !fits_four;
        const uint32_t cl = few ? kCluster : kClusterFour;
        const uint32_t wanted = (blocks * kPartEntries - 1) / kClusterEntries + 1;
        f.ways = few ? std::max(1u, std::min(kClusterParts / f.n_large, wanted)) : 1;
        const uint32_t small = q - f.n_large - tables;
        const uint32_t with_small = f.n_large * f.ways + (q + cl - 1) / cl;
        const auto rounds = [](uint32_t n) { return (n + kClusterParts - 1) / kClusterParts; };
        const bool together =
            small == 0 || (small <= kFewSmall && (!few || rounds(with_small) <= rounds(f.n_large * f.ways) + 1));
        const uint32_t clusters = small && together ? with_small : f.n_large * f.ways;
        const cudaError_t ce =
            few ? cluster_launch<kCluster>(qs.clusters, k_q_few<kCluster>, clusters, kClusterSlots, s, X, xlen, n, k,
                                           terms, seeds, offsets, f, partial, qs.done, out, qs.err)
                : cluster_launch<kClusterFour>(qs.clusters, k_q_few<kClusterFour>, clusters, kClusterSlots, s, X, xlen, n,
                                               k, terms, seeds, offsets, f, partial, qs.done, out, qs.err);
        if (ce == cudaSuccess && together) return ce;
        if (ce == cudaSuccess) blocks = 0;  // (refused: parts need no clusters)
    }
    if (e == cudaSuccess && blocks) {
        const int smem = (kPartSlots + 1 + kPartThreads / 32 * kStage) * sizeof(ulonglong2);
        const auto kernel = k > 17 ? k_q_part<true> : k_q_part<false>;  // (row_share)
        e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return e;
        note_launch();
        kernel<<<blocks, kPartThreads, smem, s>>>(X, xlen, n, k, terms, seeds, offsets, block_off, q, partial, qs.done,
                                                  out, qs.err);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess && q > tables) {
        const int smem = (kSmallSlots + 1) * sizeof(ulonglong2);
        const auto kernel = k > 17 ? k_q_small<true> : k_q_small<false>;  // (row_share)
        e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return e;
        note_launch();
        kernel<<<q, small_threads(q), smem, s>>>(X, xlen, n, k, terms, seeds, offsets, out, qs.err);
        e = cudaGetLastError();
    }
    return e;
}

uint32_t query_partials(uint32_t blocks, uint64_t table_slots) {
    return std::max(blocks + (table_slots ? kTableBlocks : 0), kClusterParts);
}

}  // namespace skim

// ---------------------------------------------------------------------------
// Allocation-free variant for callers that cannot allocate device memory.
//
// Some callers cannot call cudaMalloc: code running inside another
// framework's memory pool, inside a region where allocation would break a
// memory budget, or in processes whose allocator is owned by someone else.
// This entry point keeps the query's scratch hash table in a fixed array of
// static device memory instead (every GPU that loads the library holds it
// until the process exits).  The caller still passes the sketches, the seed
// list and the output.  All calls on a device share the one array, so calls
// whose work overlaps on the GPU race with each other; the kernel clears the
// part of the table it uses before every query.
// ---------------------------------------------------------------------------
#include <mutex>

#include "skim.h"

namespace skim {
namespace {

constexpr uint64_t kStaticSlots = 1ull << 18;  // hash slots: 2^18 keys + 2^18 values = 4 MiB
static __device__ __align__(256) uint64_t g_static_table[2 * kStaticSlots];

std::mutex g_static_mu;
constexpr int kMaxDevices = 64;
uint64_t *g_static_ptr[kMaxDevices] = {};  // device address of g_static_table, per device

__global__ void __launch_bounds__(kQThreads) k_query_static(const uint64_t *X, const uint32_t *xlen, uint32_t n,
                                                            uint32_t k, QueryTerms terms, const uint32_t *seeds,
                                                            uint32_t s, uint64_t *table, uint64_t H, double *out) {
    __shared__ unsigned long long top_tau;
    __shared__ int top_used, bad;
    __shared__ U192 wsum[kQThreads / 32];
    uint64_t *tk = table;
    uint64_t *tv = table + H;
    if (threadIdx.x == 0) {
        top_tau = 0;
        top_used = 0;
        bad = 0;
    }
    for (uint64_t i = threadIdx.x; i < H; i += blockDim.x) {
        tk[i] = kEmptyKey;
        tv[i] = 0;
    }
    __syncthreads();
    const uint64_t hmask = H - 1;
    const uint64_t work = static_cast<uint64_t>(s) * k;
    for (uint64_t e = threadIdx.x; e < work; e += blockDim.x) {
        const uint32_t u = seeds[e / k];
        const uint32_t pos = static_cast<uint32_t>(e % k);
        if (u >= n) {
            bad = 1;
            continue;
        }
        const uint32_t ln = xlen[u];
        const uint32_t body = ln == k ? k - 1 : ln;
        if (pos >= body) continue;
        const uint64_t z = X[static_cast<uint64_t>(u) * k + pos];
        const uint64_t tau = ln == k ? X[static_cast<uint64_t>(u) * k + k - 1] : ~0ull;
        if (z == kEmptyKey) {
            atomicMax(&top_tau, static_cast<unsigned long long>(tau));
            top_used = 1;
            continue;
        }
        uint64_t h = fmix(z) & hmask;
        for (uint64_t p = 0; p < H; p++) {
            unsigned long long prev = atomicCAS(reinterpret_cast<unsigned long long *>(&tk[h]),
                                                static_cast<unsigned long long>(kEmptyKey),
                                                static_cast<unsigned long long>(z));
            if (prev == kEmptyKey || prev == z) {
                atomicMax(reinterpret_cast<unsigned long long *>(&tv[h]), static_cast<unsigned long long>(tau));
                break;
            }
            h = (h + 1) & hmask;
        }
    }
    __syncthreads();
    U192 acc{{0, 0, 0}};
    for (uint64_t i = threadIdx.x; i < H; i += blockDim.x)
        if (tk[i] != kEmptyKey) {
            const double v = term_of(terms, tv[i]);
            if (v != 0.0) add192(acc, to_fixed(v));
        }
    if (threadIdx.x == 0 && top_used) {
        const double v = term_of(terms, top_tau);
        if (v != 0.0) add192(acc, to_fixed(v));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        U192 other;
        for (int w = 0; w < 3; w++) other.w[w] = __shfl_down_sync(kFull, acc.w[w], o);
        add192(acc, other);
    }
    if ((threadIdx.x & 31) == 0) wsum[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        U192 tot{{0, 0, 0}};
        for (int w = 0; w < kQThreads / 32; w++) add192(tot, wsum[w]);
        out[0] = bad ? __longlong_as_double(0x7ff8000000000000ll) : fixed_to_double(tot) / terms.div;
    }
}

}  // namespace
}  // namespace skim

extern "C" int skim_union_estimate_static(const uint64_t *x_dev, const uint32_t *len_dev, uint32_t n, uint32_t k,
                                          uint32_t l, uint32_t rank_mode, const uint32_t *seeds_dev,
                                          uint32_t n_seeds, double *est_dev, void *stream) {
    using namespace skim;
    if (!x_dev || !len_dev || !est_dev || (n_seeds && !seeds_dev)) return SKIM_EINVAL;
    if (n == 0 || k < 2 || k > 255 || l == 0 || l > 64) return SKIM_EINVAL;
    if (rank_mode > SKIM_RANKS_IC_MODEL || (rank_mode == SKIM_RANKS_IC_MODEL && l != 1)) return SKIM_EINVAL;
    // the same reading of a threshold as the context queries (query_terms_of)
    QueryTerms terms{0, 0.0, static_cast<double>(l)};
    if (rank_mode == SKIM_RANKS_PERMUTATION)
        terms = QueryTerms{1, static_cast<double>(static_cast<uint64_t>(n) * l - 1), static_cast<double>(l)};
    else if (rank_mode == SKIM_RANKS_IC_MODEL)
        terms = QueryTerms{2, static_cast<double>(n), 1.0};
    uint64_t H = 64;
    const uint64_t need = 2ull * n_seeds * (k - 1) + 2;
    while (H < need) H <<= 1;
    if (H > kStaticSlots) return SKIM_ERANGE;  // the static table holds 2^18 slots
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return SKIM_ECUDA;
    if (dev < 0 || dev >= kMaxDevices) return SKIM_ERANGE;
    uint64_t *table = nullptr;
    {
        // once per device, with that device current: the device address of
        // the static array (its name in host code is only a stand-in)
        std::lock_guard<std::mutex> lock(g_static_mu);
        if (!g_static_ptr[dev]) {
            void *p = nullptr;
            if (cudaGetSymbolAddress(&p, g_static_table) != cudaSuccess || !p) return SKIM_ECUDA;
            g_static_ptr[dev] = static_cast<uint64_t *>(p);
        }
        table = g_static_ptr[dev];
    }
    // An error left pending by the caller's earlier work is not ours to
    // consume: report it and leave it in place.
    if (cudaPeekAtLastError() != cudaSuccess) return SKIM_ECUDA;
    note_launch();
    k_query_static<<<1, kQThreads, 0, static_cast<cudaStream_t>(stream)>>>(x_dev, len_dev, n, k, terms, seeds_dev,
                                                                           n_seeds, table, H, est_dev);
    if (cudaPeekAtLastError() != cudaSuccess) {
        cudaGetLastError();  // the launch's own error
        return SKIM_ECUDA;
    }
    return SKIM_OK;
}
