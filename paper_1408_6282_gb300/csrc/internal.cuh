// internal.cuh -- launchers and argument blocks shared by the libskim
// translation units (host-visible declarations; kernels live in the .cu files).
#pragma once
#include <cstddef>
#include <cstdint>
#include <cuda_runtime.h>

#include "common.cuh"

struct skim_ctx;  // the C ABI's opaque context (capi.cu)

namespace skim {

// Live-edge threshold model (Section 6: uniform p, weighted cascade 1/indeg,
// trivalency classes).
struct CoinModel {
    int model;            // 0 uniform, 1 weighted cascade, 2 trivalency, 3 per-edge thresholds (many graphs)
    uint64_t tm1_uniform;  // floor(p * 2^64) - 1
    uint64_t tm1_class[3];
    const uint64_t *thr_wc;  // per node: floor((2^64-1) / indeg(node))
    uint64_t coin_key;
    uint64_t prob_key;
};

// Arguments of the asynchronous traversal kernels.
struct TravArgs {
    const uint32_t *ptr;  // CSR row pointers in the search direction
    const uint32_t *col;
    CoinModel cm;
    Item *q;
    uint64_t qcap;
    DevCtl *ctl;
    uint64_t timeout_ns;
    // reverse searches (lanes = ranks of a batch)
    uint64_t *hkeys;
    uint64_t *hvals;
    uint64_t hmask;             // the batch's table prefix (slots - 1), cleared before the batch
    uint64_t *rec_key;
    uint32_t *rec_val;
    uint64_t rcap;
    uint32_t tbits;             // record key = (node << tbits) | word
    uint32_t hnode;             // visited-table slots grouped by node (batches of few words)
    const uint8_t *lane_inst;   // instance of every lane of the batch
    const uint64_t *lane_g;     // per lane: (instance + 1) * G, the lane's coin-stream offset
    const uint64_t *he;         // per CSR edge: state of its coin stream, fmix(coin_key ^ (u << 32 | v))
    const uint64_t *tm1e;       // per CSR edge: live threshold (model 3)
    const uint64_t *full;       // Algorithm 2 pruning: instances whose local sketch holds k ranks
    int prune;
    uint64_t *pend;             // per table slot: lane bits whose expansion was spilled
    // residual (forward) searches (lanes = instances)
    uint64_t *covered;
    const uint64_t *seg_start;
    uint32_t *seg_len;
    uint32_t *size;
    const uint32_t *idx_nodes;
    uint32_t l;
    uint64_t *pend_trav;        // per node: instances whose expansion was spilled
    uint64_t *pend_erase;       // per node: instances whose index erasure was spilled
    // materialised instances (mat != 0): reverse searches walk the live
    // in-neighbours of (node v, instance i), col[loff[v*l+i] .. loff[v*l+i+1]),
    // forward searches the live out-neighbours the same way
    int mat;
    const uint32_t *loff;
    // sketch build over materialised instances (need != null): lane q of the
    // search is lane lane_of[q] of the batch; need, scc, hit, lbits, own as in
    // BuildArgs; words: records node << tbits | word per table entry instead
    const uint64_t *need;
    uint64_t lmask;
    const uint64_t *scc;
    uint32_t *hit;
    const uint32_t *lane_of;
    uint32_t lbits;
    int own, words;
    uint32_t *cnt;              // SKIM: per node, the batch's visits (null: not counted)
    const uint32_t *xlen;       // Algorithm 2 in the IC model: ranks of every sketch before the batch, of at most k
    uint32_t k;
    int many;                   // coins drawn in the search: the batch is expected to fill the chip
};

// graph.cu
cudaError_t launch_check_edges(const uint32_t *src, const uint32_t *dst, uint64_t m, uint32_t n, unsigned *bad,
                               cudaStream_t s);
// ptr[v] = first index with row[index] >= v, for v = 0..n (row sorted)
cudaError_t launch_row_ptr(const uint32_t *row, uint64_t m, uint32_t n, uint32_t *ptr, cudaStream_t s);
// rhe[e] = fhe[rev2fwd[e]] = edge_state(coin_key, rcol[e], rrow[e]) over the reverse CSR
cudaError_t launch_edge_states_both(const uint32_t *rcol, const uint32_t *rrow, const uint32_t *rev2fwd, uint64_t m,
                                    uint64_t coin_key, uint64_t *rhe, uint64_t *fhe, cudaStream_t s);
cudaError_t launch_make_rev_keys(const uint32_t *src, const uint32_t *dst, uint64_t m, uint64_t *key, uint32_t *val,
                                 cudaStream_t s);
cudaError_t launch_split_rev(const uint64_t *key, const uint32_t *val, uint64_t m, uint32_t *rcol, uint32_t *rrow,
                             uint32_t *rev2fwd, cudaStream_t s);
cudaError_t launch_wc_thresholds(const uint32_t *rptr, uint32_t n, uint64_t *thr, cudaStream_t s);
// Per-edge coin-stream states of a CSR: he[e] for edge (row node, col[e]);
// reverse = 1 when rows are heads (edge col[e] -> row).
// Materialised instances (Section 2: the l live-edge graphs): live masks of
// every CSR edge (bit i = coin of instance i), the nodes' live pairs (tot), and after
// an exclusive scan of those (first; n + 1 of them) the offsets off[v*l + i] of the
// node-major lists of live neighbours, which rows are not empty (nonempty, may be
// null) and the lists.
cudaError_t launch_live_masks(const uint32_t *rrow, const uint32_t *rcol, const uint64_t *rhe, const uint64_t *rtm1,
                              const uint32_t *rev2fwd, const CoinModel &cm, uint64_t m, uint32_t l, uint64_t *rmask,
                              uint64_t *fmask, cudaStream_t s);
// Rows of more than 2048 edges are counted and filled in pieces, using a
// workspace of live_pieces_bytes(m); the count pass of a CSR direction must
// precede its fill pass with the same workspace.
size_t live_pieces_bytes(uint64_t m);
cudaError_t launch_live_count(const uint32_t *ptr, const uint64_t *mask, uint32_t n, uint64_t m, uint32_t l,
                              uint64_t *tot, uint32_t *off, void *pieces_ws, cudaStream_t s);
cudaError_t launch_live_fill(const uint32_t *ptr, const uint32_t *col, const uint64_t *mask, uint32_t n, uint64_t m,
                             uint32_t l, const uint64_t *first, uint32_t *off, uint64_t *nonempty, uint32_t *live,
                             void *pieces_ws, cudaStream_t s);

// Rank order of all pairs: bucket by the top bits, then sort each bucket.
// rank of pair x = v*l+i is fmix(rank_key + G*x), or fmix(rbase[v] + G*i)
// when a per-node base is given (graphs of a batch, each with its own key).
size_t rank_sort_workspace_bytes(uint64_t nl);
// Structured permutation (Section 3.1; ic = false: pairs (v, sigma_v(c))) or
// IC-model positions (Section 3.2; ic = true: nodes) for the first `chunks`
// chunks of n positions: sorted_rank[t] = t, sorted_pair[t] = pair or node.
uint64_t perm_key(uint64_t rank_key);
size_t perm_sort_workspace_bytes(uint32_t n, uint32_t l, uint32_t chunks, bool ic);
cudaError_t perm_sort(uint64_t rank_key, uint32_t n, uint32_t l, uint32_t chunks, bool ic, uint64_t *sorted_rank,
                      uint32_t *sorted_pair, void *ws, cudaStream_t s);
cudaError_t rank_sort(uint64_t rank_key, const uint64_t *rbase, uint32_t l, uint64_t nl, uint64_t *sorted_rank,
                      uint32_t *sorted_pair, void *ws, cudaStream_t s);

// Graphs of a batch (a disjoint union): per-graph keys and models, node ->
// graph, and the per-node / per-edge tables derived from them.
struct BatchDesc {
    uint32_t count;
    const uint32_t *node_graph;  // per node
    const uint32_t *node_off;    // per graph: first node
    const uint64_t *coin_key, *rank_key, *prob_key, *tm1_uniform;  // per graph
    const int *model;            // per graph: 0 uniform, 1 wc, 2 trivalency
    uint64_t tm1_class[3];       // trivalency thresholds for p = 0.1, 0.01, 0.001
};
cudaError_t launch_node_graph(const uint32_t *node_off, uint32_t count, uint32_t *node_graph, cudaStream_t s);
cudaError_t launch_edge_states_batch(const uint32_t *ptr, const uint32_t *col, uint32_t n, const BatchDesc &b,
                                     int reverse, uint64_t *he, cudaStream_t s);
cudaError_t launch_edge_tm1_batch(const uint32_t *ptr, const uint32_t *col, uint32_t n, const BatchDesc &b,
                                  const uint64_t *thr_wc, int reverse, uint64_t *tm1, cudaStream_t s);
cudaError_t launch_rank_bases(const BatchDesc &b, uint32_t n, uint32_t l, uint64_t *rbase, cudaStream_t s);

// traverse.cu
cudaError_t launch_rev_sources(const TravArgs &a, const uint32_t *lane_pair, uint32_t B, uint32_t l,
                               const uint64_t *covered, uint64_t *alive, cudaStream_t s);
cudaError_t launch_fwd_source(const TravArgs &a, uint32_t x, cudaStream_t s);
cudaError_t launch_traverse(const TravArgs &a, bool forward, int grid, cudaStream_t s);
// Re-queue spilled work (after a drained traversal that set DevCtl::spill);
// reverse searches find it by their table slots.
cudaError_t launch_respill_rev(const TravArgs &a, cudaStream_t s);
cudaError_t launch_respill_fwd(const TravArgs &a, uint32_t n, cudaStream_t s);
int traverse_grid(bool forward, bool mat, bool many = false);  // resident blocks for the persistent traversal
// Reverse searches over materialised live rows with per-warp queues in shared
// memory (Algorithms 1 and 2): the batch's source lanes are taken by the
// kernel itself (sources = false: an earlier launch took them; covered/alive
// as for launch_rev_sources).  The source cursor DevCtl::src_next must be zero
// before the first launch of a batch.
int rev_ring_grid();
cudaError_t launch_rev_ring(const TravArgs &a, const uint32_t *lane_pair, uint32_t B, uint32_t l,
                            const uint64_t *covered, uint64_t *alive, uint64_t *leaf, bool sources, int grid,
                            cudaStream_t s);
// Behind a search with leaf lanes (traverse.cu): those of nodes whose sketch can fill
// up in this batch become records.
cudaError_t launch_leaf_records(const TravArgs &a, const uint32_t *lane_pair, uint32_t B, uint32_t l, uint64_t *leaf,
                                uint32_t k, cudaStream_t s);

// reach.cu: the residual search of seed x over materialised rows, one block per
// instance (the seed is marked chosen)
struct ReachArgs {
    const uint32_t *off;        // row bounds per (v, i) in the search direction
    const uint32_t *rows;
    uint32_t l;
    uint64_t *mask;             // per node: instances in which it has been reached (covered)
    const uint32_t *back_off, *back_rows;
    uint64_t *back_mask;
    uint2 *list;                // scratch: 2 * cap entries per instance
    uint32_t cap;
    uint64_t *pend_trav, *back_pend;  // per node: instances whose rows did not fit the scratch
    uint32_t n;
    const uint64_t *seg_start;  // index segment of every pair: first entry, entries
    uint32_t *seg_len;
    uint32_t *size;
    const uint32_t *idx_nodes;
    uint8_t *chosen;
    DevCtl *ctl;
    uint64_t timeout_ns;
};
constexpr uint32_t kSeedOfStep = 0xffffffffu;  // as x: the seed in ctl->step.best, nothing if there is none
cudaError_t launch_reach(const ReachArgs &a, uint32_t x, cudaStream_t s);
// What the nodes pivot[64 * q + i], q < starts, reach in instance i along off and
// rows, for every instance: its bit in mask (zero before), the number of nodes to count[i];
// and what reaches them, along back_off and back_rows to back_mask and count[64 + i].
// Rows that do not fit the scratch are parked in pend_trav and back_pend (zero before
// and after) and taken up when the walk runs dry.  Uses l, n, list, cap, ctl and
// timeout_ns of a too.
cudaError_t launch_reach_from(const ReachArgs &a, const uint32_t *pivot, uint32_t starts, uint32_t *count,
                              cudaStream_t s);

// build.cu: Algorithm 2 over materialised rows
struct BuildArgs {
    const uint32_t *pair;   // the batch's pairs v*l + i in rank order
    uint32_t B, l, n;
    const uint32_t *loff, *rlive;
    const uint64_t *nonempty;  // per node: instances in which its row is not empty
    const uint64_t *need;   // per node: instances in which something upstream still needs ranks
    uint64_t lmask;         // all l instances (need == lmask: the node itself may)
    const uint64_t *scc;    // per node: instances in which it is in the contracted component (null: none)
    uint32_t *hit;          // bitmap of the lanes that hit an open component
    uint64_t *rec;          // records node << lbits | lane
    uint64_t rcap;
    uint32_t lbits;
    int own;                // sources leave records too (ranks that k_merge cannot recompute)
    uint32_t *deflist, *defbits;  // deferred lanes: list, bitmap
    DevCtl *ctl;
};
struct BuildNode {
    uint32_t n, l, k;
    const uint32_t *loff, *rlive, *foff, *flive;
    const uint64_t *nonempty;
    uint32_t *len;          // row lengths (kRowDone, kRowListed)
    uint64_t rank_key;
    const uint64_t *rbase;
    int own;                // own ranks are not recorded: they are merged
    // contracted components (up null: none): per node the instances in which it
    // reaches / is in the component of its graph; per graph (first nodes
    // node_off, null for one graph) and instance the length of the hit list,
    // per graph the open lists
    const uint64_t *up, *scc;
    uint32_t graphs;
    const uint32_t *node_off;
    uint32_t *tlen;         // [graph][64]
    uint64_t *topen;
};
struct BuildScratch {
    uint64_t *over_key;     // one entry per record of a batch
    uint32_t *over_pos;
    uint64_t *buf;
    uint32_t *list, *seg;   // n entries
};
cudaError_t launch_build_search(const BuildArgs &a, cudaStream_t s);
// source pairs and instances of the D deferred lanes
cudaError_t launch_deferred_lanes(uint32_t *deflist, uint32_t D, bool all, const uint32_t *pair, uint32_t l,
                                  uint32_t *defpair, uint8_t *lane_inst, cudaStream_t s);
cudaError_t launch_append(const uint64_t *rec, uint64_t r0, uint64_t r1, uint32_t lbits, const uint32_t *defbits,
                          const uint64_t *lane_rank, uint32_t k, uint32_t *len, uint64_t *X, const BuildScratch &b,
                          DevCtl *ctl, cudaStream_t s);
// lanes of every kWordChunk of R records node << tbits | word (slots rec_val, lane bits
// hvals), to cnt
constexpr uint32_t kWordChunk = 1024;
cudaError_t launch_count_words(const uint32_t *rec_val, uint64_t R, const uint64_t *hvals, uint32_t *cnt,
                               cudaStream_t s);
// such records of a search of all lanes of a batch: the ranks of each one's lanes,
// without the node's own unless `own`
cudaError_t launch_append_words(const uint64_t *rec, const uint32_t *rec_val, uint64_t R, uint32_t tbits,
                                const uint64_t *hvals, const uint32_t *pair, uint32_t l, int own, uint32_t lbits,
                                const uint64_t *lane_rank, uint32_t k, uint32_t *len, uint64_t *X,
                                const BuildScratch &b, DevCtl *ctl, cudaStream_t s);
// rows that received more than k ranks keep the k smallest (R: records appended;
// done: and are full)
cudaError_t launch_overflow(uint64_t R, uint32_t lbits, const uint64_t *lane_rank, uint32_t k, uint32_t *len,
                            uint64_t *X, bool done, const BuildScratch &b, DevCtl *ctl, cudaStream_t s);
cudaError_t launch_need_start(uint64_t *need, uint32_t n, uint64_t lmask, cudaStream_t s);
// *next (device): the first rank not yet processed; full_list: n entries kept
// from pass to pass
cudaError_t launch_need(const BuildNode &g, const uint64_t *next, uint64_t *need, uint32_t *full_list, void *scratch,
                        uint64_t scratch_bytes, DevCtl *ctl, uint64_t timeout_ns, cudaStream_t s);
// best, pivot: 64 entries per graph
cudaError_t launch_pivots(const BuildNode &g, unsigned long long *best, uint32_t *pivot, cudaStream_t s);
// down becomes the component, up is cleared where it is not contracted
cudaError_t launch_components(const BuildNode &g, uint64_t *down, uint64_t *up, const uint32_t *ndown,
                              const uint32_t *nup, DevCtl *ctl, cudaStream_t s);
// a batch's hits into the lists hits[graph][64][k] (rec: one entry per lane of the batch)
cudaError_t launch_hits(const BuildNode &g, const uint32_t *hit, const uint32_t *pair, const uint64_t *lane_rank,
                        uint32_t B, uint32_t lbits, uint64_t *rec, uint64_t *hits, const BuildScratch &b, DevCtl *ctl,
                        cudaStream_t s);
// hits_sorted: [graph][l * k]; places: [graph][64][(l * k + 63) / 64]; total: [graph]
cudaError_t launch_merge(const BuildNode &g, uint64_t *X, uint64_t *hits, uint64_t *hits_sorted, uint64_t *places,
                         uint32_t *total, DevCtl *ctl, cudaStream_t s);

// batch.cu
cudaError_t launch_lane_inst(const uint32_t *lane_pair, const uint64_t *lane_rank, uint32_t B, uint32_t l,
                             uint8_t *lane_inst, uint64_t *lane_g, cudaStream_t s);
// Algorithm 2's acceptance of a batch's sorted records where coins are drawn
// in the searches; record r's lane bits are hvals[2 * rec_val[r]].
cudaError_t launch_accept(const uint64_t *rec_key, const uint32_t *rec_val, const uint64_t *hvals, uint64_t R,
                          uint32_t tbits, const uint8_t *lane_inst, const uint64_t *lane_rank, uint32_t l, uint32_t k,
                          uint8_t *lcnt, uint64_t *full, uint64_t *X, uint32_t *xlen, DevCtl *ctl, cudaStream_t s);

// recsort.cu: order a batch's R records by key, node by node.  cnt: n + 1
// counters, all zero on entry and on return; off: n + 1 node offsets (out);
// tmp: R scratch words; list: n scratch entries; nlist: 2 scratch counters.
cudaError_t launch_node_sort(uint64_t *rec_key, uint32_t *rec_val, uint64_t R, uint32_t tbits, uint32_t n,
                             uint64_t *cnt, uint64_t *off, uint64_t *tmp, uint32_t *list, unsigned *nlist,
                             void *scan_ws, cudaStream_t s);
// SKIM batch: the records' lane bits gathered from the visited table into
// rbits (R words), read by the steps.
cudaError_t launch_gather_bits(const uint32_t *rec_val, const uint64_t *hvals, uint64_t R, uint64_t *rbits,
                               cudaStream_t s);
// A step over the active batch's R records: the lanes [lo, B) of covered sources
// dropped (refilter), the next stop into ctl->step.best ((lane << 32) | node, ~0 if
// there is none), the lanes up to it (or all) committed.  ctl->step.cov = the last
// search's count; nothing is done and ctl->step.stalled set if it is unfinished.
struct StepArgs {
    const uint64_t *rec_key, *rbits;
    uint64_t R;
    uint32_t tbits, lo, B, l, k, refilter;
    const uint32_t *lane_pair;
    const uint64_t *covered;
    uint64_t *alive;
    const uint64_t *leaf;       // lanes committed without a record
    uint32_t *size, *lane_cnt;  // lane_cnt: zero on entry and on return
    uint64_t *lane_pos, *idx_ctr;
    uint32_t *idx_nodes;
    uint64_t *seg_start;
    uint32_t *seg_len;
    DevCtl *ctl;
    uint64_t timeout_ns;
    // of the stop, if there is one and kprime is not null: its rank to *tau, and k'
    // of Section 4.3.2 to *kprime (zero before): the largest size over the other
    // nodes without the stop lane's own part
    uint32_t n, *kprime;
    uint64_t *tau;
    const uint64_t *lane_rank;
};
cudaError_t launch_step(const StepArgs &a, cudaStream_t s);
cudaError_t launch_argmax_size(const uint32_t *size, uint32_t n, DevCtl *ctl, cudaStream_t s);
cudaError_t launch_min_unchosen(const uint8_t *chosen, uint32_t n, DevCtl *ctl, cudaStream_t s);
// query.cu
// Scratch of the queries: per-block partial sums, counters of the larger queries'
// finished blocks (zero between calls), an error flag.
struct QueryScratch {
    void *partial;
    unsigned *done;
    unsigned *err;
    void *table;            // for the largest queries, 16 bytes per slot
    uint64_t table_slots;
    bool clusters;          // may be launched (else every larger query is taken in parts)
};
// alone: the only query of its call
uint32_t query_blocks(uint64_t seeds, uint32_t k, bool alone);  // parts of a larger query, 0 for a small or largest one
uint64_t query_table_slots(uint64_t seeds, uint32_t k, bool alone);  // of a largest one's table in memory, else 0
uint32_t query_partials(uint32_t blocks, uint64_t table_slots);  // places of `partial`
size_t query_partial_bytes();
// How a threshold becomes a term of Eq. unionest, and the final divisor:
//  mode 0 (uniform 64-bit ranks): 1 / (h * 2^-64), divided by l;
//  mode 1 (structured permutation, Section 3.1): num / h with num = n*l - 1,
//          1 for a sketch that is not full, divided by l;
//  mode 2 (IC model, Section 3.2): num / h with num = n, 0 for a sketch that
//          is not full, divided by 1.
struct QueryTerms {
    int mode;
    double num;
    double div;
};
QueryTerms query_terms_of(const skim_ctx *c);
bool query_clusters_of(const skim_ctx *c);
cudaError_t launch_node_estimates(const uint64_t *X, const uint32_t *xlen, uint32_t n, uint32_t k, uint32_t l,
                                  int mode, double *out, cudaStream_t s);
// block_off: prefix sums of query_blocks; blocks: their total; h_offsets: offsets, on the host
cudaError_t launch_query_multi(const uint64_t *X, const uint32_t *xlen, uint32_t n, uint32_t k, const QueryTerms &terms,
                               const uint32_t *seeds, const uint64_t *offsets, const uint64_t *block_off, uint32_t q,
                               const uint64_t *h_offsets, uint32_t blocks, bool alone, const QueryScratch &qs,
                               double *out, cudaStream_t s);
// One query with few enough seeds (host) to be kernel arguments; out_host: pinned.  An
// error: it takes a cluster, which the device refuses (or clusters is false); the batch form does without.
constexpr uint32_t kQueryArgSeeds = 8000;
bool query_fits_args(uint64_t seeds, uint32_t k);
cudaError_t launch_query_one(const uint64_t *X, const uint32_t *xlen, uint32_t n, uint32_t k, const QueryTerms &terms,
                             const uint32_t *seeds, uint32_t s, double *out_host, bool clusters, cudaStream_t st);

}  // namespace skim
