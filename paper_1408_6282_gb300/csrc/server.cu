// server.cu -- the influence oracle as a serving loop with continuous
// batching (queries of Section 5.1, Eq. unionest, over resident sketches).
//
// Requests are seed sets submitted from any host thread.  A server thread
// admits pending requests into a launch group while in-flight slots and the
// arena of hash-table slots allow (a query of |S| seeds counts as about
// 2|S|(k-1); only the largest have a table there, the others theirs in shared
// memory), copies the group's seeds to the device and launches the batched
// query kernel on one of several streams.  Groups on different streams run
// concurrently; when a group finishes, its slots and scratch return to the
// pool and requests that arrived meanwhile are admitted into the next group.
// A burst is bound by the host: seeds go from the caller straight into one slab
// (no allocation per request), the lock is not held while a group is launched, and
// the server thread looks at its events for a while before it sleeps (a sleep
// is at least 55 us long).  3000 queries of 142 seeds on average (R-MAT 18, 64
// ranks), submitted at once: 2.8 -> 1.5 ms.
// Every query's estimate is an exact fixed-point sum rounded once, so a
// result is bitwise the same alone, in any group and on any stream.
#include <algorithm>
#include <atomic>
#include <chrono>
#include <condition_variable>
#include <cstring>
#include <deque>
#include <mutex>
#include <new>
#include <thread>
#include <unordered_map>
#include <vector>

#include "internal.cuh"
#include "skim.h"

using namespace skim;

namespace {

using Clock = std::chrono::steady_clock;

struct Request {
    uint64_t ticket;
    uint64_t count;  // seeds, in the slab behind those of the request before
    uint64_t slots;  // hash-table slots it needs
};

struct Result {
    double est;
    Clock::time_point at;
};

struct Lane {  // one stream and its buffers
    cudaStream_t st = nullptr;
    cudaEvent_t done = nullptr;
    bool busy = false;
    uint64_t arena_slots = 0;
    uint32_t *d_seeds = nullptr, *h_seeds = nullptr;
    uint64_t seed_cap = 0;
    uint64_t *d_meta = nullptr, *h_meta = nullptr;  // seed | block offsets, 2 x (group_cap + 1)
    double *d_out = nullptr, *h_out = nullptr;
    unsigned *d_err = nullptr;
    unsigned *d_done = nullptr;  // finished blocks per query, zero between groups
    void *d_part = nullptr;
    uint64_t part_cap = 0;
    void *d_table = nullptr;  // of queries above the shared-memory tables' limit (16 bytes per arena slot), or null
    uint32_t group_cap = 0;
    std::vector<uint64_t> tickets, boff;  // boff: the group's block offsets
};

uint64_t table_slots(uint64_t s, uint32_t k) {
    uint64_t need = std::max<uint64_t>(64, 2 * s * (k - 1) + 2), p = 1;
    while (p < need) p <<= 1;
    return p;
}

}  // namespace

struct skim_server {
    const uint64_t *X = nullptr;
    const uint32_t *xlen = nullptr;
    uint32_t n = 0, k = 0, l = 0;
    QueryTerms terms{0, 0.0, 1.0};
    bool clusters = true;
    uint32_t max_inflight = 0;
    std::vector<Lane> lanes;
    std::mutex mu;
    std::condition_variable cv_work, cv_done;
    std::deque<Request> pending;
    std::vector<uint32_t> slab;  // seeds of the pending requests, from slab_at on
    size_t slab_at = 0;
    std::atomic<size_t> waiting{0};  // pending.size()
    std::unordered_map<uint64_t, Result> results;
    uint64_t next_ticket = 1;
    uint32_t inflight = 0;
    bool stopping = false;
    int error = SKIM_OK;
    uint64_t groups = 0, grouped = 0;
    std::thread worker;
};

namespace {

void free_lane(Lane &ln) {
    if (ln.st) cudaStreamSynchronize(ln.st);
    if (ln.d_seeds) cudaFree(ln.d_seeds);
    if (ln.d_meta) cudaFree(ln.d_meta);
    if (ln.d_out) cudaFree(ln.d_out);
    if (ln.d_err) cudaFree(ln.d_err);
    if (ln.d_done) cudaFree(ln.d_done);
    if (ln.d_part) cudaFree(ln.d_part);
    if (ln.d_table) cudaFree(ln.d_table);
    if (ln.h_seeds) cudaFreeHost(ln.h_seeds);
    if (ln.h_meta) cudaFreeHost(ln.h_meta);
    if (ln.h_out) cudaFreeHost(ln.h_out);
    if (ln.done) cudaEventDestroy(ln.done);
    if (ln.st) cudaStreamDestroy(ln.st);
    ln = Lane{};
}

// Retire finished groups (lock held).
void retire(skim_server *s) {
    for (auto &ln : s->lanes) {
        if (!ln.busy) continue;
        cudaError_t q = cudaEventQuery(ln.done);
        if (q == cudaErrorNotReady) continue;
        const Clock::time_point now = Clock::now();
        if (q != cudaSuccess) s->error = SKIM_ECUDA;
        for (size_t i = 0; i < ln.tickets.size(); i++) s->results[ln.tickets[i]] = Result{ln.h_out[i], now};
        s->inflight -= static_cast<uint32_t>(ln.tickets.size());
        ln.tickets.clear();
        ln.busy = false;
        s->cv_done.notify_all();
    }
}

// Admit pending requests into one group on a free lane and launch it (lock
// held on entry and on return, not while the group is launched: lanes are used
// by the server thread only).
bool admit(skim_server *s, std::unique_lock<std::mutex> &lock) {
    if (s->pending.empty()) return false;
    Lane *ln = nullptr;
    for (auto &c : s->lanes)
        if (!c.busy) {
            ln = &c;
            break;
        }
    if (!ln) return false;
    uint64_t used = 0, nseeds = 0;
    uint32_t cnt = 0;
    uint64_t *h_off = ln->h_meta;
    h_off[0] = 0;
    ln->boff.assign(1, 0);
    while (!s->pending.empty() && cnt < ln->group_cap && s->inflight + cnt < s->max_inflight) {
        Request &r = s->pending.front();
        if (used + r.slots > ln->arena_slots || nseeds + r.count > ln->seed_cap) break;  // memory admission
        nseeds += r.count;
        used += r.slots;
        h_off[cnt + 1] = nseeds;
        ln->boff.push_back(ln->boff.back() + query_blocks(r.count, s->k, false));
        ln->tickets.push_back(r.ticket);
        cnt++;
        s->pending.pop_front();
    }
    if (cnt == 0) return false;
    if (nseeds) std::memcpy(ln->h_seeds, s->slab.data() + s->slab_at, nseeds * sizeof(uint32_t));
    s->slab_at += nseeds;
    if (s->pending.empty()) {
        s->slab.clear();
        s->slab_at = 0;
    } else if (s->slab_at > s->slab.size() / 2 && s->slab_at > (1u << 16)) {
        s->slab.erase(s->slab.begin(), s->slab.begin() + static_cast<ptrdiff_t>(s->slab_at));
        s->slab_at = 0;
    }
    s->waiting = s->pending.size();
    s->inflight += cnt;
    s->groups++;
    s->grouped += cnt;
    ln->busy = true;
    lock.unlock();
    bool ok = true;
    if (nseeds)
        ok &= cudaMemcpyAsync(ln->d_seeds, ln->h_seeds, nseeds * sizeof(uint32_t), cudaMemcpyHostToDevice, ln->st) ==
              cudaSuccess;
    // seed and block offsets of the group, one behind the other
    const size_t g1 = static_cast<size_t>(cnt) + 1;
    std::copy(ln->boff.begin(), ln->boff.end(), ln->h_meta + g1);
    ok &= cudaMemcpyAsync(ln->d_meta, ln->h_meta, 2 * g1 * sizeof(uint64_t), cudaMemcpyHostToDevice, ln->st) ==
          cudaSuccess;
    QueryScratch qs{ln->d_part, ln->d_done, ln->d_err, ln->d_table, ln->d_table ? ln->arena_slots : 0, s->clusters};
    ok &= launch_query_multi(s->X, s->xlen, s->n, s->k, s->terms, ln->d_seeds, ln->d_meta, ln->d_meta + g1, cnt, ln->h_meta,
                             static_cast<uint32_t>(ln->boff.back()), false, qs, ln->d_out, ln->st) == cudaSuccess;
    ok &= cudaMemcpyAsync(ln->h_out, ln->d_out, cnt * sizeof(double), cudaMemcpyDeviceToHost, ln->st) == cudaSuccess;
    ok &= cudaEventRecord(ln->done, ln->st) == cudaSuccess;
    lock.lock();
    if (!ok) s->error = SKIM_ECUDA;
    return true;
}

void serve(skim_server *s, int device) {
    cudaSetDevice(device);
    std::unique_lock<std::mutex> lock(s->mu);
    for (;;) {
        retire(s);
        while (admit(s, lock)) {
        }
        bool busy = false, free_lane = false;
        for (auto &ln : s->lanes) (ln.busy ? busy : free_lane) = true;
        const size_t left = s->pending.size();  // more than these can be admitted, or nothing until a group is done
        if (s->stopping && !busy && left == 0) break;
        if (busy) {
            // groups in flight: look at their events, and at what arrives
            lock.unlock();
            const Clock::time_point until = Clock::now() + std::chrono::microseconds(200);
            bool wake = false;
            while (!wake && Clock::now() < until) {
                for (auto &ln : s->lanes) wake |= ln.busy && cudaEventQuery(ln.done) != cudaErrorNotReady;
                wake |= free_lane && s->waiting > left;
                if (!wake) std::this_thread::yield();
            }
            if (!wake) std::this_thread::sleep_for(std::chrono::microseconds(5));
            lock.lock();
        } else {
            s->cv_work.wait(lock, [&] { return s->stopping || !s->pending.empty(); });
        }
    }
}

// Wait for a ticket's result and take it (lock held).
int take(skim_server *s, std::unique_lock<std::mutex> &lock, uint64_t ticket, uint32_t timeout_ms, Result *out) {
    auto it = s->results.end();
    const bool got = s->cv_done.wait_for(lock, std::chrono::milliseconds(timeout_ms), [&] {
        it = s->results.find(ticket);
        return it != s->results.end() || s->error != SKIM_OK;
    });
    if (!got) return SKIM_ETIMEOUT;
    if (s->error) return s->error;
    *out = it->second;
    s->results.erase(it);
    return SKIM_OK;
}

}  // namespace

extern "C" {

int skim_server_start(skim_ctx *ctx, uint32_t max_inflight, uint64_t scratch_slots, uint32_t streams,
                      skim_server **out) {
    if (!ctx || !out || max_inflight == 0 || streams == 0 || streams > 16) return SKIM_EINVAL;
    *out = nullptr;
    const uint64_t *X = nullptr;
    const uint32_t *xlen = nullptr;
    int rc = skim_sketch_pointers(ctx, &X, &xlen);
    if (rc) return rc;
    uint32_t n = 0, k = 0, l = 0;
    rc = skim_context_shape(ctx, &n, &k, &l);
    if (rc) return rc;
    skim_server *s = new skim_server();
    s->X = X;
    s->xlen = xlen;
    s->n = n;
    s->k = k;
    s->l = l;
    s->terms = query_terms_of(ctx);
    s->clusters = query_clusters_of(ctx);
    s->max_inflight = max_inflight;
    s->lanes.resize(streams);
    const uint64_t arena = std::max<uint64_t>(scratch_slots / streams, 64);
    const uint32_t gcap = std::max<uint32_t>(1, max_inflight);
    bool ok = true;
    for (auto &ln : s->lanes) {
        ln.arena_slots = arena;
        ln.group_cap = gcap;
        ln.seed_cap = arena / 2 + gcap;  // a query of |S| seeds takes at least 2|S| slots
        ok &= cudaStreamCreateWithFlags(&ln.st, cudaStreamNonBlocking) == cudaSuccess;
        ok &= cudaEventCreateWithFlags(&ln.done, cudaEventDisableTiming) == cudaSuccess;
        ok &= cudaMalloc(&ln.d_seeds, ln.seed_cap * sizeof(uint32_t)) == cudaSuccess;
        // a block per 8000 ranks, for which a query is charged 16000 slots
        const uint64_t table = query_table_slots(arena / 2 / (k - 1), k, false);  // the largest query's
        ln.part_cap = query_partials(static_cast<uint32_t>(arena / 2048 + gcap), table);
        if (table) ok &= cudaMalloc(&ln.d_table, arena * 2 * sizeof(uint64_t)) == cudaSuccess;
        ok &= cudaMalloc(&ln.d_meta, 2 * (gcap + 1) * sizeof(uint64_t)) == cudaSuccess;
        ok &= cudaMalloc(&ln.d_out, gcap * sizeof(double)) == cudaSuccess;
        ok &= cudaMalloc(&ln.d_err, sizeof(unsigned)) == cudaSuccess;
        ok &= cudaMalloc(&ln.d_done, gcap * sizeof(unsigned)) == cudaSuccess;
        ok = ok && cudaMemsetAsync(ln.d_done, 0, gcap * sizeof(unsigned), ln.st) == cudaSuccess;
        ok &= cudaMalloc(&ln.d_part, ln.part_cap * query_partial_bytes()) == cudaSuccess;
        ok &= cudaMallocHost(&ln.h_seeds, ln.seed_cap * sizeof(uint32_t)) == cudaSuccess;
        ok &= cudaMallocHost(&ln.h_meta, 2 * (gcap + 1) * sizeof(uint64_t)) == cudaSuccess;
        ok &= cudaMallocHost(&ln.h_out, gcap * sizeof(double)) == cudaSuccess;
        if (!ok) break;
    }
    if (!ok) {
        cudaGetLastError();
        for (auto &ln : s->lanes) free_lane(ln);
        delete s;
        return SKIM_ENOMEM;
    }
    int dev = 0;
    cudaGetDevice(&dev);
    s->worker = std::thread(serve, s, dev);
    *out = s;
    return SKIM_OK;
}

int skim_server_submit(skim_server *s, const uint32_t *seeds, uint32_t n_seeds, uint64_t *ticket) {
    if (!s || !ticket || (n_seeds && !seeds)) return SKIM_EINVAL;
    for (uint32_t i = 0; i < n_seeds; i++)
        if (seeds[i] >= s->n) return SKIM_EINVAL;
    const uint64_t slots = table_slots(n_seeds, s->k);
    if (slots > s->lanes[0].arena_slots || n_seeds + 1 > s->lanes[0].seed_cap) return SKIM_ERANGE;
    {
        std::lock_guard<std::mutex> lock(s->mu);
        if (s->stopping) return SKIM_EINVAL;
        if (s->error) return s->error;
        const size_t had = s->slab.size();
        try {
            s->slab.insert(s->slab.end(), seeds, seeds + n_seeds);
            s->pending.push_back(Request{s->next_ticket, n_seeds, slots});
        } catch (const std::bad_alloc &) {
            s->slab.resize(had);
            return SKIM_ENOMEM;
        }
        *ticket = s->next_ticket++;
        s->waiting = s->pending.size();
    }
    s->cv_work.notify_one();
    return SKIM_OK;
}

int skim_server_poll(skim_server *s, uint64_t ticket, int *done, double *est) {
    if (!s || !done || !est) return SKIM_EINVAL;
    std::lock_guard<std::mutex> lock(s->mu);
    auto it = s->results.find(ticket);
    if (it == s->results.end()) {
        *done = 0;
        return s->error;
    }
    *done = 1;
    *est = it->second.est;
    s->results.erase(it);
    return SKIM_OK;
}

int skim_server_wait(skim_server *s, uint64_t ticket, double *est, uint32_t timeout_ms) {
    if (!s || !est) return SKIM_EINVAL;
    std::unique_lock<std::mutex> lock(s->mu);
    Result r;
    const int rc = take(s, lock, ticket, timeout_ms, &r);
    if (rc == SKIM_OK) *est = r.est;
    return rc;
}

int skim_server_replay(skim_server *s, const double *arrival_s, const uint64_t *offsets, const uint32_t *seeds,
                       uint32_t q, double *latency_s, double *est_out) {
    if (!s || !offsets || (q && (!arrival_s || !latency_s || !est_out))) return SKIM_EINVAL;
    std::vector<uint64_t> tickets(q);
    std::vector<Clock::time_point> sent(q);
    const Clock::time_point t0 = Clock::now();
    for (uint32_t i = 0; i < q; i++) {
        const Clock::time_point at = t0 + std::chrono::duration_cast<Clock::duration>(
                                              std::chrono::duration<double>(arrival_s[i]));
        while ((sent[i] = Clock::now()) < at) {
        }
        int rc = skim_server_submit(s, seeds + offsets[i], static_cast<uint32_t>(offsets[i + 1] - offsets[i]),
                                    &tickets[i]);
        if (rc) return rc;
    }
    // The last request's result first: collecting thousands of finished ones takes the
    // lock for 0.2 ms, which the groups still in flight would wait for.
    std::unique_lock<std::mutex> lock(s->mu);
    for (uint32_t i = q; i-- > 0;) {
        Result r;
        int rc = take(s, lock, tickets[i], 60000, &r);
        if (rc) return rc;
        est_out[i] = r.est;
        latency_s[i] = std::chrono::duration<double>(r.at - sent[i]).count();
    }
    return SKIM_OK;
}

int skim_server_stats(skim_server *s, uint64_t *groups, uint64_t *queries) {
    if (!s || !groups || !queries) return SKIM_EINVAL;
    std::lock_guard<std::mutex> lock(s->mu);
    *groups = s->groups;
    *queries = s->grouped;
    return SKIM_OK;
}

int skim_server_stop(skim_server *s) {
    if (!s) return SKIM_EINVAL;
    {
        std::lock_guard<std::mutex> lock(s->mu);
        s->stopping = true;
    }
    s->cv_work.notify_all();
    if (s->worker.joinable()) s->worker.join();
    const int err = s->error;
    for (auto &ln : s->lanes) free_lane(ln);
    delete s;
    return err;
}

}  // extern "C"
