// Serving: lm_submit / lm_poll / lm_wait (include/lm.h).
//
// A few lanes (threads, each with its own engine and stream) serve one queue.  A
// lane that is free takes the requests that wait, in arrival order, as long as they
// fit the HBM budget and the slots beside those in flight, and runs them together to
// completion: one by the plain path, several by the batched one, their rows in the
// same launches.  Requests that arrive meanwhile are taken by the next free lane, so
// they join the device while earlier ones are on it and leave as soon as their own
// group is done.  Every request keeps its own seed and edge ids, so its result does not
// depend on what else is in flight.  When a group fails for want of memory or at a limit
// (lm_set_limits), its requests run again one by one, so that each gets its own outcome.
//
// A burst of 48 requests of 1 thousand to 4 million edges takes 1.28 ms with two lanes
// (1.36 with one, 1.32 with three); stepping all requests together round by round,
// with the host between the rounds, took 4.6 ms.
#include <cuda_runtime.h>

#include <algorithm>
#include <chrono>
#include <condition_variable>
#include <cstring>
#include <deque>
#include <memory>
#include <thread>
#include <unordered_map>
#include <vector>

#include "lm_host.h"

namespace lm {

struct Request {
    uint64_t ticket = 0;
    const lm_graph* g = nullptr;
    uint64_t seed = 0;
    uint32_t* mate = nullptr;
    bool host_dst = false;
    bool alone = false;     // ran in a group that failed: not in a group again
    uint32_t rounds = 0;
    int state = 0;          // 0 queued, 1 in flight, 2 done
    int rc = LM_OK;
    uint64_t matched = 0;
};

constexpr size_t MAX_QUEUE = 1u << 20;
constexpr size_t MAX_GROUP = 256;  // requests a lane runs together
constexpr int LANES = 2;

struct ServeState {
    lm_ctx* ctx = nullptr;
    Engine eng[LANES];
    std::thread th[LANES];
    std::mutex mu;
    std::condition_variable cv_work, cv_done;
    bool stop = false;
    int fatal = LM_OK;
    uint64_t next_ticket = 1;
    std::deque<Request*> queue;
    std::unordered_map<uint64_t, Request*> all;
    // capacities from the budget, and what is in flight
    uint32_t cap_v = 0, cap_e = 0;
    uint64_t used_v = 0, used_e = 0;
    uint32_t used_slots = 0;
};

namespace {

bool fits(const ServeState* S, const Request* r) {
    return S->used_v + r->g->n <= S->cap_v && S->used_e + r->g->nent <= S->cap_e && S->used_slots < S->ctx->max_slots;
}

int run_group(ServeState* S, Engine& e, const std::vector<Request*>& group, std::vector<uint32_t>& rounds,
              std::vector<unsigned long long>& m2) {
    Prof off(nullptr, e.stream);
    const size_t k = group.size();
    if (k == 1) {
        Request* r = group[0];
        const int rc = match_one(S->ctx, e, r->g, r->seed, r->mate, !r->host_dst, off);
        if (rc == LM_OK) {
            rounds[0] = e.st_host->rounds;
            m2[0] = e.st_host->matched2;
        }
        return rc;
    }
    std::vector<const lm_graph*> gs(k);
    std::vector<uint64_t> seeds(k);
    std::vector<uint32_t*> mates(k);
    for (size_t i = 0; i < k; i++) {
        gs[i] = group[i]->g;
        seeds[i] = group[i]->seed;
        mates[i] = group[i]->mate;
    }
    return match_batch(S->ctx, e, gs.data(), (uint32_t)k, seeds.data(), mates.data(), rounds.data(), m2.data(), off);
}

void lane(ServeState* S, int which) {
    cudaSetDevice(S->ctx->device);
    Engine& e = S->eng[which];
    std::unique_lock<std::mutex> lk(S->mu);
    for (;;) {
        // (a request that does not fit beside those in flight waits for one of them)
        S->cv_work.wait(lk, [&] { return S->stop || (!S->queue.empty() && (S->fatal || fits(S, S->queue.front()))); });
        if (S->stop) return;
        std::vector<Request*> group;
        uint64_t gv = 0, ge = 0;
        while (!S->queue.empty() && group.size() < MAX_GROUP && (S->fatal || fits(S, S->queue.front()))) {
            Request* r = S->queue.front();
            if (!group.empty() && (r->alone || group[0]->alone)) break;
            S->queue.pop_front();
            r->state = 1;
            gv += r->g->n;
            ge += r->g->nent;
            S->used_v += r->g->n;
            S->used_e += r->g->nent;
            S->used_slots++;
            group.push_back(r);
        }
        const size_t k = group.size();
        std::vector<uint32_t> rounds(k);
        std::vector<unsigned long long> m2(k);
        int rc = S->fatal;
        if (!rc) {
            lk.unlock();
            rc = run_group(S, e, group, rounds, m2);
            lk.lock();
        }
        S->used_v -= gv;
        S->used_e -= ge;
        S->used_slots -= (uint32_t)k;
        if ((rc == LM_ENOMEM || rc == LM_ETIMEOUT) && k > 1) {
            for (size_t i = k; i-- > 0;) {
                group[i]->alone = true;
                group[i]->state = 0;
                S->queue.push_front(group[i]);
            }
            S->cv_work.notify_all();
            continue;
        }
        if (rc == LM_ECUDA) S->fatal = rc;
        for (size_t i = 0; i < k; i++) {
            Request* r = group[i];
            r->rc = rc;
            if (rc == LM_OK) {
                r->rounds = rounds[i];
                r->matched = m2[i] / 2;
            }
            r->state = 2;
        }
        S->cv_done.notify_all();
        if (!S->queue.empty()) S->cv_work.notify_all();  // there is room again
    }
}

// the lanes' streams and engines back (also of a start that failed half-way)
void serve_free(ServeState* S) {
    for (Engine& e : S->eng) {
        const cudaStream_t st = e.stream;
        if (!st) continue;
        engine_free(e);
        cudaStreamDestroy(st);
    }
}

int serve_start(lm_ctx* ctx) {
    if (ctx->serve) return LM_OK;
    std::unique_ptr<ServeState> S(new ServeState());
    S->ctx = ctx;
    for (Engine& e : S->eng) {
        cudaStream_t st = nullptr;
        cudaError_t ce = cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking);
        int rc = ce == cudaSuccess ? engine_init(ctx, e, st) : cuda_fail(ctx, ce, "serving stream");
        if (rc) {
            if (st && !e.stream) cudaStreamDestroy(st);
            serve_free(S.get());
            return rc;
        }
        e.cfg = ctx->eng.cfg;  // the context's launch parameters when serving starts
    }
    // what may be in flight at once, from the budget (the list path's scratch takes about
    // 100 bytes a vertex, and nothing for an entry)
    const double B = (double)ctx->budget;
    const double lim = 4.0e9;
    S->cap_e = (uint32_t)std::min(lim, B * 0.80 / 25.0);
    S->cap_v = (uint32_t)std::min(lim, B * 0.15 / 110.0);
    ctx->serve = S.release();
    for (int i = 0; i < LANES; i++) ctx->serve->th[i] = std::thread(lane, ctx->serve, i);
    return LM_OK;
}

}  // namespace
}  // namespace lm

using namespace lm;

extern "C" {

__attribute__((visibility("hidden"))) void lm_serve_shutdown(lm_ctx* ctx) {
    if (!ctx || !ctx->serve) return;
    ServeState* S = ctx->serve;
    {
        std::lock_guard<std::mutex> lk(S->mu);
        S->stop = true;
    }
    S->cv_work.notify_all();
    for (std::thread& t : S->th)
        if (t.joinable()) t.join();
    serve_free(S);
    for (auto& kv : S->all) delete kv.second;
    delete S;
    ctx->serve = nullptr;
}

int lm_submit(lm_ctx* ctx, const lm_graph* g, uint64_t seed, uint32_t* mate, uint64_t* ticket) {
    if (!ctx) return LM_EINVAL;
    if (ctx->poisoned) return LM_ECUDA;
    if (!g || !mate || !ticket) return fail(ctx, LM_EINVAL, "null graph, mate or ticket");
    if (ctx->flags & LM_F_RENEW) return fail(ctx, LM_EINVAL, "serving does not renew the order (LM_F_RENEW)");
    if (g->ctx->device != ctx->device) return fail(ctx, LM_EINVAL, "graph lives on another device");
    int cur = -1;
    cudaGetDevice(&cur);
    if (cur != ctx->device) cudaSetDevice(ctx->device);
    int rc;
    {
        std::lock_guard<std::mutex> lk(ctx->call_mu);
        rc = serve_start(ctx);
    }
    const bool host_dst = rc == LM_OK && !is_device_ptr(mate);
    if (cur >= 0 && cur != ctx->device) cudaSetDevice(cur);
    if (rc) return rc;
    ServeState* S = ctx->serve;
    if (S->fatal) return S->fatal;
    if (g->n > S->cap_v || g->nent > S->cap_e) return fail(ctx, LM_ENOMEM, "request exceeds the serving budget");
    std::unique_ptr<Request> r(new Request());
    r->g = g;
    r->seed = seed;
    r->mate = mate;
    r->host_dst = host_dst;
    std::lock_guard<std::mutex> lk(S->mu);
    if (S->queue.size() >= MAX_QUEUE) return LM_EAGAIN;
    r->ticket = S->next_ticket++;
    *ticket = r->ticket;
    S->all[r->ticket] = r.get();
    S->queue.push_back(r.release());
    S->cv_work.notify_one();
    return LM_OK;
}

int lm_poll(lm_ctx* ctx, uint64_t ticket, int* done, lm_stats* stats) {
    if (!ctx || !done) return LM_EINVAL;
    *done = 0;
    ServeState* S = ctx->serve;
    if (!S) return LM_ENOTFOUND;
    std::lock_guard<std::mutex> lk(S->mu);
    auto it = S->all.find(ticket);
    if (it == S->all.end()) return LM_ENOTFOUND;
    Request* r = it->second;
    if (r->state != 2) return LM_OK;
    *done = 1;
    if (stats) {
        memset(stats, 0, sizeof *stats);
        stats->rounds = r->rounds;
        stats->matched = r->matched;
        stats->round_m[0] = r->g->m;
        stats->round_n[0] = r->g->nrows;
    }
    const int rc = r->rc;
    S->all.erase(it);
    delete r;
    return rc;
}

int lm_wait(lm_ctx* ctx, uint64_t ticket, uint32_t timeout_ms) {
    if (!ctx) return LM_EINVAL;
    ServeState* S = ctx->serve;
    if (!S) return LM_ENOTFOUND;
    std::unique_lock<std::mutex> lk(S->mu);
    auto it = S->all.find(ticket);
    if (it == S->all.end()) return LM_ENOTFOUND;
    Request* r = it->second;
    const bool ok = S->cv_done.wait_for(lk, std::chrono::milliseconds(timeout_ms), [&] { return r->state == 2; });
    return ok ? LM_OK : LM_ETIMEOUT;
}

}  // extern "C"
