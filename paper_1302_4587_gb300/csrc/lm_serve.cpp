// Serving: lm_submit / lm_poll / lm_wait (include/lm.h).
//
// A few lanes (threads) serve one queue.  A lane takes the requests that wait, in
// arrival order, as long as they fit the HBM budget and the slots beside those in
// flight, and runs them together: one by the plain path, several by the batched one,
// their rows in the same launches.  Requests that arrive meanwhile are taken by the next
// free lane, so they join the device while earlier ones are on it.  Every request keeps its
// own seed and edge ids, so its result does not depend on what else is in flight.  When a
// group fails for want of memory or at a limit (lm_set_limits), the requests that are not
// done run again one by one, so that each gets its own outcome.
//
// A graph can need many rounds (Theta(n) on a path with monotone weights).  So a lane runs a
// group in slices: after SLICE_NS the live pass gives its rows back, the group's requests
// that are done leave, and the lane takes what waits as a run of its own (an engine
// each, up to MAX_RUNS), whose slices alternate with the first one's.  A group that is
// done within a slice, as nearly all are, never notices.
//
// A burst of 48 requests of 1 thousand to 4 million edges takes 1.28 ms with two lanes
// (1.36 with one, 1.32 with three); stepping all requests together round by round,
// with the host between the rounds, took 4.6 ms.
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
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
constexpr int MAX_RUNS = 8;        // groups a lane has in progress at most
// (a pass over the largest groups measured takes about 1 ms, a launch and its wait 20 us)
constexpr unsigned long long SLICE_NS = 4000000ull;

using Clock = std::chrono::steady_clock;

struct ServeState {
    lm_ctx* ctx = nullptr;
    Engine eng[LANES][MAX_RUNS];    // the first of each lane from the start, the others when needed
    std::thread th[LANES];
    std::mutex mu;
    std::condition_variable cv_work, cv_done;
    bool stop = false;
    std::atomic<int> fatal{LM_OK};
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

// A group in progress on an engine of its own.
struct Run {
    Engine* e = nullptr;
    std::vector<Request*> req;       // by place in the group; NULL: has left
    std::vector<uint32_t*> mates;    // likewise
    ListRun list;
    bool started = false;
    unsigned long long limit_ns = 0; // the group's own time limit,
    unsigned long long waited = 0;   // and how long it stood between slices, which does not count
    Clock::time_point paused;
};
// What a slice settled: requests with their outcome, or to run again one by one.
struct Settled {
    Request* r;
    int rc;
    uint32_t rounds;
    unsigned long long matched2;
    bool again;
};

// all requests of the group that have not left, with one outcome
void settle_all(Run& run, int rc, std::vector<Settled>& out) {
    const bool again = (rc == LM_ENOMEM || rc == LM_ETIMEOUT) && run.req.size() > 1;
    for (Request*& r : run.req)
        if (r) {
            out.push_back({r, rc, 0, 0, again});
            r = nullptr;
        }
}
void settle(Run& run, size_t i, uint32_t rounds, unsigned long long matched2, std::vector<Settled>& out) {
    if (!run.req[i]) return;
    out.push_back({run.req[i], LM_OK, rounds, matched2, false});
    run.req[i] = nullptr;
    run.mates[i] = nullptr;
}

// Starts the group; what the list path does not take (no edges, 2^31 vertices) runs to its end.
int start(ServeState* S, Run& run, Prof& off, std::vector<Settled>& out) {
    Engine& e = *run.e;
    const size_t k = run.req.size();
    run.started = true;
    if (k == 1) {
        Request* r = run.req[0];
        if (r->g->nent && list_path(e, r->g))
            return list_start(S->ctx, e, r->g, r->seed, r->mate, !r->host_dst, off, true, run.list);
        const int rc = match_one(S->ctx, e, r->g, r->seed, r->mate, !r->host_dst, off);
        if (rc == LM_OK) settle(run, 0, e.st_host->rounds, e.st_host->matched2, out);
        return rc;
    }
    std::vector<const lm_graph*> gs(k);
    std::vector<uint64_t> seeds(k);
    bool listed = true;
    for (size_t i = 0; i < k; i++) {
        gs[i] = run.req[i]->g;
        seeds[i] = run.req[i]->seed;
        listed = listed && list_path(e, gs[i]);
    }
    if (listed)
        return list_batch_start(S->ctx, e, gs.data(), (uint32_t)k, seeds.data(), run.mates.data(), true, off, run.list);
    std::vector<uint32_t> rounds(k);
    std::vector<unsigned long long> m2(k);
    const int rc = match_batch(S->ctx, e, gs.data(), (uint32_t)k, seeds.data(), run.mates.data(), rounds.data(), m2.data(), off);
    if (rc == LM_OK)
        for (size_t i = 0; i < k; i++) settle(run, i, rounds[i], m2[i], out);
    return rc;
}

// A slice of the run (the first one starts it); out: the requests that it settled.
// Returns whether the run is over.
bool step(ServeState* S, Run& run, std::vector<Settled>& out) {
    lm_ctx* ctx = S->ctx;
    Engine& e = *run.e;
    Prof off(nullptr, e.stream);
    const size_t k = run.req.size();
    int rc = LM_OK;
    if (!run.started) {
        rc = start(S, run, off, out);
        if (rc || !out.empty()) {
            settle_all(run, rc, out);
            return true;
        }
        run.list.A.slice_ns = SLICE_NS;
        run.limit_ns = run.list.A.limit_ns;
    } else {
        run.waited += (unsigned long long)std::chrono::duration_cast<std::chrono::nanoseconds>(Clock::now() - run.paused).count();
        run.list.A.limit_ns = run.limit_ns + run.waited;
    }
    bool done = run.list.A.nparts == 0;
    // (a pass may also give rows back early, which wait for one another)
    const auto end = Clock::now() + std::chrono::nanoseconds(SLICE_NS);
    while (!done && rc == LM_OK) {
        rc = list_pass(ctx, e, run.list, off);
        done = rc == LM_OK && e.st_host->done;
        if (Clock::now() >= end) break;
    }
    run.paused = Clock::now();
    if (k == 1) {
        Request* r = run.req[0];
        if (rc == LM_OK && !done) return false;
        if (rc == LM_OK && r->host_dst) {
            cudaError_t ce = cudaMemcpyAsync(r->mate, e.lw.mate, (size_t)r->g->n * 4, cudaMemcpyDeviceToHost, e.stream);
            if (ce == cudaSuccess) ce = cudaStreamSynchronize(e.stream);
            if (ce != cudaSuccess) rc = cuda_fail(ctx, ce, "result of a served request");
        }
        if (rc == LM_OK) settle(run, 0, e.st_host->rounds, e.st_host->matched2, out);
        settle_all(run, rc, out);
        return true;
    }
    std::vector<uint32_t> rounds(k);
    std::vector<unsigned long long> m2(k);
    if (done) {
        rc = list_batch_finish(ctx, e, run.list, run.mates.data(), rounds.data(), m2.data());
        if (rc == LM_OK)
            for (size_t i = 0; i < k; i++) settle(run, i, rounds[i], m2[i], out);
        settle_all(run, rc, out);
        return true;
    }
    if (rc == LM_OK || rc == LM_ETIMEOUT) {
        // those that are done leave (beyond the cap: by themselves again)
        std::vector<char> fin(k);
        const int pc = list_batch_progress(ctx, e, run.list, run.mates.data(), fin.data(), rounds.data(), m2.data());
        if (pc) rc = pc;
        else
            for (size_t i = 0; i < k; i++)
                if (fin[i] && rounds[i] <= run.list.A.max_rounds) settle(run, i, rounds[i], m2[i], out);
    }
    if (rc) settle_all(run, rc, out);
    return rc != LM_OK;
}

// an engine of the lane that no run uses (NULL: none can be had)
Engine* free_engine(ServeState* S, int which, const std::vector<std::unique_ptr<Run>>& runs) {
    for (Engine& e : S->eng[which]) {
        bool used = false;
        for (const auto& r : runs) used = used || r->e == &e;
        if (used) continue;
        if (e.stream) return &e;
        cudaStream_t st = nullptr;
        if (cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking) != cudaSuccess) {
            cudaGetLastError();
            return nullptr;
        }
        if (engine_init(S->ctx, e, st)) {
            engine_free(e);
            cudaStreamDestroy(st);
            return nullptr;
        }
        e.cfg = S->eng[which][0].cfg;
        return &e;
    }
    return nullptr;
}

void lane(ServeState* S, int which) {
    cudaSetDevice(S->ctx->device);
    std::vector<std::unique_ptr<Run>> runs;
    std::vector<Settled> out;
    std::unique_lock<std::mutex> lk(S->mu);
    // (a request that does not fit beside those in flight waits for one of them)
    const auto ready = [&] { return !S->queue.empty() && (S->fatal || fits(S, S->queue.front())); };
    for (;;) {
        if (runs.empty()) S->cv_work.wait(lk, [&] { return S->stop || ready(); });
        if (S->stop) return;
        if (ready() && runs.size() < MAX_RUNS) {
            lk.unlock();
            Engine* e = free_engine(S, which, runs);
            lk.lock();
            auto run = std::make_unique<Run>();
            run->e = e;
            while (e && ready() && run->req.size() < MAX_GROUP) {
                Request* r = S->queue.front();
                if (!run->req.empty() && (r->alone || run->req[0]->alone)) break;
                S->queue.pop_front();
                r->state = 1;
                S->used_v += r->g->n;
                S->used_e += r->g->nent;
                S->used_slots++;
                run->req.push_back(r);
                run->mates.push_back(r->mate);
            }
            if (!run->req.empty()) runs.push_back(std::move(run));
        }
        for (size_t i = 0; i < runs.size();) {
            Run& run = *runs[i];
            bool over = true;
            out.clear();
            if (S->fatal) {
                settle_all(run, S->fatal, out);
            } else {
                lk.unlock();
                over = step(S, run, out);
                // only a lane's first engine keeps its scratch: the budget holds two of them
                // beside what is in flight
                if (over && run.e != &S->eng[which][0]) engine_trim(*run.e);
                lk.lock();
            }
            for (size_t j = out.size(); j-- > 0;) {
                const Settled& o = out[j];
                Request* r = o.r;
                S->used_v -= r->g->n;
                S->used_e -= r->g->nent;
                S->used_slots--;
                if (o.again) {
                    r->alone = true;
                    r->state = 0;
                    S->queue.push_front(r);
                    continue;
                }
                if (o.rc == LM_ECUDA) S->fatal = LM_ECUDA;
                r->rc = o.rc;
                r->rounds = o.rounds;
                r->matched = o.matched2 / 2;
                r->state = 2;
            }
            if (!out.empty()) {
                S->cv_done.notify_all();
                if (!S->queue.empty()) S->cv_work.notify_all();  // there is room again
            }
            if (over) runs.erase(runs.begin() + (long)i);
            else i++;
        }
    }
}

// the lanes' streams and engines back (also of a start that failed half-way)
void serve_free(ServeState* S) {
    for (auto& lane_eng : S->eng)
        for (Engine& e : lane_eng) {
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
    for (auto& lane_eng : S->eng) {
        Engine& e = lane_eng[0];
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
    // 100 bytes a vertex, and nothing for an entry; the lanes' first engines keep theirs)
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
