// The matching under a renewed order (LM_F_RENEW): the permutation that tells equal
// weights apart is drawn anew in every round, so the rounds are real ones, with all
// candidates of a round taken over the vertices that were live at its start.
//
// One cooperative kernel runs the whole job.  A round is two phases with a grid
// barrier after each:
//
//   candidates  every live row takes the heaviest of its entries, under the round's
//               keys, whose other end is live.  Nothing is compacted: an entry is read
//               again while its row lives (12 bytes), but its liveness, one bit of a
//               bitmap that L1 holds for graphs of up to 1M vertices, is looked up only
//               for entries above the heaviest live one so far.  Rows of at most
//               LIST_SHORT entries take a thread, longer ones groups, warps or chunks
//               by the graph's tasks.
//   match       rows whose candidates name each other are matched and their bits set;
//               the others are listed for the next round, those without a live
//               neighbour are dropped.
//
// Once little work is left one block finishes the job without grid barriers.
//
// The line to the rounds of launches (lm_kernels.cu) lies at 2^31 vertices and at batches,
// whose graphs that path takes side by side.  One graph is faster here at every size and
// weight tried: R-MAT scale 22 unit 1.58 ms (launches 2.63) and weighted 1.81 (2.10), a
// unit grid of 1M vertices 195 us (317), 5,000 edges 75 us (167).
//
// Bound by the passes over the entries in the first three rounds (R-MAT scale 20, unit
// weights, 15.7M edges, 8 rounds: 524 us; rounds as launches with the
// entries compacted after each one, 919 us, which read and wrote 16 bytes an entry
// and gathered every neighbour's state).
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "../../include/lm.h"
#include "lm_device.cuh"
#include "lm_internal.h"

namespace lm {

namespace {

constexpr uint32_t RT = 256, RW = RT / 32;
constexpr uint32_t RMINB = 4;   // (3 a SM: 2 to 10% slower on large graphs, 4% faster on small ones; 5: spills, 5 to 12%)
// one block finishes the job once its warps' share of a round is short: 512 short rows, 64 of up
// to 64 entries, 32 of up to 256, 8 longer ones or 4 chunks (2048 short rows: 10 to 20% slower;
// any 512 rows: a complete graph of 1000 vertices 723 us, this 151)
__device__ __forceinline__ bool tail(const uint32_t cnt[5]) {
    return 16ull * cnt[0] + 8ull * cnt[1] + 2ull * cnt[2] + cnt[3] + cnt[4] / 8 <= 64;
}
constexpr uint32_t NONE = 0x7FFFFFFFu;  // (vertex ids are below it)
constexpr unsigned long long BAR_LIMIT_NS = 20000000000ull;  // a barrier gives up after 20 s
// kinds of rows: chunks of the longest, then the other kinds of task, then short rows
constexpr int KINDS = 5;
// counters: lengths of the lists of either buffer, units taken (by the round's parity), barrier
constexpr int UNITS = 2 * KINDS, BAR = UNITS + 2;

struct Smem {
    uint32_t ok;
    uint32_t red[2][RW];
    unsigned long long ent[RW];
};

struct Ctx {
    const RenewArgs& a;      // (kernel parameters: constant memory)
    const ListSeg& g;
    uint32_t round, k0, k1;
    uint32_t buf;            // the live rows' lists of this round
    uint32_t cnt[KINDS];     // their lengths
};

// bits change between phases only: through L1, which the barrier's acquire clears
__device__ __forceinline__ uint32_t ld_ca(const uint32_t* p) {
    uint32_t x;
    asm volatile("ld.global.ca.u32 %0, [%1];" : "=r"(x) : "l"(p));
    return x;
}
__device__ __forceinline__ uint32_t ld_acq(const uint32_t* p) {
    uint32_t x;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(x) : "l"(p) : "memory");
    return x;
}
__device__ __forceinline__ bool is_dead(const Ctx& c, uint32_t v) { return (ld_ca(c.a.dead + (v >> 5)) >> (v & 31)) & 1u; }

__device__ __forceinline__ uint32_t kind_from(const ListSeg& g, int k) { return k ? g.ntask[k - 1] : 0u; }
// place i of kind k's list: chunks' lists lie in the chunks' records, the rows' kinds
// side by side in list[buf] (a row is of one kind: together at most n)
__device__ __forceinline__ uint32_t* place(const Ctx& c, int k, uint32_t buf, uint32_t i) {
    if (k == 0) return reinterpret_cast<uint32_t*>(c.a.part + (size_t)i * LIST_KEPT + 1) + buf;
    return c.a.list[buf] + (kind_from(c.g, k) - c.g.ntask[0]) + i;
}
// item i of kind k: a task or (kind 4) a row; the first round has them all
__device__ __forceinline__ uint32_t item(const Ctx& c, int k, uint32_t i) {
    if (c.round) return *place(c, k, c.buf, i);
    return k < 4 ? kind_from(c.g, k) + i : i;
}

__device__ __forceinline__ uint64_t key_at(const Ctx& c, uint64_t ent, uint32_t e) {
    return (ent & 0xFFFFFFFF00000000ull) | perm_seed(e, c.k0, c.k1);
}
template <int G>
__device__ __forceinline__ uint64_t group_max64(uint64_t x) {
    if constexpr (G == 32) {
        const uint32_t hi = __reduce_max_sync(FULL, (uint32_t)(x >> 32));
        const uint32_t lw = __reduce_max_sync(FULL, (uint32_t)(x >> 32) == hi ? (uint32_t)x : 0u);
        return ((uint64_t)hi << 32) | lw;
    } else {
#pragma unroll
        for (int d = 1; d < G; d <<= 1) {
            const uint64_t o = __shfl_xor_sync(FULL, x, d);
            x = o > x ? o : x;
        }
        return x;
    }
}

// a row of at most LIST_SHORT entries by one thread, four entries at a time
template <bool COUNT>
__device__ __forceinline__ void short_row(const Ctx& c, uint32_t r, unsigned long long& ent) {
    const uint32_t o = __ldg(c.g.roff + r), d = __ldg(c.g.roff + r + 1) - o, v = __ldg(c.g.vid + r);
    if (d > LIST_SHORT) return;
    uint64_t best = 0, x[4], nx[4];
    uint32_t bn = NONE, e[4], ne[4];
    auto load = [&](uint64_t y[4], uint32_t z[4], uint32_t j) {
#pragma unroll
        for (int q = 0; q < 4; q++) {
            y[q] = j + q < d ? __ldg(c.g.ent + o + j + q) : 0ull;
            z[q] = j + q < d ? __ldg(c.g.eid + o + j + q) : 0u;
        }
    };
    load(x, e, 0);
    for (uint32_t j = 0; j < d; j += 4) {
        uint32_t live = 0;
        load(nx, ne, j + 4);
#pragma unroll
        for (int q = 0; q < 4; q++)
            if (j + q < d && (c.round == 0 || !is_dead(c, (uint32_t)x[q]))) live |= 1u << q;
#pragma unroll
        for (int q = 0; q < 4; q++) {
            const uint64_t k = key_at(c, x[q], e[q]);
            if (((live >> q) & 1u) && k > best) {
                best = k;
                bn = (uint32_t)x[q];
            }
            x[q] = nx[q];
            e[q] = ne[q];
        }
        if (COUNT) ent += __popc(live);
    }
    c.a.cur[v] = bn;
}

// The heaviest live entry of entries s .. s + d - 1 (at most E G) by the lanes of a group
// of G; best and bn are its key and neighbour so far, the same for all its lanes.
// Whole warps; d = 0: none.
template <bool COUNT, int G, int E>
__device__ __forceinline__ void group_step(const Ctx& c, const uint64_t x[E], const uint32_t e[E], uint32_t d,
                                           uint64_t& best, uint32_t& bn, unsigned long long& ent) {
    const uint32_t lane = threadIdx.x & 31, sub = lane & (G - 1);
    uint64_t k[E];
#pragma unroll
    for (int q = 0; q < E; q++) k[q] = q * G + sub < d ? key_at(c, x[q], e[q]) : 0ull;
    // liveness of the entries that would become the candidate (all of them at a row's first
    // step, few later on), their lookups side by side
    if (COUNT || c.round) {
        uint32_t gone = 0;
#pragma unroll
        for (int q = 0; q < E; q++)
            if (k[q] > (COUNT ? 0ull : best) && c.round && is_dead(c, (uint32_t)x[q])) gone |= 1u << q;
#pragma unroll
        for (int q = 0; q < E; q++) {
            if ((gone >> q) & 1u) k[q] = 0;
            if (COUNT) ent += k[q] ? 1u : 0u;
        }
    }
    uint64_t m = 0;
    uint32_t n = 0;
#pragma unroll
    for (int q = 0; q < E; q++)
        if (k[q] > m) {
            m = k[q];
            n = (uint32_t)x[q];
        }
    if (!__any_sync(FULL, m > best)) return;
    const uint64_t b = group_max64<G>(m);
    // (keys differ: one lane of the group holds it)
    const uint32_t own = __ballot_sync(FULL, m == b && b > best) >> (lane & ~(G - 1)) & (G == 32 ? FULL : (1u << (G & 31)) - 1u);
    const uint32_t who = __shfl_sync(FULL, n, (lane & ~(G - 1)) + (own ? __ffs(own) - 1 : 0));
    if (own) {
        best = b;
        bn = who;
    }
}

// rows of LIST_SHORT + 1 .. LIST_GROUP entries, two at a time
template <bool COUNT>
__device__ __forceinline__ void group_rows(const Ctx& c, uint32_t w, unsigned long long& ent) {
    constexpr int G = LIST_GROUP / 4;
    const uint32_t lane = threadIdx.x & 31, sub = lane & (G - 1);
    const uint32_t i = w * (32 / G) + lane / G;
    uint4 d4 = make_uint4(0, 0, 0, 0);
    if (i < c.cnt[3]) d4 = __ldg(c.g.task + item(c, 3, i));
    uint64_t x[4], best = 0;
    uint32_t e[4], bn = NONE;
#pragma unroll
    for (int q = 0; q < 4; q++) {
        x[q] = q * G + sub < d4.z ? __ldg(c.g.ent + d4.y + q * G + sub) : 0ull;
        e[q] = q * G + sub < d4.z ? __ldg(c.g.eid + d4.y + q * G + sub) : 0u;
    }
    group_step<COUNT, G, 4>(c, x, e, d4.z, best, bn, ent);
    if (sub == 0 && d4.z) c.a.cur[d4.x] = bn;
}

// a row of more than LIST_GROUP entries, or a chunk, by a warp: 128 entries a step, the
// next step's on their way
template <bool COUNT>
__device__ __forceinline__ void long_row(const Ctx& c, uint32_t t, unsigned long long& ent) {
    const uint32_t lane = threadIdx.x & 31;
    const uint4 d4 = __ldg(c.g.task + t);
    const uint32_t v = d4.x, len = d4.z, ch = d4.w;
    const bool whole = len <= LIST_CHUNK;
    const uint32_t s = whole ? d4.y : d4.y + ch * LIST_CHUNK, d = whole ? len : min(len - ch * LIST_CHUNK, LIST_CHUNK);
    uint64_t best = 0, x[4], nx[4];
    uint32_t bn = NONE, e[4], ne[4];
    auto load = [&](uint64_t y[4], uint32_t z[4], uint32_t p) {
#pragma unroll
        for (int q = 0; q < 4; q++) {
            const bool in = p + q * 32 + lane < d;
            y[q] = in ? __ldg(c.g.ent + s + p + q * 32 + lane) : 0ull;
            z[q] = in ? __ldg(c.g.eid + s + p + q * 32 + lane) : 0u;
        }
    };
    load(x, e, 0);
    for (uint32_t p = 0; p < d; p += 128) {
        load(nx, ne, p + 128);
        group_step<COUNT, 32, 4>(c, x, e, min(d - p, 128u), best, bn, ent);
#pragma unroll
        for (int q = 0; q < 4; q++) {
            x[q] = nx[q];
            e[q] = ne[q];
        }
    }
    if (whole) {
        if (lane == 0) c.a.cur[v] = bn;
        return;
    }
    // a chunk: the row's last one to finish takes the heaviest of all
    const uint32_t first = t - ch, nch = (len + LIST_CHUNK - 1) / LIST_CHUNK;
    if (lane == 0) c.a.part[(size_t)t * LIST_KEPT] = make_uint4((uint32_t)best, (uint32_t)(best >> 32), bn, 0);
    __syncwarp();
    uint32_t old = 0;
    if (lane == 0) old = atom_add_acq_rel(&c.a.pcnt[first], 1u);
    old = __shfl_sync(FULL, old, 0);
    __syncwarp();
    if (old != nch - 1) return;
    best = 0;
    bn = NONE;
    for (uint32_t b = 0; b < nch; b += 32) {
        uint4 rec = make_uint4(0, 0, NONE, 0);
        if (b + lane < nch) rec = __ldcg(c.a.part + (size_t)(first + b + lane) * LIST_KEPT);
        const uint64_t k = ((uint64_t)rec.y << 32) | rec.x, m = group_max64<32>(k);
        if (m > best) {   // (uniform)
            best = m;
            bn = __shfl_sync(FULL, rec.z, __ffs(__ballot_sync(FULL, k == m)) - 1);
        }
    }
    if (lane == 0) {
        c.a.pcnt[first] = 0;
        c.a.cur[v] = bn;
    }
}

// Every block of the grid (blocks = 1: one block is left) arrives, and none goes on
// before; false: one did not within the limit.
__device__ __forceinline__ bool barrier(uint32_t* ctr, uint32_t& target, uint32_t blocks, DevState* st, Smem& S) {
    __threadfence();
    __syncthreads();
    if (blocks == 1) return true;
    target += blocks;
    if (threadIdx.x == 0) {
        uint32_t ok = 1;
        atom_add_acq_rel(ctr, 1u);
        const uint64_t t0 = globaltimer_ns();
        for (uint32_t i = 1; (int32_t)(ld_acq(ctr) - target) < 0; i++)
            if ((i & 255u) == 0 && globaltimer_ns() - t0 > BAR_LIMIT_NS) {
                set_err(st, ERR_TIMEOUT, 0x40000000u | blocks);
                ok = 0;
                break;
            }
        __threadfence();
        S.ok = ok;
    }
    __syncthreads();
    return S.ok != 0;
}

template <bool COUNT>
__global__ void __launch_bounds__(RT, RMINB) k_renew(const __grid_constant__ RenewArgs a) {
    __shared__ Smem S;
    const ListSeg& g = a.g;
    DevState* st = a.st;
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    uint32_t* ctr = a.ctr;
    uint32_t blocks = gridDim.x, target = 0;
    Ctx c{a, g, 0, 0, 0, 0, {}};
    const uint64_t t0 = globaltimer_ns();
    if (blockIdx.x == 0) {
        for (uint32_t i = tid; i < 64; i += RT) { st->ring_m[i] = 0; st->ring_n[i] = 0; }
        if (tid == 0) {
            st->err = 0; st->err_info = 0; st->rounds = 0; st->done = 0;
            st->matched2 = 0; st->tail = 0; st->tail_round = 0; st->round = 0;
            st->t0_ns = t0;
        }
    }
    for (uint64_t v = (uint64_t)blockIdx.x * RT + tid; v < g.n; v += (uint64_t)blocks * RT) {
        g.dst[v] = NIL;
        if ((v & 31) == 0) c.a.dead[v >> 5] = 0;
    }
#pragma unroll
    for (int k = 0; k < KINDS; k++) c.cnt[k] = k < 4 ? g.ntask[k] - kind_from(g, k) : g.nrows;
    for (;; c.round++) {
        const uint64_t z = splitmix64_at(g.seed, c.round);
        c.k0 = (uint32_t)z;
        c.k1 = (uint32_t)(z >> 32);
        unsigned long long ent = 0;
        // candidates: warps take units of work from a counter, the largest first, a few at
        // a time (row lengths depend on vertex ids, so that a fixed share for each warp left
        // half of them waiting)
        {
            const uint32_t u0 = c.cnt[0] + c.cnt[1], u1 = u0 + c.cnt[2], u2 = u1 + (c.cnt[3] + 7) / 8,
                           u3 = u2 + (c.cnt[4] + 31) / 32;
            const uint32_t W = blocks * RW, grab = max(1u, u3 / (W * 8));
            uint32_t* units = ctr + UNITS + (c.round & 1);
            uint32_t from = (blockIdx.x * RW + warp) * grab;   // (the first without the counter)
            while (from < u3) {
                uint32_t next = 0;
                if (u3 > W * grab && lane == 0) next = atomicAdd(units, grab);
                for (uint32_t u = from; u < min(from + grab, u3); u++) {
                    if (u < u1) {
                        const int kind = u < c.cnt[0] ? 0 : u < u0 ? 1 : 2;
                        long_row<COUNT>(c, item(c, kind, u - (kind == 0 ? 0u : kind == 1 ? c.cnt[0] : u0)), ent);
                    } else if (u < u2) {
                        for (uint32_t i = 4 * (u - u1); i < min(4 * (u - u1) + 4, (c.cnt[3] + 1) / 2); i++)
                            group_rows<COUNT>(c, i, ent);
                    } else {
                        const uint32_t i = 32 * (u - u2) + lane;
                        if (i < c.cnt[4]) short_row<COUNT>(c, item(c, 4, i), ent);
                    }
                }
                if (u3 <= W * grab) break;
                from = __shfl_sync(FULL, next, 0) + W * grab;
            }
        }
        const uint32_t out = c.buf ^ 1u;
        if (blockIdx.x == 0 && tid < KINDS) ctr[out * KINDS + tid] = 0;
        if (!barrier(ctr + BAR, target, blocks, st, S)) break;
        // match
        uint32_t live = 0, matched = 0;
        if (blockIdx.x == 0 && tid == 0) ctr[UNITS + ((c.round + 1) & 1)] = 0;
        {
            // all kinds in one row of numbers, 128 a warp and step, so that their chains of
            // loads run side by side
            uint32_t end[KINDS], all = 0;
#pragma unroll
            for (int k = 0; k < KINDS; k++) end[k] = all += c.cnt[k];
            auto end_of = [&](int k) {   // (by selects, so that end stays in registers)
                uint32_t x = 0;
#pragma unroll
                for (int z = 0; z < KINDS; z++) x = k == z ? end[z] : x;
                return x;
            };
            auto kind_of = [&](uint32_t i) {
                int k = 0;
#pragma unroll
                for (int z = 0; z < KINDS - 1; z++) k += i >= end[z];
                return k;
            };
            for (uint32_t b = (blockIdx.x * RW + warp) * 128; b < all; b += blocks * RW * 128) {
                uint32_t it[4], v[4], u[4], w[4], keep = 0, mine = 0;
#pragma unroll
                for (int q = 0; q < 4; q++) {
                    const uint32_t i = b + 32 * q + lane;
                    const int k = kind_of(i);
                    it[q] = i < all ? item(c, k, i - end_of(k - 1)) : NIL;
                }
#pragma unroll
                for (int q = 0; q < 4; q++) {
                    v[q] = NONE;
                    if (it[q] == NIL) continue;
                    if (b + 32 * q + lane < end[3]) {
                        const uint4 d4 = __ldg(g.task + it[q]);
                        v[q] = d4.x;
                        // (a row's later chunks go with the first)
                        if (b + 32 * q + lane >= end[0] || d4.w == 0) mine |= 1u << q;
                    } else {
                        mine |= 1u << q;
                        if (c.round || __ldg(g.roff + it[q] + 1) - __ldg(g.roff + it[q]) <= LIST_SHORT)
                            v[q] = __ldg(g.vid + it[q]);
                    }
                }
#pragma unroll
                for (int q = 0; q < 4; q++) u[q] = v[q] != NONE ? __ldcg(c.a.cur + v[q]) : NONE;
#pragma unroll
                for (int q = 0; q < 4; q++) w[q] = u[q] != NONE ? __ldcg(c.a.cur + u[q]) : NONE;
#pragma unroll
                for (int q = 0; q < 4; q++) {
                    if (u[q] == NONE) continue;
                    live += (mine >> q) & 1u;
                    if (w[q] != v[q]) {
                        keep |= 1u << q;
                    } else if ((mine >> q) & 1u) {
                        g.dst[v[q]] = u[q];
                        atomicOr(c.a.dead + (v[q] >> 5), 1u << (v[q] & 31));
                        matched++;
                    }
                }
                const int k1 = kind_of(min(b + 127, all - 1));
                for (int k = kind_of(b); k <= k1; k++) {
                    const uint32_t lo = end_of(k - 1), hi = end_of(k);
                    uint32_t bal[4], total = 0;
#pragma unroll
                    for (int q = 0; q < 4; q++) {
                        const uint32_t i = b + 32 * q + lane;
                        bal[q] = __ballot_sync(FULL, ((keep >> q) & 1u) && i >= lo && i < hi);
                        total += __popc(bal[q]);
                    }
                    uint32_t at = 0;
                    if (lane == 0 && total) at = atomicAdd(&ctr[out * KINDS + k], total);
                    at = __shfl_sync(FULL, at, 0);
#pragma unroll
                    for (int q = 0; q < 4; q++) {
                        if ((bal[q] >> lane) & 1u) *place(c, k, out, at + __popc(bal[q] & lanemask_lt())) = it[q];
                        at += __popc(bal[q]);
                    }
                }
            }
        }
        // the round's tallies
        live = __reduce_add_sync(FULL, live);
        matched = __reduce_add_sync(FULL, matched);
        if (COUNT)
            for (int o = 16; o > 0; o >>= 1) ent += __shfl_xor_sync(FULL, ent, o);
        __syncthreads();
        if (lane == 0) {
            S.red[0][warp] = live;
            S.red[1][warp] = matched;
            S.ent[warp] = ent;
        }
        __syncthreads();
        if (tid == 0) {
            uint32_t l = 0, m = 0;
            unsigned long long en = 0;
            for (uint32_t x = 0; x < RW; x++) {
                l += S.red[0][x];
                m += S.red[1][x];
                en += S.ent[x];
            }
            if (m) atomicAdd(&st->matched2, (unsigned long long)m);
            if (COUNT && c.round < 64) {
                if (l) atomicAdd(reinterpret_cast<unsigned long long*>(&st->ring_n[c.round]), (unsigned long long)l);
                if (en) atomicAdd(reinterpret_cast<unsigned long long*>(&st->ring_m[c.round]), en);
            }
            if (l) {
                atomicMax(&st->rounds, c.round + 1);
                if (c.round + 1 > a.max_rounds) set_err(st, ERR_TIMEOUT, c.round + 1);
            }
            if (blockIdx.x == 0 && globaltimer_ns() - t0 > a.limit_ns) set_err(st, ERR_TIMEOUT, c.round);
        }
        if (!barrier(ctr + BAR, target, blocks, st, S)) break;
        // (the error bits and lengths change again only after the next barrier)
        uint32_t total = 0;
#pragma unroll
        for (int k = 0; k < KINDS; k++) total += c.cnt[k] = __ldcg(ctr + out * KINDS + k);
        c.buf = out;
        if (total == 0 || ld_volatile_u32(&st->err)) break;
        if (blocks > 1 && tail(c.cnt)) {
            if (blockIdx.x) return;
            blocks = 1;
        }
    }
    if (blockIdx.x) return;
    __syncthreads();
    if (COUNT)
        for (uint32_t i = tid; i < 64; i += RT) st->ring_m[i] /= 2;   // both ends counted every edge
    if (tid == 0) st->done = 1;
    __threadfence();
    __syncthreads();
    if (a.host) state_to_host(a.host, st, RT);
}

}  // namespace

// (every block resident, and no more than have work)
int launch_renew(void* stream, const RenewArgs& a, bool counts) {
    int dev = 0;
    cudaGetDevice(&dev);
    const uint32_t* t = a.g.ntask;
    const uint64_t warps = (uint64_t)t[2] + (t[3] - t[2] + 7) / 8 + (a.g.nrows + 31) / 32;
    const uint64_t most = (uint64_t)device_sm_count(dev) * RMINB;
    // (a graph with few edges: blocks that clear its result, 64 vertices a thread; by its rows'
    // block alone 5M vertices and 100 edges took 749 us)
    const uint64_t want = std::max((warps + RW - 1) / RW, (uint64_t)a.g.n / (64 * RT));
    const uint32_t grid = (uint32_t)(want < 1 ? 1 : want < most ? want : most);
    static_assert(BAR < RENEW_CTRS, "counters");
    const cudaError_t e = cudaMemsetAsync(a.ctr, 0, RENEW_CTRS * sizeof(uint32_t), (cudaStream_t)stream);
    if (e != cudaSuccess) return (int)e;
    void* params[] = {const_cast<RenewArgs*>(&a)};
    const void* f = counts ? (const void*)k_renew<true> : (const void*)k_renew<false>;
    return (int)cudaLaunchCooperativeKernel(f, dim3(grid), dim3(RT), params, 0, (cudaStream_t)stream);
}

}  // namespace lm
