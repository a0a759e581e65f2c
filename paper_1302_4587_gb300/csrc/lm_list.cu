// The list path of the matching: local max without compaction and without rounds.
//
// A vertex only ever looks at the heaviest few of its edges before it is
// matched or runs out of live neighbours (2.3 to 2.5 entries a row on random,
// grid and R-MAT graphs, 9% to 40% of the adjacency entries).  So one pass over
// the adjacency arrays (k_top) keeps the heaviest neighbours of every row, in
// order -- four, eight of the longer rows --, and no entry is read again unless
// those are used up:
//
//   k_top   every row's candidate (Sec. 2.1, step 2) and the next of its list
//   k_live  the live rows until none is left.  A row looks at its candidate's
//           word: chosen back, it is matched (step 3); matched to another, the row
//           moves on to the next of its list that is not (steps 4 to 6 without
//           moving an edge: an edge is dead when the word of its other end says so),
//           and scans its adjacency once more for the heaviest live ones
//           when the list is used up; otherwise it stays as it is.
//
// A vertex's word is its candidate, with DEAD set once it is matched (to it).
// Only the thread that holds the row writes the word, and a row passes over a
// neighbour only once that one is matched for good.  So when two words name each
// other, everything heavier at either end is gone and the edge is in the greedy
// matching, whenever either thread looks: the result needs no barrier between
// rounds, and a word that is seen late only delays its reader.
//
// The rounds of the synchronous algorithm are recovered exactly where they are
// wanted (64-bit words): an edge is chosen in the round after the last of the
// heavier edges at its ends went, so a matched vertex's word carries its round,
// a live one's the latest round among the neighbours it has passed over.
#include <cuda_runtime.h>
#include <stdint.h>
#include <string.h>

#include "../../include/lm.h"
#include "lm_device.cuh"
#include "lm_internal.h"

namespace lm {

namespace {

constexpr uint32_t DEAD = 0x80000000u, VMASK = 0x7FFFFFFFu;

// ---------------------------------------------------------------- words
// W = uint32_t: candidate | DEAD.  W = uint64_t: the same in the low half; above it
// 1 + the round the vertex was matched in (DEAD), or the largest such number among
// the neighbours the row has passed over (0: none).
__device__ __forceinline__ uint32_t lo(uint32_t w) { return w; }
__device__ __forceinline__ uint32_t lo(uint64_t w) { return (uint32_t)w; }
__device__ __forceinline__ uint32_t info(uint32_t) { return 0; }
__device__ __forceinline__ uint32_t info(uint64_t w) { return (uint32_t)(w >> 32); }
template <class W>
__device__ __forceinline__ W word(uint32_t c, uint32_t inf) {
    if (sizeof(W) == 4) return (W)c;
    return (W)(((uint64_t)inf << 32) | c);
}
template <class W>
__device__ __forceinline__ W* words(const ListArgs& a) { return reinterpret_cast<W*>(a.cur); }
// words change while others read them: always from L2
__device__ __forceinline__ uint32_t look(const uint32_t* p) { return __ldcg(p); }
__device__ __forceinline__ uint64_t look(const uint64_t* p) {
    return __ldcg(reinterpret_cast<const unsigned long long*>(p));
}

// ---------------------------------------------------------------- a row's list
// The candidate is the row's word; the next three neighbours and the flags sit in
// lst[v] (x, y, z, w), four more in wide[v] if WIDE is set.  MORE: the row holds
// entries beyond its list.  An empty place is NIL.  Where rounds are wanted and the
// list comes from a refill (HASR), rl[v] and rw[v] hold beside every place the latest
// round (plus one) among the neighbours above it that were matched by then: the row
// passes over them with that place.
struct RowLists {
    uint4 *lst, *wide, *rl, *rw;
};
__device__ __forceinline__ RowLists row_lists(const ListArgs& a, uint32_t vbase) {
    return {a.lst + vbase, a.wide + vbase, a.rl ? a.rl + vbase : nullptr, a.rw ? a.rw + vbase : nullptr};
}
// Above the flags: the largest ord(w) that an entry beyond the list can have (its low
// bits lost): a scan of a long row need not look at the ends of heavier ones, which are
// all matched (rows of at most 128 entries look at all ends at once).
constexpr uint32_t MORE = 1u, WIDE = 2u, HASR = 4u, FLAGS = 7u;
constexpr int KS = 4, KL = LIST_KEPT;   // list lengths: rows of at most LIST_SHORT entries, longer ones

// entry i of a graph: ord(w), its neighbour, its full key
__device__ __forceinline__ uint32_t ord_at(const ListSeg& g, uint32_t i) {
    return __ldg(reinterpret_cast<const uint32_t*>(g.ent) + 2 * (size_t)i + 1);
}
__device__ __forceinline__ uint32_t nbr_at(const ListSeg& g, uint32_t i) {
    return __ldg(reinterpret_cast<const uint32_t*>(g.ent) + 2 * (size_t)i);
}
__device__ __forceinline__ uint64_t key_of(const ListSeg& g, uint32_t ord, uint32_t i) {
    return ((uint64_t)ord << 32) | perm_seed(__ldg(g.eid + i), g.k0, g.k1);
}

// Entries are compared by ord(w) alone where that decides: perm_seed tells equal
// ones apart, and only rows where it matters (two of the list, or its last and one
// left out, are equal) are taken again by their full keys.
//
// Up to 256 entries are compared as 32-bit numbers: ord(w) with its low bits
// replaced by the entry's place in the row (smaller first), so that an exchange is
// one minimum and one maximum and no two are equal.  Entries whose ord agrees above
// those bits count as equal.
__device__ __forceinline__ uint32_t packed(uint32_t ord, uint32_t idx, uint32_t mask) {
    return (ord & ~mask) | (mask - idx);
}
__device__ __forceinline__ void order2(uint32_t& a, uint32_t& b) {
    const uint32_t hi = max(a, b);
    b = min(a, b);
    a = hi;
}
template <int E>
__device__ __forceinline__ void order(uint32_t x[E]);
template <>
__device__ __forceinline__ void order<4>(uint32_t x[4]) {
    order2(x[0], x[1]); order2(x[2], x[3]);
    order2(x[0], x[2]); order2(x[1], x[3]);
    order2(x[1], x[2]);
}
template <>
__device__ __forceinline__ void order<8>(uint32_t x[8]) {   // Batcher's odd-even merge sort
    order<4>(x);
    order<4>(x + 4);
    order2(x[0], x[4]); order2(x[1], x[5]); order2(x[2], x[6]); order2(x[3], x[7]);
    order2(x[2], x[4]); order2(x[3], x[5]);
    order2(x[1], x[2]); order2(x[3], x[4]); order2(x[5], x[6]);
}

// a thread's four largest of any number of such entries, taken four at a time
struct Top4 {
    uint32_t k[4] = {0, 0, 0, 0};
    uint32_t out = 0;                 // largest one left out
    // the larger of each pair taken head to tail from two ordered fours is one of the
    // four largest (a bitonic four), then put in order
    __device__ __forceinline__ void take(uint32_t x[4]) {
        order<4>(x);
        out = max(out, max(max(min(k[0], x[3]), min(k[1], x[2])), max(min(k[2], x[1]), min(k[3], x[0]))));
#pragma unroll
        for (int i = 0; i < 4; i++) k[i] = max(k[i], x[3 - i]);
        order2(k[0], k[2]); order2(k[1], k[3]);
        order2(k[0], k[1]); order2(k[2], k[3]);
    }
};
// equal neighbours in an ordered list r of K, the last against the largest left out (a
// place without an entry packs to a number of at most `mask`, below every entry's)
template <int K>
__device__ __forceinline__ bool any_tie(const uint32_t r[K], uint32_t out, uint32_t mask) {
    bool t = out > mask && (r[K - 1] ^ out) <= mask;
#pragma unroll
    for (int i = 1; i < K; i++) t |= r[i] > mask && (r[i - 1] ^ r[i]) <= mask;
    return t;
}
// maximum over an aligned group of G lanes
template <int G>
__device__ __forceinline__ uint32_t group_max(uint32_t x) {
    if constexpr (G == 32) {
        return __reduce_max_sync(FULL, x);
    } else {
#pragma unroll
        for (int d = 1; d < G; d <<= 1) x = max(x, __shfl_xor_sync(FULL, x, d));
        return x;
    }
}
template <int G>
__device__ __forceinline__ uint64_t group_max64(uint64_t x) {
#pragma unroll
    for (int d = 1; d < G; d <<= 1) {
        const uint64_t o = __shfl_xor_sync(FULL, x, d);
        x = o > x ? o : x;
    }
    return x;
}
// The K largest of a group's entries, E packed ones a lane: every lane in order, then
// the largest head K times.  r: the same for all lanes; returns the largest left out.
template <int G, int E, int K>
__device__ __forceinline__ uint32_t group_top(uint32_t x[E], uint32_t r[K]) {
    order<E>(x);
#pragma unroll
    for (int i = 0; i < K; i++) {
        const uint32_t h = group_max<G>(x[0]);
        r[i] = h;
        const bool mine = x[0] == h;
#pragma unroll
        for (int e = 0; e + 1 < E; e++) x[e] = mine ? x[e + 1] : x[e];
        x[E - 1] = mine ? 0u : x[E - 1];
    }
    return group_max<G>(x[0]);
}
// the same by full key among the entries in `live` (bit e; entry e * G + the lane's
// place): positions (NIL: none) and keys; returns whether others are left
template <int G, int E, int K>
__device__ __forceinline__ bool group_top_keyed(const uint64_t key[E], uint32_t live, uint32_t sub, uint32_t p[K],
                                                uint64_t k[K]) {
    uint32_t left = live;
#pragma unroll
    for (int i = 0; i < K; i++) {
        uint64_t m = 0;
        uint32_t at = NIL;
#pragma unroll
        for (int e = 0; e < E; e++)
            if (((left >> e) & 1u) && key[e] > m) { m = key[e]; at = e; }
        const uint64_t b = group_max64<G>(m);
        const bool own = b && b == m;
        p[i] = ~group_max<G>(own ? ~(at * G + sub) : 0u);   // (the owner's position; NIL without one)
        if (own) left &= ~(1u << at);
        k[i] = b;
    }
    return group_max<G>(left) != 0;
}

// A warp's KL largest of any number of entries, in order, one to a lane (lane i < KL
// has the i-th): by ord(w) with the position, or by full key with the neighbour.  The
// other lanes hold 0.
struct LaneTop32 {
    uint32_t o = 0, p = NIL;
    __device__ __forceinline__ uint32_t last() const { return __shfl_sync(FULL, o, KL - 1); }
    __device__ __forceinline__ void put(uint32_t h, uint32_t hp) {   // h differs from all of the list
        const uint32_t lane = threadIdx.x & 31;
        const uint32_t at = __popc(__ballot_sync(FULL, o > h));
        const uint32_t uo = __shfl_up_sync(FULL, o, 1), up = __shfl_up_sync(FULL, p, 1);
        if (lane >= at && lane < KL) {
            o = lane == at ? h : uo;
            p = lane == at ? hp : up;
        }
    }
};
struct LaneTop64 {
    uint64_t k = 0;
    uint32_t n = NIL;
    __device__ __forceinline__ uint64_t last() const { return __shfl_sync(FULL, k, KL - 1); }
    __device__ __forceinline__ void put(uint64_t h, uint32_t hn) {
        const uint32_t lane = threadIdx.x & 31;
        const uint32_t at = __popc(__ballot_sync(FULL, k > h));
        const uint64_t uk = __shfl_up_sync(FULL, k, 1);
        const uint32_t un = __shfl_up_sync(FULL, n, 1);
        if (lane >= at && lane < KL) {
            k = lane == at ? h : uk;
            n = lane == at ? hn : un;
        }
    }
    // every lane offers (key, neighbour), 0 for none: those above the last go in
    __device__ __forceinline__ void offer(uint64_t key, uint32_t nb) {
        for (uint64_t bar = last(); __any_sync(FULL, key > bar); bar = last()) {
            const uint32_t hi = __reduce_max_sync(FULL, (uint32_t)(key >> 32));
            const uint32_t lw = __reduce_max_sync(FULL, ((uint32_t)(key >> 32) == hi) ? (uint32_t)key : 0u);
            const uint64_t best = ((uint64_t)hi << 32) | lw;
            const int L = __ffs(__ballot_sync(FULL, key == best)) - 1;
            put(best, __shfl_sync(FULL, nb, L));
            if ((int)(threadIdx.x & 31) == L) key = 0;
        }
    }
};

// A list into row `at`'s places: lane (or group lane) i has the i-th neighbour c (NIL:
// none) and, with rounds, the r that goes with it; lane 0's r joins the word.
template <class W, int K>
__device__ __forceinline__ void put_list(W* cur, const RowLists& R, size_t at, uint32_t sub, uint32_t c, uint32_t r,
                                         uint32_t flags) {
    uint32_t* l = reinterpret_cast<uint32_t*>(R.lst + at);
    if (sub == 0) cur[at] = word<W>(c, r);
    else if (sub < 3) l[sub - 1] = c;
    else if (sub == 3) *reinterpret_cast<uint2*>(l + 2) = make_uint2(c, flags);
    else if (sub < K) reinterpret_cast<uint32_t*>(R.wide + at)[sub - 4] = c;
    if (sizeof(W) == 8 && (flags & HASR)) {
        if (sub > 0 && sub < 4) reinterpret_cast<uint32_t*>(R.rl + at)[sub - 1] = r;
        else if (sub >= 4 && sub < K) reinterpret_cast<uint32_t*>(R.rw + at)[sub - 4] = r;
    }
}

// A job's arguments and a graph's record are read from shared memory: from global
// memory through two pointers they were loaded again after every barrier and atomic, or
// held in registers that the rows need.
template <class T>
__device__ __forceinline__ void copy_words(T* to, const T* from, uint32_t threads) {
    static_assert(sizeof(T) % 4 == 0, "words");
    for (uint32_t i = threadIdx.x; i < sizeof(T) / 4; i += threads)
        reinterpret_cast<uint32_t*>(to)[i] = reinterpret_cast<const uint32_t*>(from)[i];
}

// ---------------------------------------------------------------- k_top
constexpr int TT = 256, TWARPS = TT / 32;
constexpr uint32_t MPW = 2;       // long-row tasks a warp takes,
constexpr uint32_t WPW = 8;       // rows of LIST_GROUP + 1 .. LIST_WARP entries,
constexpr uint32_t GPW = 16;      // and rows of LIST_SHORT + 1 .. LIST_GROUP
static_assert(LIST_SHORT == 32 && LIST_GROUP == 8 * 8 && LIST_WARP == 8 * 32, "eight entries a lane");

// A row of at most LIST_SHORT entries by one thread, four entries at a time, the next
// four on their way.  Neighbouring threads' rows are neighbours in the arrays, so
// their loads share sectors through L1 (staging the entries through shared memory
// first cost more instructions than it saved wavefronts).
template <class W>
__device__ __forceinline__ void top_short(const ListArgs& a, const ListSeg& g, uint32_t r) {
    uint32_t o = 0, d = 0, v = 0;
    if (r < g.nrows) {
        o = __ldg(g.roff + r);
        d = __ldg(g.roff + r + 1) - o;
        v = __ldg(g.vid + r);
    }
    if (d == 0 || d > LIST_SHORT) return;
    constexpr uint32_t MASK = LIST_SHORT - 1;
    Top4 t;
    uint32_t x[4], nx[4];
    auto load = [&](uint32_t y[4], uint32_t j) {
#pragma unroll
        for (uint32_t q = 0; q < 4; q++) y[q] = j + q < d ? ord_at(g, o + j + q) : 0u;
    };
    load(x, 0);
#pragma unroll
    for (uint32_t j = 0; j < LIST_SHORT; j += 4) {   // (unrolled: the places are constants)
        if (j >= d) break;
        if (j + 4 < LIST_SHORT) load(nx, j + 4);
#pragma unroll
        for (uint32_t q = 0; q < 4; q++) x[q] = packed(x[q], j + q, MASK);
        t.take(x);
#pragma unroll
        for (int q = 0; q < 4; q++) x[q] = nx[q];
    }
    uint32_t p[4];
#pragma unroll
    for (int i = 0; i < 4; i++) p[i] = MASK - (t.k[i] & MASK);
    if (any_tie<4>(t.k, t.out, MASK)) {
        // by full key
        uint64_t k[4] = {0, 0, 0, 0};
        for (uint32_t j = 0; j < d; j++) {
            uint64_t x64 = key_of(g, ord_at(g, o + j), o + j);
            uint32_t px = j;
#pragma unroll
            for (int i = 0; i < 4; i++) {
                const bool gt = x64 > k[i];
                const uint64_t tk = k[i];
                const uint32_t tp = p[i];
                k[i] = gt ? x64 : tk;
                p[i] = gt ? px : tp;
                x64 = gt ? tk : x64;
                px = gt ? tp : px;
            }
        }
    }
    const size_t at = (size_t)g.vbase + v;
    words<W>(a)[at] = word<W>(nbr_at(g, o + p[0]), 0);
    a.lst[at] = make_uint4(d > 1 ? nbr_at(g, o + p[1]) : NIL, d > 2 ? nbr_at(g, o + p[2]) : NIL,
                           d > 3 ? nbr_at(g, o + p[3]) : NIL, d > 4 ? MORE | (t.k[3] & ~FLAGS) | (MASK & ~FLAGS) : 0u);
}

// Rows of more than LIST_SHORT entries, eight entries to each of the G lanes of a group
// (32 / G rows at a time), straight from the arrays into registers; the next rows'
// entries are on their way while these are compared.
template <class W, int G>
__device__ __forceinline__ void top_group(const ListArgs& a, const ListSeg& g, uint32_t t0, uint32_t cnt) {
    constexpr uint32_t ROWS = 32 / G, MASK = 8 * G - 1;
    const uint32_t lane = threadIdx.x & 31, sub = lane & (G - 1), grp = lane / G;
    uint4 d4 = make_uint4(0, 0, 0, 0);
    if (lane < cnt) d4 = __ldg(g.task + t0 + lane);
    uint32_t v = 0, s = 0, d = 0, x[8];
    auto fetch = [&](uint32_t i) {
        v = __shfl_sync(FULL, d4.x, (i + grp) & 31u);
        s = __shfl_sync(FULL, d4.y, (i + grp) & 31u);
        d = __shfl_sync(FULL, d4.z, (i + grp) & 31u);
        if (i + grp >= cnt) d = 0;
#pragma unroll
        for (int e = 0; e < 8; e++) x[e] = e * G + sub < d ? ord_at(g, s + e * G + sub) : 0u;
    };
    fetch(0);
    for (uint32_t i = 0; i < cnt; i += ROWS) {
        const uint32_t cv = v, cs = s, cd = d;
#pragma unroll
        for (int e = 0; e < 8; e++) x[e] = packed(x[e], e * G + sub, MASK);
        uint32_t r[KL];
        const uint32_t out = group_top<G, 8, KL>(x, r);
        uint32_t mine = r[0];
#pragma unroll
        for (int q = 1; q < KL; q++) mine = (sub & 7u) == (uint32_t)q ? r[q] : mine;
        uint32_t p = MASK - (mine & MASK);
        if (__any_sync(FULL, any_tie<KL>(r, out, MASK))) {
            uint64_t key[8], kk[KL];
            uint32_t pk[KL];
#pragma unroll
            for (int e = 0; e < 8; e++)
                key[e] = e * G + sub < cd ? key_of(g, ord_at(g, cs + e * G + sub), cs + e * G + sub) : 0ull;
            group_top_keyed<G, 8, KL>(key, 0xFFu, sub, pk, kk);
            p = pk[0];
#pragma unroll
            for (int q = 1; q < KL; q++) p = (sub & 7u) == (uint32_t)q ? pk[q] : p;
        }
        uint32_t c = 0;
        if (cd && sub < KL) c = nbr_at(g, cs + p);
        if (i + ROWS < cnt) fetch(i + ROWS);
        if (cd) put_list<W, KL>(words<W>(a) + g.vbase, row_lists(a, g.vbase), cv, sub, c, 0,
                                WIDE | MORE | ((r[KL - 1] | MASK) & ~FLAGS));
    }
}

// Long-row tasks (a row of more than LIST_WARP entries, or a LIST_CHUNK-entry chunk of
// one longer than that), the warp together: 256 entries a step in 16-byte loads, the
// next step's on their way.  An entry is compared as its ord(w) with the low three
// bits replaced by its place among the lane's eight; equal ones above those bits
// are a tie.  The first step's list comes from the lanes' ordered eights; a later
// step whose entries all lie below the list costs a maximum and a vote, and one that
// does not is put in with a warp maximum.
template <class W>
__device__ __forceinline__ void top_long(const ListArgs& a, const ListSeg& g, uint32_t t) {
    const uint32_t lane = threadIdx.x & 31;
    const uint4 d4 = __ldg(g.task + t);
    const uint32_t v = d4.x, len = d4.z, c = d4.w;
    const bool whole = len <= LIST_CHUNK;
    const uint32_t s = d4.y + c * LIST_CHUNK, e = whole ? d4.y + len : d4.y + min(len, (c + 1) * LIST_CHUNK);
    LaneTop32 top;
    // pairs start at an even entry (the array is 256-byte aligned)
    auto load = [&](uint32_t y[8], uint64_t pos) {
        if (pos >= s && pos + 256 <= e) {
#pragma unroll
            for (int q = 0; q < 4; q++) {
                const uint4 w = __ldg(reinterpret_cast<const uint4*>(g.ent + pos + 64 * q + 2 * lane));
                y[2 * q] = w.y;
                y[2 * q + 1] = w.w;
            }
        } else {
#pragma unroll
            for (int q = 0; q < 8; q++) {
                const uint64_t i = pos + 64 * (q >> 1) + 2 * lane + (q & 1);
                y[q] = i >= s && i < e ? ord_at(g, (uint32_t)i) : 0u;
            }
        }
    };
    // the entry a packed number of lane L stands for
    auto place = [&](uint32_t pos, uint32_t h, uint32_t L) {
        const uint32_t z = 7u - (h & 7u);
        return pos + 64 * (z >> 1) + 2 * L + (z & 1);
    };
    uint32_t x[8], y[8];
    uint64_t pos = s & ~1u;
    load(x, pos);
    load(y, pos + 256);
    bool tie;
    {
#pragma unroll
        for (uint32_t z = 0; z < 8; z++) x[z] = packed(x[z], z, 7u);
        order<8>(x);
        uint32_t prev = ~0u, left = 0;
        bool same = false;
#pragma unroll
        for (int i = 0; i <= KL; i++) {
            const uint32_t h = __reduce_max_sync(FULL, x[0]);
            const uint32_t own = __ballot_sync(FULL, x[0] == h);
            same |= h > 7u && ((prev ^ h) <= 7u || (own & (own - 1)));
            prev = h;
            if (i == KL) { left = h; break; }
            const uint32_t L = __ffs(own) - 1;
            if (h > 7u && (int)lane == i) {
                top.o = h & ~7u;
                top.p = place((uint32_t)pos, h, L);
            }
            const bool mine = lane == L;
#pragma unroll
            for (int z = 0; z < 7; z++) x[z] = mine ? x[z + 1] : x[z];
            x[7] = mine ? 0u : x[7];
        }
        (void)left;
        tie = same;
    }
    uint32_t bar = max(top.last(), 8u);
    auto step = [&](uint32_t w[8]) {
        uint32_t m = max(max(max(w[0], w[1]), max(w[2], w[3])), max(max(w[4], w[5]), max(w[6], w[7])));
        if (!__any_sync(FULL, m >= bar)) return;
#pragma unroll
        for (uint32_t z = 0; z < 8; z++) w[z] = packed(w[z], z, 7u);
        for (;;) {
            m = max(max(max(w[0], w[1]), max(w[2], w[3])), max(max(w[4], w[5]), max(w[6], w[7])));
            const uint32_t h = __reduce_max_sync(FULL, m);
            if (h < bar) return;
            const uint32_t own = __ballot_sync(FULL, m == h);
            if (__any_sync(FULL, top.o == (h & ~7u)) || (own & (own - 1))) {
                tie = true;
                return;
            }
            top.put(h & ~7u, place((uint32_t)pos, h, __ffs(own) - 1));
#pragma unroll
            for (int z = 0; z < 8; z++) w[z] = m == h && w[z] == h ? 0u : w[z];
            bar = max(top.last(), 8u);
        }
    };
    pos += 256;
    while (pos < e && !tie) {
        load(x, pos + 256);
        step(y);
        pos += 256;
        if (pos >= e || tie) break;
        load(y, pos + 256);
        step(x);
        pos += 256;
    }
    uint32_t p = top.p;
    if (tie) {
        LaneTop64 kt;
        // four entries a lane and step, so that their loads go side by side (1000 rows of 4000
        // equal weights: 110 us one by one, 75 so); by places within the row: positions
        // may end close to 2^32
        const uint32_t d = e - s;
        for (uint32_t k = 0; k < div_up(d, 128); k++) {
            uint32_t o[4], id[4];
#pragma unroll
            for (uint32_t q = 0; q < 4; q++) {
                const uint32_t j = 128 * k + 32 * q + lane;
                o[q] = j < d ? ord_at(g, s + j) : 0u;
                id[q] = j < d ? __ldg(g.eid + s + j) : 0u;
            }
#pragma unroll
            for (uint32_t q = 0; q < 4; q++)   // (no entry has ord 0)
                kt.offer(o[q] ? ((uint64_t)o[q] << 32) | perm_seed(id[q], g.k0, g.k1) : 0ull,
                         s + 128 * k + 32 * q + lane);
        }
        p = kt.n;
        top.o = (uint32_t)(kt.k >> 32);
    }
    if (lane >= KL) p = NIL;
    if (whole) {
        const uint32_t last = top.last();
        put_list<W, KL>(words<W>(a) + g.vbase, row_lists(a, g.vbase), v, lane, p != NIL ? nbr_at(g, p) : NIL, 0,
                        WIDE | MORE | (last & ~FLAGS));
        return;
    }
    // a chunk: its list with the full keys; the last chunk of the row to finish merges all
    const uint32_t first = t - c;   // the row's chunk 0 in the task list
    const uint32_t nch = (len + LIST_CHUNK - 1) / LIST_CHUNK;
    if (lane < KL) {
        uint4 rec = make_uint4(0, 0, NIL, 0);
        if (p != NIL) {
            const uint64_t K = key_of(g, ord_at(g, p), p);
            rec = make_uint4((uint32_t)K, (uint32_t)(K >> 32), nbr_at(g, p), 0);
        }
        a.part[((size_t)g.lbase + t) * KL + lane] = rec;
    }
    __syncwarp();
    uint32_t old = 0;
    if (lane == 0) old = atom_add_acq_rel(&a.pcnt[(size_t)g.lbase + first], 1u);
    old = __shfl_sync(FULL, old, 0);
    __syncwarp();
    if (old != nch - 1) return;
    LaneTop64 kt;
    const uint4* P = a.part + ((size_t)g.lbase + first) * KL;
    for (uint32_t b = 0; b < nch * KL; b += 32) {
        uint4 rec = make_uint4(0, 0, NIL, 0);
        if (b + lane < nch * KL) rec = __ldcg(P + b + lane);
        kt.offer(((uint64_t)rec.y << 32) | rec.x, rec.z);
    }
    if (lane == 0) a.pcnt[(size_t)g.lbase + first] = 0;
    put_list<W, KL>(words<W>(a) + g.vbase, row_lists(a, g.vbase), v, lane, kt.n, 0,
                    WIDE | MORE | ((uint32_t)(kt.last() >> 32) & ~FLAGS));
}

// Blocks of k_top for one graph, in this order: long tasks, rows of a warp, rows of a
// group, and all rows 256 at a time for the short ones.
struct TopBlocks {
    uint32_t l, w, g, s;
};
__host__ __device__ __forceinline__ TopBlocks top_blocks(const uint32_t task[4], uint32_t nrows) {
    TopBlocks b;
    b.l = (task[1] + TWARPS * MPW - 1) / (TWARPS * MPW);
    b.w = (task[2] - task[1] + TWARPS * WPW - 1) / (TWARPS * WPW);
    b.g = (task[3] - task[2] + TWARPS * GPW - 1) / (TWARPS * GPW);
    b.s = (nrows + TT - 1) / TT;
    return b;
}

constexpr int TMINB = 6;
// Every block also clears its share of the result, and block 0 resets the job's state.  A
// graph with few edges has blocks of its vertices alone: its rows' block, 5M vertices and
// 100 edges, took 450 us to clear the result, these 1221 blocks 8.
constexpr uint32_t CLEAR = 4096;
template <class W>
__global__ void __launch_bounds__(TT, TMINB) k_top(const __grid_constant__ ListArgs a) {
    __shared__ ListSeg g;
    const uint32_t tid = threadIdx.x, warp = tid >> 5;
    if (blockIdx.x == 0) {
        DevState* st = a.st;
        for (uint32_t i = tid; i < 64; i += TT) { st->ring_m[i] = 0; st->ring_n[i] = 0; }
        if (tid < 4) st->task[tid] = 0;
        if (tid == 0) {
            st->exit_v = 0;
            st->left = 0;
            st->err = 0; st->err_info = 0; st->rounds = 0; st->done = 0;
            st->matched2 = 0; st->tail = 0; st->tail_round = 0;
            st->round = 0;
            st->t0_ns = globaltimer_ns();
        }
    }
    copy_words(&g, a.bmap ? a.segs + a.bmap[blockIdx.x] : &a.one, TT);
    __syncthreads();
    uint32_t b = blockIdx.x - g.blk0;
    {
        const uint32_t per = (uint32_t)(((uint64_t)g.n + g.nblk - 1) / g.nblk);
        const uint64_t from = (uint64_t)b * per, to = from + per < g.n ? from + per : g.n;
        for (uint64_t v = from + tid; v < to; v += TT) g.dst[v] = NIL;
    }
    const TopBlocks nb = top_blocks(g.ntask, g.nrows);
    if (b < nb.l) {
        const uint32_t t0 = (b * TWARPS + warp) * MPW;
        for (uint32_t t = t0; t < min(t0 + MPW, g.ntask[1]); t++) top_long<W>(a, g, t);
    } else if ((b -= nb.l) < nb.w) {
        const uint32_t t0 = g.ntask[1] + (b * TWARPS + warp) * WPW;
        if (t0 < g.ntask[2]) top_group<W, 32>(a, g, t0, min(WPW, g.ntask[2] - t0));
    } else if ((b -= nb.w) < nb.g) {
        const uint32_t t0 = g.ntask[2] + (b * TWARPS + warp) * GPW;
        if (t0 < g.ntask[3]) top_group<W, 8>(a, g, t0, min(GPW, g.ntask[3] - t0));
    } else {
        top_short<W>(a, g, (b - nb.g) * TT + tid);
    }
}

// ---------------------------------------------------------------- refills
// The K heaviest live entries of rows of at most G E entries, a group of G lanes
// each; d = 0: no row.  Returns whether one is left (uniform over the group).
template <class W, int G, int E, int K>
__device__ __forceinline__ bool refill_group(const ListSeg& g, W* cur, const RowLists& R, uint32_t v, uint32_t s,
                                             uint32_t d) {
    static_assert(G >= 4 && (K == KS || G >= 8), "a lane for every place");
    constexpr uint32_t MASK = G * E - 1;
    constexpr bool ROUNDS = sizeof(W) == 8;
    const uint32_t sub = threadIdx.x & (G - 1);
    uint32_t x[E], live = 0;
    W t[E];
    {
        uint32_t n[E];
#pragma unroll
        for (int e = 0; e < E; e++) {
            const uint64_t w = e * G + sub < d ? __ldg(g.ent + s + e * G + sub) : 0ull;
            x[e] = (uint32_t)(w >> 32);
            n[e] = (uint32_t)w;
        }
#pragma unroll
        for (int e = 0; e < E; e++) t[e] = e * G + sub < d ? look(cur + n[e]) : (W)DEAD;
    }
#pragma unroll
    for (int e = 0; e < E; e++)
        if (!(lo(t[e]) & DEAD)) live |= 1u << e;
    uint32_t p[K];
    uint32_t last = 0;   // ord(w) of the list's last place
    bool rest = false, exact = ROUNDS;
    uint32_t mr = 0;   // with rounds: the place's r
    if (!ROUNDS) {
        uint32_t y[E], r[K];
#pragma unroll
        for (int e = 0; e < E; e++) y[e] = packed(((live >> e) & 1u) ? x[e] : 0u, e * G + sub, MASK);
        const uint32_t out = group_top<G, E, K>(y, r);
#pragma unroll
        for (int i = 0; i < K; i++) p[i] = r[i] > MASK ? MASK - (r[i] & MASK) : NIL;
        rest = out > MASK;
        last = r[K - 1] | MASK;
        exact = __any_sync(FULL, any_tie<K>(r, out, MASK));
    }
    if (exact) {
        uint64_t key[E], k[K];
#pragma unroll
        for (int e = 0; e < E; e++) key[e] = e * G + sub < d ? key_of(g, x[e], s + e * G + sub) : 0ull;
        rest = group_top_keyed<G, E, K>(key, live, sub, p, k);
        if (ROUNDS) {
#pragma unroll
            for (int i = 0; i < K; i++) {
                uint32_t r = 0;
#pragma unroll
                for (int e = 0; e < E; e++)
                    if (e * G + sub < d && !((live >> e) & 1u) && key[e] > k[i]) r = max(r, info(t[e]));
                r = group_max<G>(r);
                mr = sub == (uint32_t)i ? r : mr;
            }
        }
    }
    if (d && p[0] != NIL) {
        uint32_t mp = p[0];
#pragma unroll
        for (int i = 1; i < K; i++) mp = sub == (uint32_t)i ? p[i] : mp;
        uint32_t c = NIL;
        if (sub < K && mp != NIL) c = nbr_at(g, s + mp);
        if (ROUNDS && sub == 0) mr = max(mr, info(look(cur + v)));
        put_list<W, K>(cur, R, v, sub, c, mr, 
                       (K == KL ? WIDE : 0u) | (rest ? MORE : 0u) | (ROUNDS ? HASR : 0u) | (last & ~FLAGS));
        return true;
    }
    return false;
}

// The same for longer rows: part `q` of `parts` of the row's 128-entry steps by this
// warp.  Only entries between the last of the list so far and ub have their end looked up.
template <class W>
__device__ __forceinline__ void refill_scan(const ListSeg& g, const W* cur, uint32_t s, uint32_t d, uint32_t ub,
                                            uint32_t q, uint32_t parts, LaneTop64& t) {
    const uint32_t lane = threadIdx.x & 31;
    const uint64_t stride = 128ull * parts;
    uint64_t x[4], nx[4];
    auto load = [&](uint64_t y[4], uint64_t b) {
#pragma unroll
        for (int i = 0; i < 4; i++) y[i] = b + 32 * i + lane < d ? __ldg(g.ent + s + (uint32_t)b + 32 * i + lane) : 0ull;
    };
    load(x, 128ull * q);
    uint32_t bar = 1;
    for (uint64_t b = 128ull * q; b < d; b += stride) {
        load(nx, b + stride);
        bool in[4];
#pragma unroll
        for (int i = 0; i < 4; i++) in[i] = (uint32_t)(x[i] >> 32) >= bar && (uint32_t)(x[i] >> 32) <= ub;
        if (__any_sync(FULL, in[0] | in[1] | in[2] | in[3])) {
            uint32_t y[4], e[4];   // (the indices together with the words, not one by one)
#pragma unroll
            for (int i = 0; i < 4; i++) {
                y[i] = in[i] ? lo(look(cur + (uint32_t)x[i])) : DEAD;
                e[i] = in[i] ? __ldg(g.eid + s + (uint32_t)b + 32 * i + lane) : 0u;
            }
#pragma unroll
            for (int i = 0; i < 4; i++) {
                const bool on = !(y[i] & DEAD) && (uint32_t)(x[i] >> 32) >= bar;
                if (!__any_sync(FULL, on)) continue;
                t.offer(on ? (x[i] & 0xFFFFFFFF00000000ull) | perm_seed(e[i], g.k0, g.k1) : 0ull, (uint32_t)x[i]);
                bar = max((uint32_t)(t.last() >> 32), 1u);
            }
        }
#pragma unroll
        for (int i = 0; i < 4; i++) x[i] = nx[i];
    }
}
// lane i < KL: the latest round (plus one) among the row's matched neighbours above the
// list's i-th key (part `q` of `parts` of the row)
__device__ __forceinline__ uint32_t refill_passed(const ListSeg& g, const uint64_t* cur, uint32_t s, uint32_t d,
                                                  uint32_t q, uint32_t parts, const LaneTop64& t) {
    uint64_t k[KL];
    uint32_t r[KL];
#pragma unroll
    for (int i = 0; i < KL; i++) {
        k[i] = __shfl_sync(FULL, t.k, i);
        r[i] = 0;
    }
    const uint32_t low = (uint32_t)(k[KL - 1] >> 32);
    // four entries a lane and step, their words and indices side by side
    for (uint64_t b = 128ull * q + (threadIdx.x & 31); b < d; b += 128ull * parts) {
        uint64_t w[4], y[4];
        uint32_t e[4];
#pragma unroll
        for (int z = 0; z < 4; z++) w[z] = b + 32 * z < d ? __ldg(g.ent + s + (uint32_t)b + 32 * z) : 0ull;
#pragma unroll
        for (int z = 0; z < 4; z++) {
            const bool on = b + 32 * z < d && (uint32_t)(w[z] >> 32) >= low;
            y[z] = on ? look(cur + (uint32_t)w[z]) : 0ull;
            e[z] = on ? __ldg(g.eid + s + (uint32_t)b + 32 * z) : 0u;
        }
#pragma unroll
        for (int z = 0; z < 4; z++) {
            if (!(lo(y[z]) & DEAD)) continue;
            const uint64_t key = (w[z] & 0xFFFFFFFF00000000ull) | perm_seed(e[z], g.k0, g.k1);
#pragma unroll
            for (int j = 0; j < KL; j++)
                if (key > k[j]) r[j] = max(r[j], info(y[z]));
        }
    }
    uint32_t mine = 0;
#pragma unroll
    for (int j = 0; j < KL; j++) {
        const uint32_t x = __reduce_max_sync(FULL, r[j]);
        mine = (threadIdx.x & 31) == (uint32_t)j ? x : mine;
    }
    return mine;
}
// t, r: lanes 0 .. KL - 1
template <class W>
__device__ __forceinline__ void refill_put(W* cur, const RowLists& R, uint32_t v, const LaneTop64& t, uint32_t r) {
    const uint32_t lane = threadIdx.x & 31;
    // (with a full list there may be more)
    const uint32_t flags = WIDE | (__shfl_sync(FULL, t.n, KL - 1) != NIL ? MORE : 0u) | (sizeof(W) == 8 ? HASR : 0u) |
                           ((uint32_t)(t.last() >> 32) & ~FLAGS);
    if (sizeof(W) == 8 && lane == 0) r = max(r, info(look(cur + v)));
    put_list<W, KL>(cur, R, v, lane, t.k ? t.n : NIL, r, flags);
}

// ---------------------------------------------------------------- k_live
constexpr int LT = 128, LW = LT / 32;
// blocks an SM, chosen on 32-bit words: 8 need no spills but 10 cover more latency (R-MAT scale 23
// 1.32 and 1.28 ms, 4096 graphs 3.88 and 3.80; 12: 1.30, 3.72, but coarsening 9.9 ms for 9.5).
// 64-bit words take the same 48 registers and spill 426 bytes of stores there.
constexpr int LMINB = 10;
constexpr uint32_t BLOCK_ROW = 1024;  // longer rows are refilled by the whole block
constexpr uint32_t IDLE_MAX = 48;     // passes without a change before a block gives its rows back

// places for the lanes that are on, from a counter
__device__ __forceinline__ uint32_t warp_slot(uint32_t* ctr, bool on) {
    const uint32_t b = __ballot_sync(FULL, on);
    if (!b) return 0;
    uint32_t base = 0;
    if ((threadIdx.x & 31) == 0) base = atomicAdd(ctr, (uint32_t)__popc(b));
    return __shfl_sync(FULL, base, 0) + __popc(b & lanemask_lt());
}
__device__ __forceinline__ void warp_append(uint32_t* ctr, uint32_t* out, bool on, uint32_t v) {
    const uint32_t q = warp_slot(ctr, on);
    if (on) out[q] = v;
}

// A part: every nparts-th run of 2^run consecutive rows of one graph (the long rows of a graph
// that numbers its vertices by degree, R-MAT's, a coarsened one's, would otherwise be in a
// few parts, which the others wait for: fifth level of R-MAT
// scale 20, 47 rounds: 2.26 ms by consecutive rows, 0.96 by runs of 8 to 64; runs of 8 cost
// graphs with local edges coalescing, a unit grid of 1M 115 and 138 us), its
// live rows compacted in its own range of the list buffers, its rows to refill in its
// range of the queue (vertex, row offset, length, heaviest entry to look at; rows of at
// most LIST_SHORT entries from the front, longer ones from the back).
template <class W>
struct Part {
    ListSeg g;
    W* cur;
    RowLists R;
    uint4* queue;
    uint32_t first, rows;  // its first run, and the rows it has
    size_t home;           // first slot of the part
    // (g is there)
    __device__ __forceinline__ void init(const ListArgs& a, uint32_t part) {
        const uint32_t p = part - g.part0, np = g.nparts;
        const uint32_t RUN = 1u << g.run;
        const uint32_t runs = (g.nrows + RUN - 1) >> g.run, q = runs / np, r = runs - q * np;
        const uint32_t missing = RUN * runs - g.nrows, owner = (runs - 1) % np;   // of the last run
        first = p;
        rows = RUN * (q + (p < r)) - (owner == p ? missing : 0u);
        home = (size_t)g.vbase + RUN * (p * q + min(p, r)) - (owner < p ? missing : 0u);
        cur = words<W>(a) + g.vbase;
        R = row_lists(a, g.vbase);
        queue = a.queue + home;
    }
    // the vertex of its row i
    __device__ __forceinline__ uint32_t vertex(uint32_t i) const {
        return __ldg(g.vid + ((((i >> g.run) * (size_t)g.nparts + first) << g.run) + (i & ((1u << g.run) - 1u))));
    }
};
struct PartCounts {
    uint32_t live, nshort, nlong;
};
struct Tally {
    uint32_t matched = 0, last = 0;   // rows matched; 1 + their latest round (the rounds that it takes)
    bool changed = false;
};

// One pass over `cnt` live rows (list NULL: all of the part's) by the block: a row that
// is chosen back is matched, one whose candidate is matched to another moves on in its
// list; live rows go to `out`, rows with a used-up list to the queue.
template <class W>
__device__ __forceinline__ void poll_rows(const ListArgs& a, const Part<W>& P, const uint32_t* list, uint32_t cnt,
                                          uint32_t* out, PartCounts& S, Tally& T) {
    constexpr bool ROUNDS = sizeof(W) == 8;
    const ListSeg& g = P.g;
    W* cur = P.cur;
    uint32_t v, nv;
    W w, nw, t;
    uint4 l, nl;
    // the next row's word and list are on their way while this one is decided
    auto fetch = [&](uint32_t at) { nv = at >= cnt ? NIL : list ? list[at] : P.vertex(at); };
    auto fetch_words = [&]() {
        nw = nv != NIL ? look(cur + nv) : (W)0;
        nl = nv != NIL ? P.R.lst[nv] : make_uint4(NIL, NIL, NIL, 0);
    };
    fetch(threadIdx.x);
    fetch_words();
    for (uint32_t base = 0; base < cnt; base += LT) {
        v = nv;
        w = nw;
        l = nl;
        if (v != NIL && lo(w) >= g.n) { set_err(a.st, ERR_BOUNDS, lo(w)); v = NIL; }
        t = v != NIL ? look(cur + lo(w)) : (W)0;
        fetch(base + LT + threadIdx.x);
        const bool gone = v != NIL && (lo(t) & DEAD) && (lo(t) & VMASK) != v;
        W n[3];
        n[0] = gone && l.x != NIL ? look(cur + l.x) : (W)DEAD;
        n[1] = gone && l.y != NIL ? look(cur + l.y) : (W)DEAD;
        n[2] = gone && l.z != NIL ? look(cur + l.z) : (W)DEAD;
        fetch_words();
        bool live = v != NIL, refill = false;
        uint32_t s = 0, d = 0;
        if (live) {
            uint32_t u = lo(w), passed = info(w);
            W y = t;
            if (gone) {
                T.changed = true;
                // the first of the list that is not matched (an empty place: DEAD, no round)
                const bool d0 = lo(n[0]) & DEAD, d1 = lo(n[1]) & DEAD, d2 = lo(n[2]) & DEAD;
                if (ROUNDS) {
                    passed = max(passed, info(y));
                    if (d0) passed = max(passed, info(n[0]));
                    if (d0 && d1) passed = max(passed, info(n[1]));
                    if (d0 && d1 && d2) passed = max(passed, info(n[2]));
                }
                const uint32_t at = v;
                const bool hasr = ROUNDS && (l.w & HASR);
                if (!(d0 && d1 && d2)) {
                    u = !d0 ? l.x : !d1 ? l.y : l.z;
                    y = !d0 ? n[0] : !d1 ? n[1] : n[2];
                    if (hasr) {
                        const uint4 r = P.R.rl[at];
                        passed = max(passed, !d0 ? r.x : !d1 ? r.y : r.z);
                        P.R.rl[at] = make_uint4(!d0 ? r.y : r.z, r.z, 0, 0);
                    }
                    cur[v] = word<W>(u, passed);
                    P.R.lst[at] = make_uint4(!d0 ? l.y : !d1 ? l.z : NIL, !d0 ? l.z : NIL, NIL, l.w);
                } else {
                    live = false;
                    if (l.w & WIDE) {
                        // the second half of a long row's list takes the first's place
                        const uint4 l2 = P.R.wide[at];
                        const W m0 = l2.x != NIL ? look(cur + l2.x) : (W)DEAD;
                        const W m1 = l2.y != NIL ? look(cur + l2.y) : (W)DEAD;
                        const W m2 = l2.z != NIL ? look(cur + l2.z) : (W)DEAD;
                        const W m3 = l2.w != NIL ? look(cur + l2.w) : (W)DEAD;
                        const bool e0 = lo(m0) & DEAD, e1 = e0 && (lo(m1) & DEAD), e2 = e1 && (lo(m2) & DEAD),
                                   e3 = e2 && (lo(m3) & DEAD);
                        if (ROUNDS) {
                            if (e0) passed = max(passed, info(m0));
                            if (e1) passed = max(passed, info(m1));
                            if (e2) passed = max(passed, info(m2));
                            if (e3) passed = max(passed, info(m3));
                        }
                        l.w &= ~WIDE;
                        if (!e3) {
                            live = true;
                            u = !e0 ? l2.x : !e1 ? l2.y : !e2 ? l2.z : l2.w;
                            y = !e0 ? m0 : !e1 ? m1 : !e2 ? m2 : m3;
                            if (hasr) {
                                const uint4 r = P.R.rw[at];
                                passed = max(passed, !e0 ? r.x : !e1 ? r.y : !e2 ? r.z : r.w);
                                P.R.rl[at] = make_uint4(!e0 ? r.y : !e1 ? r.z : r.w, !e0 ? r.z : r.w, r.w, 0);
                            }
                            cur[v] = word<W>(u, passed);
                            P.R.lst[at] = make_uint4(!e0 ? l2.y : !e1 ? l2.z : !e2 ? l2.w : NIL,
                                                   !e0 ? l2.z : !e1 ? l2.w : NIL, !e0 ? l2.w : NIL, l.w);
                        }
                    }
                    refill = !live && (l.w & MORE);
                    if (refill) {
                        s = __ldg(g.off + v);
                        d = __ldg(g.off + v + 1) - s;
                        if (ROUNDS) cur[v] = word<W>(u, passed);
                    }
                }
            }
            if (live && (lo(y) & VMASK) == v) {
                // chosen back
                uint32_t r = 0;
                if (ROUNDS) {
                    // its word, if matched already, has the round; else both ends' passed ones give it
                    r = (lo(y) & DEAD) ? info(y) : max(passed, info(y)) + 1u;
                    T.last = max(T.last, r);
                }
                cur[v] = word<W>(u | DEAD, r);
                g.dst[v] = u;
                T.matched++;
                live = false;
                T.changed = true;
            }
        }
        warp_append(&S.live, out, live, v);
        if (__any_sync(FULL, refill)) {
            const bool few = refill && d <= LIST_SHORT, many = refill && d > LIST_SHORT;
            const uint32_t q0 = warp_slot(&S.nshort, few), q1 = warp_slot(&S.nlong, many);
            // (the rounds of matched ends are wanted again, however heavy their edges)
            if (refill) P.queue[few ? q0 : P.rows - 1 - q1] = make_uint4(v, s, d, ROUNDS ? ~0u : l.w | FLAGS);
        }
    }
}

// the queued rows of a part by the block, its warps taking them from two counters; the
// live ones join `out`
struct RefillSmem {
    uint64_t k[LW][KL];
    uint32_t n[LW][KL];
};
template <class W>
__device__ __forceinline__ void refill_rows(const ListArgs& a, const Part<W>& P, uint32_t k0, uint32_t k1,
                                            uint32_t* out, uint32_t* nlive, uint32_t next[2], RefillSmem& S) {
    constexpr bool ROUNDS = sizeof(W) == 8;
    const ListSeg& g = P.g;
    W* cur = P.cur;
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint4 none = make_uint4(0, 0, 0, 0);
    auto take = [&](uint32_t* ctr, uint32_t k) {
        uint32_t b = 0;
        if (lane == 0) b = atomicAdd(ctr, k);
        return __shfl_sync(FULL, b, 0);
    };
    bool huge = false;
    // longer rows first
    for (uint32_t b = take(&next[1], 2); b < k1; b = take(&next[1], 2)) {
        // two rows by half a warp each if both are of at most 64 entries, else one by one
        const uint32_t i = b + lane / 16;
        const uint4 q2 = i < k1 ? P.queue[P.rows - 1 - i] : none;
        if (__all_sync(FULL, q2.z <= 64)) {
            const bool live = refill_group<W, 16, 4, KL>(g, cur, P.R, q2.x, q2.y, q2.z);
            warp_append(nlive, out, live && (lane & 15) == 0, q2.x);
            continue;
        }
        for (int k = 0; k < 2; k++) {
            const uint32_t v = __shfl_sync(FULL, q2.x, 16 * k), s = __shfl_sync(FULL, q2.y, 16 * k),
                           d = __shfl_sync(FULL, q2.z, 16 * k), ub = __shfl_sync(FULL, q2.w, 16 * k);
            if (d == 0) continue;
            if (d > BLOCK_ROW) {
                huge = true;
                continue;
            }
            bool live;
            if (d <= 128) {
                live = refill_group<W, 32, 4, KL>(g, cur, P.R, v, s, d);
            } else {
                LaneTop64 t;
                refill_scan<W>(g, cur, s, d, ub, 0, 1, t);
                live = __shfl_sync(FULL, t.k, 0) != 0;
                uint32_t r = 0;
                if (ROUNDS && live) r = refill_passed(g, reinterpret_cast<const uint64_t*>(cur), s, d, 0, 1, t);
                if (live) refill_put<W>(cur, P.R, v, t, r);
            }
            warp_append(nlive, out, live && lane == 0, v);
        }
    }
    // rows of at most LIST_SHORT: eight at a time by four lanes each if they are of at
    // most 16 entries, else four by eight lanes
    for (uint32_t b = take(&next[0], 8); b < k0; b = take(&next[0], 8)) {
        const uint32_t i = b + lane / 4;
        const uint4 q = i < k0 ? P.queue[i] : none;
        if (__all_sync(FULL, q.z <= 16)) {
            const bool live = refill_group<W, 4, 4, KS>(g, cur, P.R, q.x, q.y, q.z);
            warp_append(nlive, out, live && (lane & 3) == 0, q.x);
            continue;
        }
        for (int h = 0; h < 2; h++) {
            const int from = 16 * h + 4 * (lane / 8);
            const uint32_t v = __shfl_sync(FULL, q.x, from), s = __shfl_sync(FULL, q.y, from),
                           d = __shfl_sync(FULL, q.z, from);
            const bool live = refill_group<W, 8, 4, KS>(g, cur, P.R, v, s, d);
            warp_append(nlive, out, live && (lane & 7) == 0, v);
        }
    }
    if (!__syncthreads_or(huge)) return;
    for (uint32_t i = 0; i < k1; i++) {
        const uint4 q4 = P.queue[P.rows - 1 - i];
        const uint32_t v = q4.x, s = q4.y, d = q4.z;
        if (d <= BLOCK_ROW) continue;
        {
            LaneTop64 t;
            refill_scan<W>(g, cur, s, d, q4.w, warp, LW, t);
            if (lane < KL) {
                S.k[warp][lane] = t.k;
                S.n[warp][lane] = t.n;
            }
        }
        __syncthreads();
        LaneTop64 r;   // every warp merges all
        for (uint32_t z = lane; z < LW * KL; z += 32) r.offer(S.k[z / KL][z % KL], S.n[z / KL][z % KL]);
        static_assert(LW * KL % 32 == 0, "whole warps offer");
        const bool live = __shfl_sync(FULL, r.k, 0) != 0;
        if (ROUNDS) {
            __syncthreads();   // every warp has read the lists
            if (live) {
                const uint32_t x = refill_passed(g, reinterpret_cast<const uint64_t*>(cur), s, d, warp, LW, r);
                if (lane < KL) S.n[warp][lane] = x;
            }
            __syncthreads();
        }
        if (warp == 0) {
            uint32_t x = 0;
            if (ROUNDS && live && lane < KL)
                for (int w = 0; w < LW; w++) x = max(x, S.n[w][lane]);
            if (live) refill_put<W>(cur, P.R, v, r, x);
            warp_append(nlive, out, live && lane == 0, v);
        }
        __syncthreads();
    }
}

template <class W>
struct LiveSmem {
    ListArgs a;
    Part<W> p;
    RefillSmem r;
    PartCounts c;
    uint32_t part, changed, stop, next[2];
    uint32_t red[2][LW];
    uint64_t begin;   // when the block started
};

// Blocks take parts from a counter and pass over a part's live rows until none is
// left.  A part may wait for words that another block writes, but no block waits for
// good: after IDLE_MAX passes without a change it puts the part's rows back for the
// next launch, which the last block to leave asks for.  A part's block stops after the
// pass that matched a row beyond the round cap, the others when they see the error: with
// rounds at their next pass, else (no cap then, only the time limit) within 16.  With a
// slice, a block also puts back what is left of its parts once that time is over, each after
// one pass at least, so that a host that shares the GPU among jobs gets it back.  (pa: the
// arguments in device memory, for a launch in a graph.)
template <class W>
__global__ void __launch_bounds__(LT, LMINB) k_live(const __grid_constant__ ListArgs av,
                                                       const ListArgs* __restrict__ pa, cudaGraphConditionalHandle h) {
    __shared__ LiveSmem<W> S;
    copy_words(&S.a, pa ? pa : &av, LT);
    __syncthreads();
    const ListArgs& a = S.a;
    const Part<W>& P = S.p;
    DevState* st = a.st;
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t launch = ld_volatile_u32(&st->round);
    uint32_t left = 0;   // thread 0: rows given back
    if (sizeof(W) == 8 && tid == 0) S.begin = globaltimer_ns();
    for (;;) {
        if (tid == 0) S.part = atomicAdd(&st->task[0], 1u);
        __syncthreads();
        const uint32_t part = S.part;
        if (part >= a.nparts) break;
        const uint32_t si = a.pmap ? a.pmap[part] : 0u;
        copy_words(&S.p.g, a.pmap ? a.segs + si : &a.one, LT);
        __syncthreads();
        if (tid == 0) S.p.init(a, part);
        __syncthreads();
        const uint32_t pc = launch ? a.pcount[part] : P.rows << 1;
        uint32_t cnt = pc >> 1, buf = pc & 1u;
        const uint32_t* list = launch ? a.list[buf] + P.home : nullptr;
        Tally T;
        uint32_t idle = 0;
        for (uint32_t pass = 0; cnt; pass++) {
            uint32_t* out = a.list[buf ^ 1u] + P.home;
            // (thread 0: asked for ahead of the pass and looked at after it)
            const uint32_t err = sizeof(W) == 8 && tid == 0 ? ld_volatile_u32(&st->err) : 0u;
            if (tid == 0) {
                S.c.live = S.c.nshort = S.c.nlong = 0;
                S.next[0] = S.next[1] = 0;
                S.changed = 0;
                S.stop = 0;
                const uint64_t now = globaltimer_ns();
                if (now - st->t0_ns > a.limit_ns) {
                    set_err(st, ERR_TIMEOUT, pass);
                    S.stop = 1;
                } else if (sizeof(W) == 8 && a.slice_ns && now - S.begin > a.slice_ns) {
                    S.stop = 1;
                } else if (sizeof(W) == 4 && (pass & 15u) == 15u && ld_volatile_u32(&st->err)) {
                    S.stop = 1;
                }
            }
            __syncthreads();
            T.changed = false;
            poll_rows<W>(a, P, list, cnt, out, S.c, T);
            if (T.changed) S.changed = 1;
            if (sizeof(W) == 8) {
                const bool over = T.last > a.max_rounds;
                if (over) set_err(st, ERR_TIMEOUT, T.last);
                if (over || err) S.stop = 1;
            }
            __syncthreads();
            const uint32_t k0 = S.c.nshort, k1 = S.c.nlong;
            if (k0 | k1) {
                refill_rows<W>(a, P, k0, k1, out, &S.c.live, S.next, S.r);
                __syncthreads();
            }
            cnt = S.c.live;
            const uint32_t ch = S.changed, stop = S.stop;
            list = out;
            buf ^= 1u;
            __syncthreads();  // read before the next pass resets them
            idle = ch ? 0u : idle + 1u;
            if (stop || idle > IDLE_MAX) break;
        }
        // the part's matched rows and their latest round
        const uint32_t m = __reduce_add_sync(FULL, T.matched), r = __reduce_max_sync(FULL, T.last);
        if (lane == 0) {
            S.red[0][warp] = m;
            S.red[1][warp] = r;
        }
        __syncthreads();
        if (tid == 0) {
            unsigned long long t = 0;
            uint32_t l = 0;
            for (int i = 0; i < LW; i++) {
                t += S.red[0][i];
                l = max(l, S.red[1][i]);
            }
            if (t) atomicAdd(a.gmatched ? &a.gmatched[si] : &st->matched2, t);
            if (sizeof(W) == 8 && l) atomicMax(a.grounds ? &a.grounds[si] : &st->rounds, l);
            a.pcount[part] = cnt << 1 | buf;
            left += cnt;
        }
    }
    if (tid == 0) {
        if (left) atomicAdd(&st->left, left);
        __threadfence();
        S.stop = atomicAdd(&st->exit_v, 1u) == gridDim.x - 1;
        if (S.stop) {
            __threadfence();
            st->exit_v = 0;
            st->task[0] = 0;
            const uint32_t rest = ld_volatile_u32(&st->left);
            st->left = 0;
            st->round = launch + 1;
            if (rest == 0) st->done = 1;
            if (pa) cudaGraphSetConditional(h, rest && !ld_volatile_u32(&st->err) ? 1u : 0u);
            __threadfence();
        }
    }
    __syncthreads();
    if (S.stop && a.host) state_to_host(a.host, st, LT);
}

// ---------------------------------------------------------------- per-round counts
// An edge is live up to the earlier match of its ends (the result is maximal: one of
// them is matched), a matched row up to its own match, another up to the last of its
// neighbours'.  k_round_bytes packs the match rounds (63: that or later, 255:
// unmatched) so that the gathers of k_round_counts stay in L2; ring_m / ring_n get the
// edges and rows by their last live round.  Counters are a thread's own columns of a
// shared table: nearly all lanes count the same few rounds.
__global__ void k_round_bytes(const __grid_constant__ ListArgs a, uint8_t* mr) {
    const uint32_t n = a.one.n;
    const uint64_t* cur = words<uint64_t>(a);
    const uint32_t* dst = a.one.dst;
    for (uint64_t v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (uint64_t)gridDim.x * blockDim.x)
        mr[v] = dst[v] == NIL ? 255 : (uint8_t)min(info(cur[v]) - 1u, 63u);
}
__global__ void __launch_bounds__(256) k_round_counts(const __grid_constant__ ListArgs a,
                                                      const uint8_t* __restrict__ mr) {
    __shared__ uint32_t h[64][128];   // two threads a column: counts of either by halves of 16 bits
    const ListSeg& g = a.one;
    const uint32_t tid = threadIdx.x;
    uint16_t* col = reinterpret_cast<uint16_t*>(&h[0][0]) + tid;   // [round][thread]
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (int kind = 0; kind < 2; kind++) {
        unsigned long long* ring = reinterpret_cast<unsigned long long*>(kind ? a.st->ring_n : a.st->ring_m);
        const uint64_t total = kind ? g.nrows : g.m;
        // (steps of at most 32768 counts a thread, so that 16 bits hold them)
        for (uint64_t base = 0; base < total; base += stride * 32768) {
            for (int i = 0; i < 64; i++) col[i * 256] = 0;
            const uint64_t end = total - base < stride * 32768 ? total : base + stride * 32768;
            for (uint64_t i = base + blockIdx.x * blockDim.x + tid; i < ((end + 31) & ~31ull); i += stride) {
                uint32_t r = NIL;
                if (kind == 0) {
                    // four edges a step: their gathers in flight together
                    uint64_t rec[4];
                    uint32_t q[4];
#pragma unroll
                    for (int z = 0; z < 4; z++) rec[z] = i + z * stride < end ? __ldg(g.edges + i + z * stride) : 0ull;
#pragma unroll
                    for (int z = 0; z < 4; z++) q[z] = min((uint32_t)__ldg(mr + (uint32_t)rec[z]), (uint32_t)__ldg(mr + (uint32_t)(rec[z] >> 32)));
#pragma unroll
                    for (int z = 0; z < 4; z++)
                        if (i + z * stride < end && q[z] < 64) col[q[z] * 256]++;
                    i += 3 * stride;
                } else {
                    // a thread a row: a matched one has its round, a short unmatched one looks at
                    // its neighbours, longer ones are done by the warp one after the other
                    uint32_t s0 = 0, d = 0;
                    if (i < end) {
                        r = mr[g.vid[i]];
                        if (r == 255) {
                            s0 = g.roff[i];
                            d = g.roff[i + 1] - s0;
                            r = 0;
                            if (d <= 16)
                                for (uint32_t j = 0; j < d; j += 4) {
                                    uint32_t x[4];
#pragma unroll
                                    for (uint32_t z = 0; z < 4; z++) x[z] = nbr_at(g, s0 + min(j + z, d - 1));
#pragma unroll
                                    for (uint32_t z = 0; z < 4; z++) r = max(r, (uint32_t)__ldg(mr + x[z]));
                                }
                        }
                    }
                    for (uint32_t todo = __ballot_sync(FULL, d > 16); todo; todo &= todo - 1) {
                        const int L = __ffs(todo) - 1;
                        const uint32_t sl = __shfl_sync(FULL, s0, L), dl = __shfl_sync(FULL, d, L);
                        uint32_t x = 0;
                        for (uint64_t j = tid & 31; j < dl; j += 32) x = max(x, (uint32_t)__ldg(mr + nbr_at(g, sl + (uint32_t)j)));
                        x = __reduce_max_sync(FULL, x);
                        if ((int)(tid & 31) == L) r = x;
                    }
                }
                if (r < 64) col[r * 256]++;
            }
            __syncthreads();
            // warp w sums rounds w, w + 8, ...
            for (uint32_t i = tid >> 5; i < 64; i += 8) {
                uint32_t s = 0;
                for (uint32_t j = tid & 31; j < 128; j += 32) s += (h[i][j] & 0xFFFFu) + (h[i][j] >> 16);
                s = __reduce_add_sync(FULL, s);
                if ((tid & 31) == 0 && s) atomicAdd(&ring[i], (unsigned long long)s);
            }
            __syncthreads();
        }
    }
}

// graph of every block of k_top and of every part
__global__ void k_list_map(const __grid_constant__ ListArgs a, uint32_t* bmap, uint32_t* pmap) {
    const uint32_t w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (w >= a.nsegs) return;
    const ListSeg& g = a.segs[w];
    for (uint32_t b = lane; b < g.nblk; b += 32) bmap[g.blk0 + b] = w;
    for (uint32_t b = lane; b < g.nparts; b += 32) pmap[g.part0 + b] = w;
}

int sms() {
    int dev = 0;
    cudaGetDevice(&dev);
    return device_sm_count(dev);
}
uint32_t live_grid() { return (uint32_t)sms() * LMINB; }   // every block resident

}  // namespace

uint32_t list_live_blocks(int device) { return (uint32_t)device_sm_count(device) * LMINB; }
uint32_t list_blocks(const uint32_t task[4], uint32_t nrows, uint32_t n) {
    const TopBlocks b = top_blocks(task, nrows);
    const uint32_t t = b.l + b.w + b.g + b.s, c = div_up(n, CLEAR);
    return t > c ? t : c ? c : 1u;
}
int launch_list_map(void* stream, const ListArgs& d, uint32_t nsegs, uint32_t* bmap, uint32_t* pmap) {
    k_list_map<<<(nsegs + 7) / 8, 256, 0, (cudaStream_t)stream>>>(d, bmap, pmap);
    return (int)cudaGetLastError();
}
int launch_top(void* stream, const ListArgs& d, uint32_t blocks, bool rounds) {
    if (rounds) k_top<uint64_t><<<blocks, TT, 0, (cudaStream_t)stream>>>(d);
    else k_top<uint32_t><<<blocks, TT, 0, (cudaStream_t)stream>>>(d);
    return (int)cudaGetLastError();
}
// (more blocks than parts would only come and go)
int launch_live(void* stream, const ListArgs& d, uint32_t nparts, bool rounds) {
    const uint32_t grid = nparts < live_grid() ? nparts : live_grid();
    const cudaGraphConditionalHandle none{};
    if (rounds) k_live<uint64_t><<<grid, LT, 0, (cudaStream_t)stream>>>(d, nullptr, none);
    else k_live<uint32_t><<<grid, LT, 0, (cudaStream_t)stream>>>(d, nullptr, none);
    return (int)cudaGetLastError();
}
int launch_round_counts(void* stream, const ListArgs& d, void* bytes) {
    k_round_bytes<<<sms() * 8, 256, 0, (cudaStream_t)stream>>>(d, (uint8_t*)bytes);
    k_round_counts<<<sms() * 6, 256, 0, (cudaStream_t)stream>>>(d, (const uint8_t*)bytes);
    return (int)cudaGetLastError();
}

// k_live, and again while it leaves rows (asynchronous matches: the host does not look)
int build_list_graph(const ListArgs* dargs, bool rounds, void** exec_out) {
    *exec_out = nullptr;
    cudaGraph_t g = nullptr;
    cudaError_t e = cudaGraphCreate(&g, 0);
    if (e != cudaSuccess) return (int)e;
    cudaGraphConditionalHandle h{};
    ListArgs unused;
    memset(&unused, 0, sizeof unused);
    void* params[3] = {&unused, &dargs, &h};
    cudaKernelNodeParams kp{};
    kp.func = rounds ? (void*)k_live<uint64_t> : (void*)k_live<uint32_t>;
    kp.gridDim = dim3(live_grid());
    kp.blockDim = dim3(LT);
    kp.kernelParams = params;
    do {
        if ((e = cudaGraphConditionalHandleCreate(&h, g, 1, cudaGraphCondAssignDefault))) break;
        cudaGraphNode_t first, loop, again;
        if ((e = cudaGraphAddKernelNode(&first, g, nullptr, 0, &kp))) break;
        alignas(cudaGraphNodeParams) unsigned char cp_raw[sizeof(cudaGraphNodeParams)];
        memset(cp_raw, 0, sizeof cp_raw);
        cudaGraphNodeParams& cp = *reinterpret_cast<cudaGraphNodeParams*>(cp_raw);
        cp.type = cudaGraphNodeTypeConditional;
        cp.conditional.handle = h;
        cp.conditional.type = cudaGraphCondTypeWhile;
        cp.conditional.size = 1;
        if ((e = cudaGraphAddNode(&loop, g, &first, nullptr, 1, &cp))) break;
        if ((e = cudaGraphAddKernelNode(&again, cp.conditional.phGraph_out[0], nullptr, 0, &kp))) break;
        cudaGraphExec_t ex = nullptr;
        if ((e = cudaGraphInstantiate(&ex, g, 0))) break;
        *exec_out = ex;
    } while (0);
    cudaGraphDestroy(g);
    return (int)e;
}

}  // namespace lm
