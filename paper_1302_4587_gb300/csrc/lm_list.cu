// The list path of the matching: local max without compaction and without rounds.
//
// A vertex only ever looks at the heaviest few of its edges before it is
// matched or runs out of live neighbours (2.3 to 2.5 entries a row on random,
// grid and R-MAT graphs, 9% to 40% of the adjacency entries).  So one pass over
// the adjacency arrays (k_top) keeps the four heaviest neighbours of every row,
// in order, and no entry is read again unless those four are used up:
//
//   k_top   every row's candidate (Sec. 2.1, step 2) and the next three
//   k_live  the live rows until none is left.  A row looks at its candidate's
//           word: chosen back, it is matched (step 3); matched to another, the row
//           moves on to the next of its list that is not (steps 4 to 6 without
//           moving an edge: an edge is dead when the word of its other end says so),
//           and scans its adjacency once more for the four heaviest live ones
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
constexpr uint32_t TOPN = 4;   // neighbours kept per row (its word and lst)

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

// ---------------------------------------------------------------- the four heaviest entries
// Entries are compared by ord(w) alone where that decides: perm_seed tells equal
// ones apart, and only rows where it matters (two of the four, or the fourth
// and one left out, are equal) are taken again by their full keys.

// One unit's (a thread's, a group of lanes') four largest of up to 256 entries as
// 32-bit numbers: ord(w) with its low BITS bits replaced by the entry's place in
// the row (smaller first), so that an exchange is one minimum and one maximum.
// Entries whose ord agrees above those bits count as equal.
__device__ __forceinline__ uint32_t packed(uint32_t ord, uint32_t idx, uint32_t mask) {
    return (ord & ~mask) | (mask - idx);
}
struct TopP {
    uint32_t k[4] = {0, 0, 0, 0};
    uint32_t out = 0;                 // largest one left out
    __device__ __forceinline__ void add(uint32_t x) {
#pragma unroll
        for (int i = 0; i < 4; i++) {
            const uint32_t hi = max(k[i], x);
            x = min(k[i], x);
            k[i] = hi;
        }
        out = max(out, x);
    }
    // the four largest of two ordered fours: the larger of each pair taken head to tail
    // is one of them (a bitonic four), then put in order
    __device__ __forceinline__ void merge(const uint32_t o[4], uint32_t oout) {
        out = max(out, oout);
#pragma unroll
        for (int i = 0; i < 4; i++) out = max(out, min(k[i], o[3 - i]));
#pragma unroll
        for (int i = 0; i < 4; i++) k[i] = max(k[i], o[3 - i]);
        order(0, 2);
        order(1, 3);
        order(0, 1);
        order(2, 3);
    }
    __device__ __forceinline__ void order(int a, int b) {
        const uint32_t hi = max(k[a], k[b]);
        k[b] = min(k[a], k[b]);
        k[a] = hi;
    }
    // over the lanes of aligned groups of G, each lane's four in order on entry
    template <int G>
    __device__ __forceinline__ void across() {
#pragma unroll
        for (int d = 1; d < G; d <<= 1) {
            uint32_t o[4];
#pragma unroll
            for (int i = 0; i < 4; i++) o[i] = __shfl_xor_sync(FULL, k[i], d);
            const uint32_t oo = __shfl_xor_sync(FULL, out, d);
            merge(o, oo);
        }
    }
    __device__ __forceinline__ bool tied(uint32_t mask) const {
        return (k[1] && (k[0] ^ k[1]) <= mask) || (k[2] && (k[1] ^ k[2]) <= mask) ||
               (k[3] && ((k[2] ^ k[3]) <= mask || (out && (k[3] ^ out) <= mask)));
    }
};

// A warp's four largest (uniform over its lanes) of any number of entries, by
// ord(w), with their positions; an equal one is for the caller to notice (has()).
struct Top32 {
    uint32_t o0 = 0, o1 = 0, o2 = 0, o3 = 0;
    uint32_t p0 = 0, p1 = 0, p2 = 0, p3 = 0;
    __device__ __forceinline__ void swap_in(uint32_t& o, uint32_t& p, uint32_t& x, uint32_t& px) {
        const bool g = x > o;
        const uint32_t hi = max(o, x), lw = min(o, x), ph = g ? px : p, pl = g ? p : px;
        o = hi; p = ph; x = lw; px = pl;
    }
    __device__ __forceinline__ void add(uint32_t x, uint32_t px) {
        swap_in(o0, p0, x, px);
        swap_in(o1, p1, x, px);
        swap_in(o2, p2, x, px);
        swap_in(o3, p3, x, px);
    }
    __device__ __forceinline__ bool has(uint32_t x) const { return x == o0 || x == o1 || x == o2 || x == o3; }
};
struct Top64 {
    uint64_t k0 = 0, k1 = 0, k2 = 0, k3 = 0;
    uint32_t p0 = NIL, p1 = NIL, p2 = NIL, p3 = NIL;
    __device__ __forceinline__ void swap_in(uint64_t& k, uint32_t& p, uint64_t& x, uint32_t& px) {
        if (x > k) {
            const uint64_t t = k; k = x; x = t;
            const uint32_t q = p; p = px; px = q;
        }
    }
    __device__ __forceinline__ void add(uint64_t x, uint32_t px) {
        swap_in(k0, p0, x, px);
        swap_in(k1, p1, x, px);
        swap_in(k2, p2, x, px);
        swap_in(k3, p3, x, px);
    }
};

__device__ __forceinline__ uint32_t hi32(const uint64_t* pk, uint32_t i) {
    return __ldg(reinterpret_cast<const uint32_t*>(pk) + 2 * (size_t)i + 1);
}
__device__ __forceinline__ uint64_t full_key(uint64_t w, uint32_t k0, uint32_t k1) {
    return (w & 0xFFFFFFFF00000000ull) | perm_seed((uint32_t)w, k0, k1);
}

// every lane offers (key, p), 0 for none: the warp's keys above t.k3 go in, largest first
__device__ __forceinline__ void warp_add(Top64& t, uint64_t key, uint32_t p) {
    while (__any_sync(FULL, key > t.k3)) {
        const uint32_t hi = __reduce_max_sync(FULL, (uint32_t)(key >> 32));
        const uint32_t lo = __reduce_max_sync(FULL, ((uint32_t)(key >> 32) == hi) ? (uint32_t)key : 0u);
        const uint64_t best = ((uint64_t)hi << 32) | lo;
        const uint32_t own = __ballot_sync(FULL, key == best);
        const int L = __ffs(own) - 1;
        t.add(best, __shfl_sync(FULL, p, L));
        if ((int)(threadIdx.x & 31) == L) key = 0;
    }
}

// the four heaviest entries [s, e) by full key, the warp together; p: positions
__device__ __noinline__ void warp_top_keyed(const ListSeg& g, uint32_t s, uint32_t e, Top64& t) {
    const uint32_t lane = threadIdx.x & 31;
    uint64_t nx = s + lane < e ? __ldg(g.pk + s + lane) : 0ull;
    for (uint32_t b = s; b < e; b += 32) {
        const uint64_t w = nx;
        const uint32_t i = b + lane, j = i + 32;
        nx = (j < e && j > i) ? __ldg(g.pk + j) : 0ull;
        warp_add(t, i < e ? full_key(w, g.k0, g.k1) : 0ull, i);
    }
}

// row v's list: four neighbours (NIL: none), more = entries beyond them were left out
template <class W>
__device__ __forceinline__ void put_row(const ListArgs& a, size_t at, uint32_t c0, uint32_t c1, uint32_t c2,
                                        uint32_t c3, bool more) {
    words<W>(a)[at] = word<W>(c0, 0);
    a.lst[at] = make_uint4(c1, c2, c3, more ? 1u : 0u);
}

// ---------------------------------------------------------------- k_top
constexpr int TT = 256, TWARPS = TT / 32;
constexpr uint32_t SBUF = 512;    // entries of short rows a warp stages at a time
constexpr uint32_t MPW = 2;       // long-row tasks a warp takes,
constexpr uint32_t WPW = 8;       // rows of LIST_GROUP + 1 .. LIST_WARP entries,
constexpr uint32_t GPW = 16;      // and rows of LIST_SHORT + 1 .. LIST_GROUP
static_assert(LIST_SHORT <= 32 && LIST_GROUP == 8 * 8 && LIST_WARP == 8 * 32, "eight entries a lane");

struct TopSmem {
    uint32_t o[TWARPS][SBUF];     // ord(w) of the staged entries
    uint32_t n[TWARPS][SBUF];     // their neighbours
};

// 32 rows of at most LIST_SHORT entries (longer ones among them are skipped), a
// thread each.  Runs of neighbouring short rows are contiguous in the arrays:
// the warp copies them to shared memory coalesced and each thread walks its own
// row there, so a row costs its length in warp steps shared by 32 rows instead
// of a segmented scan over its entries.
template <class W>
__device__ void top_short(const ListArgs& a, const ListSeg& g, uint32_t r0, uint32_t* so, uint32_t* sn) {
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t r = r0 + lane;
    uint32_t o = 0, e = 0, v = 0;
    if (r < g.nrows) {
        o = __ldg(g.roff + r);
        e = __ldg(g.roff + r + 1);
        v = __ldg(g.vid + r);
    }
    const uint32_t d = e - o;
    const bool mine = d > 0 && d <= LIST_SHORT;
    uint32_t todo = __ballot_sync(FULL, mine);
    while (todo) {
        // stage runs of short rows until the buffer is full
        uint32_t used = 0, my = 0, taken = 0;
        while (todo) {
            const int f = __ffs(todo) - 1;
            const uint32_t run = todo >> f;
            const int len = run == (FULL >> f) ? 32 - f : __ffs(~run) - 1;
            const uint32_t s = __shfl_sync(FULL, o, f);
            // rows f .. of the run that still fit
            const bool fit = (int)lane >= f && (int)lane < f + len && e - s <= SBUF - used;
            const uint32_t fits = __ballot_sync(FULL, fit);
            if (!fits) break;
            const int last = 31 - __clz(fits);
            const uint32_t cnt = __shfl_sync(FULL, e, last) - s;
            if (fit) my = used + (o - s);
            for (uint32_t i = lane; i < cnt; i += 128) {
                uint32_t x[4], y[4];
#pragma unroll
                for (int q = 0; q < 4; q++)
                    if (i + 32 * q < cnt) { x[q] = hi32(g.pk, s + i + 32 * q); y[q] = __ldg(g.nbr + s + i + 32 * q); }
#pragma unroll
                for (int q = 0; q < 4; q++)
                    if (i + 32 * q < cnt) { so[used + i + 32 * q] = x[q]; sn[used + i + 32 * q] = y[q]; }
            }
            used += cnt;
            taken |= fits;
            todo &= ~fits;
            if (last < f + len - 1) break;  // the buffer is full
        }
        __syncwarp();
        if ((taken >> lane) & 1u) {
            constexpr uint32_t MASK = LIST_SHORT - 1;
            TopP t;
            for (uint32_t j = 0; j < d; j++) t.add(packed(so[my + j], j, MASK));
            uint32_t p[4];
#pragma unroll
            for (int i = 0; i < 4; i++) p[i] = MASK - (t.k[i] & MASK);
            if (t.tied(MASK)) {
                Top64 k;
                for (uint32_t j = 0; j < d; j++) k.add(full_key(__ldg(g.pk + o + j), g.k0, g.k1), j);
                p[0] = k.p0; p[1] = k.p1; p[2] = k.p2; p[3] = k.p3;
            }
            put_row<W>(a, (size_t)g.vbase + v, sn[my + p[0]], d > 1 ? sn[my + p[1]] : NIL, d > 2 ? sn[my + p[2]] : NIL,
                       d > 3 ? sn[my + p[3]] : NIL, d > TOPN);
        }
        __syncwarp();
    }
}

// The four heaviest of a row held by a group of G lanes, eight entries a lane (entry
// 8-fold: e * G + the lane's place), among those in `live` (bit e), by full key: the
// exact form.  Positions (NIL: none) and keys; rest: others are left.
template <int G>
__device__ __forceinline__ void group_keyed(const uint64_t K[8], uint32_t live, uint32_t sub, uint32_t p[4],
                                            uint64_t k[4], bool& rest) {
    uint32_t left = live;
#pragma unroll
    for (int i = 0; i < 4; i++) {
        uint64_t m = 0;
        uint32_t at = NIL;
#pragma unroll
        for (int e = 0; e < 8; e++)
            if (((left >> e) & 1u) && K[e] > m) { m = K[e]; at = e; }
        uint64_t b = m;
#pragma unroll
        for (int d = 1; d < G; d <<= 1) {
            const uint64_t o = __shfl_xor_sync(FULL, b, d);
            b = o > b ? o : b;
        }
        const bool own = b && b == m;
        uint32_t pos = own ? at * G + sub : NIL;
#pragma unroll
        for (int d = 1; d < G; d <<= 1) pos = min(pos, __shfl_xor_sync(FULL, pos, d));
        p[i] = pos;
        if (own) left &= ~(1u << at);
        k[i] = b;
    }
    uint32_t any = left;
#pragma unroll
    for (int d = 1; d < G; d <<= 1) any |= __shfl_xor_sync(FULL, any, d);
    rest = any != 0;
}

// `per` rows of more than LIST_SHORT entries a warp, eight entries to each of the G
// lanes of a group (32 / G rows at a time), straight from the arrays into registers;
// the next rows' entries are on their way while these are compared.
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
        for (int e = 0; e < 8; e++) x[e] = e * G + sub < d ? hi32(g.pk, s + e * G + sub) : 0u;
    };
    fetch(0);
    for (uint32_t i = 0; i < cnt; i += ROWS) {
        const uint32_t cv = v, cs = s, cd = d;
        TopP t;
#pragma unroll
        for (int e = 0; e < 8; e++) t.add(x[e] ? packed(x[e], e * G + sub, MASK) : 0u);
        t.across<G>();
        uint32_t p[4];
#pragma unroll
        for (int q = 0; q < 4; q++) p[q] = MASK - (t.k[q] & MASK);
        if (__any_sync(FULL, t.tied(MASK))) {
            uint64_t K[8], kk[4];
            uint32_t pk[4];
            bool rest;
#pragma unroll
            for (int e = 0; e < 8; e++)
                K[e] = e * G + sub < cd ? full_key(__ldg(g.pk + cs + e * G + sub), g.k0, g.k1) : 0ull;
            group_keyed<G>(K, 0xFFu, sub, pk, kk, rest);
#pragma unroll
            for (int q = 0; q < 4; q++) p[q] = pk[q];
        }
        const uint32_t mp = sub == 0 ? p[0] : sub == 1 ? p[1] : sub == 2 ? p[2] : p[3];
        uint32_t c = 0;
        if (cd && sub < TOPN) c = __ldg(g.nbr + cs + mp);
        if (i + ROWS < cnt) fetch(i + ROWS);
        if (cd) {
            const size_t at = (size_t)g.vbase + cv;
            if (sub == 0) words<W>(a)[at] = word<W>(c, 0);
            else if (sub < TOPN) reinterpret_cast<uint32_t*>(a.lst + at)[sub - 1] = c;
            else if (sub == TOPN) reinterpret_cast<uint32_t*>(a.lst + at)[3] = 1u;
        }
    }
}

// Up to MPW long-row tasks (a row of more than LIST_WARP entries, or a
// LIST_CHUNK-entry chunk of one longer than that), the warp together: 128
// entries a step, the next 128 (of the next task, if need be) on their way.  A
// step whose entries all lie below the fourth-heaviest seen so far costs a
// maximum and a vote; an entry that does not is put in with a warp maximum.
template <class W>
__device__ void top_long(const ListArgs& a, const ListSeg& g, uint32_t t0, uint32_t cnt) {
    const uint32_t lane = threadIdx.x & 31;
    uint4 d4 = make_uint4(0, 0, 0, 0);
    if (lane < cnt) d4 = __ldg(g.task + t0 + lane);
    // task k: row vertex, [s, e) of the pass
    auto bounds = [&](uint32_t k, uint32_t& v, uint32_t& s, uint32_t& e, uint32_t& len, uint32_t& c) {
        v = __shfl_sync(FULL, d4.x, k);
        const uint32_t rs = __shfl_sync(FULL, d4.y, k);
        len = __shfl_sync(FULL, d4.z, k);
        c = __shfl_sync(FULL, d4.w, k);
        s = rs + c * LIST_CHUNK;
        e = rs + min(len, (c + 1) * LIST_CHUNK);
        if (len <= LIST_CHUNK) e = rs + len;
    };
    auto load = [&](uint32_t x[4], uint32_t pos, uint32_t e) {
#pragma unroll
        for (int q = 0; q < 4; q++) {
            const uint32_t i = pos + 32 * q + lane;
            x[q] = (i < e && i >= pos) ? hi32(g.pk, i) : 0u;
        }
    };
    uint32_t v, s, e, len, c;
    bounds(0, v, s, e, len, c);
    uint32_t x[4], nx[4];
    load(x, s, e);
    uint32_t pos = s, k = 0;
    Top32 t;
    bool tie = false;
    // the neighbours of the previous row's four are stored when the next row is done,
    // so that their loads do not stall the steps between
    uint32_t pend_v = NIL, pend_c = NIL;
    auto flush = [&]() {
        if (pend_v != NIL) {
            const size_t at = (size_t)g.vbase + pend_v;
            if (lane == 0) words<W>(a)[at] = word<W>(pend_c, 0);
            else if (lane < TOPN) reinterpret_cast<uint32_t*>(a.lst + at)[lane - 1] = pend_c;
            else if (lane == TOPN) reinterpret_cast<uint32_t*>(a.lst + at)[3] = 1u;
            pend_v = NIL;
        }
    };
    for (;;) {
        // where the next step reads
        uint32_t nv = v, ns = s, ne = e, nlen = len, nc = c, npos = pos + 128, nk = k;
        if (npos >= e || npos < pos) {
            nk = k + 1;
            if (nk < cnt) {
                bounds(nk, nv, ns, ne, nlen, nc);
                npos = ns;
            }
        }
        if (nk < cnt) load(nx, npos, ne);
        if (!tie) {
            uint32_t m = max(max(x[0], x[1]), max(x[2], x[3]));
            while (__any_sync(FULL, m && m >= t.o3)) {
                const uint32_t h = __reduce_max_sync(FULL, m);
                const uint32_t own = __ballot_sync(FULL, m == h);
                const uint32_t eq = (uint32_t)(x[0] == h) + (x[1] == h) + (x[2] == h) + (x[3] == h);
                const int L = __ffs(own) - 1;
                if (t.has(h) || (own & (own - 1)) || __shfl_sync(FULL, eq, L) > 1) {
                    tie = true;
                    break;
                }
                const uint32_t q = x[0] == h ? 0u : x[1] == h ? 1u : x[2] == h ? 2u : 3u;
                t.add(h, __shfl_sync(FULL, pos + 32 * q + lane, L));
                if ((int)lane == L) {
#pragma unroll
                    for (int z = 0; z < 4; z++)
                        if (x[z] == h) x[z] = 0;
                    m = max(max(x[0], x[1]), max(x[2], x[3]));
                }
            }
        }
        if (nk != k) {
            // the task's four, in order, one to a lane
            uint32_t p;
            if (tie) {
                Top64 kt;
                warp_top_keyed(g, s, e, kt);
                p = lane == 0 ? kt.p0 : lane == 1 ? kt.p1 : lane == 2 ? kt.p2 : kt.p3;
            } else {
                // (a row or chunk may hold fewer than four entries: a chunk's remainder)
                const uint32_t oo = lane == 0 ? t.o0 : lane == 1 ? t.o1 : lane == 2 ? t.o2 : t.o3;
                p = lane == 0 ? t.p0 : lane == 1 ? t.p1 : lane == 2 ? t.p2 : t.p3;
                if (!oo) p = NIL;
            }
            flush();
            if (len <= LIST_CHUNK) {
                pend_v = v;
                pend_c = lane < TOPN ? __ldg(g.nbr + p) : 0u;
            } else {
                // a chunk: its four with their full keys; the last chunk of the row to
                // finish merges all of them
                const uint32_t first = t0 + k - c;   // the row's chunk 0 in the task list
                const uint32_t nch = (len + LIST_CHUNK - 1) / LIST_CHUNK;
                if (lane < TOPN) {
                    uint4 rec = make_uint4(0, 0, NIL, 0);
                    if (p != NIL) {
                        const uint64_t K = full_key(__ldg(g.pk + p), g.k0, g.k1);
                        rec = make_uint4((uint32_t)K, (uint32_t)(K >> 32), __ldg(g.nbr + p), 0);
                    }
                    a.part[((size_t)g.lbase + t0 + k) * TOPN + lane] = rec;
                }
                __syncwarp();
                uint32_t old = 0;
                if (lane == 0) old = atom_add_acq_rel(&a.pcnt[(size_t)g.lbase + first], 1u);
                old = __shfl_sync(FULL, old, 0);
                __syncwarp();
                if (old == nch - 1) {
                    Top64 kt;
                    const uint4* P = a.part + ((size_t)g.lbase + first) * TOPN;
                    for (uint32_t b = 0; b < nch * TOPN; b += 32) {
                        uint4 rec = make_uint4(0, 0, NIL, 0);
                        if (b + lane < nch * TOPN) rec = __ldcg(P + b + lane);
                        warp_add(kt, ((uint64_t)rec.y << 32) | rec.x, rec.z);
                    }
                    if (lane == 0) {
                        a.pcnt[(size_t)g.lbase + first] = 0;
                        put_row<W>(a, (size_t)g.vbase + v, kt.p0, kt.p1, kt.p2, kt.p3, true);
                    }
                }
            }
            t = Top32();
            tie = false;
            if (nk >= cnt) break;
        }
#pragma unroll
        for (int q = 0; q < 4; q++) x[q] = nx[q];
        v = nv; s = ns; e = ne; len = nlen; c = nc; pos = npos; k = nk;
    }
    flush();
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

// Every block also clears its share of the result, and block 0 resets the job's state.
template <class W>
__global__ void __launch_bounds__(TT) k_top(const ListArgs* __restrict__ pa) {
    extern __shared__ __align__(16) unsigned char top_raw[];
    TopSmem& S = *reinterpret_cast<TopSmem*>(top_raw);
    const ListArgs& a = *pa;
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
    const uint32_t sg = a.bmap ? a.bmap[blockIdx.x] : 0u;
    const ListSeg& g = a.segs[sg];
    uint32_t b = blockIdx.x - g.blk0;
    {
        const uint32_t per = (uint32_t)(((uint64_t)g.n + g.nblk - 1) / g.nblk);
        const uint64_t from = (uint64_t)b * per, to = from + per < g.n ? from + per : g.n;
        for (uint64_t v = from + tid; v < to; v += TT) g.dst[v] = NIL;
    }
    const TopBlocks nb = top_blocks(g.ntask, g.nrows);
    if (b < nb.l) {
        const uint32_t t0 = (b * TWARPS + warp) * MPW;
        if (t0 < g.ntask[1]) top_long<W>(a, g, t0, min(MPW, g.ntask[1] - t0));
    } else if ((b -= nb.l) < nb.w) {
        const uint32_t t0 = g.ntask[1] + (b * TWARPS + warp) * WPW;
        if (t0 < g.ntask[2]) top_group<W, 32>(a, g, t0, min(WPW, g.ntask[2] - t0));
    } else if ((b -= nb.w) < nb.g) {
        const uint32_t t0 = g.ntask[2] + (b * TWARPS + warp) * GPW;
        if (t0 < g.ntask[3]) top_group<W, 8>(a, g, t0, min(GPW, g.ntask[3] - t0));
    } else {
        const uint32_t r0 = (b - nb.g) * TT + warp * 32;
        if (r0 < g.nrows) top_short<W>(a, g, r0, S.o[warp], S.n[warp]);
    }
}

// ---------------------------------------------------------------- refills
// The four heaviest live entries of rows of at most 8 G entries, a group of G lanes
// each; d = 0: no row.  Returns whether one is left (uniform over the group).
template <class W, int G>
__device__ __forceinline__ bool refill_group(const ListArgs& a, const ListSeg& g, uint32_t v, uint32_t s, uint32_t d) {
    constexpr uint32_t MASK = 8 * G - 1;
    constexpr bool ROUNDS = sizeof(W) == 8;
    const uint32_t sub = threadIdx.x & (G - 1);
    W* cur = words<W>(a) + g.vbase;
    uint4* lst = a.lst + g.vbase;
    uint32_t x[8], n[8], live = 0;
    W t[8];
#pragma unroll
    for (int e = 0; e < 8; e++) {
        const bool in = e * G + sub < d;
        x[e] = in ? hi32(g.pk, s + e * G + sub) : 0u;
        n[e] = in ? __ldg(g.nbr + s + e * G + sub) : 0u;
    }
#pragma unroll
    for (int e = 0; e < 8; e++) t[e] = e * G + sub < d ? look(cur + n[e]) : (W)DEAD;
#pragma unroll
    for (int e = 0; e < 8; e++)
        if (!(lo(t[e]) & DEAD)) live |= 1u << e;
    uint32_t p[4];
    bool rest = false, exact = ROUNDS;
    uint32_t passed = 0;
    if (!ROUNDS) {
        TopP q;
#pragma unroll
        for (int e = 0; e < 8; e++) q.add(((live >> e) & 1u) ? packed(x[e], e * G + sub, MASK) : 0u);
        q.across<G>();
#pragma unroll
        for (int i = 0; i < 4; i++) p[i] = q.k[i] ? MASK - (q.k[i] & MASK) : NIL;
        rest = q.out != 0;
        exact = __any_sync(FULL, q.tied(MASK));
    }
    if (exact) {
        uint64_t K[8], k[4];
#pragma unroll
        for (int e = 0; e < 8; e++)
            K[e] = e * G + sub < d ? full_key(__ldg(g.pk + s + e * G + sub), g.k0, g.k1) : 0ull;
        group_keyed<G>(K, live, sub, p, k, rest);
        if (ROUNDS) {
            // the latest round among the matched neighbours above the new candidate; the
            // list ends at the heaviest matched one below it, whose round counts for
            // every candidate after that
            uint64_t cut = 0;
#pragma unroll
            for (int e = 0; e < 8; e++) {
                if (e * G + sub >= d || ((live >> e) & 1u)) continue;
                if (K[e] > k[0]) passed = max(passed, info(t[e]));
                else cut = K[e] > cut ? K[e] : cut;
            }
#pragma unroll
            for (int z = 1; z < G; z <<= 1) {
                passed = max(passed, __shfl_xor_sync(FULL, passed, z));
                const uint64_t o = __shfl_xor_sync(FULL, cut, z);
                cut = o > cut ? o : cut;
            }
#pragma unroll
            for (int i = 1; i < 4; i++)
                if (p[i] != NIL && k[i] < cut) {
                    p[i] = NIL;
                    rest = true;
                }
        }
    }
    if (d && p[0] != NIL) {
        const uint32_t mp = sub == 0 ? p[0] : sub == 1 ? p[1] : sub == 2 ? p[2] : p[3];
        uint32_t c = NIL;
        if (sub < TOPN && mp != NIL) c = __ldg(g.nbr + s + mp);
        if (sub == 0) {
            cur[v] = word<W>(c, ROUNDS ? max(passed, info(look(cur + v))) : 0u);
            lst[v].w = rest ? 1u : 0u;
        } else if (sub < TOPN) {
            reinterpret_cast<uint32_t*>(lst + v)[sub - 1] = c;
        }
        return true;
    }
    return false;
}

// The same for longer rows: part `q` of `parts` of the row's 128-entry steps by this
// warp.  Only entries at or above the fourth-heaviest live one so far have their end
// looked up.
template <class W>
__device__ __forceinline__ void refill_scan(const ListSeg& g, const W* cur, uint32_t s, uint32_t d, uint32_t q,
                                            uint32_t parts, Top64& t) {
    const uint32_t lane = threadIdx.x & 31;
    const uint64_t stride = 128ull * parts;
    uint32_t x[4], nx[4];
    auto load = [&](uint32_t y[4], uint64_t b) {
#pragma unroll
        for (int i = 0; i < 4; i++) y[i] = b + 32 * i + lane < d ? hi32(g.pk, s + (uint32_t)b + 32 * i + lane) : 0u;
    };
    load(x, 128ull * q);
    for (uint64_t b = 128ull * q; b < d; b += stride) {
        load(nx, b + stride);
        const uint32_t bar = (uint32_t)(t.k3 >> 32);
        uint32_t m = max(max(x[0], x[1]), max(x[2], x[3]));
        if (__any_sync(FULL, m && m >= bar)) {
            uint32_t n[4];
            W y[4];
            uint64_t key[4];
#pragma unroll
            for (int i = 0; i < 4; i++) n[i] = x[i] && x[i] >= bar ? __ldg(g.nbr + s + (uint32_t)b + 32 * i + lane) : NIL;
#pragma unroll
            for (int i = 0; i < 4; i++) {
                y[i] = n[i] != NIL ? look(cur + n[i]) : (W)DEAD;
                key[i] = n[i] != NIL ? __ldg(g.pk + s + (uint32_t)b + 32 * i + lane) : 0ull;
            }
#pragma unroll
            for (int i = 0; i < 4; i++)
                warp_add(t, !(lo(y[i]) & DEAD) ? full_key(key[i], g.k0, g.k1) : 0ull, n[i]);
        }
#pragma unroll
        for (int i = 0; i < 4; i++) x[i] = nx[i];
    }
}
// the latest round among the row's matched neighbours above key k0, and the heaviest
// matched one's key below it (as far as it lies above `low`)
struct Passed {
    uint32_t round;
    uint64_t cut;
};
__device__ __forceinline__ Passed refill_passed(const ListSeg& g, const uint64_t* cur, uint32_t s, uint32_t d,
                                                uint32_t q, uint32_t parts, uint64_t k0, uint64_t low) {
    uint32_t r = 0;
    uint64_t cut = 0;
    for (uint64_t i = 32ull * q + (threadIdx.x & 31); i < d; i += 32ull * parts) {
        const uint64_t w = __ldg(g.pk + s + (uint32_t)i);
        if ((uint32_t)(w >> 32) < (uint32_t)(low >> 32)) continue;
        const uint64_t y = look(cur + __ldg(g.nbr + s + (uint32_t)i));
        if (!(lo(y) & DEAD)) continue;
        const uint64_t key = full_key(w, g.k0, g.k1);
        if (key > k0) r = max(r, info(y));
        else if (key > cut) cut = key;
    }
    r = __reduce_max_sync(FULL, r);
    const uint32_t hi = __reduce_max_sync(FULL, (uint32_t)(cut >> 32));
    const uint32_t l = __reduce_max_sync(FULL, ((uint32_t)(cut >> 32) == hi) ? (uint32_t)cut : 0u);
    return {r, ((uint64_t)hi << 32) | l};
}
template <class W>
__device__ __forceinline__ void refill_put(W* cur, uint4* lst, uint32_t v, const Top64& t, const Passed& ps) {
    cur[v] = word<W>(t.p0, sizeof(W) == 8 ? max(ps.round, info(look(cur + v))) : 0u);
    // (with four live ones there may be more of them; the list ends at ps.cut)
    lst[v] = make_uint4(t.k1 > ps.cut ? t.p1 : NIL, t.k2 > ps.cut ? t.p2 : NIL, t.k3 > ps.cut ? t.p3 : NIL,
                        t.k3 || (t.k1 && t.k1 <= ps.cut) || (t.k2 && t.k2 <= ps.cut) ? 1u : 0u);
}

// ---------------------------------------------------------------- k_live
constexpr int LT = 256, LV = 2;
constexpr uint32_t BLOCK_ROW = 1024;  // longer rows are refilled by the whole block
constexpr uint32_t IDLE_MAX = 48;     // passes without a change before a block gives its rows back

struct LiveSmem {
    Top64 top[LT / 32];
    uint64_t cut[LT / 32];
    uint32_t passed[LT / 32];
    uint32_t part, nlive, nq0, nq1, nq2, changed, stop;
    uint32_t red[LT / 32];
};

// append the warp's rows (one a lane where on)
__device__ __forceinline__ void warp_append(uint32_t* ctr, uint32_t* out, bool on, uint32_t v) {
    const uint32_t b = __ballot_sync(FULL, on);
    if (!b) return;
    uint32_t base = 0;
    if ((threadIdx.x & 31) == 0) base = atomicAdd(ctr, (uint32_t)__popc(b));
    base = __shfl_sync(FULL, base, 0);
    if (on) out[base + __popc(b & lanemask_lt())] = v;
}

// Blocks take parts (consecutive rows of one graph) from a counter and pass over a
// part's live rows, compacted after every pass in the part's own range of the list
// buffers, until none is left.  A part may wait for words that another block writes,
// but no block waits for good: after IDLE_MAX passes without a change it puts
// the part's rows back for the next launch, which the last block to leave asks for.
template <class W>
__global__ void __launch_bounds__(LT, 4) k_live(const ListArgs* __restrict__ pa, cudaGraphConditionalHandle h,
                                                uint32_t in_graph) {
    constexpr bool ROUNDS = sizeof(W) == 8;
    __shared__ LiveSmem S;
    const ListArgs& a = *pa;
    DevState* st = a.st;
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t launch = ld_volatile_u32(&st->round);
    uint32_t left = 0;   // thread 0: rows given back
    for (;;) {
        if (tid == 0) S.part = atomicAdd(&st->task[0], 1u);
        __syncthreads();
        const uint32_t part = S.part;
        if (part >= a.nparts) break;
        const uint32_t si = a.pmap ? a.pmap[part] : 0u;
        const ListSeg& g = a.segs[si];
        const uint32_t per = (g.nrows + g.nparts - 1) / g.nparts;
        const uint32_t from = min(g.nrows, (part - g.part0) * per);
        uint32_t cnt = min(g.nrows, from + per) - from, buf = 0;
        const uint32_t* list = g.vid + from;
        const size_t home = (size_t)g.vbase + from;   // the part's range of the buffers
        if (launch) {
            cnt = a.pcount[part] >> 1;
            buf = a.pcount[part] & 1u;
            list = a.list[buf] + home;
        }
        W* cur = words<W>(a) + g.vbase;
        uint4* lst = a.lst + g.vbase;
        uint32_t matched = 0, last = 0, idle = 0;
        for (uint32_t pass = 0; cnt; pass++) {
            uint32_t* out = a.list[buf ^ 1u] + home;
            uint32_t* q0 = a.queue[0] + home;     // rows to refill: short ones,
            uint32_t* q1 = a.queue[1] + home;     // a warp's,
            uint32_t* q2 = a.queue[2] + home;     // the block's
            if (tid == 0) {
                S.nlive = S.nq0 = S.nq1 = S.nq2 = 0;
                S.changed = 0;
                S.stop = 0;
                if (globaltimer_ns() - st->t0_ns > a.limit_ns) {
                    set_err(st, ERR_TIMEOUT, pass);
                    S.stop = 1;
                } else if ((pass & 15u) == 15u && ld_volatile_u32(&st->err)) {
                    S.stop = 1;
                }
            }
            __syncthreads();
            bool changed = false;
            for (uint32_t base = 0; base < cnt; base += LT * LV) {
                uint32_t v[LV];
                W w[LV], t[LV];
                uint4 l[LV];
#pragma unroll
                for (int i = 0; i < LV; i++) {
                    const uint32_t at = base + i * LT + tid;
                    v[i] = at < cnt ? list[at] : NIL;
                }
#pragma unroll
                for (int i = 0; i < LV; i++) {
                    w[i] = v[i] != NIL ? look(cur + v[i]) : (W)0;
                    l[i] = v[i] != NIL ? lst[v[i]] : make_uint4(NIL, NIL, NIL, 0);
                }
#pragma unroll
                for (int i = 0; i < LV; i++) {
                    if (v[i] != NIL && lo(w[i]) >= g.n) { set_err(st, ERR_BOUNDS, lo(w[i])); v[i] = NIL; }
                    t[i] = v[i] != NIL ? look(cur + lo(w[i])) : (W)0;
                }
                W n[LV][3];
#pragma unroll
                for (int i = 0; i < LV; i++) {
                    const bool gone = v[i] != NIL && (lo(t[i]) & DEAD) && (lo(t[i]) & VMASK) != v[i];
                    n[i][0] = gone && l[i].x != NIL ? look(cur + l[i].x) : (W)DEAD;
                    n[i][1] = gone && l[i].y != NIL ? look(cur + l[i].y) : (W)DEAD;
                    n[i][2] = gone && l[i].z != NIL ? look(cur + l[i].z) : (W)DEAD;
                }
#pragma unroll
                for (int i = 0; i < LV; i++) {
                    bool live = false, refill = false;
                    uint32_t d = 0;
                    if (v[i] != NIL) {
                        uint32_t u = lo(w[i]), passed = info(w[i]);
                        W y = t[i];
                        live = true;
                        if ((lo(y) & DEAD) && (lo(y) & VMASK) != v[i]) {
                            changed = true;
                            const uint32_t c[3] = {l[i].x, l[i].y, l[i].z};
                            passed = max(passed, info(y));
                            int k = 0;
                            for (; k < 3; k++) {
                                if (c[k] == NIL) { k = 3; break; }
                                if (!(lo(n[i][k]) & DEAD)) break;
                                passed = max(passed, info(n[i][k]));
                            }
                            if (k < 3) {
                                u = c[k];
                                y = n[i][k];
                                cur[v[i]] = word<W>(u, passed);
                                lst[v[i]] = k == 0 ? make_uint4(c[1], c[2], NIL, l[i].w)
                                          : k == 1 ? make_uint4(c[2], NIL, NIL, l[i].w)
                                                   : make_uint4(NIL, NIL, NIL, l[i].w);
                            } else {
                                live = false;
                                refill = l[i].w != 0;
                                if (refill) {
                                    d = __ldg(g.off + v[i] + 1) - __ldg(g.off + v[i]);
                                    if (ROUNDS) cur[v[i]] = word<W>(u, passed);
                                }
                            }
                        }
                        if (live && (lo(y) & VMASK) == v[i]) {
                            // chosen back
                            uint32_t r = 0;
                            if (ROUNDS) {
                                // its word, if matched already, has the round; else both ends' passed ones give it
                                r = (lo(y) & DEAD) ? info(y) : max(passed, info(y)) + 1u;
                                last = max(last, r);
                            }
                            cur[v[i]] = word<W>(u | DEAD, r);
                            g.dst[v[i]] = u;
                            matched++;
                            live = false;
                            changed = true;
                        }
                    }
                    warp_append(&S.nlive, out, live, v[i]);
                    warp_append(&S.nq0, q0, refill && d <= 32, v[i]);
                    warp_append(&S.nq1, q1, refill && d > 32 && d <= BLOCK_ROW, v[i]);
                    warp_append(&S.nq2, q2, refill && d > BLOCK_ROW, v[i]);
                }
            }
            if (changed) S.changed = 1;
            __syncthreads();
            // rows whose list is used up
            const uint32_t k0 = S.nq0, k1 = S.nq1, k2 = S.nq2;
            for (uint32_t b = warp * 8; b < k0; b += LT / 4) {
                const uint32_t i = b + lane / 4;
                uint32_t v = 0, s = 0, d = 0;
                if (i < k0) {
                    v = q0[i];
                    s = __ldg(g.off + v);
                    d = __ldg(g.off + v + 1) - s;
                }
                const bool live = refill_group<W, 4>(a, g, v, s, d);
                warp_append(&S.nlive, out, live && (lane & 3) == 0, v);
            }
            for (uint32_t i = warp; i < k1; i += LT / 32) {
                const uint32_t v = q1[i], s = __ldg(g.off + v), d = __ldg(g.off + v + 1) - s;
                bool live;
                if (d <= 256) {
                    live = refill_group<W, 32>(a, g, v, s, d);
                } else {
                    Top64 t;
                    refill_scan<W>(g, cur, s, d, 0, 1, t);
                    live = t.k0 != 0;
                    Passed ps = {0, 0};
                    if (ROUNDS && live)
                        ps = refill_passed(g, reinterpret_cast<const uint64_t*>(cur), s, d, 0, 1, t.k0, t.k3);
                    if (live && lane == 0) refill_put<W>(cur, lst, v, t, ps);
                }
                warp_append(&S.nlive, out, live && lane == 0, v);
            }
            for (uint32_t i = 0; i < k2; i++) {
                const uint32_t v = q2[i], s = __ldg(g.off + v), d = __ldg(g.off + v + 1) - s;
                {
                    Top64 t;
                    refill_scan<W>(g, cur, s, d, warp, LT / 32, t);
                    if (lane == 0) S.top[warp] = t;
                }
                __syncthreads();
                Top64 r;
                {
                    const Top64& q = S.top[lane >> 2];   // 8 warps x 4: every warp merges all
                    const uint32_t z = lane & 3;
                    warp_add(r, z == 0 ? q.k0 : z == 1 ? q.k1 : z == 2 ? q.k2 : q.k3,
                             z == 0 ? q.p0 : z == 1 ? q.p1 : z == 2 ? q.p2 : q.p3);
                }
                if (ROUNDS) {
                    if (r.k0) {
                        const Passed x = refill_passed(g, reinterpret_cast<const uint64_t*>(cur), s, d, warp,
                                                       LT / 32, r.k0, r.k3);
                        if (lane == 0) {
                            S.passed[warp] = x.round;
                            S.cut[warp] = x.cut;
                        }
                    }
                    __syncthreads();
                }
                if (warp == 0) {
                    Passed ps = {0, 0};
                    if (ROUNDS && r.k0)
                        for (int w = 0; w < LT / 32; w++) {
                            ps.round = max(ps.round, S.passed[w]);
                            ps.cut = S.cut[w] > ps.cut ? S.cut[w] : ps.cut;
                        }
                    if (r.k0 && lane == 0) refill_put<W>(cur, lst, v, r, ps);
                    warp_append(&S.nlive, out, r.k0 && lane == 0, v);
                }
                __syncthreads();
            }
            __syncthreads();
            cnt = S.nlive;
            const uint32_t ch = S.changed, stop = S.stop;
            list = out;
            buf ^= 1u;
            __syncthreads();  // read before the next pass resets them
            idle = ch ? 0u : idle + 1u;
            if (stop || idle > IDLE_MAX) break;
        }
        if (tid == 0) a.pcount[part] = cnt << 1 | buf;
        matched = __reduce_add_sync(FULL, matched);
        if (lane == 0) S.red[warp] = matched;
        if (ROUNDS) {
            last = __reduce_max_sync(FULL, last);
            if (lane == 0) S.passed[warp] = last;
        }
        __syncthreads();
        if (tid == 0) {
            left += cnt;
            unsigned long long t = 0;
            uint32_t r = 0;
            for (int i = 0; i < LT / 32; i++) {
                t += S.red[i];
                if (ROUNDS) r = max(r, S.passed[i]);
            }
            if (t) atomicAdd(a.gmatched ? &a.gmatched[si] : &st->matched2, t);
            if (ROUNDS && r) {
                atomicMax(a.grounds ? &a.grounds[si] : &st->rounds, r);
                if (r > a.max_rounds) set_err(st, ERR_TIMEOUT, r);
            }
        }
    }
    if (tid == 0) {
        if (left) atomicAdd(&st->left, left);
        __threadfence();
        if (atomicAdd(&st->exit_v, 1u) == gridDim.x - 1) {
            __threadfence();
            st->exit_v = 0;
            st->task[0] = 0;
            const uint32_t rest = ld_volatile_u32(&st->left);
            st->left = 0;
            st->round = launch + 1;
            if (rest == 0) st->done = 1;
            if (in_graph) cudaGraphSetConditional(h, rest && !ld_volatile_u32(&st->err) ? 1u : 0u);
            __threadfence();
        }
    }
}

// ---------------------------------------------------------------- per-round counts
// An edge is live up to the earlier match of its ends (the result is maximal: one of
// them is matched), a matched row up to its own match, another up to the last of its
// neighbours'.  k_round_bytes packs the match rounds (63: that or later, 255:
// unmatched) so that the gathers of k_round_counts stay in L2; ring_m / ring_n get the
// edges and rows by their last live round.  Counters are a thread's own columns of a
// shared table: nearly all lanes count the same few rounds.
__global__ void k_round_bytes(const ListArgs* __restrict__ pa, uint8_t* mr) {
    const ListArgs& a = *pa;
    const uint32_t n = a.segs[0].n;
    const uint64_t* cur = words<uint64_t>(a);
    const uint32_t* dst = a.segs[0].dst;
    for (uint64_t v = blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (uint64_t)gridDim.x * blockDim.x)
        mr[v] = dst[v] == NIL ? 255 : (uint8_t)min(info(cur[v]) - 1u, 63u);
}
__global__ void __launch_bounds__(256) k_round_counts(const ListArgs* __restrict__ pa,
                                                      const uint8_t* __restrict__ mr) {
    __shared__ uint32_t h[64][128];   // two threads a column: counts of either by halves of 16 bits
    const ListArgs& a = *pa;
    const ListSeg& g = a.segs[0];
    const uint32_t tid = threadIdx.x;
    uint16_t* col = reinterpret_cast<uint16_t*>(&h[0][0]) + tid;   // [round][thread]
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (int kind = 0; kind < 2; kind++) {
        unsigned long long* ring = reinterpret_cast<unsigned long long*>(kind ? a.st->ring_n : a.st->ring_m);
        const uint64_t total = kind ? (uint64_t)g.nrows * 8 : g.m;
        // (steps of at most 32768 counts a thread, so that 16 bits hold them)
        for (uint64_t base = 0; base < total; base += stride * 32768) {
            for (int i = 0; i < 64; i++) col[i * 256] = 0;
            const uint64_t end = total - base < stride * 32768 ? total : base + stride * 32768;
            for (uint64_t i = base + blockIdx.x * blockDim.x + tid; i < ((end + 31) & ~31ull); i += stride) {
                uint32_t r = NIL;
                if (kind == 0) {
                    if (i < end) {
                        const uint64_t rec = __ldg(g.edges + i);
                        r = min((uint32_t)__ldg(mr + (uint32_t)rec), (uint32_t)__ldg(mr + (uint32_t)(rec >> 32)));
                    }
                } else {
                    // eight lanes a row
                    uint32_t own = 0;
                    if (i < end) {
                        const uint32_t row = (uint32_t)(i >> 3), v = g.vid[row];
                        own = mr[v];
                        if (own == 255) {
                            own = 0;
                            for (uint64_t j = (uint64_t)g.roff[row] + (i & 7); j < g.roff[row + 1]; j += 8)
                                own = max(own, (uint32_t)__ldg(mr + g.nbr[j]));
                        }
                    }
                    own = max(own, __shfl_xor_sync(FULL, own, 1));
                    own = max(own, __shfl_xor_sync(FULL, own, 2));
                    own = max(own, __shfl_xor_sync(FULL, own, 4));
                    if (i < end && (i & 7) == 0) r = own;
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
__global__ void k_list_map(const ListArgs* __restrict__ pa, uint32_t* bmap, uint32_t* pmap) {
    const ListArgs& a = *pa;
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
uint32_t live_grid() { return (uint32_t)sms() * 4; }

}  // namespace

uint32_t list_blocks(const uint32_t task[4], uint32_t nrows) {
    const TopBlocks b = top_blocks(task, nrows);
    const uint32_t t = b.l + b.w + b.g + b.s;
    return t ? t : 1u;
}
int launch_list_map(void* stream, const ListArgs* d, uint32_t nsegs, uint32_t* bmap, uint32_t* pmap) {
    k_list_map<<<(nsegs + 7) / 8, 256, 0, (cudaStream_t)stream>>>(d, bmap, pmap);
    return (int)cudaGetLastError();
}
int launch_top(void* stream, const ListArgs* d, uint32_t blocks, bool rounds) {
    if (rounds) k_top<uint64_t><<<blocks, TT, sizeof(TopSmem), (cudaStream_t)stream>>>(d);
    else k_top<uint32_t><<<blocks, TT, sizeof(TopSmem), (cudaStream_t)stream>>>(d);
    return (int)cudaGetLastError();
}
// (more blocks than parts would only come and go)
int launch_live(void* stream, const ListArgs* d, uint32_t nparts, bool rounds) {
    const uint32_t grid = nparts < live_grid() ? nparts : live_grid();
    const cudaGraphConditionalHandle none{};
    if (rounds) k_live<uint64_t><<<grid, LT, 0, (cudaStream_t)stream>>>(d, none, 0u);
    else k_live<uint32_t><<<grid, LT, 0, (cudaStream_t)stream>>>(d, none, 0u);
    return (int)cudaGetLastError();
}
int launch_round_counts(void* stream, const ListArgs* d, void* bytes) {
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
    uint32_t yes = 1;
    void* params[3] = {&dargs, &h, &yes};
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
