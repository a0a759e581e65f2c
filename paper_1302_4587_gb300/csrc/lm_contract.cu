// Contraction of a matching: the step that multilevel graph partitioning
// repeats on maximal matchings (Sec. 1 names it as the main use of the
// matching).  Reading: a matched pair becomes one coarse vertex and an
// unmatched vertex stays alone; coarse ids number the representatives (the
// unmatched vertices and the smaller end of each pair) in vertex order; a
// coarse vertex weighs the sum of its members; edges inside a pair vanish;
// the original edges between two coarse vertices become one coarse edge,
// placed and oriented as the first of them in the input order, whose weight
// is their sum (accumulated in double in input order, rounded once to float32).
//
// Device steps (all of them here): representatives and their prefix ranks;
// the coarse map and vertex weights; every edge gets a 32-bit hash of its unordered
// coarse pair, and its coarse endpoints are stored.  The crossing edges go to
// partitions by the hash's top bits (k_c_part); in each partition a bitmap in shared
// memory finds the edges that share their slot of the hash with another (most pairs
// have one edge, which then is done), and a hash table the ones whose full hash repeats
// (k_c_groups).  Each such run (a group of several edges, or pairs whose hashes collide)
// is put in input order and walked (k_c_walk): its groups' first edges lead, every later
// member loses its crossing bit, and a leader of several edges records the group's
// weight summed over its edges in order.  An edge alone with its hash is alone in its
// group and leads it.  Runs too long or too mixed for that walk are taken out in input
// order and sorted by the pair itself.  Prefix counts of the remaining bits (the leaders)
// give each coarse edge its place, and the leaders write the coarse edges.
// Lists that partitions don't suit (see contract_part_bits, and one with a partition of
// more than twice the average) are sorted instead: a stable LSD radix sort by the low B
// bits of the hash (8-bit passes, as few as leave about 2048 edges to a bucket of equal
// low bits; edges inside a pair have the key 0xFFFFFFFF, and no pair's hash ends in the
// byte 0xFF, so that they end up last) brings each pair's edges into one bucket, still in
// input order, and k_c_buckets finds the runs.
// R-MAT scale 22 (64M edges): sort 2.18 ms, partitions 1.40 (part 525, groups 327, walk
// 125, emit 266 us, the rest map, scans and a host round trip).
#include <cstdint>
#include <type_traits>
#include <cuda_runtime.h>
#include "../../include/lm.h"
#include "lm_internal.h"

namespace lm {

namespace {

constexpr uint32_t CT = 256;
constexpr uint32_t C_ERR_MATE = 1u, C_ERR_EDGE = 2u;

uint32_t grid_for(uint64_t count) {
    int dev = 0;
    cudaGetDevice(&dev);
    const uint64_t b = (count + CT - 1) / CT;
    const uint64_t cap = (uint64_t)device_sm_count(dev) * 16;
    return (uint32_t)(b < 1 ? 1 : (b > cap ? cap : b));
}

// (vertex numbers of a step beyond n may not fit 32 bits)
__global__ void k_c_rep(const uint32_t* __restrict__ mate, uint32_t n, uint32_t* __restrict__ flag,
                        uint32_t* __restrict__ err) {
    for (uint64_t v = blockIdx.x * CT + threadIdx.x; v < n; v += gridDim.x * CT) {
        const uint32_t u = mate[v];
        bool rep = true;
        if (u != NIL) {
            if (u >= n || u == v || mate[u] != v) { atomicOr(err, C_ERR_MATE); rep = false; }
            else rep = v < u;
        }
        flag[v] = rep ? 1u : 0u;
    }
}

__global__ void k_c_map(const uint32_t* __restrict__ mate, uint32_t n, const uint32_t* __restrict__ rank,
                        const uint32_t* __restrict__ vw, uint32_t* __restrict__ cmap, uint32_t* __restrict__ cvw) {
    for (uint64_t i = blockIdx.x * CT + threadIdx.x; i < n; i += gridDim.x * CT) {
        const uint32_t v = (uint32_t)i;
        uint32_t u = mate[v];
        if (u >= n) u = v;  // unmatched (an invalid mate was flagged by k_c_rep)
        const uint32_t c = rank[u < v ? u : v];
        cmap[v] = c;
        atomicAdd(&cvw[c], vw ? vw[v] : 1u);
    }
}

// the unordered coarse pair of an edge as a 64-bit word, min(c, d) << 32 | max(c, d)
__device__ __forceinline__ unsigned long long pair_word(uint32_t c, uint32_t d) {
    return ((unsigned long long)min(c, d) << 32) | max(c, d);
}
// 32-bit hash of a pair word (a 64-bit finaliser's upper half) whose low byte is never
// 0xFF: sorted by any number of low bytes, the pairs come before the edges inside a
// pair (key 0xFFFFFFFF)
__device__ __forceinline__ uint32_t pair_hash(unsigned long long x) {
    x ^= x >> 33;
    x *= 0xFF51AFD7ED558CCDull;
    x ^= x >> 33;
    x *= 0xC4CEB9FE1A85EC53ull;
    x ^= x >> 33;
    const uint32_t h = (uint32_t)(x >> 32);
    return (h & 0xFFu) == 0xFFu ? h ^ 1u : h;
}

// Edge kernels take four consecutive edges per thread (vector loads when the
// arrays are 16-byte aligned) and a warp 128 edges: four whole words of a bitmask
// over the edges, lanes 8q .. 8q+7 sharing word q.
template <bool VEC>
__device__ __forceinline__ uint4 load4(const uint32_t* a, uint64_t i, uint32_t count) {
    if (VEC && i + 4 <= count) return __ldg(reinterpret_cast<const uint4*>(a + i));
    uint4 v;
    v.x = i < count ? a[i] : 0u;
    v.y = i + 1 < count ? a[i + 1] : 0u;
    v.z = i + 2 < count ? a[i + 2] : 0u;
    v.w = i + 3 < count ? a[i + 3] : 0u;
    return v;
}
__device__ __forceinline__ uint32_t at(const uint4& v, int j) { return j == 0 ? v.x : j == 1 ? v.y : j == 2 ? v.z : v.w; }

// every edge in input order, keyed by a hash of its unordered coarse pair (equal
// pairs get equal keys); an edge inside a pair (or with an endpoint >= n) gets the
// key 0xFFFFFFFF, above every pair's, so the sort puts it at the end.  Bit e of
// cross: edge e joins two coarse vertices (counted in counts[0]); cpair: the
// coarse endpoints of every edge; hist: each tile's counts of the keys' low byte,
// the sort's first digit.  A warp takes 64 groups of four edges per step, their
// loads issued together.
template <bool VEC>
__global__ void __launch_bounds__(CT) k_c_keys(const uint32_t* __restrict__ eu, const uint32_t* __restrict__ ev,
                                               uint32_t m, uint32_t n, const uint32_t* __restrict__ cmap,
                                               uint32_t* __restrict__ key, uint32_t* __restrict__ cpair,
                                               uint32_t* __restrict__ cross, uint32_t* __restrict__ counts,
                                               uint32_t* __restrict__ hist, uint32_t* __restrict__ err) {
    __shared__ uint32_t h[256];
    h[threadIdx.x] = 0;
    __syncthreads();
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t mine = 0;
    // a block takes the 4096 edges of one tile of the sort that follows (1024 groups
    // of four); g0: the warp's first group of a step (a multiple of 64, so of 8)
    for (uint32_t it = 0; it < 2; it++) {
        const uint64_t g0 = (uint64_t)blockIdx.x * 1024 + warp * 128 + it * 64;
        uint4 a[2], b[2];
#pragma unroll
        for (int u = 0; u < 2; u++) {
            const uint64_t e0 = 4 * (g0 + 32 * u + lane);
            a[u] = load4<VEC>(eu, e0, m);
            b[u] = load4<VEC>(ev, e0, m);
        }
        uint32_t cu[2][4], cv[2][4];
#pragma unroll
        for (int u = 0; u < 2; u++) {
            const uint64_t e0 = 4 * (g0 + 32 * u + lane);
#pragma unroll
            for (int j = 0; j < 4; j++) {
                const uint32_t x = at(a[u], j), y = at(b[u], j);
                const bool ok = e0 + j < m && x < n && y < n;
                if (e0 + j < m && !ok) atomicOr(err, C_ERR_EDGE);
                cu[u][j] = ok ? cmap[x] : 0u;
                cv[u][j] = ok ? cmap[y] : 0u;
            }
        }
#pragma unroll
        for (int u = 0; u < 2; u++) {
            const uint64_t g = g0 + 32 * u + lane;
            const uint64_t e0 = 4 * g;
            uint32_t nib = 0, k[4];
#pragma unroll
            for (int j = 0; j < 4; j++) {
                k[j] = 0xFFFFFFFFu;
                if (e0 + j >= m) continue;
                if (cu[u][j] != cv[u][j]) {
                    k[j] = pair_hash(pair_word(cu[u][j], cv[u][j]));
                    nib |= 1u << j;
                }
                atomicAdd(&h[k[j] & 0xFFu], 1u);  // the sort's first digit
            }
            if (e0 + 4 <= m) {  // key and cpair are 16-byte aligned scratch
                *reinterpret_cast<uint4*>(key + e0) = make_uint4(k[0], k[1], k[2], k[3]);
                *reinterpret_cast<uint4*>(cpair + 2 * e0) = make_uint4(cu[u][0], cv[u][0], cu[u][1], cv[u][1]);
                *reinterpret_cast<uint4*>(cpair + 2 * e0 + 4) = make_uint4(cu[u][2], cv[u][2], cu[u][3], cv[u][3]);
            } else {
#pragma unroll
                for (int j = 0; j < 4; j++)
                    if (e0 + j < m) {
                        key[e0 + j] = k[j];
                        cpair[2 * (e0 + j)] = cu[u][j];
                        cpair[2 * (e0 + j) + 1] = cv[u][j];
                    }
            }
            mine += __popc(nib);
            uint32_t w = nib << (4 * (g & 7));
            w |= __shfl_xor_sync(0xFFFFFFFFu, w, 1);
            w |= __shfl_xor_sync(0xFFFFFFFFu, w, 2);
            w |= __shfl_xor_sync(0xFFFFFFFFu, w, 4);
            if ((g & 7) == 0 && e0 < m) cross[g >> 3] = w;
        }
    }
    // one atomic per warp on the count
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mine += __shfl_xor_sync(0xFFFFFFFFu, mine, o);
    if (lane == 0 && mine) atomicAdd(&counts[0], mine);
    __syncthreads();
    hist[threadIdx.x * gridDim.x + blockIdx.x] = h[threadIdx.x];  // digit-major, as the sort's counts
}

// ---- partitions --------------------------------------------------------------
// The crossing edges go to 2^pb partitions by the top bits of their hash, as (hash, edge)
// items in no particular order, each partition in a room of cap items of its own
// (gcur: its items; more than cap: counts[4] is set, the items are not kept).  A block
// maps and keys a tile of PT_TILE edges, counts them by partition in shared memory
// (each item's rank is what the count returned), takes a run of every partition's room with
// one atomic, and writes the tile out in partition order, so that runs of 8 items and
// more are written together.  Also writes cpair, cross and counts[0], as k_c_keys.
// R-MAT scale 21, 31.8M edges: 268 us, of which the gathers of cmap 92, the items' stores
// 26, cpair 33, the rest the phases in shared memory.  Three blocks an SM (spills), 8 or
// 24 edges a thread, 256 or 1024 threads: 3 to 15% slower over all.
constexpr uint32_t PT_T = 512, PT_E = 16, PT_TILE = PT_E * PT_T;
template <uint32_t D>  // partitions a thread: at most D PT_T
struct PtSmem {
    uint32_t key[PT_TILE];
    uint16_t edge[PT_TILE];  // its place in the tile
    uint32_t cnt[D * PT_T];   // items of each partition, then where its run starts in it
    uint32_t gofs[D * PT_T];  // the run's place in the partition's room, minus that
    uint32_t ws[PT_T / 32];
};
static_assert(PT_E % 8 == 0 && PT_TILE <= 65536, "eight edges a step, 16-bit places");

template <bool VEC, uint32_t D>
__global__ void __launch_bounds__(PT_T, 2)
    k_c_part(const uint32_t* __restrict__ eu, const uint32_t* __restrict__ ev, uint32_t m, uint32_t n,
             const uint32_t* __restrict__ cmap, uint32_t pb, uint32_t cap, uint32_t* __restrict__ gcur,
             uint2* __restrict__ items, uint32_t* __restrict__ cpair, uint32_t* __restrict__ cross,
             uint32_t* __restrict__ counts, uint32_t* __restrict__ err) {
    extern __shared__ __align__(16) unsigned char pt_raw[];
    PtSmem<D>& S = *reinterpret_cast<PtSmem<D>*>(pt_raw);
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t dsh = 32 - pb;
    for (uint32_t i = tid; i < D * PT_T; i += PT_T) S.cnt[i] = 0;
    __syncthreads();
    uint32_t mine = 0, key[PT_E], rk[PT_E / 2];
#pragma unroll
    for (int it = 0; it < (int)PT_E / 8; it++) {
        uint4 a[2], b[2];
#pragma unroll
        for (int u = 0; u < 2; u++) {
            const uint64_t e0 = (uint64_t)blockIdx.x * PT_TILE + 4 * ((2 * it + u) * PT_T + tid);
            a[u] = load4<VEC>(eu, e0, m);
            b[u] = load4<VEC>(ev, e0, m);
        }
        uint32_t cu[2][4], cv[2][4];
#pragma unroll
        for (int u = 0; u < 2; u++) {
            const uint64_t e0 = (uint64_t)blockIdx.x * PT_TILE + 4 * ((2 * it + u) * PT_T + tid);
#pragma unroll
            for (int j = 0; j < 4; j++) {
                const uint32_t x = at(a[u], j), y = at(b[u], j);
                const bool ok = e0 + j < m && x < n && y < n;
                if (e0 + j < m && !ok) atomicOr(err, C_ERR_EDGE);
                cu[u][j] = ok ? cmap[x] : 0u;
                cv[u][j] = ok ? cmap[y] : 0u;
            }
        }
#pragma unroll
        for (int u = 0; u < 2; u++) {
            const uint64_t e0 = (uint64_t)blockIdx.x * PT_TILE + 4 * ((2 * it + u) * PT_T + tid);
            uint32_t nib = 0;
#pragma unroll
            for (int j = 0; j < 4; j++) {
                const int i = 8 * it + 4 * u + j;
                key[i] = 0xFFFFFFFFu;
                uint32_t r = 0;
                if (cu[u][j] != cv[u][j]) {  // (never past m: both are 0 there)
                    key[i] = pair_hash(pair_word(cu[u][j], cv[u][j]));
                    nib |= 1u << j;
                    r = atomicAdd(&S.cnt[key[i] >> dsh], 1u);
                }
                if (i & 1) rk[i >> 1] |= r << 16;
                else rk[i >> 1] = r;
            }
            if (e0 + 4 <= m) {
                *reinterpret_cast<uint4*>(cpair + 2 * e0) = make_uint4(cu[u][0], cv[u][0], cu[u][1], cv[u][1]);
                *reinterpret_cast<uint4*>(cpair + 2 * e0 + 4) = make_uint4(cu[u][2], cv[u][2], cu[u][3], cv[u][3]);
            } else {
#pragma unroll
                for (int j = 0; j < 4; j++)
                    if (e0 + j < m) {
                        cpair[2 * (e0 + j)] = cu[u][j];
                        cpair[2 * (e0 + j) + 1] = cv[u][j];
                    }
            }
            mine += __popc(nib);
            uint32_t w = nib << (4 * (lane & 7));
            w |= __shfl_xor_sync(0xFFFFFFFFu, w, 1);
            w |= __shfl_xor_sync(0xFFFFFFFFu, w, 2);
            w |= __shfl_xor_sync(0xFFFFFFFFu, w, 4);
            if ((lane & 7) == 0 && e0 < m) cross[e0 >> 5] = w;
        }
    }
    mine = __reduce_add_sync(0xFFFFFFFFu, mine);
    if (lane == 0 && mine) atomicAdd(&counts[0], mine);
    __syncthreads();
    // thread t: partitions D t .. D t + D - 1
    uint32_t c[D], x = 0;
#pragma unroll
    for (uint32_t i = 0; i < D; i++) x += c[i] = S.cnt[D * tid + i];
    const uint32_t sum = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, o);
        if (lane >= (uint32_t)o) x += y;
    }
    if (lane == 31) S.ws[warp] = x;
    __syncthreads();
    uint32_t start = x - sum, total = 0;
    for (uint32_t w = 0; w < PT_T / 32; w++) {
        if (w < warp) start += S.ws[w];
        total += S.ws[w];
    }
#pragma unroll
    for (uint32_t i = 0; i < D; i++) {
        if (c[i]) {
            const uint32_t had = atomicAdd(&gcur[D * tid + i], c[i]);
            if (had + c[i] > cap) atomicOr(&counts[4], 1u);
            S.gofs[D * tid + i] = had - start;
        }
        S.cnt[D * tid + i] = start;
        start += c[i];
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < (int)PT_E; i++) {
        if (key[i] == 0xFFFFFFFFu) continue;
        const uint32_t p = S.cnt[key[i] >> dsh] + ((rk[i >> 1] >> (16 * (i & 1))) & 0xFFFFu);
        S.key[p] = key[i];
        S.edge[p] = (uint16_t)(4 * ((i >> 2) * PT_T + tid) + (i & 3));
    }
    __syncthreads();
    for (uint32_t p = tid; p < total; p += PT_T) {
        const uint32_t x = S.key[p], d = x >> dsh, o = S.gofs[d] + p;
        if (o < cap) items[(size_t)d * cap + o] = make_uint2(x, blockIdx.x * PT_TILE + S.edge[p]);
    }
}

// ---- buckets of the partial hash sort --------------------------------------
// The sort orders the items by the low B bits of their keys only, so a bucket
// (the items sharing those bits) holds every edge of each of its pairs, in input
// order.  A block takes the buckets that start in its chunk of BK_C sorted items.
// It reads a window of BK_W keys from the chunk's first bucket on into registers,
// enters the keys of its buckets in a shared-memory hash table with a count per
// key, and lists the items whose key repeats grouped by key.  Each such run (a
// group of several edges, or pairs whose hashes collide) is put back in input
// order and walked by one thread: with at most GR_PAIRS distinct pairs among at
// most GR_MAX items (the case on simple graphs, where a group has at most four
// edges) it finds the groups in registers -- a group's first edge leads it, every
// later member loses its crossing bit as soon as it is seen, and a leader of
// several edges gets its multi bit and the group's weight summed in double in
// input order once the run is known to fit.  A bucket that runs past the window
// is done in a second window that starts at it.  A bucket longer than a window,
// and any run that does not fit the walk, is flagged in ofl (a bit per edge) for the
// general path below: taken out in order with its pair as the key and sorted by the pair
// (which clears the same bits again).
constexpr uint32_t GR_MAX = 64, GR_PAIRS = 4, GR_SHORT = 8;
constexpr uint32_t BK_T = 512, BK_J = 12, BK_W = BK_T * BK_J, BK_C = 4096, BK_TS = 8192, BK_TS_BITS = 13;
constexpr uint32_t BK_AVG = 2048;  // the sort takes as few bytes as leave at most this many items to a bucket
constexpr uint32_t BK_EMPTY = 0xFFFFFFFFu;
constexpr uint32_t RUN_START = 0x80000000u, RUN_NONE = 0xFFFFFFFFu;  // (edges are below 2^31 - 1)
static_assert(BK_TS == 1u << BK_TS_BITS && BK_TS / 16 == BK_T && BK_W < BK_TS && BK_W < 65536 && BK_C < BK_W,
              "table of at most 3/4 load, 16-bit counts and window indices, a chunk shorter than a window");

struct BkSmem {
    union {
        uint32_t tab[BK_TS];    // keys of the table (BK_EMPTY: free), linear probing; then
        uint32_t dl[BK_W];      // items of runs, slot << 16 | window index, grouped by slot
    };
    uint32_t cnt[BK_TS / 2];    // a 16-bit field per slot: its items, then where its run goes in dl
    uint32_t dupb[BK_TS / 32];  // slots whose key repeats,
    uint32_t longb[BK_TS / 32]; // and those of more than GR_MAX items
    uint32_t hand[BK_J * (BK_T / 32) + 1];  // each warp's last keys, and the key before the window
    uint32_t wsum[BK_T / 32];
    uint32_t first, lastp1, end, ndup, nmid;
};

template <uint32_t TSB>
__device__ __forceinline__ uint32_t bk_slot(uint32_t k) {
    return (k * 0x9E3779B1u) >> (32 - TSB);
}

__device__ __forceinline__ unsigned long long upair(const uint32_t* __restrict__ cpair, uint32_t e) {
    const uint2 p = *reinterpret_cast<const uint2*>(cpair + 2 * (size_t)e);
    return ((unsigned long long)min(p.x, p.y) << 32) | max(p.x, p.y);
}

// The items lo <= q < hi of a window (item q: thread q % T, k[q / T]) with edges val[q]: those
// whose key repeats, by the table in S, which is cleared (val in input order, or
// BYVAL: in any).
template <uint32_t T, uint32_t J, uint32_t TSB, bool BYVAL, class SM>
__device__ __forceinline__ void bk_table(SM& S, const uint32_t (&k)[J], uint32_t lo, uint32_t hi, const uint32_t* val,
                                         uint32_t* __restrict__ list, uint32_t* __restrict__ ofl,
                                         uint32_t* __restrict__ counts) {
    constexpr uint32_t TS = 1u << TSB;
    static_assert(TS / 16 == T && T * J < TS && T * J < 65536, "16 slots a thread, a free slot always");
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // every item of [lo, hi) into the table; its slot kept in 16 bits of sp
    uint32_t sp[(J + 1) / 2];
#pragma unroll
    for (int j = 0; j < (int)J; j++) {
        const uint32_t q = j * T + tid;
        uint32_t sl = 0;
        if (q >= lo && q < hi) {
            sl = bk_slot<TSB>(k[j]);
            // (at most the window < TS keys: a free slot or the key is always found)
            for (uint32_t probe = 0; probe < TS; probe++) {
                const uint32_t old = atomicCAS(&S.tab[sl], BK_EMPTY, k[j]);
                if (old == BK_EMPTY || old == k[j]) break;
                sl = (sl + 1) & (TS - 1);
            }
            atomicAdd(&S.cnt[sl >> 1], 1u << (16 * (sl & 1)));
        }
        if (j & 1) sp[j >> 1] |= sl << 16;
        else sp[j >> 1] = sl;
    }
    __syncthreads();
    // slots of two or more items, and where each one's run starts in dl (thread t:
    // slots 16 t .. 16 t + 15, cnt words 8 t .. 8 t + 7)
    {
        uint4* cq = reinterpret_cast<uint4*>(S.cnt) + 2 * tid;
        uint32_t tot = 0, bits = 0, lng = 0;
#pragma unroll
        for (int v = 0; v < 2; v++) {
            const uint4 x = cq[v];
            const uint32_t wv[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
            for (int h = 0; h < 8; h++) {
                const uint32_t c = (wv[h >> 1] >> (16 * (h & 1))) & 0xFFFFu;
                if (c >= 2) {
                    tot += c;
                    bits |= 1u << (8 * v + h);
                    if (c > GR_MAX) lng |= 1u << (8 * v + h);
                }
            }
        }
        uint32_t x = tot;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, o);
            if (lane >= (uint32_t)o) x += y;
        }
        if (lane == 31) S.wsum[warp] = x;
        __syncthreads();
        uint32_t run = x - tot;
        for (uint32_t v = 0; v < warp; v++) run += S.wsum[v];
#pragma unroll
        for (int v = 0; v < 2; v++) {
            if (!((bits >> (8 * v)) & 0xFFu)) continue;
            const uint4 x4 = cq[v];
            uint32_t wv[4] = {x4.x, x4.y, x4.z, x4.w};
#pragma unroll
            for (int h = 0; h < 8; h++) {
                if (!((bits >> (8 * v + h)) & 1u)) continue;
                const uint32_t sh = 16 * (h & 1);
                const uint32_t c = (wv[h >> 1] >> sh) & 0xFFFFu;
                wv[h >> 1] = (wv[h >> 1] & ~(0xFFFFu << sh)) | (run << sh);
                run += c;
            }
            cq[v] = make_uint4(wv[0], wv[1], wv[2], wv[3]);
        }
        reinterpret_cast<uint16_t*>(S.dupb)[tid] = (uint16_t)bits;  // bit 16 t + h: slot 16 t + h
        reinterpret_cast<uint16_t*>(S.longb)[tid] = (uint16_t)lng;
        if (tid == T - 1) {
            S.ndup = run;
            S.nmid = 0;
        }
    }
    __syncthreads();
    // the items of repeated keys into dl, grouped by slot
#pragma unroll
    for (int j = 0; j < (int)J; j++) {
        const uint32_t q = j * T + tid;
        if (q >= lo && q < hi) {
            const uint32_t sl = (sp[j >> 1] >> (16 * (j & 1))) & 0xFFFFu;
            if ((S.dupb[sl >> 5] >> (sl & 31)) & 1u) {
                const uint32_t sh = 16 * (sl & 1);
                const uint32_t pos = (atomicAdd(&S.cnt[sl >> 1], 1u << sh) >> sh) & 0xFFFFu;
                S.dl[pos] = (sl << 16) | q;
            }
        }
    }
    __syncthreads();
    // each run back in input order, by the window index or by the edge: short ones by the
    // thread that holds their first entry (an insertion sort; its entries share their slot
    // bits, which is all that other threads read of them), those of more than GR_SHORT
    // by a warp; long ones are flagged below.  (Slots' cnt: where their runs end.)
    const uint32_t nd = S.ndup;
    uint32_t* mid = S.tab + T * J;   // their first entries and lengths, behind dl
    static_assert(T * J / (GR_SHORT + 1) <= TS - T * J && GR_MAX <= 64, "room for them, two items a lane");
    for (uint32_t i = tid; i < nd; i += T) {
        const uint32_t sl = S.dl[i] >> 16;
        if ((i > 0 && (S.dl[i - 1] >> 16) == sl) || ((S.longb[sl >> 5] >> (sl & 31)) & 1u)) continue;
        const uint32_t len = ((S.cnt[sl >> 1] >> (16 * (sl & 1))) & 0xFFFFu) - i;
        if (len > GR_SHORT) {
            mid[atomicAdd(&S.nmid, 1u)] = len << 16 | i;
            continue;
        }
        for (uint32_t a = 1; a < len; a++) {
            const uint32_t y = S.dl[i + a], vy = BYVAL ? val[y & 0xFFFFu] : y;
            uint32_t b = a;
            for (; b > 0; b--) {
                const uint32_t z = S.dl[i + b - 1];
                if ((BYVAL ? val[z & 0xFFFFu] : z) < vy) break;
                S.dl[i + b] = z;
            }
            S.dl[i + b] = y;
        }
    }
    if (tid == 0 && nd) S.wsum[0] = atomicAdd(&counts[5], nd);
    __syncthreads();
    const uint32_t nmid = S.nmid;
    for (uint32_t k = warp; k < nmid; k += T / 32) {
        const uint32_t i = mid[k] & 0xFFFFu, len = mid[k] >> 16;
        // items lane and lane + 32, in order by a bitonic network (no item: above all)
        uint32_t x[2], v[2];
#pragma unroll
        for (int h = 0; h < 2; h++) {
            const uint32_t q = lane + 32 * h;
            x[h] = q < len ? S.dl[i + q] : 0u;
            v[h] = q >= len ? 0xFFFFFFFFu : BYVAL ? val[x[h] & 0xFFFFu] : x[h];
        }
#pragma unroll
        for (uint32_t w = 2; w <= 64; w *= 2)
#pragma unroll
            for (uint32_t d = w / 2; d > 0; d /= 2) {
                if (d == 32) {
                    if (v[0] > v[1]) {
                        const uint32_t tv = v[0], tx = x[0];
                        v[0] = v[1]; x[0] = x[1];
                        v[1] = tv; x[1] = tx;
                    }
                    continue;
                }
#pragma unroll
                for (int h = 0; h < 2; h++) {
                    const uint32_t ov = __shfl_xor_sync(0xFFFFFFFFu, v[h], d), ox = __shfl_xor_sync(0xFFFFFFFFu, x[h], d);
                    const bool up = ((lane + 32 * h) & w) == 0, low = (lane & d) == 0;
                    if ((ov < v[h]) == (up == low) && ov != v[h]) {
                        v[h] = ov;
                        x[h] = ox;
                    }
                }
            }
#pragma unroll
        for (int h = 0; h < 2; h++)
            if (lane + 32 * h < len) S.dl[i + lane + 32 * h] = x[h];
    }
    if (nmid) __syncthreads();
    const uint32_t lbase = S.wsum[0];
    uint32_t lng = 0;
    for (uint32_t i = tid; i < nd; i += T) {
        const uint32_t x = S.dl[i], sl = x >> 16, e = val[x & 0xFFFFu];
        const bool start = i == 0 || (S.dl[i - 1] >> 16) != sl;
        if ((S.longb[sl >> 5] >> (sl & 31)) & 1u) {   // to the general path
            list[lbase + i] = RUN_NONE;
            atomicOr(&ofl[e >> 5], 1u << (e & 31));
            lng++;
        } else {
            list[lbase + i] = e | (start ? RUN_START : 0u);
        }
    }
    lng = __reduce_add_sync(0xFFFFFFFFu, lng);
    if (lane == 0 && lng) atomicAdd(&counts[1], lng);
}

// The runs of list (counts[5] entries: edges in input order, RUN_START on a run's first; runs
// of at most GR_MAX), a thread each: settled here, or flagged for the general path.  A
// kernel of its own: the gathers of pairs and weights are all that it does, with every
// warp that an SM holds to cover them (as the last phase of the table's block, which
// has 32 warps an SM, they took 84 us on R-MAT scale 21, here 54).
__global__ void __launch_bounds__(CT) k_c_walk(const uint32_t* __restrict__ list,
                                               const uint32_t* __restrict__ cpair, const float* __restrict__ w,
                                               uint32_t* __restrict__ cross, uint32_t* __restrict__ multi,
                                               uint32_t* __restrict__ gsum, uint32_t* __restrict__ ofl,
                                               uint32_t* __restrict__ counts) {
    const uint32_t nlist = counts[5];
    for (uint32_t i0 = blockIdx.x * CT + threadIdx.x; i0 < nlist; i0 += gridDim.x * CT) {
        const uint32_t first = list[i0];
        if (!(first & RUN_START) || first == RUN_NONE) continue;
        uint32_t len = 1;
        while (len <= GR_MAX && i0 + len < nlist && !(list[i0 + len] & RUN_START)) len++;
        unsigned long long gp[GR_PAIRS];
        uint32_t gl[GR_PAIRS], gn[GR_PAIRS];
        double gs[GR_PAIRS];
        uint32_t ng = 0;
        bool over = false;
        for (uint32_t j0 = 0; j0 < len && !over; j0 += 4) {
            uint32_t e[4];
            unsigned long long pj[4];
            float wj[4];
#pragma unroll
            for (uint32_t t = 0; t < 4; t++) e[t] = j0 + t < len ? list[i0 + j0 + t] & ~RUN_START : 0u;
#pragma unroll
            for (uint32_t t = 0; t < 4; t++) {
                pj[t] = j0 + t < len ? upair(cpair, e[t]) : 0ull;
                wj[t] = j0 + t < len ? w[e[t]] : 0.0f;
            }
#pragma unroll
            for (uint32_t t = 0; t < 4; t++) {
                if (j0 + t >= len || over) continue;
                bool found = false;
#pragma unroll
                for (uint32_t g = 0; g < GR_PAIRS; g++)
                    if (!found && g < ng && gp[g] == pj[t]) {
                        gs[g] += (double)wj[t];
                        gn[g]++;
                        found = true;
                    }
                // a later member of a group: not a leader, whatever the rest of the run
                // holds (a run left to the general path has the same bits cleared there)
                if (found) atomicAnd(&cross[e[t] >> 5], ~(1u << (e[t] & 31)));
                if (!found) {
                    if (ng == GR_PAIRS) {
                        over = true;
                    } else {
#pragma unroll
                        for (uint32_t g = 0; g < GR_PAIRS; g++)
                            if (g == ng) {
                                gp[g] = pj[t];
                                gl[g] = e[t];
                                gn[g] = 1;
                                gs[g] = (double)wj[t];
                            }
                        ng++;
                    }
                }
            }
        }
        if (over) {
            for (uint32_t a = 0; a < len; a++) {
                const uint32_t p = list[i0 + a] & ~RUN_START;
                atomicOr(&ofl[p >> 5], 1u << (p & 31));
            }
            atomicAdd(&counts[1], len);
            continue;
        }
#pragma unroll
        for (uint32_t g = 0; g < GR_PAIRS; g++)
            if (g < ng && gn[g] > 1) {
                atomicOr(&multi[gl[g] >> 5], 1u << (gl[g] & 31));
                gsum[gl[g]] = __float_as_uint((float)gs[g]);
            }
    }
}

// key: the sorted keys of the cnt crossing items (sorted by the bits in mask);
// val: their edge indices
__global__ void __launch_bounds__(BK_T, 2)
    k_c_buckets(const uint32_t* __restrict__ key, const uint32_t* __restrict__ val, uint32_t cnt, uint32_t mask,
                uint32_t* __restrict__ list, uint32_t* __restrict__ ofl, uint32_t* __restrict__ counts) {
    extern __shared__ __align__(16) unsigned char bk_raw[];
    BkSmem& S = *reinterpret_cast<BkSmem*>(bk_raw);
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // (cnt < 2^31: every index below fits in 32 bits)
    const uint32_t c0 = blockIdx.x * BK_C;
    const uint32_t cend = min(cnt, c0 + BK_C);  // this block's buckets start in [c0, cend)
    uint32_t ws = c0;                           // the window: sorted items ws .. ws + BK_W - 1
    for (;;) {
        // item q of the window (thread q % BK_T, slot q / BK_T) ...
        uint32_t k[BK_J];
#pragma unroll
        for (int j = 0; j < (int)BK_J; j++) {
            const uint32_t p = ws + j * BK_T + tid;
            k[j] = p < cnt ? key[p] : BK_EMPTY;
        }
        for (uint32_t i = tid; i < BK_TS / 4; i += BK_T)
            reinterpret_cast<uint4*>(S.tab)[i] = make_uint4(BK_EMPTY, BK_EMPTY, BK_EMPTY, BK_EMPTY);
        for (uint32_t i = tid; i < BK_TS / 8; i += BK_T) reinterpret_cast<uint4*>(S.cnt)[i] = make_uint4(0, 0, 0, 0);
        if (tid == 0) {
            S.first = ~0u;
            S.lastp1 = 0;
            S.end = ~0u;
        }
        // ... starts a bucket when its key's low bits differ from the previous item's:
        // the first and last bucket starts in the chunk, and the first one after it
        // (each warp's last lane hands its keys to the next warp's first lane)
        const uint32_t chunk_q = cend > ws ? cend - ws : 0u;
        if (lane == 31)
#pragma unroll
            for (int j = 0; j < (int)BK_J; j++) S.hand[j * (BK_T / 32) + warp] = k[j];
        if (tid == 0) S.hand[BK_J * (BK_T / 32)] = ws > 0 ? key[ws - 1] : 0u;
        __syncthreads();
        uint32_t f = ~0u, l = 0, e = ~0u;
#pragma unroll
        for (int j = 0; j < (int)BK_J; j++) {
            const uint32_t q = j * BK_T + tid;
            const uint32_t p = ws + q;
            uint32_t prev = __shfl_up_sync(0xFFFFFFFFu, k[j], 1);
            if (lane == 0)
                prev = S.hand[warp > 0 ? j * (BK_T / 32) + warp - 1 : j > 0 ? j * (BK_T / 32) - 1 : BK_J * (BK_T / 32)];
            if (p < cnt && (p == 0 || ((k[j] ^ prev) & mask) != 0)) {
                if (q < chunk_q) {
                    f = min(f, q);
                    l = max(l, q + 1);
                } else {
                    e = min(e, q);
                }
            }
        }
        f = __reduce_min_sync(0xFFFFFFFFu, f);
        l = __reduce_max_sync(0xFFFFFFFFu, l);
        e = __reduce_min_sync(0xFFFFFFFFu, e);
        if (lane == 0) {
            if (f != ~0u) atomicMin(&S.first, f);
            if (l) atomicMax(&S.lastp1, l);
            if (e != ~0u) atomicMin(&S.end, e);
        }
        __syncthreads();
        const uint32_t s = S.first, last = S.lastp1 - 1u;
        uint32_t end = S.end;
        if (ws + BK_W >= cnt) end = min(end, cnt - ws);
        if (s == ~0u) return;  // no bucket starts in this block's chunk
        // the buckets done in this window: [lo, hi)
        uint32_t lo = s, hi = s;
        bool again = false;
        if (end != ~0u) {
            hi = end;
        } else if (last > s) {
            hi = last;  // the last one runs past the window: a window of its own
            again = true;
        } else if (s > 0) {
            again = true;  // the only one runs past the window: a window of its own
        } else {
            // a bucket longer than a window: all of it to the general path
            const uint32_t bv = key[ws] & mask;
            uint32_t mine = 0;
            for (uint32_t p = ws + tid;; p += BK_T) {
                const bool in = p < cnt && (key[p] & mask) == bv;
                if (!__syncthreads_or(in)) break;
                if (in) {
                    const uint32_t x = val[p];
                    atomicOr(&ofl[x >> 5], 1u << (x & 31));
                    mine++;
                }
            }
            mine = __reduce_add_sync(0xFFFFFFFFu, mine);
            if (lane == 0 && mine) atomicAdd(&counts[1], mine);
            return;
        }
        bk_table<BK_T, BK_J, BK_TS_BITS, false>(S, k, lo, hi, val + ws, list, ofl, counts);
        if (!again) return;
        __syncthreads();  // (dl and the table are free again)
        ws += hi > s ? hi : s;
    }
}

// One partition a block: all edges of each of its pairs.  Most pairs have one edge; a
// bitmap over slots of the hash (seen, and rep: seen again) finds the items that share
// their slot (about an eighth by chance, at 8 slots an item, and the groups), and only
// these go through the table, GP_CAP of them at a time: when there are more, those
// of one residue of the hash at a time, each a pass over the partition (from L2).  A
// residue with more than GP_CAP is left to the general path.
// Two blocks of 512 threads an SM; one of 1024 with bitmaps, table and lists twice as
// large where a partition has more than 32768 items (scale 21, 31K items: 763 and 800 us
// over all; scale 22, 62K items: 2150 and 1424).  R-MAT scale 21: 154 us, of which both
// passes over the items 120 (a bitmap in L2 instead, by atomics of the keys' kernel, cost
// it 240 us: 130 G atomics/s).
// counts[4]: a partition outgrew its room, and the list is sorted instead.
constexpr uint32_t GP_J = 12;
template <int B>  // 512 << B threads
struct GpSmem {
    static constexpr uint32_t GP_T = 512u << B, GP_CAP = GP_T * GP_J, GP_TSB = 13 + B, GP_BITS = 18 + B;
    uint32_t rep[1u << (GP_BITS - 5)];
    union {
        uint32_t seen[1u << (GP_BITS - 5)];
        uint32_t keyl[GP_CAP];
        uint32_t tab[1u << GP_TSB];
        uint32_t dl[GP_CAP];
    };
    uint32_t cnt[1u << (GP_TSB - 1)];
    uint32_t vall[GP_CAP];
    uint32_t dupb[(1u << GP_TSB) / 32], longb[(1u << GP_TSB) / 32];
    uint32_t wsum[GP_T / 32];
    uint32_t ndup, nmid, nc;
};

template <int B>
__global__ void __launch_bounds__(512 << B, 2 >> B)
    k_c_groups(const uint2* __restrict__ items, const uint32_t* __restrict__ gcur, uint32_t cap, uint32_t pb,
               uint32_t gb, uint32_t* __restrict__ list, uint32_t* __restrict__ ofl, uint32_t* __restrict__ counts) {
    using SM = GpSmem<B>;
    constexpr uint32_t GP_T = SM::GP_T, GP_CAP = SM::GP_CAP, GP_TSB = SM::GP_TSB;
    extern __shared__ __align__(16) unsigned char gp_raw[];
    SM& S = *reinterpret_cast<SM*>(gp_raw);
    const uint32_t tid = threadIdx.x, lane = tid & 31;
    // (few pairs with many edges each, 4M edges among 64 vertices: all blocks' work for
    // nothing took 1.1 ms before the sort's 2.4)
    if (counts[4]) return;
    const uint32_t total = gcur[blockIdx.x];
    const uint2* it = items + (size_t)blockIdx.x * cap;
    for (uint32_t i = tid; i < 1u << (gb - 5); i += GP_T) S.seen[i] = S.rep[i] = 0;
    __syncthreads();
    const uint32_t gsh = 32 - gb;  // a slot: the gb bits of the key below the partition's
    for (uint32_t i0 = tid; i0 < total; i0 += 8 * GP_T) {
        uint32_t k[8];
#pragma unroll
        for (int q = 0; q < 8; q++) k[q] = i0 + q * GP_T < total ? it[i0 + q * GP_T].x : 0u;
#pragma unroll
        for (int q = 0; q < 8; q++) {
            const uint32_t s = (k[q] << pb) >> gsh, bit = 1u << (s & 31);
            if (i0 + q * GP_T < total && (atomicOr(&S.seen[s >> 5], bit) & bit)) atomicOr(&S.rep[s >> 5], bit);
        }
    }
    __syncthreads();
    uint32_t rounds = 1;  // residues (a power of two)
    for (uint32_t r = 0; r < rounds;) {
        if (tid == 0) S.nc = 0;
        __syncthreads();
        for (uint32_t i0 = tid; i0 - tid < total; i0 += 8 * GP_T) {  // (whole warps)
            uint2 v[8];
#pragma unroll
            for (int q = 0; q < 8; q++) v[q] = i0 + q * GP_T < total ? it[i0 + q * GP_T] : make_uint2(0, 0);
#pragma unroll
            for (int q = 0; q < 8; q++) {
                const uint32_t s = (v[q].x << pb) >> gsh;
                const bool in = i0 + q * GP_T < total && (v[q].x & (rounds - 1)) == r && ((S.rep[s >> 5] >> (s & 31)) & 1u);
                const uint32_t b = __ballot_sync(0xFFFFFFFFu, in);
                uint32_t p = 0;
                if (b && lane == 0) p = atomicAdd(&S.nc, __popc(b));
                p = __shfl_sync(0xFFFFFFFFu, p, 0) + __popc(b & ((1u << lane) - 1u));
                if (in && p < GP_CAP) {
                    S.keyl[p] = v[q].x;
                    S.vall[p] = v[q].y;
                }
            }
        }
        __syncthreads();
        const uint32_t nc = S.nc;
        if (nc > GP_CAP) {
            if (rounds == 1) {  // from the start, by residues that leave a margin
                while (rounds < 4096 && nc > (rounds * GP_CAP) / 8 * 7) rounds *= 2;
                __syncthreads();
                continue;
            }
            for (uint32_t i = tid; i < total; i += GP_T) {
                const uint2 v = it[i];
                const uint32_t s = (v.x << pb) >> gsh;
                if ((v.x & (rounds - 1)) == r && ((S.rep[s >> 5] >> (s & 31)) & 1u))
                    atomicOr(&ofl[v.y >> 5], 1u << (v.y & 31));
            }
            if (tid == 0) atomicAdd(&counts[1], nc);
        } else if (nc > 1) {
            uint32_t k[GP_J];
#pragma unroll
            for (int j = 0; j < (int)GP_J; j++) k[j] = j * GP_T + tid < nc ? S.keyl[j * GP_T + tid] : BK_EMPTY;
            __syncthreads();
            for (uint32_t i = tid; i < (1u << GP_TSB) / 4; i += GP_T)
                reinterpret_cast<uint4*>(S.tab)[i] = make_uint4(BK_EMPTY, BK_EMPTY, BK_EMPTY, BK_EMPTY);
            for (uint32_t i = tid; i < (1u << GP_TSB) / 8; i += GP_T)
                reinterpret_cast<uint4*>(S.cnt)[i] = make_uint4(0, 0, 0, 0);
            __syncthreads();
            bk_table<GP_T, GP_J, GP_TSB, true>(S, k, 0, nc, S.vall, list, ofl, counts);
        }
        __syncthreads();  // (the lists are free again)
        r++;
    }
}

// The general path: the flagged edges, a tile of 4096 per block, thread t holding
// chunks c = 0..3 of four edges at tile offset 1024 c + 4 t.  One launch counts
// them per tile; after a scan of the counts the second takes them out in order.
constexpr uint32_t RN_TILE = 4096;

// bit j: edge i + j is flagged (i a multiple of 4)
__device__ __forceinline__ uint32_t run_bits(const uint32_t* __restrict__ ofl, uint64_t i, uint32_t cnt) {
    return i < cnt ? (ofl[i >> 5] >> (i & 31)) & 0xFu : 0u;
}

__global__ void __launch_bounds__(CT) k_c_runs_count(const uint32_t* __restrict__ ofl, uint32_t cnt,
                                                     uint32_t* __restrict__ tcount) {
    __shared__ uint32_t ws[CT / 32];
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint64_t base = (uint64_t)blockIdx.x * RN_TILE + 4 * threadIdx.x;
    uint32_t x = 0;
#pragma unroll
    for (int c = 0; c < 4; c++) x += __popc(run_bits(ofl, base + 1024 * c, cnt));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xFFFFFFFFu, x, o);
    if (lane == 0) ws[warp] = x;
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t t = 0;
        for (int w = 0; w < (int)(CT / 32); w++) t += ws[w];
        tcount[blockIdx.x] = t;
    }
}

// the flagged edges in input order, with
// (min, max) of their coarse pair as the key of a second sort; counts[3] = how many.
// The tile's run items are listed in shared memory first, so that the gathers of
// their pairs spread over all threads.
__global__ void __launch_bounds__(CT) k_c_runs_take(const uint32_t* __restrict__ ofl, uint32_t cnt,
                                                    const uint32_t* __restrict__ toffs,
                                                    const uint32_t* __restrict__ cpair, uint32_t bits,
                                                    unsigned long long* __restrict__ skey,
                                                    uint32_t* __restrict__ sval, uint32_t* __restrict__ counts) {
    __shared__ uint32_t ws[4][CT / 32];
    __shared__ uint32_t list[RN_TILE];
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint64_t tile0 = (uint64_t)blockIdx.x * RN_TILE;
    const uint64_t base = tile0 + 4 * threadIdx.x;
    uint32_t f[4], incl[4];
#pragma unroll
    for (int c = 0; c < 4; c++) {
        f[c] = run_bits(ofl, base + 1024 * c, cnt);
        uint32_t x = __popc(f[c]);
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, o);
            if (lane >= (uint32_t)o) x += y;
        }
        incl[c] = x;
        if (lane == 31) ws[c][warp] = x;
    }
    __syncthreads();
    uint32_t run = 0;
#pragma unroll
    for (int c = 0; c < 4; c++) {
        uint32_t before = 0, total = 0;
        for (uint32_t w = 0; w < CT / 32; w++) {
            before += w < warp ? ws[c][w] : 0u;
            total += ws[c][w];
        }
        uint32_t q = run + before + incl[c] - __popc(f[c]);
        for (uint32_t bl = f[c]; bl; bl &= bl - 1) list[q++] = 1024 * c + 4 * threadIdx.x + __ffs(bl) - 1;
        run += total;
    }
    __syncthreads();
    const uint32_t off = toffs[blockIdx.x];
    for (uint32_t q = threadIdx.x; q < run; q += CT) {
        const uint32_t e = (uint32_t)tile0 + list[q];
        const uint2 cp = *reinterpret_cast<const uint2*>(cpair + 2 * (size_t)e);
        const uint32_t x = cp.x, y = cp.y;
        skey[off + q] = ((unsigned long long)min(x, y) << bits) | max(x, y);  // coarse ids take `bits` bits
        sval[off + q] = e;
    }
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) counts[3] = off + run;
}

// ---- stable LSD radix sort of (key, value) pairs, 8 bits per pass ----------
// A pass is three launches.  The first counts each tile's digits; an exclusive
// scan over (digit, tile) then gives every tile the output position of its first
// item of each digit; the third ranks each tile's items stably (warp by warp, 32
// items at a time in input order: lanes with the same digit from one ballot per
// digit bit, earlier rounds and warps by shared counters), puts the tile in digit
// order in shared memory and writes it out.  No block waits on another.
constexpr uint32_t RS_T = 256, RS_I = 16, RS_TILE = RS_T * RS_I, RS_W = RS_T / 32;

template <class K>
struct RsSmem {
    uint32_t wcnt[RS_W][256];  // items of each digit seen so far by each warp, then where the warp's start
    uint32_t gofs[256];        // output position of the tile's first item of each digit, minus its tile start
    uint32_t wsum[RS_W];
    K sk[RS_TILE];
    uint32_t sv[RS_TILE];
};

// digit counts of every tile, digit-major (hist[d * tiles + t]) for the scan
template <class K>
__global__ void __launch_bounds__(RS_T) k_rs_hist(const K* __restrict__ key, uint32_t cnt, uint32_t shift,
                                                  uint32_t tiles, uint32_t* __restrict__ hist) {
    __shared__ uint32_t h[RS_W][256];
    for (uint32_t i = threadIdx.x; i < RS_W * 256; i += RS_T) (&h[0][0])[i] = 0;
    __syncthreads();
    const uint32_t warp = threadIdx.x >> 5;
    const uint32_t base = blockIdx.x * RS_TILE + threadIdx.x;
    K k[RS_I];
#pragma unroll
    for (int j = 0; j < (int)RS_I; j++) {
        const uint32_t q = base + j * RS_T;
        k[j] = q < cnt ? key[q] : (K)0;
    }
#pragma unroll
    for (int j = 0; j < (int)RS_I; j++)
        if (base + j * RS_T < cnt) atomicAdd(&h[warp][(uint32_t)(k[j] >> shift) & 0xFFu], 1u);
    __syncthreads();
    uint32_t x = 0;
#pragma unroll
    for (int w = 0; w < (int)RS_W; w++) x += h[w][threadIdx.x];
    hist[threadIdx.x * tiles + blockIdx.x] = x;
}

// val_in NULL: the values are the items' indices
template <class K>
__global__ void __launch_bounds__(RS_T, sizeof(K) == 4 ? 3 : 2)
    k_rs_scatter(const K* __restrict__ key_in, const uint32_t* __restrict__ val_in, uint32_t cnt, uint32_t shift,
                 uint32_t tiles, const uint32_t* __restrict__ offs, K* __restrict__ key_out,
                 uint32_t* __restrict__ val_out) {
    extern __shared__ __align__(16) unsigned char rs_raw[];
    RsSmem<K>& S = *reinterpret_cast<RsSmem<K>*>(rs_raw);
    auto& wcnt = S.wcnt;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t lt = (1u << lane) - 1u;
    const uint32_t tile = blockIdx.x, dg = threadIdx.x;  // (one digit per thread below)
    const uint32_t gstart = offs[dg * tiles + tile];
    for (uint32_t i = threadIdx.x; i < RS_W * 256; i += RS_T) (&wcnt[0][0])[i] = 0;
    // warp w owns items [w * 32 RS_I, (w + 1) * 32 RS_I) of the tile, 32 per round in order
    const uint32_t tile0 = tile * RS_TILE;
    const uint32_t base = tile0 + warp * 32 * RS_I;
    const uint32_t nin = cnt > tile0 ? min(RS_TILE, cnt - tile0) : 0u;
    K k[RS_I];
    uint32_t v[RS_I], r[RS_I];
#pragma unroll
    for (int j = 0; j < (int)RS_I; j++) {
        const uint32_t q = base + j * 32 + lane;
        const bool ok = q < cnt;
        k[j] = ok ? key_in[q] : (K)0;
        v[j] = ok ? (val_in ? val_in[q] : q) : 0u;  // no values: each item's own index
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < (int)RS_I; j++) {
        const bool ok = base + j * 32 + lane < cnt;
        const uint32_t d = (uint32_t)(k[j] >> shift) & 0xFFu;
        // the lanes holding the same digit, from one ballot per digit bit (lanes past
        // the end match nobody)
        uint32_t peers = __ballot_sync(0xFFFFFFFFu, ok);
#pragma unroll
        for (int b = 0; b < 8; b++) {
            const uint32_t bal = __ballot_sync(0xFFFFFFFFu, (d >> b) & 1u);
            peers &= ((d >> b) & 1u) ? bal : ~bal;
        }
        // the whole warp reads, then each digit's last lane writes: no branch splits
        // the warp by digit
        const uint32_t before = ok ? wcnt[warp][d] : 0u;
        r[j] = before + __popc(peers & lt);
        __syncwarp();
        if (ok && (peers >> lane) == 1u) wcnt[warp][d] = before + __popc(peers);
        __syncwarp();
    }
    __syncthreads();
    {
        uint32_t run = 0;
        for (int w = 0; w < (int)RS_W; w++) run += wcnt[w][dg];
        // exclusive scan of the 256 digit totals across the tile
        uint32_t x = run;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) S.wsum[warp] = x;
        __syncthreads();
        uint32_t before = 0;
        for (int w = 0; w < warp; w++) before += S.wsum[w];
        const uint32_t dst = before + x - run;
        uint32_t acc = dst;
        for (int w = 0; w < (int)RS_W; w++) {
            const uint32_t c = wcnt[w][dg];
            wcnt[w][dg] = acc;
            acc += c;
        }
        S.gofs[dg] = gstart - dst;
    }
    __syncthreads();
    // the tile in digit order in shared memory ...
#pragma unroll
    for (int j = 0; j < (int)RS_I; j++) {
        if (base + j * 32 + lane >= cnt) continue;
        const uint32_t p = wcnt[warp][(uint32_t)(k[j] >> shift) & 0xFFu] + r[j];
        S.sk[p] = k[j];
        S.sv[p] = v[j];
    }
    __syncthreads();
    // ... then written out: consecutive threads take consecutive items, which within
    // a digit land on consecutive addresses
    for (uint32_t p = threadIdx.x; p < nin; p += RS_T) {
        const K kk = S.sk[p];
        const uint32_t o = S.gofs[(uint32_t)(kk >> shift) & 0xFFu] + p;
        if (o < cnt) {
            key_out[o] = kk;
            val_out[o] = S.sv[p];
        }
    }
}

// groups in pair order (runs of equal keys; a run's first item is its leader, the
// smallest edge index, since the sort is stable and a pair's edges entered in
// input order).  Every other member loses its bit in cross; the leader of a
// group of several edges gets a bit in multi and, in gsum, the float32 bits of
// the group's weight: the sum in double over its edges in input order, rounded once.
__global__ void k_c_marks(const unsigned long long* __restrict__ key, const uint32_t* __restrict__ val, uint32_t cnt,
                          const float* __restrict__ w, uint32_t* __restrict__ cross, uint32_t* __restrict__ multi,
                          uint32_t* __restrict__ gsum) {
    for (uint32_t i = blockIdx.x * CT + threadIdx.x; i < cnt; i += gridDim.x * CT) {
        const unsigned long long k = key[i];
        const uint32_t e = val[i];
        if (i > 0 && k == key[i - 1]) {
            atomicAnd(&cross[e >> 5], ~(1u << (e & 31)));
        } else if (i + 1 < cnt && key[i + 1] == k) {
            double sum = (double)w[e];
            uint32_t j = i + 1;
            // members four at a time: their loads issue together, the additions stay in order
            for (bool more = true; more;) {
                uint32_t vj[4];
                bool in[4];
#pragma unroll
                for (int t = 0; t < 4; t++) {
                    in[t] = j + t < cnt && key[j + t] == k;
                    vj[t] = in[t] ? val[j + t] : 0u;
                }
                float wj[4];
#pragma unroll
                for (int t = 0; t < 4; t++) wj[t] = in[t] ? w[vj[t]] : 0.0f;
#pragma unroll
                for (int t = 0; t < 4; t++)
                    if (in[t]) sum += (double)wj[t];
                more = in[3];
                j += 4;
            }
            atomicOr(&multi[e >> 5], 1u << (e & 31));
            gsum[e] = __float_as_uint((float)sum);
        }
    }
}

// leaders per word of cross (wlead[words] = 0, so that the scan's last entry is the total)
__global__ void k_c_wcount(const uint32_t* __restrict__ cross, uint32_t words, uint32_t* __restrict__ wlead) {
    for (uint32_t i = blockIdx.x * CT + threadIdx.x; i <= words; i += gridDim.x * CT)
        wlead[i] = i < words ? __popc(cross[i]) : 0u;
}

// the leaders, in input order, write their coarse edge at their rank among the
// leaders, with their group's weight (a single edge's own weight, which double and
// back leaves unchanged)
template <bool VEC>
__global__ void __launch_bounds__(CT) k_c_emit(uint32_t m, const uint32_t* __restrict__ cpair,
                                               const float* __restrict__ w, const uint32_t* __restrict__ cross,
                                               const uint32_t* __restrict__ wpos, const uint32_t* __restrict__ multi,
                                               const uint32_t* __restrict__ gsum, uint32_t* __restrict__ ceu,
                                               uint32_t* __restrict__ cev, float* __restrict__ cw) {
    // a block takes 1024 edges (32 words of cross) at a time; their leaders fill one
    // run of the output, staged here and written out contiguously
    __shared__ uint32_t su[4 * CT], sv2[4 * CT], sw[4 * CT];
    const uint32_t groups = (uint32_t)(((uint64_t)m + 3) / 4);
    const uint32_t words = (uint32_t)(((uint64_t)m + 31) / 32);
    const uint32_t* wb = reinterpret_cast<const uint32_t*>(w);
    for (uint32_t c0 = blockIdx.x * CT; c0 < groups; c0 += gridDim.x * CT) {
        const uint32_t g = c0 + threadIdx.x;
        const uint32_t w0 = c0 >> 3, w1 = min(w0 + CT / 8, words);
        const uint32_t obase = wpos[w0], ocount = wpos[w1] - obase;
        if (g < groups) {
            const uint64_t e0 = 4ull * g;
            // every load of the group at once (most edges lead); cpair is aligned scratch
            const uint32_t word = cross[g >> 3], wp = wpos[g >> 3], mw = __ldg(&multi[g >> 3]);
            const uint4 x = load4<VEC>(wb, e0, m);
            const uint4 p0 = load4<true>(cpair, 2 * e0, 2 * m), p1 = load4<true>(cpair, 2 * e0 + 4, 2 * m);
            const uint32_t sh = 4 * (g & 7);
            const uint32_t nib = (word >> sh) & 0xFu, mb = (mw >> sh) & 0xFu;
            uint32_t p = wp - obase + __popc(word & ((1u << sh) - 1u));
            const uint32_t cu[4] = {p0.x, p0.z, p1.x, p1.z}, cv[4] = {p0.y, p0.w, p1.y, p1.w};
#pragma unroll
            for (int j = 0; j < 4; j++) {
                if (!((nib >> j) & 1u)) continue;
                su[p] = cu[j];
                sv2[p] = cv[j];
                sw[p] = ((mb >> j) & 1u) ? gsum[(uint32_t)e0 + j] : at(x, j);
                p++;
            }
        }
        __syncthreads();
        for (uint32_t i = threadIdx.x; i < ocount; i += CT) {
            ceu[obase + i] = su[i];
            cev[obase + i] = sv2[i];
            cw[obase + i] = __uint_as_float(sw[i]);
        }
        __syncthreads();
    }
}

// What the host waits for, written to its memory: counts[0 .. 4], the coarse vertices, the
// error bits, the coarse edges (0 without edges).  One launch instead of a copy each.
__global__ void k_c_report(const uint32_t* __restrict__ counts, const uint32_t* __restrict__ nc,
                           const uint32_t* __restrict__ err, const uint32_t* __restrict__ mc,
                           volatile uint32_t* host) {
    for (int i = 0; i < 5; i++) host[i] = counts[i];
    host[5] = *nc;
    host[6] = *err;
    host[7] = mc ? *mc : 0u;
}

uint32_t bits_for(uint32_t x) {  // bits to write 0 .. x
    uint32_t b = 1;
    while (b < 32 && (x >> b)) b++;
    return b;
}

}  // namespace

// log2 of the partitions, or 0: the list is sorted by the hash.  About 8192 edges to a
// partition up to 1024 partitions, which are written in runs of 8 items; then as many as
// a bitmap of 8 slots an item allows (R-MAT scale 22, 64M edges: 1.42 ms with 1024, 1.54
// with 2048), and from there up to 4096 (scale 23, 129M: 4.34 ms with 1024, 3.19 with
// 2048; 300M: 10.5 with 2048, 8.4 with 4096).  Partitions beat the sort from the
// smallest lists (fewer launches: 1,000 edges 99 us against 122, 1M edges 142 against
// 210) to the largest measured (590M edges 23.8 ms against 29.4), with a gain that shrinks
// as the slots are shared; so the line lies at 2^30 edges.  A caller that sets the
// sort's width gets the sort.
static uint32_t contract_part_bits(uint32_t m, uint32_t sort_bits) {
    if (sort_bits || m > 1u << 30) return 0;
    uint32_t b = 1;
    while (b < 10 && (m >> b) > 8192) b++;
    while (b < 12 && (m >> b) > 1u << (GpSmem<1>::GP_BITS - 3)) b++;
    return b;
}

size_t contract_sort_words(uint32_t m) {
    const uint64_t tiles = ((uint64_t)m + RS_TILE - 1) / RS_TILE;
    return (size_t)(2 * (256 * tiles + 4));
}

int launch_contract(void* stream, const ContractArgs& c, uint32_t* host) {
    cudaStream_t s = (cudaStream_t)stream;
    cudaError_t e;
    if ((e = cudaMemsetAsync(c.err, 0, sizeof(uint32_t), s))) return (int)e;
    if ((e = cudaMemsetAsync(c.flag + c.n, 0, sizeof(uint32_t), s))) return (int)e;
    if ((e = cudaMemsetAsync(c.cvw, 0, (size_t)c.n * sizeof(uint32_t), s))) return (int)e;
    k_c_rep<<<grid_for(c.n), CT, 0, s>>>(c.mate, c.n, c.flag, c.err);
    if (int r = launch_exclusive_scan(s, c.flag, c.rank, c.n + 1, c.scan_tmp, c.scan_words)) return r;
    k_c_map<<<grid_for(c.n), CT, 0, s>>>(c.mate, c.n, c.rank, c.vw, c.cmap, c.cvw);
    const uint32_t words = (uint32_t)(((uint64_t)c.m + 31) / 32);
    auto report = [&](bool last) -> int {
        k_c_report<<<1, 1, 0, s>>>(c.counts, c.rank + c.n, c.err, last && c.m ? c.wpos + words : nullptr, host);
        return (int)cudaGetLastError();
    };
    if (c.m == 0) return report(true);
    if ((e = cudaFuncSetAttribute(k_rs_scatter<uint32_t>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)sizeof(RsSmem<uint32_t>)))) return (int)e;
    if ((e = cudaFuncSetAttribute(k_rs_scatter<unsigned long long>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)sizeof(RsSmem<unsigned long long>)))) return (int)e;
    // stable sort by the low `bits` bits of the keys (8-bit digits), ping-ponging
    // between the two buffers; *cur tells which holds the result
    // (ident: the values are the items' indices, and v0 is not read)
    // (counted0: the first pass's per-tile digit counts are in place already)
    auto radix = [&](auto* k0, auto* k1, uint32_t* v0, uint32_t* v1, uint32_t cnt, uint32_t bits, bool ident,
                     bool counted0, int* cur) -> int {
        using K = typename std::remove_pointer<decltype(k0)>::type;
        K* kk[2] = {k0, k1};
        uint32_t* vv[2] = {v0, v1};
        *cur = 0;
        if (cnt < 2) return 0;
        const uint32_t tiles = (cnt + RS_TILE - 1) / RS_TILE;
        uint32_t* hist = c.shist;
        uint32_t* offs = c.shist + ((256 * (size_t)tiles + 4) & ~(size_t)3);
        for (uint32_t p = 0; p * 8 < bits; p++) {
            if (!(counted0 && p == 0)) k_rs_hist<K><<<tiles, RS_T, 0, s>>>(kk[*cur], cnt, 8 * p, tiles, hist);
            if (int r = launch_exclusive_scan(s, hist, offs, 256 * tiles, c.scan_tmp, c.scan_words)) return r;
            const uint32_t* vin = (ident && p == 0) ? nullptr : vv[*cur];
            k_rs_scatter<K><<<tiles, RS_T, sizeof(RsSmem<K>), s>>>(kk[*cur], vin, cnt, 8 * p, tiles, offs,
                                                                   kk[*cur ^ 1], vv[*cur ^ 1]);
            *cur ^= 1;
        }
        return (int)cudaGetLastError();
    };
    uint32_t* hk[2] = {reinterpret_cast<uint32_t*>(c.key[0]), reinterpret_cast<uint32_t*>(c.key[1])};
    const uint32_t egrid = grid_for(((uint64_t)c.m + 3) / 4);
    const bool vec = ((reinterpret_cast<uintptr_t>(c.eu) | reinterpret_cast<uintptr_t>(c.ev) |
                       reinterpret_cast<uintptr_t>(c.w)) & 15u) == 0;
    uint32_t* ofl = c.wlead;  // (free until the leaders are counted)
    const size_t bitmap = ((size_t)c.m / 32 + 2) * sizeof(uint32_t);
    uint32_t mc = 0, nc = 0;  // crossing edges, coarse vertices
    bool done = false;
    // counts to the host: crossing edges, coarse vertices, edges left to the general path, a
    // partition outgrew its room
    auto read_counts = [&]() -> int {
        if (int r = report(false)) return r;
        if (cudaError_t x = cudaStreamSynchronize(s)) return (int)x;
        mc = host[0];
        nc = host[5];
        return 0;
    };
    // 1. partitions, where their rule holds: the crossing bits become the leader bits, every
    //    group member but the first cleared
    if (const uint32_t pb = contract_part_bits(c.m, c.sort_bits)) {
        // twice the average (key[0] and key[1], which follows it), less what makes the rooms' distance
        // an odd number of cache lines (R-MAT scale 22 1.42 and 1.40 ms)
        uint32_t cap = (uint32_t)(2ull * c.m >> pb);
        if (cap > 4096) cap = (((cap >> 4) - 1) | 1u) << 4;
        uint32_t gb = 10;
        while (gb < GpSmem<1>::GP_BITS && (1ull << gb) < (8ull * c.m >> pb)) gb++;
        uint2* items = reinterpret_cast<uint2*>(c.key[0]);
        const int d = pb > 10 ? pb - 9 : 1;   // (log2 of) partitions a thread
        auto part = d == 1 ? (vec ? k_c_part<true, 2> : k_c_part<false, 2>)
                  : d == 2 ? (vec ? k_c_part<true, 4> : k_c_part<false, 4>)
                           : (vec ? k_c_part<true, 8> : k_c_part<false, 8>);
        const size_t psmem = d == 1 ? sizeof(PtSmem<2>) : d == 2 ? sizeof(PtSmem<4>) : sizeof(PtSmem<8>);
        const int big = gb > GpSmem<0>::GP_BITS;
        auto groups = big ? k_c_groups<1> : k_c_groups<0>;
        const size_t gsmem = big ? sizeof(GpSmem<1>) : sizeof(GpSmem<0>);
        if ((e = cudaFuncSetAttribute(part, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)psmem)) ||
            (e = cudaFuncSetAttribute(groups, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)gsmem)) ||
            (e = cudaMemsetAsync(c.counts, 0, 8 * sizeof(uint32_t), s)) ||
            (e = cudaMemsetAsync(c.shist, 0, sizeof(uint32_t) << pb, s)) ||
            (e = cudaMemsetAsync(c.multi, 0, bitmap, s)) || (e = cudaMemsetAsync(ofl, 0, bitmap, s)))
            return (int)e;
        part<<<(uint32_t)(((uint64_t)c.m + PT_TILE - 1) / PT_TILE), PT_T, psmem, s>>>(
            c.eu, c.ev, c.m, c.n, c.cmap, pb, cap, c.shist, items, c.cpair, c.cross, c.counts, c.err);
        groups<<<1u << pb, 512u << big, gsmem, s>>>(items, c.shist, cap, pb, gb, c.val[0], ofl, c.counts);
        k_c_walk<<<egrid, CT, 0, s>>>(c.val[0], c.cpair, c.w, c.cross, c.multi, c.gref, ofl, c.counts);
        if (int r = read_counts()) return r;
        done = host[4] == 0;
    }
    // or every edge keyed by its pair's hash in input order; the stable sort keeps input
    // order among equal keys and puts the edges inside pairs last, after the mc crossing
    // edges; then the buckets
    if (!done) {
        if ((e = cudaMemsetAsync(c.counts, 0, 8 * sizeof(uint32_t), s))) return (int)e;
        static_assert(RS_TILE == 4096 && CT == 256, "k_c_keys takes one tile of the sort per block");
        const uint32_t kgrid = (uint32_t)(((uint64_t)c.m + RS_TILE - 1) / RS_TILE);  // the sort's tiles
        auto keys = vec ? k_c_keys<true> : k_c_keys<false>;
        keys<<<kgrid, CT, 0, s>>>(c.eu, c.ev, c.m, c.n, c.cmap, hk[0], c.cpair, c.cross, c.counts, c.shist, c.err);
        if (int r = read_counts()) return r;
        host[1] = 0;
        // the sort's bits: as few bytes as leave at most BK_AVG crossing edges to a bucket
        uint32_t sbits = c.sort_bits;
        if (!sbits)
            for (sbits = 8; sbits < 32 && (uint64_t)mc > ((uint64_t)BK_AVG << sbits); sbits += 8) {
            }
        const uint32_t mask = sbits >= 32 ? ~0u : (1u << sbits) - 1u;
        int hc = 0;
        if ((e = cudaMemsetAsync(c.multi, 0, bitmap, s))) return (int)e;
        if (mc > 1) {
            if (int r = radix(hk[0], hk[1], c.val[0], c.val[1], c.m, sbits, true, true, &hc)) return r;
            if ((e = cudaMemsetAsync(ofl, 0, bitmap, s)) ||
                (e = cudaFuncSetAttribute(k_c_buckets, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(BkSmem))) ||
                (e = cudaFuncSetAttribute(k_c_buckets, cudaFuncAttributePreferredSharedMemoryCarveout,
                                          (int)cudaSharedmemCarveoutMaxShared)))
                return (int)e;
            k_c_buckets<<<(mc + BK_C - 1) / BK_C, BK_T, sizeof(BkSmem), s>>>(hk[hc], c.val[hc], mc, mask, c.val[hc ^ 1], ofl,
                                                                           c.counts);
            k_c_walk<<<egrid, CT, 0, s>>>(c.val[hc ^ 1], c.cpair, c.w, c.cross, c.multi, c.gref, ofl, c.counts);
            if (int r = read_counts()) return r;
        }
    }
    // 2. the flagged edges are taken out in order with their pair as the key, sorted by the
    //    pair and marked
    if (host[1]) {
        const uint32_t bits = bits_for(nc ? nc - 1 : 0);
        const uint32_t tiles = (c.m + RN_TILE - 1) / RN_TILE;
        uint32_t* toffs = c.tsum + ((size_t)c.m / RN_TILE + 2);
        k_c_runs_count<<<tiles, CT, 0, s>>>(ofl, c.m, c.tsum);
        if (int r = launch_exclusive_scan(s, c.tsum, toffs, tiles, c.scan_tmp, c.scan_words)) return r;
        k_c_runs_take<<<tiles, CT, 0, s>>>(ofl, c.m, toffs, c.cpair, bits, c.key[0], c.val[0], c.counts);
        if (int r = read_counts()) return r;
        const uint32_t nsub = host[3];
        int cur = 0;
        if (nsub) {
            if (int r = radix(c.key[0], c.key[1], c.val[0], c.val[1], nsub, 2 * bits, false, false, &cur)) return r;
            k_c_marks<<<grid_for(nsub), CT, 0, s>>>(c.key[cur], c.val[cur], nsub, c.w, c.cross, c.multi, c.gref);
        }
    }
    // 3. leaders ranked by words of the bitmask; the leaders write the coarse edges
    k_c_wcount<<<grid_for((uint64_t)words + 1), CT, 0, s>>>(c.cross, words, c.wlead);
    if (int r = launch_exclusive_scan(s, c.wlead, c.wpos, words + 1, c.scan_tmp, c.scan_words)) return r;
    if (mc) {
        if (vec)
            k_c_emit<true><<<egrid, CT, 0, s>>>(c.m, c.cpair, c.w, c.cross, c.wpos, c.multi, c.gref, c.ceu, c.cev,
                                                c.cw);
        else
            k_c_emit<false><<<egrid, CT, 0, s>>>(c.m, c.cpair, c.w, c.cross, c.wpos, c.multi, c.gref, c.ceu, c.cev,
                                                 c.cw);
    }
    return report(true);
}

}  // namespace lm
