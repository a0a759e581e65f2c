// lm_match_small_noalloc: local max for one small graph whose edge list is already on
// the device, in one launch of one thread-block cluster and without allocation.
//
// Edge-centric rounds (the Combining CRCW formulation of Sec. 2): every live edge
// offers its key to both ends with an atomic maximum, an edge that is the best offer
// at both is matched, edges with a matched end leave.  The offers live in the cluster's
// shared memory (vertex x: slot x / C of block x % C) and a barrier of the cluster
// ends a phase.  They are 32-bit, which shared memory takes in one operation (a 64-bit
// maximum is a loop of compare-and-swaps, 136 us for the case below): first ord(w)
// alone, then perm_seed among the edges that reached a vertex's largest ord.  A
// matched vertex is marked in the next round's offers, above every ord; the two
// sets of offers alternate, one cleared while the other is read.  Up to NA_R edges a
// thread stay in registers with their keys for the whole run, more are kept as lists
// of edge ids in the static scratch.
//
// 10,000 vertices and 50,000 edges, 7 rounds: 314 us with one block and 64-bit offers in
// global memory (every phase waiting on L2), 75 us with sixteen blocks here.  Waited for
// call by call: 92 us with sixteen blocks, 122 with eight, 99 with 512 threads a block and
// twice the edges each.
#include <cuda_runtime.h>
#include <stdint.h>

#include <mutex>

#include "../../include/lm.h"
#include "lm_device.cuh"
#include "lm_internal.h"

namespace lm {

namespace {

constexpr uint32_t NA_MAX_N = LM_NOALLOC_MAX_N, NA_MAX_M = LM_NOALLOC_MAX_M;
constexpr uint32_t NA_T = 1024, NA_R = 8;   // threads, edges in a thread's registers
constexpr uint32_t NA_CMIN = 8, NA_CMAX = 16; // blocks of the cluster: 16 where the device takes it
constexpr uint32_t NA_SLOTS = NA_MAX_N / NA_CMIN;     // vertices of a block, at most
constexpr uint32_t NA_MATCHED = 0xFFFFFFFFu;          // above every ord(w) (only a NaN's is that large)
static_assert(NA_MAX_N <= 65536, "two vertex ids to a word");
static_assert(2 * sizeof(uint32_t) * NA_MAX_M == LM_NOALLOC_SCRATCH_BYTES, "scratch size as documented");
static __device__ __align__(256) unsigned char g_noalloc_scratch[LM_NOALLOC_SCRATCH_BYTES];

struct NaSmem {
    uint32_t hi[2][NA_SLOTS];   // largest ord(w) offered at each vertex (NA_MATCHED: matched), by round parity
    uint32_t lo[2][NA_SLOTS];   // largest perm_seed among the edges of that ord
    unsigned long long msg[2][NA_CMAX];  // every block's (error, live edges), by call parity
    uint32_t cnt, err;
};

template <int C>
__device__ __forceinline__ uint32_t na_addr(const void* p, uint32_t rank) {
    const uint32_t a = (uint32_t)__cvta_generic_to_shared(p);
    if (C == 1) return a;
    uint32_t out;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(out) : "r"(a), "r"(rank));
    return out;
}
template <int C>
__device__ __forceinline__ void na_sync() {
    if (C == 1) {
        __syncthreads();
    } else {
        __syncwarp();
        asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    }
}
// vertex x's slot in an array of its block
template <int C>
__device__ __forceinline__ uint32_t na_slot(const uint32_t* p, uint32_t x) {
    return na_addr<C>(p, x % C) + x / C * 4;
}
__device__ __forceinline__ void na_max(uint32_t at, uint32_t k) {
    asm volatile("red.relaxed.cluster.shared::cluster.max.u32 [%0], %1;" :: "r"(at), "r"(k) : "memory");
}
__device__ __forceinline__ uint32_t na_ld(uint32_t at) {
    uint32_t v;
    asm volatile("ld.relaxed.cluster.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(at) : "memory");
    return v;
}
__device__ __forceinline__ void na_st(uint32_t at, uint32_t x) {
    asm volatile("st.relaxed.cluster.shared::cluster.u32 [%0], %1;" :: "r"(at), "r"(x) : "memory");
}
// sum over the blocks (a barrier of the cluster); slot alternates between calls
template <int C>
__device__ __forceinline__ unsigned long long na_sum(NaSmem& S, uint32_t slot, uint32_t rank, unsigned long long x) {
    if (threadIdx.x < C) {
        const uint32_t at = na_addr<C>(&S.msg[slot][rank], threadIdx.x);
        asm volatile("st.relaxed.cluster.shared::cluster.u64 [%0], %1;" :: "r"(at), "l"(x) : "memory");
    }
    na_sync<C>();
    unsigned long long t = 0;
#pragma unroll
    for (int c = 0; c < C; c++) t += S.msg[slot][c];
    return t;
}

// REG: at most NA_R edges a thread, kept in registers; else lists of edge ids
template <int C, bool REG>
__global__ void __launch_bounds__(NA_T, 1) k_match_small(uint32_t n, uint32_t m, const uint32_t* __restrict__ eu,
                                                         const uint32_t* __restrict__ ev, const float* __restrict__ w,
                                                         uint32_t k0, uint32_t k1, uint32_t* mate, uint32_t* status,
                                                         uint32_t* lists) {
    extern __shared__ __align__(16) unsigned char na_raw[];
    NaSmem& S = *reinterpret_cast<NaSmem*>(na_raw);
    const uint32_t tid = threadIdx.x;
    uint32_t rank = 0;
    if (C > 1) asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    const uint32_t slots = (n + C - 1) / C;
    for (uint32_t v = rank * NA_T + tid; v < n; v += C * NA_T) mate[v] = NIL;
    for (uint32_t i = tid; i < slots; i += NA_T) S.hi[0][i] = S.hi[1][i] = S.lo[0][i] = S.lo[1][i] = 0;
    if (tid == 0) {
        S.cnt = 0;
        S.err = 0;
    }
    na_sync<C>();   // every block's slots are clear before an offer arrives
    const uint32_t per = (m + C - 1) / C, from = min(m, rank * per), share = min(m, from + per) - from;
    // edge e: ends, ord(w); false if it is not an edge of the graph
    auto get = [&](uint32_t e, uint32_t& uv, uint32_t& o) {
        const uint32_t u = __ldg(eu + e), v = __ldg(ev + e), wb = __float_as_uint(__ldg(w + e));
        const bool nan = ((wb & 0x7F800000u) == 0x7F800000u) && (wb & 0x007FFFFFu);
        uv = u | v << 16;
        o = ord_of_bits(wb);
        return u < n && v < n && u != v && !nan;
    };
    auto offer = [&](uint32_t b, uint32_t uv, uint32_t o) {
        na_max(na_slot<C>(S.hi[b], uv & 0xFFFFu), o);
        na_max(na_slot<C>(S.hi[b], uv >> 16), o);
    };
    // bit 0, 1: the edge has its first, second end's largest ord, and offers its perm there
    auto claim = [&](uint32_t b, uint32_t uv, uint32_t o, uint32_t e) {
        const uint32_t x = na_ld(na_slot<C>(S.hi[b], uv & 0xFFFFu)), y = na_ld(na_slot<C>(S.hi[b], uv >> 16));
        const uint32_t at = (x == o ? 1u : 0u) | (y == o ? 2u : 0u);
        if (at) {
            const uint32_t p = perm_seed(e, k0, k1);
            if (at & 1u) na_max(na_slot<C>(S.lo[b], uv & 0xFFFFu), p);
            if (at & 2u) na_max(na_slot<C>(S.lo[b], uv >> 16), p);
        }
        return at == 3u;
    };
    // an edge that claimed both ends: matched if its perm is the largest there
    auto settle = [&](uint32_t b, uint32_t uv, uint32_t e) {
        const uint32_t u = uv & 0xFFFFu, v = uv >> 16, p = perm_seed(e, k0, k1);
        if (na_ld(na_slot<C>(S.lo[b], u)) != p || na_ld(na_slot<C>(S.lo[b], v)) != p) return;
        mate[u] = v;
        mate[v] = u;
        na_st(na_slot<C>(S.hi[b ^ 1u], u), NA_MATCHED);
        na_st(na_slot<C>(S.hi[b ^ 1u], v), NA_MATCHED);
    };
    // an edge with no matched end stays and offers for the next round
    auto stay = [&](uint32_t b, uint32_t uv, uint32_t o) {
        const uint32_t su = na_slot<C>(S.hi[b ^ 1u], uv & 0xFFFFu), sv = na_slot<C>(S.hi[b ^ 1u], uv >> 16);
        const uint32_t x = na_ld(su), y = na_ld(sv);
        if (x == NA_MATCHED || y == NA_MATCHED) return false;
        if (x < o) na_max(su, o);
        if (y < o) na_max(sv, o);
        return true;
    };
    uint32_t uv[REG ? NA_R : 1], ord[REG ? NA_R : 1], alive = 0, both = 0;   // bit j: the thread's edge j
    auto list = [&](uint32_t b) { return lists + (b ? NA_MAX_M : 0u) + from; };   // the block's live edges, by round parity
    uint32_t cnt = share, bad = 0;
    if (REG) {
#pragma unroll
        for (uint32_t j = 0; j < NA_R; j++) {
            const uint32_t i = j * NA_T + tid;
            uv[j] = ord[j] = 0;
            if (i < share) {
                if (get(from + i, uv[j], ord[j])) alive |= 1u << j;
                else bad = 1;
            }
        }
#pragma unroll
        for (uint32_t j = 0; j < NA_R; j++)
            if ((alive >> j) & 1u) offer(0, uv[j], ord[j]);
    } else {
        for (uint32_t i = tid; i < share; i += NA_T) {
            uint32_t x, o;
            if (get(from + i, x, o)) offer(0, x, o);
            else bad = 1;
        }
    }
    if (bad) S.err = 1;
    __syncthreads();
    uint32_t slot = 0;
    const unsigned long long sum = na_sum<C>(S, slot, rank, ((unsigned long long)S.err << 32) | share);
    slot ^= 1u;
    uint32_t st = sum >> 32 ? 1u : 0u, total = st ? 0u : (uint32_t)sum;
    for (uint32_t round = 0; total > 0; round++) {
        if (round > m) {  // every round matches at least one edge
            st = 2u;
            break;
        }
        const uint32_t b = round & 1u;
        if (REG) {
            both = 0;
#pragma unroll
            for (uint32_t j = 0; j < NA_R; j++)
                if (((alive >> j) & 1u) && claim(b, uv[j], ord[j], from + j * NA_T + tid)) both |= 1u << j;
        } else {
            for (uint32_t i = tid; i < cnt; i += NA_T) {
                const uint32_t e = round == 0 ? from + i : __ldcg(list(b) + i);
                uint32_t x, o;
                get(e, x, o);
                claim(b, x, o, e);
            }
        }
        if (round > 0)   // the previous round's offers go back to nothing
            for (uint32_t i = tid; i < slots; i += NA_T) S.hi[b ^ 1u][i] = S.lo[b ^ 1u][i] = 0;
        if (tid == 0) S.cnt = 0;
        na_sync<C>();
        if (REG) {
#pragma unroll
            for (uint32_t j = 0; j < NA_R; j++)
                if ((both >> j) & 1u) settle(b, uv[j], from + j * NA_T + tid);
        } else {
            for (uint32_t i = tid; i < cnt; i += NA_T) {
                const uint32_t e = round == 0 ? from + i : __ldcg(list(b) + i);
                uint32_t x, o;
                get(e, x, o);
                if (na_ld(na_slot<C>(S.hi[b], x & 0xFFFFu)) == o && na_ld(na_slot<C>(S.hi[b], x >> 16)) == o) settle(b, x, e);
            }
        }
        na_sync<C>();
        if (REG) {
#pragma unroll
            for (uint32_t j = 0; j < NA_R; j++)
                if (((alive >> j) & 1u) && !stay(b, uv[j], ord[j])) alive &= ~(1u << j);
            const uint32_t left = __reduce_add_sync(FULL, (uint32_t)__popc(alive));
            if ((tid & 31) == 0 && left) atomicAdd(&S.cnt, left);
        } else {
            for (uint32_t i0 = 0; i0 < cnt; i0 += NA_T) {
                const uint32_t i = i0 + tid;
                uint32_t x = 0, o = 0, e = 0;
                bool keep = false;
                if (i < cnt) {
                    e = round == 0 ? from + i : __ldcg(list(b) + i);
                    get(e, x, o);
                    keep = stay(b, x, o);
                }
                const uint32_t bal = __ballot_sync(FULL, keep);
                uint32_t base = 0;
                if ((tid & 31) == 0 && bal) base = atomicAdd(&S.cnt, (uint32_t)__popc(bal));
                base = __shfl_sync(FULL, base, 0);
                if (keep) list(b ^ 1u)[base + __popc(bal & lanemask_lt())] = e;
            }
        }
        __syncthreads();
        cnt = S.cnt;
        total = (uint32_t)na_sum<C>(S, slot, rank, cnt);
        slot ^= 1u;
    }
    // a round cap that tripped leaves no partial result behind: every vertex unmatched
    if (st == 2u)
        for (uint32_t v = rank * NA_T + tid; v < n; v += C * NA_T) mate[v] = NIL;
    if (rank == 0 && tid == 0) *status = st;
    if (C > 1) na_sync<C>();  // no block leaves while another may still reach its shared memory
}

template <int C, bool REG>
int launch_small(void* stream, uint32_t n, uint32_t m, const uint32_t* eu, const uint32_t* ev, const float* w,
                 uint32_t k0, uint32_t k1, uint32_t* mate, uint32_t* status, uint32_t* lists) {
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute at[1];
    cfg.gridDim = dim3(C);
    cfg.blockDim = dim3(NA_T);
    cfg.dynamicSmemBytes = sizeof(NaSmem);
    cfg.stream = (cudaStream_t)stream;
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = C;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = C > 1 ? 1 : 0;
    return (int)cudaLaunchKernelEx(&cfg, k_match_small<C, REG>, n, m, eu, ev, w, k0, k1, mate, status, lists);
}
// the kernels' attributes, once per device; blocks: the cluster size the device takes
template <int C, bool REG>
cudaError_t small_attribute() {
    cudaError_t e = cudaFuncSetAttribute(k_match_small<C, REG>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)sizeof(NaSmem));
    if (e == cudaSuccess && C > 8)
        e = cudaFuncSetAttribute(k_match_small<C, REG>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    return e;
}
int small_attributes(uint32_t* blocks) {
    cudaError_t e = small_attribute<1, true>();
    if (e == cudaSuccess) e = small_attribute<NA_CMIN, true>();
    if (e == cudaSuccess) e = small_attribute<NA_CMIN, false>();
    if (e == cudaSuccess) e = small_attribute<NA_CMAX, true>();
    if (e == cudaSuccess) e = small_attribute<NA_CMAX, false>();
    if (e != cudaSuccess) return (int)e;
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute at[1];
    cfg.gridDim = dim3(NA_CMAX);
    cfg.blockDim = dim3(NA_T);
    cfg.dynamicSmemBytes = sizeof(NaSmem);
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = NA_CMAX;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int fit = 0;
    if (cudaOccupancyMaxActiveClusters(&fit, k_match_small<NA_CMAX, false>, &cfg) != cudaSuccess) {
        cudaGetLastError();
        fit = 0;
    }
    *blocks = fit > 0 ? NA_CMAX : NA_CMIN;
    return 0;
}
template <int C>
int launch_cluster(void* stream, uint32_t n, uint32_t m, const uint32_t* eu, const uint32_t* ev, const float* w,
                   uint32_t k0, uint32_t k1, uint32_t* mate, uint32_t* status, uint32_t* lists) {
    if (m <= C * NA_T * NA_R) return launch_small<C, true>(stream, n, m, eu, ev, w, k0, k1, mate, status, lists);
    return launch_small<C, false>(stream, n, m, eu, ev, w, k0, k1, mate, status, lists);
}

}  // namespace
}  // namespace lm

// The scratch's address on each device, looked up once with that device current.
namespace {
constexpr int NA_MAX_DEVICES = 64;
std::mutex g_na_mu;
void* g_na_ptr[NA_MAX_DEVICES] = {};
uint32_t g_na_blocks[NA_MAX_DEVICES] = {};
}  // namespace

extern "C" int lm_match_small_noalloc(uint32_t n, uint32_t m, const uint32_t* eu, const uint32_t* ev,
                                      const float* w, uint64_t seed, uint32_t* mate, uint32_t* status,
                                      void* stream) {
    if (n > LM_NOALLOC_MAX_N || m > LM_NOALLOC_MAX_M) return LM_EINVAL;
    if (!status || (n > 0 && !mate) || (m > 0 && (!eu || !ev || !w))) return LM_EINVAL;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) {
        cudaGetLastError();
        return LM_ECUDA;
    }
    if (dev < 0 || dev >= NA_MAX_DEVICES) return LM_EINVAL;
    // every array must be global memory of the current device: a pointer into host
    // memory or into another GPU would be dereferenced by the kernel as it is
    const void* arrays[5] = {eu, ev, w, mate, status};
    const bool needed[5] = {m > 0, m > 0, m > 0, n > 0, true};
    for (int i = 0; i < 5; i++) {
        if (!needed[i]) continue;
        cudaPointerAttributes at;
        if (cudaPointerGetAttributes(&at, arrays[i]) != cudaSuccess) {
            cudaGetLastError();
            return LM_EINVAL;
        }
        if ((at.type != cudaMemoryTypeDevice && at.type != cudaMemoryTypeManaged) || at.device != dev)
            return LM_EINVAL;
    }
    void* scratch = nullptr;
    uint32_t blocks = 0;
    {
        std::lock_guard<std::mutex> lk(g_na_mu);
        if (!g_na_ptr[dev]) {
            void* p = nullptr;
            cudaError_t e = cudaGetSymbolAddress(&p, lm::g_noalloc_scratch);
            if (e == cudaSuccess) e = (cudaError_t)lm::small_attributes(&g_na_blocks[dev]);
            if (e != cudaSuccess || !p) {
                cudaGetLastError();
                return LM_ECUDA;
            }
            g_na_ptr[dev] = p;
        }
        scratch = g_na_ptr[dev];
        blocks = g_na_blocks[dev];
    }
    const uint64_t z = lm::splitmix64_first(seed);
    const uint32_t k0 = (uint32_t)z, k1 = (uint32_t)(z >> 32);
    uint32_t* list = static_cast<uint32_t*>(scratch);
    int e;
    // one block as long as its slots and its threads' registers hold the graph: it needs
    // no cluster barrier
    if (n <= lm::NA_SLOTS && m <= lm::NA_T * lm::NA_R / 2)
        e = lm::launch_small<1, true>(stream, n, m, eu, ev, w, k0, k1, mate, status, list);
    else if (blocks == lm::NA_CMAX)
        e = lm::launch_cluster<lm::NA_CMAX>(stream, n, m, eu, ev, w, k0, k1, mate, status, list);
    else
        e = lm::launch_cluster<lm::NA_CMIN>(stream, n, m, eu, ev, w, k0, k1, mate, status, list);
    if (e) {
        cudaGetLastError();
        return LM_ECUDA;
    }
    return LM_OK;
}
