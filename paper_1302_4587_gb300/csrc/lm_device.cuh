// Device helpers shared by the matching kernels (lm_kernels.cu, lm_list.cu): the
// edge order, warp utilities, error recording.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "lm_internal.h"

namespace lm {

#define FULL 0xFFFFFFFFu

// ---------------------------------------------------------------- order
// MurmurHash3 32-bit finaliser (Appleby, public domain).
__device__ __forceinline__ uint32_t fmix32(uint32_t h) {
    h ^= h >> 16;
    h *= 0x85EBCA6Bu;
    h ^= h >> 13;
    h *= 0xC2B2AE35u;
    h ^= h >> 16;
    return h;
}
__device__ __forceinline__ uint32_t perm_seed(uint32_t e, uint32_t k0, uint32_t k1) {
    return fmix32(fmix32(e ^ k0) ^ k1);
}
// inverse of x -> x * a (mod 2^32) for odd a, by Newton's iteration
__host__ __device__ constexpr uint32_t inv_mul(uint32_t a) {
    uint32_t x = a;  // correct to 3 bits for odd a
    x *= 2u - a * x;
    x *= 2u - a * x;
    x *= 2u - a * x;
    x *= 2u - a * x;
    x *= 2u - a * x;
    return x;
}
constexpr uint32_t INV_M1 = inv_mul(0x85EBCA6Bu), INV_M2 = inv_mul(0xC2B2AE35u);
static_assert(0x85EBCA6Bu * INV_M1 == 1u && 0xC2B2AE35u * INV_M2 == 1u, "modular inverses");
__device__ __forceinline__ uint32_t fmix32_inv(uint32_t h) {
    h ^= h >> 16;                       // h ^ (h >> 16) is its own inverse on 32 bits
    h *= INV_M2;
    h ^= (h >> 13) ^ (h >> 26);         // inverse of h ^= h >> 13
    h *= INV_M1;
    h ^= h >> 16;
    return h;
}
// e = perm_seed^-1(x)
__device__ __forceinline__ uint32_t perm_seed_inv(uint32_t x, uint32_t k0, uint32_t k1) {
    return fmix32_inv(fmix32_inv(x) ^ k1) ^ k0;
}
// SplitMix64 (Steele, Lea, Flood 2014): the r-th output (r >= 0) for state `seed`
__device__ __forceinline__ uint64_t splitmix64_at(uint64_t seed, uint32_t r) {
    uint64_t z = seed + (uint64_t)(r + 1u) * 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}
// monotone float32 -> uint32 (-0 == +0); NaN is rejected before this runs
__device__ __forceinline__ uint32_t ord_of_bits(uint32_t b) {
    if (b == 0x80000000u) b = 0u;
    return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}

// ---------------------------------------------------------------- utilities
__device__ __forceinline__ uint32_t ld_volatile_u32(const uint32_t* p) {
    return *reinterpret_cast<const volatile uint32_t*>(p);
}
__device__ __forceinline__ uint32_t lanemask_lt() {
    uint32_t m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}
__device__ __forceinline__ uint32_t lanemask_le() {
    uint32_t m;
    asm("mov.u32 %0, %%lanemask_le;" : "=r"(m));
    return m;
}
__device__ __forceinline__ uint32_t warp_incl_scan(uint32_t x, int lane) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(FULL, x, o);
        if (lane >= o) x += y;
    }
    return x;
}
// device-scope fetch-and-add with acquire-release ordering
__device__ __forceinline__ uint32_t atom_add_acq_rel(uint32_t* p, uint32_t v) {
    uint32_t old;
    asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], %2;" : "=r"(old) : "l"(p), "r"(v) : "memory");
    return old;
}
__device__ __forceinline__ void set_err(DevState* st, uint32_t bit, uint32_t info) {
    if ((atomicOr(&st->err, bit) & bit) == 0) st->err_info = info;
    atomicOr(&st->err_any, bit);  // not reset by the next job's init (asynchronous matches)
}
// the job's state into the host's mirror by the last block to leave (`threads` threads): a
// copy in the stream would cost a small job 5 us more
__device__ __forceinline__ void state_to_host(DevState* host, const DevState* st, uint32_t threads) {
    static_assert(sizeof(DevState) % 4 == 0, "words");
    for (uint32_t i = threadIdx.x; i < sizeof(DevState) / 4; i += threads)
        reinterpret_cast<volatile uint32_t*>(host)[i] = __ldcg(reinterpret_cast<const uint32_t*>(st) + i);
}
__device__ __forceinline__ uint64_t globaltimer_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

}  // namespace lm
