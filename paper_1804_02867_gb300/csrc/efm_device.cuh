// efm_device.cuh -- device helpers shared by the kernel files.
#pragma once
#include "efm_internal.cuh"

namespace efm {
namespace {

constexpr unsigned FULL = 0xFFFFFFFFu;

__device__ __forceinline__ uint64_t mix64(uint64_t x)
{
    // splitmix64 finaliser (Steele, Lea, Flood 2014)
    x ^= x >> 30;
    x *= 0xbf58476d1ce4e5b9ull;
    x ^= x >> 27;
    x *= 0x94d049bb133111ebull;
    x ^= x >> 31;
    return x;
}

__device__ __forceinline__ uint64_t gcd64(uint64_t a, uint64_t b)
{
    // binary gcd (Stein)
    if (a == 0) return b;
    if (b == 0) return a;
    const int sh = __ffsll((long long)(a | b)) - 1;
    a >>= __ffsll((long long)a) - 1;
    while (b != 0) {
        b >>= __ffsll((long long)b) - 1;
        if (a > b) {
            const uint64_t t = a;
            a = b;
            b = t;
        }
        b -= a;
    }
    return a << sh;
}

__device__ __forceinline__ uint32_t gcd32(uint32_t a, uint32_t b)
{
    if (a == 0) return b;
    if (b == 0) return a;
    const int sh = __ffs((int)(a | b)) - 1;
    a >>= __ffs((int)a) - 1;
    while (b != 0) {
        b >>= __ffs((int)b) - 1;
        if (a > b) {
            const uint32_t t = a;
            a = b;
            b = t;
        }
        b -= a;
    }
    return a << sh;
}

__device__ __forceinline__ uint64_t abs64(int64_t x) { return x < 0 ? (uint64_t)(-x) : (uint64_t)x; }

__device__ __forceinline__ bool bit_of(const uint64_t *U, int k) { return (U[k >> 6] >> (k & 63)) & 1ull; }

__device__ __forceinline__ unsigned long long load_volatile(unsigned long long *p)
{
    return *(volatile unsigned long long *)p;
}

__device__ __forceinline__ uint64_t global_ns()
{
    uint64_t t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}

constexpr uint64_t kWatchdogNs = 20ull * 1000000000ull;  // a level that runs longer gives up
constexpr int kMaxRounds = 1 << 22;

// Record the first failed self-check (code, offending value, its limit) and
// raise the error bit; the caller skips the access.
__device__ __forceinline__ void record_diag(unsigned long long *ctr, unsigned bit, unsigned long long code, long long value,
                            long long limit, int level)
{
    atomicOr(&ctr[C_ERR], (unsigned long long)bit);
    if (atomicCAS(&ctr[C_DIAG], 0ull, code) == 0ull) {
        ctr[C_DIAG + 1] = (unsigned long long)value;
        ctr[C_DIAG + 2] = (unsigned long long)limit;
        ctr[C_DIAG + 3] = (unsigned long long)level;
    }
}

enum { INS_NEW = 1, INS_DUP = 0, INS_ARENA_FULL = -1, INS_TIMEOUT = -2, INS_TABLE_FULL = -3 };

__device__ __forceinline__ void slot_tag_pos(uint64_t h, uint64_t mask, uint64_t &pos, uint32_t &tag)
{
    const uint64_t f = mix64(h);
    pos = f & mask;
    tag = (uint32_t)(f >> 32);
    if (tag == 0xFFFFFFFFu) tag = 0xFFFFFFFEu;
}

// pivot key (degree << 16 | row) -> state meta: row | degree << 10 | |U| << 23
__device__ __forceinline__ uint32_t pack_meta(uint32_t key, int pc)
{
    return (key & 0x3FFu) | ((key >> 16) << 10) | ((uint32_t)pc << 23);
}

// The meta word's degree field counts the branches a state has: the list of
// the pivot's side, plus (subtractive variant) the opposite list.
__device__ __forceinline__ uint32_t branch_key(const uint32_t *bl, const NetView &nv, uint32_t key, int sub)
{
    if (!sub) return key;
    const int m = (int)(key & 0xFFFFu);
    const uint32_t deg = (bl[nv.o_consptr + m + 1] - bl[nv.o_consptr + m]) + (bl[nv.o_prodptr + m + 1] - bl[nv.o_prodptr + m]);
    return (deg << 16) | (key & 0xFFFFu);
}

}  // namespace
}  // namespace efm
