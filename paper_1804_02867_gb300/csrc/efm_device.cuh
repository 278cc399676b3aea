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

constexpr uint32_t kPadKey = 0xFFFFFFFFu;

__device__ __forceinline__ uint32_t mag(int32_t v) { return (uint32_t)(v < 0 ? -v : v); }

// gcd of magnitudes that are mostly small (Euclid: one or two divisions)
__device__ __forceinline__ uint32_t gcd_small(uint32_t a, uint32_t b)
{
    while (a) {
        const uint32_t t = b % a;
        b = a;
        a = t;
    }
    return b;
}

__device__ __forceinline__ uint64_t blob_u64(const uint32_t *bl, int o)
{
    return *reinterpret_cast<const uint64_t *>(bl + o);
}

// pivot key from the two masks (kPadKey when balanced)
__device__ __forceinline__ uint32_t mask_key(const uint32_t *bl, const NetView &nv, uint64_t pm, uint64_t nm)
{
    const uint32_t kp = pm ? bl[nv.o_keyr + __ffsll((long long)pm) - 1] : kPadKey;
    const uint32_t kn = nm ? bl[nv.o_keyr + 64 + __ffsll((long long)nm) - 1] : kPadKey;
    return kp < kn ? kp : kn;
}

// ---------------------------------------------------------------------------
// the superset rule's index (CellIndex): filing a result
// ---------------------------------------------------------------------------

__device__ __forceinline__ uint64_t col_bit(int c) { return 1ull << ((uint32_t)(c * 0x9E3779B1u) >> 26); }

__device__ __forceinline__ uint32_t cell_slot(uint32_t key, uint32_t mask)
{
    uint32_t x = key * 0x85EBCA6Bu;
    x ^= x >> 15;
    x *= 0xC2B2AE35u;
    return (x ^ (x >> 13)) & mask;
}

// One warp files result r, the support of the n <= 64 columns cols (shared
// memory), a column a lane: a lane's atomics are a chain, the lanes' are not.
// Its sentinels are its two columns with the fewest results at this moment
// (any other column of a result is a valid sentinel).
__device__ __noinline__ void file_result(const CellIndex &ix, int W, int64_t r, const int *cols, int n, uint64_t e0,
                                         uint64_t e1)
{
    const int lane = threadIdx.x & 31;
    if (n <= 1) {  // a one-column result: every child adding that column contains it
        if (lane == 0 && n == 1) ix.single[cols[0]] = 1u;
        return;
    }
    int c[2];
    unsigned long long key[2];
    uint64_t sig = 0;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        c[h] = lane + 32 * h < n ? cols[lane + 32 * h] : -1;
        key[h] = ~0ull;
        if (c[h] >= 0) {
            key[h] = ((unsigned long long)atomicAdd(&ix.cnt[c[h]], 1) << 16) | (unsigned)c[h];
            sig |= col_bit(c[h]);
        }
    }
    unsigned long long k1 = min(key[0], key[1]), k2 = max(key[0], key[1]);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        const unsigned long long o1 = __shfl_xor_sync(FULL, k1, off), o2 = __shfl_xor_sync(FULL, k2, off);
        k2 = min(min(k2, o2), max(k1, o1));  // the second of the four
        k1 = min(k1, o1);
        sig |= __shfl_xor_sync(FULL, sig, off);
    }
    const int m1 = (int)(k1 & 0xFFFFull), m2 = (int)(k2 & 0xFFFFull);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int k = c[h];
        if (k < 0) continue;
        const int s = k == m1 ? m2 : m1;
        const int64_t id = r * ix.ent_stride + lane + 32 * h;
        if (W <= 2) {
            atomicOr((unsigned long long *)&ix.ksig[2 * k + (s >> 6)], 1ull << (s & 63));
            const uint32_t next = atomicExch(reinterpret_cast<uint32_t *>(ix.cells) + 128 * k + s, (uint32_t)id);
            ix.ent[2 * id] = make_uint4((uint32_t)e0, (uint32_t)(e0 >> 32), (uint32_t)e1, (uint32_t)(e1 >> 32));
            ix.ent[2 * id + 1] = make_uint4(next, (uint32_t)r, 0u, 0u);
            continue;
        }
        atomicOr((unsigned long long *)&ix.ksig[k], (unsigned long long)col_bit(s));
        const uint32_t want = ((uint32_t)k << 12) | (uint32_t)s;
        uint32_t p = cell_slot(want, ix.mask);
        for (uint32_t probe = 0; probe <= ix.mask; ++probe) {
            const uint32_t v = atomicCAS(&ix.cells[p].x, kNoRecord, want);
            if (v == kNoRecord || v == want) {
                const uint32_t next = atomicExch(&ix.cells[p].y, (uint32_t)id);
                ix.ent[id] = make_uint4((uint32_t)sig, (uint32_t)(sig >> 32), next, (uint32_t)r);
                break;
            }
            p = (p + 1) & ix.mask;
        }
    }
    __syncwarp();
}

// Ascending columns of a support into cols (shared memory, room for 64); lane
// l holds its words l and l + 32.  Returns their number (columns past the
// 64th are not written).
__device__ __forceinline__ int support_columns(uint64_t u0, uint64_t u1, int *cols)
{
    const int lane = threadIdx.x & 31;
    const int n0 = __popcll(u0), n1 = __popcll(u1);
    int s0 = n0, s1 = n1;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const int x0 = __shfl_up_sync(FULL, s0, off), x1 = __shfl_up_sync(FULL, s1, off);
        if (lane >= off) {
            s0 += x0;
            s1 += x1;
        }
    }
    const int tot0 = __shfl_sync(FULL, s0, 31);
    int pos0 = s0 - n0, pos1 = tot0 + s1 - n1;
    for (uint64_t x = u0; x && pos0 < 64; x &= x - 1) cols[pos0++] = lane * 64 + __ffsll((long long)x) - 1;
    for (uint64_t x = u1; x && pos1 < 64; x &= x - 1) cols[pos1++] = (lane + 32) * 64 + __ffsll((long long)x) - 1;
    __syncwarp();
    return tot0 + __shfl_sync(FULL, s1, 31);
}

}  // namespace
}  // namespace efm
