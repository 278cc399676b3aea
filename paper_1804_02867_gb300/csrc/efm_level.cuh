// efm_level.cuh -- device code of the traversal's level pass, for the whole grid
// (efm_sparse.cu) or one CTA (the batched traversal, efm_kernels.cu).
//
// A state keeps only what it holds: its support and the unbalanced entries of
// its extra-flux row.  Most entries of a row are zero (a state of the
// 58-row core-shaped network holds about 10 unbalanced rows, one of the
// 850-row genome-shaped network 8 to 19), so a state takes about 100 bytes.
//
// Layout (Arena): per row of the arena a 16-byte header, and a payload in
// 16-byte units somewhere in the arena's pool:
//   hdr  x = payload offset in units, y = meta (0: the row carries no state),
//        z = number of entries | bits of max|EF| << 11, w = EF of the pivot
//   pay  the row hash rh = sum_m EF_m R[m] (mod 2^64) with R[m] =
//        mix64(0x9E3779B97F4A7C15 (m + 1)), linear in EF, so that a child's
//        follows from its parent's and column k's; the sum of the columns'
//        hash constants (lists only); then the support: at most 128 columns,
//        a bitset of 2 words (one unit); else the columns, 16 bits each, in
//        the order they were added, padded with 0xFFFF to a unit; then the entries, 8 bytes each, in no order,
//        padded to a unit: (pivot key of the row's side, degree << 16 | row;
//        value); the key of a flux entry is 0xFFFF0000 | row, of padding ~0.
// Narrow networks (at most 64 rows and 128 columns) instead: rh and the mask
// of the nonzero rows; the bitset; the masks of the positive and of the
// negative entries, each row at its rank in the order of that side's pivot
// keys; then the values in row order, 4 bytes each, padded with zeros.
// In the subtractive variant (Eq. 5) the entries go on with the flux of every
// column k of U at row M + k.
//
// Measured against the dense rows it replaced (the whole row by a group of
// lanes, in up to five passes), one GB300, calls through the library: four
// genome-shaped targets at a 2^22 budget 361 -> 23.7 ms (1817 -> about 110
// warp instructions a child, 3.5 KB -> about 130 bytes written), six targets
// of a 400-row network at 2^17 23.4 -> 5.4, first-K = 1000 on three genome
// targets 103 -> 44.5, eight targets of the core-shaped network at 2^17 20.4
// -> 13.6 and at 2^26 539 -> 471, its subtractive variant 12.1 -> 8.2.
//
// The AND update EF' = A EF + C S_int[:, k] is then a copy of the parent's
// entries (times A) in 16-byte units, with the few rows of column k changed
// in place, appended or removed: a lane per child, no order to keep.  The
// smallest key among the entries names the pivot.
#pragma once
#include "efm_device.cuh"

namespace efm {
namespace {

constexpr uint32_t kFluxKey = 0xFFFF0000u;  // keys from here on are no balance rows

__device__ __forceinline__ uint64_t column_hash(int k) { return mix64(0x51ed27f3a5b1c3d9ull * (uint64_t)(k + 1)); }
__device__ __forceinline__ uint64_t row_hash(int m) { return mix64(0x9E3779B97F4A7C15ull * (uint64_t)(m + 1)); }

// Fingerprint of a state: 63 bits.  The top bit marks a reserved row without
// one: kDeadFp, or a child that the dedup pass finishes first (an open child:
// its parent's row, column k and flags; see kOpen...).
__device__ __forceinline__ uint64_t state_fp(uint64_t rows, uint64_t cols)
{
    return (rows ^ mix64(cols + 0x632BE59BD9B4E019ull)) >> 1;
}

constexpr uint64_t kOpenFp = 1ull << 63;
constexpr uint64_t kOpenInU = 1ull << 44;   // a secondary step (k is in U)
constexpr uint64_t kOpenSub = 1ull << 45;   // Eq. 5: flux taken away from k
constexpr uint64_t kOpenPruned = 1ull << 46;  // the superset rule holds
constexpr uint64_t kOpenDead = 1ull << 47;  // first-K: cannot balance any more
constexpr uint64_t kOpenBal = 1ull << 48;   // balanced: to the arbiter

__device__ __forceinline__ void prefetch_l2(const void *p)
{
    asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
}

__device__ __forceinline__ int max_bits(uint32_t om) { return om ? 32 - __clz((int)om) : 0; }

// 16-bit column i of a payload's list
__device__ __forceinline__ int list_col(const uint4 *pay, int i)
{
    return reinterpret_cast<const uint16_t *>(pay)[8 + i];
}

// ---------------------------------------------------------------------------
// Supports.  F (NetView::form) = 1, 2: a bitset of two words (at most 128
// columns); F = 0: a list.  A child's support is its parent's plus column k (k < 0: the same).
// ---------------------------------------------------------------------------

template <int F>
__device__ __forceinline__ int support_units(int pc)
{
    return F == 2 ? 3 : (F == 1 ? 2 : sparse_list_units(pc));
}

__device__ __forceinline__ uint64_t bits_hash(uint64_t u0, uint64_t u1)
{
    return mix64(u0 ^ 0x2545f4914f6cdd1dull) + mix64(u1 ^ 0x4a8be9229ed9ba3aull);
}

__device__ __forceinline__ void add_bit(uint64_t &u0, uint64_t &u1, int k)
{
    if (k < 64) u0 |= 1ull << k;
    else u1 |= 1ull << (k - 64);
}

// hash of the support U + {k}
template <int F>
__device__ __forceinline__ uint64_t support_hash_of(const uint4 *pay, int k)
{
    if (F) {
        uint64_t u0 = reinterpret_cast<const uint64_t *>(pay)[2], u1 = reinterpret_cast<const uint64_t *>(pay)[3];
        if (k >= 0) add_bit(u0, u1, k);
        return bits_hash(u0, u1);
    }
    return reinterpret_cast<const uint64_t *>(pay)[1] + (k >= 0 ? column_hash(k) : 0ull);
}

// Insert the support U + {k} into the set of supports judged in this
// traversal (one thread; the arbiter reads bitset words).
template <int F>
__device__ __noinline__ int insert_candidate(const LevelArgs &a, int W, const uint4 *pay, int pc, int k)
{
    uint64_t p;
    uint32_t tag;
    slot_tag_pos(support_hash_of<F>(pay, k), a.cslot_mask, p, tag);
    for (uint64_t probe = 0; probe <= a.cslot_mask; ++probe) {
        unsigned long long v = atomicCAS(&a.cslots[p], kEmpty, ((unsigned long long)tag << 32) | kPending);
        if (v == kEmpty) {
            const unsigned long long idx = atomicAdd(&a.ctr[C_CAND_N], 1ull);
            if ((int64_t)idx >= a.cand_cap) {
                atomicOr(&a.ctr[C_ERR], (unsigned long long)ERR_CAND_CAP);
                atomicExch(&a.cslots[p], ((unsigned long long)tag << 32) | kOverflowIdx);
                return INS_ARENA_FULL;
            }
            uint64_t *dst = a.cand + (size_t)idx * W;
            if (F) {
                uint64_t u[2] = {reinterpret_cast<const uint64_t *>(pay)[2], reinterpret_cast<const uint64_t *>(pay)[3]};
                if (k >= 0) add_bit(u[0], u[1], k);
                for (int w = 0; w < W; ++w) dst[w] = w ? u[1] : u[0];
            } else {
                for (int w = 0; w < W; ++w) dst[w] = 0ull;
                for (int i = 0; i < pc; ++i) {
                    const int c = list_col(pay, i);
                    dst[c >> 6] |= 1ull << (c & 63);
                }
                if (k >= 0) dst[k >> 6] |= 1ull << (k & 63);
            }
            __threadfence();
            atomicExch(&a.cslots[p], ((unsigned long long)tag << 32) | idx);
            return INS_NEW;
        }
        if ((uint32_t)(v >> 32) == tag) {
            int spins = 0;
            while ((uint32_t)v == kPending) {
                if (++spins > kWaitSpinLimit) {
                    atomicOr(&a.ctr[C_ERR], (unsigned long long)ERR_TIMEOUT);
                    return INS_TIMEOUT;
                }
                __nanosleep(64);
                v = load_volatile(&a.cslots[p]);
            }
            const uint32_t idx = (uint32_t)v;
            if (idx == kOverflowIdx) return INS_ARENA_FULL;
            const uint64_t *src = a.cand + (size_t)idx * W;
            bool eq = true;
            if (F) {
                uint64_t u[2] = {reinterpret_cast<const uint64_t *>(pay)[2], reinterpret_cast<const uint64_t *>(pay)[3]};
                if (k >= 0) add_bit(u[0], u[1], k);
                for (int w = 0; w < W && eq; ++w) eq = __ldcg(src + w) == (w ? u[1] : u[0]);
            } else {
                // equal: as many columns, and each of them there
                int n = 0;
                for (int w = 0; w < W; ++w) n += __popcll(__ldcg(src + w));
                eq = n == pc + (k >= 0 ? 1 : 0);
                for (int i = 0; i < pc && eq; ++i) {
                    const int c = list_col(pay, i);
                    eq = (__ldcg(src + (c >> 6)) >> (c & 63)) & 1ull;
                }
                if (k >= 0 && eq) eq = (__ldcg(src + (k >> 6)) >> (k & 63)) & 1ull;
            }
            if (eq) return INS_DUP;
        }
        p = (p + 1) & a.cslot_mask;
    }
    atomicOr(&a.ctr[C_ERR], (unsigned long long)ERR_TABLE_FULL);
    return INS_TABLE_FULL;
}

// ---------------------------------------------------------------------------
// the superset rule (see CellIndex in efm_internal.cuh)
// ---------------------------------------------------------------------------

// Does a result E with k in E lie inside U + {k}?  One lane.  Only the cells
// (k, s) of the sentinels s in U are looked up.
__device__ __forceinline__ bool pruned_bits(const CellIndex &ix, const uint4 *pay, int k)
{
    uint64_t u0 = reinterpret_cast<const uint64_t *>(pay)[2], u1 = reinterpret_cast<const uint64_t *>(pay)[3];
    const ulonglong2 ks = reinterpret_cast<const ulonglong2 *>(ix.ksig)[k];
    uint64_t m[2] = {ks.x & u0, ks.y & u1};
    if (ix.single[k]) return true;
    if ((m[0] | m[1]) == 0) return false;
    add_bit(u0, u1, k);
    const uint32_t *heads = reinterpret_cast<const uint32_t *>(ix.cells) + 128 * k;
#pragma unroll
    for (int w = 0; w < 2; ++w)
        for (uint64_t x = m[w]; x; x &= x - 1) {
            uint32_t head = heads[64 * w + __ffsll((long long)x) - 1];
            // a list holds each result at most once
            for (int64_t n = 0; head != kNoRecord && n < ix.room; ++n) {
                const ulonglong2 e = *reinterpret_cast<const ulonglong2 *>(ix.ent + 2 * (size_t)head);
                if (((e.x & ~u0) | (e.y & ~u1)) == 0) return true;
                head = ix.ent[2 * (size_t)head + 1].x;
            }
        }
    return false;
}

// The same on lists: a cell's results are tested by a 64-bit signature, then
// column by column.
__device__ __noinline__ bool pruned_list(const CellIndex &ix, const uint16_t *rcols, const uint4 *pay, int pc, int k)
{
    if (ix.single[k]) return true;
    const uint64_t ks = ix.ksig[k];
    if (ks == 0) return false;
    uint64_t su = col_bit(k);
    for (int i = 0; i < pc; ++i) su |= col_bit(list_col(pay, i));
    if ((ks & su) == 0) return false;
    for (int i = 0; i < pc; ++i) {
        const int s = list_col(pay, i);
        if (!(ks & col_bit(s)) || s == k) continue;
        const uint32_t key = ((uint32_t)k << 12) | (uint32_t)s;
        uint32_t p = cell_slot(key, ix.mask);
        uint32_t head = kNoRecord;
        for (uint32_t probe = 0; probe <= ix.mask; ++probe) {
            const uint2 cell = ix.cells[p];
            if (cell.x == key) {
                head = cell.y;
                break;
            }
            if (cell.x == kNoRecord) break;
            p = (p + 1) & ix.mask;
        }
        for (int64_t n = 0; head != kNoRecord && n < ix.room; ++n) {
            const uint4 e = ix.ent[head];
            const uint64_t sig = (uint64_t)e.x | ((uint64_t)e.y << 32);
            if ((sig & ~su) == 0) {
                const uint16_t *lst = rcols + (size_t)e.w * kRcolStride;
                const int m = lst[0];
                bool sub = m <= pc + 1;
                for (int j = 1; j <= m && sub; ++j) {
                    const int c = lst[j];
                    if (c == k) continue;
                    sub = false;
                    for (int q = 0; q < pc && !sub; ++q) sub = list_col(pay, q) == c;
                }
                if (sub) return true;
            }
            head = e.z;
        }
    }
    return false;
}

// ---------------------------------------------------------------------------
// the AND update
// ---------------------------------------------------------------------------

// pivot key of an entry of row `row` with the sign of t
template <bool SUB>
__device__ __forceinline__ uint32_t entry_key(const NetView &nv, const uint32_t *bl, int row, bool positive)
{
    if (SUB && row >= nv.M) return kFluxKey | (uint32_t)row;
    return bl[(positive ? nv.o_keypos : nv.o_keyneg) + row];
}

struct Child {
    int n;          // entries
    uint32_t key;   // smallest key (kFluxKey or above: no balance row is left)
    int32_t pv;     // the entry of that key
    uint32_t om;    // OR of the magnitudes
    uint32_t g;     // gcd of the entries (1 as soon as it is known to be 1)
    uint64_t rh;    // wide_child only
    bool zflux;     // the flux of k is not positive any more (Prop. 3)
    bool ovf;       // an entry outside int32 after the division (wide_child only)
};

// Column entries: words [cb, ce) of the column CSR, rows ascending; in the
// subtractive view one more, flux 1 on k at row M + k.
template <bool SUB>
__device__ __forceinline__ void column_entry(const NetView &nv, const uint32_t *bl, int cb, int ce, int q, int k,
                                             int &row, int32_t &val)
{
    if (SUB && cb + q == ce) {
        row = nv.M + k;
        val = 1;
        return;
    }
    const uint32_t f = bl[nv.o_colent + cb + q];
    row = ent_index(f);
    val = ent_coef(f);
}

// One child, when every entry is known to fit int32, the parent has at most
// 64 entries and the column at most 32 (dst null: nothing is written).
template <bool SUB>
__device__ __forceinline__ void fast_child(const NetView &nv, const uint32_t *bl, const uint4 *pe, int np, int32_t A,
                                           int32_t C, int cb, int ce, uint64_t mask, int k, uint4 *dst, Child &r)
{
    uint32_t key = kPadKey, om = 0, mn = 0xFFFFFFFFu;  // mn: smallest magnitude
    int32_t pv = 0;
    uint64_t hits = 0;  // parent entries on a row whose mask bit column k sets
    for (int i = 0; 2 * i < np; ++i) {
        const uint4 e = pe[i];
        const int32_t v0 = A * (int32_t)e.y, v1 = A * (int32_t)e.w;
        const uint32_t h0 = (uint32_t)(mask >> (e.x & 63u)) & 1u;
        const uint32_t h1 = e.w ? (uint32_t)(mask >> (e.z & 63u)) & 1u : 0u;  // (padding is no hit)
        hits |= (uint64_t)(h0 | (h1 << 1)) << (2 * i);
        const uint32_t a0 = h0 ? 0u : mag(v0), a1 = h1 ? 0u : mag(v1);
        om |= a0 | a1;
        mn = min(mn, min(a0 - 1u, a1 - 1u));  // less one: a hit or padding counts as none
        const uint32_t k0 = h0 ? kPadKey : e.x, k1 = h1 ? kPadKey : e.z;
        if (k0 < key) {
            key = k0;
            pv = v0;
        }
        if (k1 < key) {
            key = k1;
            pv = v1;
        }
        if (dst) dst[i] = make_uint4(e.x, (uint32_t)v0, e.z, (uint32_t)v1);
    }
    const int2 *p2 = reinterpret_cast<const int2 *>(pe);
    int2 *d2 = reinterpret_cast<int2 *>(dst);
    const int nq = ce - cb + (SUB ? 1 : 0);
    uint32_t matched = 0, g = 0;  // column entries met; gcd of the changed entries (while it is needed)
    uint64_t holes = 0;
    bool zflux = false;
    int n = np;
    auto take = [&](uint32_t kk, int32_t t) {
        const uint32_t at = mag(t);
        om |= at;
        mn = min(mn, at - 1u);
        if (mn != 0u) g = gcd_small(g, at);
        if (kk < key) {
            key = kk;
            pv = t;
        }
    };
    for (uint64_t h = hits; h; h &= h - 1) {
        const int i = __ffsll((long long)h) - 1;
        const int2 e = p2[i];
        const int row = e.x & 0xFFFF;
        int32_t cv = 0;
        for (int q = 0; q < nq; ++q) {
            int rq;
            int32_t vq;
            column_entry<SUB>(nv, bl, cb, ce, q, k, rq, vq);
            if (rq == row) {
                cv = vq;
                matched |= 1u << q;
                break;
            }
        }
        const int32_t t = A * e.y + C * cv;
        if (SUB && row == nv.M + k && t <= 0) zflux = true;
        if (t == 0) {
            holes |= 1ull << i;
            continue;
        }
        const uint32_t kk = cv == 0 ? (uint32_t)e.x : entry_key<SUB>(nv, bl, row, t > 0);
        take(kk, t);
        if (d2) d2[i] = make_int2((int)kk, t);
    }
    for (int q = 0; q < nq; ++q) {
        if ((matched >> q) & 1u) continue;
        int row;
        int32_t cv;
        column_entry<SUB>(nv, bl, cb, ce, q, k, row, cv);
        const int32_t t = C * cv;
        if (SUB && row >= nv.M && t <= 0) zflux = true;
        const uint32_t kk = entry_key<SUB>(nv, bl, row, t > 0);
        take(kk, t);
        int at = n;
        if (holes) {
            at = __ffsll((long long)holes) - 1;
            holes &= holes - 1;
        } else {
            ++n;
        }
        if (d2) d2[at] = make_int2((int)kk, t);
    }
    while (holes) {  // close what is left with entries from the end
        const int last = --n;
        if (last < 64 && ((holes >> last) & 1ull)) {
            holes &= ~(1ull << last);
            continue;
        }
        const int at = __ffsll((long long)holes) - 1;
        holes &= holes - 1;
        if (d2) d2[at] = d2[last];
    }
    if (d2 && (n & 1)) d2[n] = make_int2((int)kPadKey, 0);
    // the gcd: 1 with an entry of magnitude 1, or when the changed entries (which
    // every common divisor divides) share none, or only powers of two beside
    // an odd entry; else by the unchanged entries, until it is 1
    if (mn == 0u || ((om & 1u) && g != 0u && (g & (g - 1u)) == 0u)) g = 1u;
    if (g != 1u)
        for (int i = 0; i < np && g != 1u; ++i)
            if (!((hits >> i) & 1ull)) g = gcd_small(g, mag(A * p2[i].y));
    r.n = n;
    r.key = key;
    r.pv = pv;
    r.om = om;
    r.g = g;
    r.zflux = zflux;
}

// One child of any number of entries, when every one is known to fit int32
// (networks whose reactions have dozens of metabolites, where states have as
// many entries): the coefficients from the dense copy of S_int, the rows that
// the parent has as bits in local memory, the entries written one after the
// other.
template <bool SUB>
__device__ __noinline__ void long_child(const NetView &nv, const uint32_t *bl, const uint4 *pe, int np, int32_t A,
                                        int32_t C, int cb, int ce, int k, uint4 *dst, Child &r)
{
    const int2 *p2 = reinterpret_cast<const int2 *>(pe);
    int2 *d2 = reinterpret_cast<int2 *>(dst);
    const int32_t *col = reinterpret_cast<const int32_t *>(bl + nv.o_dcols) + (size_t)k * nv.Mpad;
    const int rows = nv.M + (SUB ? nv.N : 0);  // at most EFM_MAX_INTERNAL
    uint32_t has[EFM_MAX_INTERNAL / 32];
    for (int w = 0; 32 * w < rows; ++w) has[w] = 0u;
    uint32_t key = kPadKey, om = 0, g = 0;
    int32_t pv = 0;
    bool zflux = false;
    int n = 0;
    auto put = [&](uint32_t kk, int32_t t) {
        const uint32_t at = mag(t);
        om |= at;
        if (g != 1u) g = gcd_small(g, at);
        if (kk < key) {
            key = kk;
            pv = t;
        }
        if (d2) d2[n] = make_int2((int)kk, t);
        ++n;
    };
    for (int i = 0; i < np; ++i) {
        const int2 e = p2[i];
        const int row = e.x & 0xFFFF;
        const int32_t cv = col[row];
        has[row >> 5] |= 1u << (row & 31);
        const int32_t t = A * e.y + C * cv;
        if (SUB && row == nv.M + k && t <= 0) zflux = true;
        if (t != 0) put(cv == 0 ? (uint32_t)e.x : entry_key<SUB>(nv, bl, row, t > 0), t);
    }
    const int nq = ce - cb + (SUB ? 1 : 0);
    for (int q = 0; q < nq; ++q) {
        int row;
        int32_t cv;
        column_entry<SUB>(nv, bl, cb, ce, q, k, row, cv);
        if ((has[row >> 5] >> (row & 31)) & 1u) continue;
        const int32_t t = C * cv;
        if (SUB && row >= nv.M && t <= 0) zflux = true;
        put(entry_key<SUB>(nv, bl, row, t > 0), t);
    }
    if (d2 && (n & 1)) d2[n] = make_int2((int)kPadKey, 0);
    r.n = n;
    r.key = key;
    r.pv = pv;
    r.om = om;
    r.g = g;
    r.zflux = zflux;
}

// --- narrow networks ---

// values below row r in a state with nonzero rows zm
__device__ __forceinline__ int value_at(uint64_t zm, int r) { return __popcll(zm & ((1ull << r) - 1ull)); }

struct NarrowMasks {
    uint64_t zm, pm, nm;
};

// One child of a narrow network, when every entry is known to fit int32: the
// masks follow from the rows of column k alone, the other values are copied
// (times A) to their places.  LONG: a column of more than kNarrowCol entries,
// whose new values are computed twice instead of kept.
template <bool LONG = false>
__device__ __forceinline__ void narrow_child(const NetView &nv, const uint32_t *bl, const uint4 *pp, int32_t A,
                                             int32_t C, int cb, int nc, int k, int32_t *dst, Child &r, NarrowMasks &z)
{
    const uint64_t zm = reinterpret_cast<const uint64_t *>(pp)[1];
    const int32_t *vals = reinterpret_cast<const int32_t *>(pp + 3);
    const int ox = nv.o_colx + 10 * k;
    const uint64_t mask = blob_u64(bl, ox + 4);
    const uint2 *ent = reinterpret_cast<const uint2 *>(bl + nv.o_nent) + cb;
    int32_t t[LONG ? 1 : kNarrowCol];
    uint32_t om = 0, mn = 0xFFFFFFFFu;  // OR of the magnitudes; smallest magnitude less one
    uint64_t newz = 0, newp = 0, newn = 0;
    auto value = [&](const uint2 &e) -> int32_t {  // the child's, on a row of column k
        const int row = (int)(e.x & 63u);
        int32_t v = 0;
        if ((zm >> row) & 1ull) v = vals[value_at(zm, row)];
        return A * v + C * (int32_t)e.y;
    };
    auto note = [&](const uint2 &e, int32_t x) {
        newz |= (uint64_t)(x != 0) << (e.x & 63u);
        newp |= (uint64_t)(x > 0) << ((e.x >> 8) & 63u);
        newn |= (uint64_t)(x < 0) << ((e.x >> 16) & 63u);
        const uint32_t a = mag(x);
        om |= a;
        mn = min(mn, a - 1u);
    };
    if (LONG) {
        for (int q = 0; q < nc; ++q) {
            const uint2 e = ent[q];
            note(e, value(e));
        }
    } else {
#pragma unroll
        for (int q = 0; q < kNarrowCol; ++q) {
            t[q] = 0;
            if (q < nc) {
                const uint2 e = ent[q];
                t[q] = value(e);
                note(e, t[q]);
            }
        }
    }
    const uint64_t keep = zm & ~mask;
    z.zm = keep | newz;
    z.pm = (reinterpret_cast<const uint64_t *>(pp)[4] & ~blob_u64(bl, ox)) | newp;
    z.nm = (reinterpret_cast<const uint64_t *>(pp)[5] & ~blob_u64(bl, ox + 2)) | newn;
    // the unchanged rows, a 32-bit half at a time
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const uint32_t zh = (uint32_t)(zm >> (32 * h)), yh = (uint32_t)(z.zm >> (32 * h));
        const int32_t *src = vals + (h ? __popc((uint32_t)zm) : 0);
        int32_t *to = dst + (h ? __popc((uint32_t)z.zm) : 0);
        for (uint32_t x = (uint32_t)(keep >> (32 * h)); x; x &= x - 1u) {
            const uint32_t below = (x & (0u - x)) - 1u;
            const int32_t v = A * src[__popc(zh & below)];
            const uint32_t a = mag(v);
            om |= a;
            mn = min(mn, a - 1u);
            if (dst) to[__popc(yh & below)] = v;
        }
    }
    r.n = __popcll(z.zm);
    r.key = mask_key(bl, nv, z.pm, z.nm);
    r.om = om;
    // the gcd: 1 with an entry of magnitude 1; a power of two as the smallest
    // magnitude beside an odd entry; else by the entries, until it is 1
    uint32_t g = mn + 1u;
    if ((om & 1u) && (g & (g - 1u)) == 0u) g = 1u;
    const int piv = (int)(r.key & 63u);
    int32_t pv = 0;
    auto place = [&](const uint2 &e, int32_t x) {
        const int row = (int)(e.x & 63u);
        if (row == piv) pv = x;
        if (x != 0) {
            if (g != 1u) g = gcd_small(g, mag(x));
            if (dst) dst[value_at(z.zm, row)] = x;
        }
    };
    if (LONG) {
        for (int q = 0; q < nc; ++q) {
            const uint2 e = ent[q];
            place(e, value(e));
        }
    } else {
#pragma unroll
        for (int q = 0; q < kNarrowCol; ++q)
            if (q < nc) place(ent[q], t[q]);
    }
    if (g != 1u)
        for (uint64_t x = keep; x && g != 1u; x &= x - 1) g = gcd_small(g, mag(A * vals[value_at(zm, __ffsll((long long)x) - 1)]));
    if (r.key < kFluxKey && ((keep >> piv) & 1ull)) pv = A * vals[value_at(zm, piv)];
    r.pv = pv;
    r.g = g;
    r.zflux = false;
    if (dst)
        for (int i = r.n; i & 3; ++i) dst[i] = 0;
}

__device__ __noinline__ void narrow_child_long(const NetView &nv, const uint32_t *bl, const uint4 *pp, int32_t A,
                                               int32_t C, int cb, int nc, int k, int32_t *dst, Child &r, NarrowMasks &z)
{
    narrow_child<true>(nv, bl, pp, A, C, cb, nc, k, dst, r, z);
}

// gcd and exact division of the children below: most are there for a common
// divisor and fit 32 bits, where both take a fraction of the 64-bit time (one
// such child holds up a small level)
__device__ __forceinline__ uint64_t gcd_any(uint64_t g, uint64_t x)
{
    if (g == 1ull) return 1ull;
    return (g | x) >> 32 ? gcd64(g, x) : (uint64_t)gcd32((uint32_t)g, (uint32_t)x);
}

__device__ __forceinline__ int32_t div_any(int64_t t, uint64_t g)
{
    if (g == 1ull) return (int32_t)t;
    if (g < (1ull << 31) && t == (int64_t)(int32_t)t) return (int32_t)t / (int32_t)g;
    return (int32_t)(t / (int64_t)g);
}

// does x / g leave int32?
__device__ __forceinline__ bool past_int32(uint64_t x, uint64_t g) { return x > 2147483647ull && x / g > 2147483647ull; }

// gcd over a warp (g: 0 for a lane without an entry).  Mostly small numbers that
// share a small divisor: Euclid against the smallest, all lanes at once, ends
// after a step or two.
__device__ __forceinline__ uint64_t warp_gcd(uint64_t g)
{
    if (__any_sync(FULL, (g >> 32) != 0)) {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) g = gcd64(g, __shfl_xor_sync(FULL, g, off));
        return g;
    }
    uint32_t x = (uint32_t)g;
    for (;;) {
        const uint32_t m = __reduce_min_sync(FULL, x - 1u) + 1u;  // (less one: no entry counts as the largest)
        if (m == 1u) return 1ull;
        const uint32_t rest = x % m;
        if (!__any_sync(FULL, rest != 0u)) return m;
        x = rest ? rest : (x ? m : 0u);
    }
}

__device__ __forceinline__ uint64_t warp_sum(uint64_t x)
{
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) x += __shfl_xor_sync(FULL, x, off);
    return x;
}

// Any child of a narrow network, in 64 bits, by one warp: lane l holds rows l
// and l + 32 (see wide_child).
__device__ __forceinline__ void wide_narrow(const NetView &nv, const uint32_t *bl, const uint4 *pp, int32_t A, int32_t C,
                                         int cb, int k, int32_t *dst, Child &r, NarrowMasks &z, int lane)
{
    const uint64_t zm = reinterpret_cast<const uint64_t *>(pp)[1];
    const int32_t *vals = reinterpret_cast<const int32_t *>(pp + 3);
    const uint2 *ent = reinterpret_cast<const uint2 *>(bl + nv.o_nent) + cb;
    const uint64_t mask = blob_u64(bl, nv.o_colx + 10 * k + 4);
    int64_t t[2];
    uint64_t g = 0;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int row = lane + 32 * h;
        t[h] = 0;
        if ((zm >> row) & 1ull) t[h] = (int64_t)A * vals[value_at(zm, row)];
        if ((mask >> row) & 1ull) t[h] += (int64_t)C * (int32_t)ent[value_at(mask, row)].y;  // (rows ascend in the column)
        g = gcd_any(g, abs64(t[h]));
    }
    r.n = 0;
    r.key = kPadKey;
    r.pv = 0;
    r.om = 0;
    r.rh = 0;
    r.g = 1;
    r.zflux = r.ovf = false;
    z.zm = z.pm = z.nm = 0;
    if (!__any_sync(FULL, g != 0)) return;  // balanced (key stays kPadKey)
    g = warp_gcd(g);
    if (__any_sync(FULL, past_int32(abs64(t[0]), g) || past_int32(abs64(t[1]), g))) {
        r.ovf = true;
        r.key = 0;
        return;
    }
    int32_t v[2];
    uint64_t pm = 0, nm = 0, rh = 0;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int row = lane + 32 * h;
        v[h] = div_any(t[h], g);
        z.zm |= (uint64_t)__ballot_sync(FULL, v[h] != 0) << (32 * h);
        if (v[h] == 0) continue;
        const uint32_t rk = bl[nv.o_rank + row];
        if (v[h] > 0) pm |= 1ull << (rk & 0xFFu);
        else nm |= 1ull << ((rk >> 8) & 0xFFu);
        rh += (uint64_t)(int64_t)v[h] * row_hash(row);
    }
    r.om = __reduce_or_sync(FULL, mag(v[0]) | mag(v[1]));
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        z.pm |= (uint64_t)__reduce_or_sync(FULL, (uint32_t)(pm >> (32 * h))) << (32 * h);
        z.nm |= (uint64_t)__reduce_or_sync(FULL, (uint32_t)(nm >> (32 * h))) << (32 * h);
    }
    r.rh = warp_sum(rh);
    r.n = __popcll(z.zm);
    r.key = mask_key(bl, nv, z.pm, z.nm);
    const int piv = (int)(r.key & 63u);
    r.pv = __shfl_sync(FULL, piv < 32 ? v[0] : v[1], piv & 31);
    if (dst) {
#pragma unroll
        for (int h = 0; h < 2; ++h)
            if (v[h] != 0) dst[value_at(z.zm, lane + 32 * h)] = v[h];
        if (lane < ((4 - r.n) & 3)) dst[r.n + lane] = 0;
    }
}

// The same by one lane (see slow_child).
__device__ __noinline__ void slow_narrow(const NetView &nv, const uint32_t *bl, const uint4 *pp, int32_t A, int32_t C,
                                         int cb, int ce, int k, int32_t *dst, Child &r, NarrowMasks &z)
{
    const uint64_t zm = reinterpret_cast<const uint64_t *>(pp)[1];
    const int32_t *vals = reinterpret_cast<const int32_t *>(pp + 3);
    const uint2 *ent = reinterpret_cast<const uint2 *>(bl + nv.o_nent);
    const uint64_t mask = blob_u64(bl, nv.o_colx + 10 * k + 4);
    uint64_t g = 0, mx = 0;
    r.n = 0;
    r.key = kPadKey;
    r.pv = 0;
    r.om = 0;
    r.rh = 0;
    r.zflux = r.ovf = false;
    z.zm = z.pm = z.nm = 0;
    for (int pass = 0; pass < 2; ++pass) {
        int q = cb;  // rows ascend in the column and in the state
        for (uint64_t x = zm | mask; x; x &= x - 1) {
            const int row = __ffsll((long long)x) - 1;
            int64_t t = 0;
            if ((zm >> row) & 1ull) t = (int64_t)A * vals[value_at(zm, row)];
            while (q < ce && (int)(ent[q].x & 63u) < row) ++q;
            if (q < ce && (int)(ent[q].x & 63u) == row) t += (int64_t)C * (int32_t)ent[q].y;
            if (t == 0) continue;
            if (pass == 0) {
                const uint64_t at = abs64(t);
                g = gcd_any(g, at);
                mx = at > mx ? at : mx;
                continue;
            }
            const int32_t v = div_any(t, g);
            const uint32_t kk = bl[(v > 0 ? nv.o_keypos : nv.o_keyneg) + row];
            const uint32_t rk = bl[nv.o_rank + row];
            z.zm |= 1ull << row;
            if (v > 0) z.pm |= 1ull << (rk & 0xFFu);
            else z.nm |= 1ull << ((rk >> 8) & 0xFFu);
            r.om |= mag(v);
            r.rh += (uint64_t)(int64_t)v * row_hash(row);
            if (kk < r.key) {
                r.key = kk;
                r.pv = v;
            }
            if (dst) dst[r.n] = v;
            ++r.n;
        }
        if (pass == 0) {
            if (g == 0) return;  // balanced (key stays kPadKey)
            if (past_int32(mx, g)) {
                r.ovf = true;
                r.key = 0;
                return;
            }
        }
    }
    r.g = 1;
    if (dst)
        for (int i = r.n; i & 3; ++i) dst[i] = 0;
}

// payload units of n entries (values on narrow networks)
template <int F>
__device__ __forceinline__ int entry_units(int n)
{
    return F == 2 ? (n + 3) >> 2 : (n + 1) >> 1;
}

// Any child, by one warp: the entries in 64 bits, a lane each; the gcd and the
// range over all of them, then the divided entries.  For the child that may
// leave int32, shares a divisor, or has more entries than a lane of the
// generate pass takes: rare where reactions have a few metabolites, every
// child where they have dozens.
template <bool SUB>
__device__ __forceinline__ void wide_child(const NetView &nv, const uint32_t *bl, const uint4 *pe, int np, int32_t A,
                                        int32_t C, int cb, int ce, int k, uint4 *dst, Child &r, int lane)
{
    const int2 *p2 = reinterpret_cast<const int2 *>(pe);
    int2 *d2 = reinterpret_cast<int2 *>(dst);
    const int nq = ce - cb + (SUB ? 1 : 0);  // at most 1024
    // the child's value at parent entry i; at: its place in the column (-1: none)
    auto parent_entry = [&](int i, int &row, int &at) -> int64_t {
        const int2 e = p2[i];
        row = e.x & 0xFFFF;
        int lo = 0, hi = nq;  // first column entry with a row >= row (they ascend)
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            int rq;
            int32_t vq;
            column_entry<SUB>(nv, bl, cb, ce, mid, k, rq, vq);
            if (rq < row) lo = mid + 1;
            else hi = mid;
        }
        int64_t t = (int64_t)A * e.y;
        at = -1;
        if (lo < nq) {
            int rq;
            int32_t vq;
            column_entry<SUB>(nv, bl, cb, ce, lo, k, rq, vq);
            if (rq == row) {
                t += (int64_t)C * vq;
                at = lo;
            }
        }
        return t;
    };
    uint32_t matched = 0;  // lane w: which of the column entries 32 w .. 32 w + 31 the parent has
    uint64_t g = 0, mx = 0;
    bool unbal = false, zflux = false;
    auto see = [&](int row, int64_t t) {
        if (SUB && row == nv.M + k && t <= 0) zflux = true;
        if (t == 0) return;
        const uint64_t at = abs64(t);
        g = gcd_any(g, at);
        mx = at > mx ? at : mx;
        if (!SUB || row < nv.M) unbal = true;
    };
    for (int i0 = 0; i0 < np; i0 += 32) {
        int row = 0, at = -1;
        if (i0 + lane < np) {
            const int64_t t = parent_entry(i0 + lane, row, at);
            see(row, t);
        }
        for (int w = 0; 32 * w < nq; ++w) {
            const uint32_t m = __reduce_or_sync(FULL, at >= 0 && (at >> 5) == w ? 1u << (at & 31) : 0u);
            if (lane == w) matched |= m;
        }
    }
    // the column entries that the parent does not have
    auto fresh = [&](int q0) -> bool {
        const uint32_t w = __shfl_sync(FULL, matched, q0 >> 5);
        return q0 + lane < nq && !((w >> lane) & 1u);
    };
    for (int q0 = 0; q0 < nq; q0 += 32)
        if (fresh(q0)) {
            int row;
            int32_t cv;
            column_entry<SUB>(nv, bl, cb, ce, q0 + lane, k, row, cv);
            see(row, (int64_t)C * cv);
        }
    r.n = 0;
    r.key = kPadKey;
    r.pv = 0;
    r.om = 0;
    r.rh = 0;
    r.g = 1;
    r.zflux = __any_sync(FULL, zflux);
    r.ovf = false;
    if (!__any_sync(FULL, unbal)) return;  // balanced (key stays kPadKey)
    g = warp_gcd(g);
    if (__any_sync(FULL, past_int32(mx, g))) {
        r.ovf = true;
        r.key = 0;
        return;
    }
    uint32_t key = kPadKey, om = 0;
    int32_t pv = 0;
    uint64_t rh = 0;
    int n = 0;
    auto put = [&](int row, int64_t t) {
        const unsigned m = __ballot_sync(FULL, t != 0);
        if (t != 0) {
            const int32_t v = div_any(t, g);
            const uint32_t kk = entry_key<SUB>(nv, bl, row, v > 0);
            om |= mag(v);
            rh += (uint64_t)(int64_t)v * row_hash(row);
            if (kk < key) {
                key = kk;
                pv = v;
            }
            if (d2) d2[n + __popc(m & ((1u << lane) - 1u))] = make_int2((int)kk, v);
        }
        n += __popc(m);
    };
    for (int i0 = 0; i0 < np; i0 += 32) {
        int row = 0, at;
        int64_t t = 0;
        if (i0 + lane < np) t = parent_entry(i0 + lane, row, at);
        put(row, t);
    }
    for (int q0 = 0; q0 < nq; q0 += 32) {
        int row = 0;
        int64_t t = 0;
        if (fresh(q0)) {
            int32_t cv;
            column_entry<SUB>(nv, bl, cb, ce, q0 + lane, k, row, cv);
            t = (int64_t)C * cv;
        }
        put(row, t);
    }
    r.n = n;
    r.key = __reduce_min_sync(FULL, key);
    r.pv = __shfl_sync(FULL, pv, __ffs((int)__ballot_sync(FULL, key == r.key)) - 1);  // (keys are distinct)
    r.om = __reduce_or_sync(FULL, om);
    r.rh = warp_sum(rh);
    if (d2 && lane == 0 && (n & 1)) d2[n] = make_int2((int)kPadKey, 0);
}

// The same by one lane: where many such children come to a warp, 32 chains side
// by side take less than 32 one after the other.
template <bool SUB>
__device__ __noinline__ void slow_child(const NetView &nv, const uint32_t *bl, const uint4 *pe, int np, int32_t A,
                                        int32_t C, int cb, int ce, int k, uint4 *dst, Child &r)
{
    const int2 *p2 = reinterpret_cast<const int2 *>(pe);
    int2 *d2 = reinterpret_cast<int2 *>(dst);
    const int nq = ce - cb + (SUB ? 1 : 0);
    uint32_t matched[(EFM_MAX_INTERNAL + 32) / 32];
    for (int i = 0; 32 * i < nq; ++i) matched[i] = 0;
    uint64_t g = 0, mx = 0;
    r.n = 0;
    r.key = kPadKey;
    r.pv = 0;
    r.om = 0;
    r.rh = 0;
    r.zflux = r.ovf = false;
    int nbal = 0;
    for (int pass = 0; pass < 2; ++pass) {
        auto take = [&](int row, int64_t t) {
            if (SUB && row == nv.M + k && t <= 0) r.zflux = true;
            if (t == 0) return;
            if (pass == 0) {
                const uint64_t at = abs64(t);
                g = gcd_any(g, at);
                mx = at > mx ? at : mx;
                if (!SUB || row < nv.M) ++nbal;
                return;
            }
            const int32_t v = div_any(t, g);
            const uint32_t kk = entry_key<SUB>(nv, bl, row, v > 0);
            r.om |= mag(v);
            r.rh += (uint64_t)(int64_t)v * row_hash(row);
            if (kk < r.key) {
                r.key = kk;
                r.pv = v;
            }
            if (d2) d2[r.n] = make_int2((int)kk, v);
            ++r.n;
        };
        for (int i = 0; i < np; ++i) {
            const int2 e = p2[i];
            const int row = e.x & 0xFFFF;
            int64_t t = (int64_t)A * e.y;
            int lo = 0, hi = nq;  // first column entry with a row >= row (they ascend)
            while (lo < hi) {
                const int mid = (lo + hi) >> 1;
                int rq;
                int32_t vq;
                column_entry<SUB>(nv, bl, cb, ce, mid, k, rq, vq);
                if (rq < row) lo = mid + 1;
                else hi = mid;
            }
            if (lo < nq) {
                int rq;
                int32_t vq;
                column_entry<SUB>(nv, bl, cb, ce, lo, k, rq, vq);
                if (rq == row) {
                    t += (int64_t)C * vq;
                    matched[lo >> 5] |= 1u << (lo & 31);
                }
            }
            take(row, t);
        }
        for (int q = 0; q < nq; ++q) {
            if ((matched[q >> 5] >> (q & 31)) & 1u) continue;
            int row;
            int32_t cv;
            column_entry<SUB>(nv, bl, cb, ce, q, k, row, cv);
            take(row, (int64_t)C * cv);
        }
        if (pass == 0) {
            if (nbal == 0) return;  // balanced (key stays kPadKey)
            if (past_int32(mx, g)) {
                r.ovf = true;
                r.key = 0;
                return;
            }
        }
    }
    r.g = 1;
    if (d2 && (r.n & 1)) d2[r.n] = make_int2((int)kPadKey, 0);
}

// ---------------------------------------------------------------------------
// first-K length-cap rules: rows touched by a support, as bitmaps over the
// internal rows (lane w of a warp holds word w; at most 1024 rows)
// ---------------------------------------------------------------------------

struct CapScratch {
    uint32_t pc[32], pp[32];  // rows the parent's columns consume / produce
    uint32_t cc[32], cp[32];  // the child's
    uint32_t u[EFM_MAX_COLUMNS / 32];  // columns of the parent
};

template <int F>
__device__ void cap_parent(const NetView &nv, const uint32_t *bl, CapScratch &s, const uint4 *pay, int pc, int lane)
{
    __syncwarp();
    s.pc[lane] = 0;
    s.pp[lane] = 0;
    for (int i = lane; i < EFM_MAX_COLUMNS / 32; i += 32) s.u[i] = 0;
    __syncwarp();
    const int n = F ? 128 : pc;
    for (int i = lane; i < n; i += 32) {
        int c = i;
        if (F) {
            if (!((reinterpret_cast<const uint64_t *>(pay)[2 + (i >> 6)] >> (i & 63)) & 1ull)) continue;
        } else {
            c = list_col(pay, i);
        }
        atomicOr(&s.u[c >> 5], 1u << (c & 31));
        for (int q = (int)bl[nv.o_colptr + c]; q < (int)bl[nv.o_colptr + c + 1]; ++q) {
            const uint32_t f = bl[nv.o_colent + q];
            const int r = ent_index(f);
            atomicOr(ent_coef(f) < 0 ? &s.pc[r >> 5] : &s.pp[r >> 5], 1u << (r & 31));
        }
    }
    __syncwarp();
}

// One child U + {k} (k < 0: U) of the parent in s: can a traversal with
// `room` (0 or 1) more columns still balance it?  A row that U touches with
// one sign only keeps its imbalance under secondary steps, so a child with
// such rows needs one more column that gives each of them the missing sign
// and finds the opposite sign in U for every row of its own (twin rule kept).
// The warp tries the columns able to fix the one-sided row with the shortest
// list.  False when the child can never balance.
__device__ bool cap_child(const NetView &nv, const uint32_t *bl, CapScratch &s, int k, int room, int lane)
{
    uint32_t c = s.pc[lane], p = s.pp[lane];
    if (k >= 0) {
        for (int q = (int)bl[nv.o_colptr + k]; q < (int)bl[nv.o_colptr + k + 1]; ++q) {
            const uint32_t f = bl[nv.o_colent + q];
            const int r = ent_index(f);
            if ((r >> 5) == lane) {
                if (ent_coef(f) < 0) c |= 1u << (r & 31);
                else p |= 1u << (r & 31);
            }
        }
    }
    const uint32_t x = c ^ p;  // one-sided rows of this lane's word
    const int nd = (int)__reduce_add_sync(FULL, (unsigned)__popc(x));
    if (nd == 0) return true;
    if (room == 0) return false;
    uint32_t pick = 0xFFFFFFFFu;  // list length << 20 | surplus << 19 | row
    for (uint32_t y = x; y; y &= y - 1) {
        const int b = __ffs((int)y) - 1;
        const int r = 32 * lane + b;
        const bool sur = (p >> b) & 1u;  // produced only: a surplus
        const int lp = (sur ? nv.o_consptr : nv.o_prodptr) + r;
        const uint32_t len = min(bl[lp + 1] - bl[lp], 4095u);
        const uint32_t cand = (len << 20) | (sur ? 1u << 19 : 0u) | (uint32_t)r;
        pick = cand < pick ? cand : pick;
    }
    pick = __reduce_min_sync(FULL, pick);
    __syncwarp();
    s.cc[lane] = c;
    s.cp[lane] = p;
    __syncwarp();
    const int r0 = (int)(pick & 0x7FFFFu);
    const bool sur0 = (pick >> 19) & 1u;
    const int lp0 = (sur0 ? nv.o_consptr : nv.o_prodptr) + r0;
    const int b0 = (int)bl[lp0], n0 = (int)bl[lp0 + 1] - b0;
    const int eo0 = sur0 ? nv.o_consent : nv.o_prodent;
    bool found = false;
    for (int i0 = 0; i0 < n0 && !found; i0 += 32) {
        bool ok = i0 + lane < n0;
        if (ok) {
            const int kc = ent_index(bl[eo0 + b0 + i0 + lane]);
            const int tw = (int)bl[nv.o_twin + kc];
            ok = !(tw >= 0 && (tw == k || ((s.u[tw >> 5] >> (tw & 31)) & 1u)));
            int hit = 0;
            for (int q = (int)bl[nv.o_colptr + kc]; ok && q < (int)bl[nv.o_colptr + kc + 1]; ++q) {
                const uint32_t f = bl[nv.o_colent + q];
                const int r = ent_index(f);
                const uint32_t wc = (s.cc[r >> 5] >> (r & 31)) & 1u, wp = (s.cp[r >> 5] >> (r & 31)) & 1u;
                // the column produces r: U must consume it, and the reverse
                ok = (ent_coef(f) > 0 ? wc : wp) != 0u;
                hit += (int)(wc ^ wp);
            }
            ok = ok && hit == nd;
        }
        found = __any_sync(FULL, ok);
    }
    return found;
}

// First-K bound, supports of equal size: does U + {k} come after the bound?
// The support holding the lowest column of their difference comes first.
struct BoundScratch {
    uint32_t bits[EFM_MAX_COLUMNS / 32];
    uint16_t cols[64];
    int n;
};

template <int F>
__device__ __noinline__ bool after_bound(const BoundScratch &b, const uint4 *pay, int pc, int k)
{
    if (F) {
        uint64_t u[2] = {reinterpret_cast<const uint64_t *>(pay)[2], reinterpret_cast<const uint64_t *>(pay)[3]};
        if (k >= 0) add_bit(u[0], u[1], k);
        for (int w = 0; w < 2; ++w) {
            const uint64_t d = u[w] ^ ((uint64_t)b.bits[2 * w] | ((uint64_t)b.bits[2 * w + 1] << 32));
            if (d) return (u[w] & (d & (~d + 1))) == 0;
        }
        return false;
    }
    int own = 0x7FFFFFFF;  // the lowest column of U + {k} outside the bound
    for (int i = 0; i < pc + (k >= 0 ? 1 : 0); ++i) {
        const int c = i < pc ? list_col(pay, i) : k;
        if (!((b.bits[c >> 5] >> (c & 31)) & 1u)) own = c < own ? c : own;
    }
    for (int j = 0; j < b.n; ++j) {  // ascending
        const int c = (int)b.cols[j];
        if (c > own) return false;
        bool in = c == k;
        for (int i = 0; i < pc && !in; ++i) in = list_col(pay, i) == c;
        if (!in) return true;
    }
    return false;
}

// the hashes and the support of a child U + {k} (k < 0: U)
template <int F>
__device__ __forceinline__ void write_support(uint4 *dst, const uint4 *pp, int pc, int k, uint64_t rh, uint64_t uh,
                                              const NarrowMasks &z)
{
    if (F) {
        uint64_t u0 = reinterpret_cast<const uint64_t *>(pp)[2], u1 = reinterpret_cast<const uint64_t *>(pp)[3];
        if (k >= 0) add_bit(u0, u1, k);
        const uint64_t s = F == 2 ? z.zm : 0ull;
        dst[0] = make_uint4((uint32_t)rh, (uint32_t)(rh >> 32), (uint32_t)s, (uint32_t)(s >> 32));
        dst[1] = make_uint4((uint32_t)u0, (uint32_t)(u0 >> 32), (uint32_t)u1, (uint32_t)(u1 >> 32));
        if (F == 2)
            dst[2] = make_uint4((uint32_t)z.pm, (uint32_t)(z.pm >> 32), (uint32_t)z.nm, (uint32_t)(z.nm >> 32));
    } else {
        dst[0] = make_uint4((uint32_t)rh, (uint32_t)(rh >> 32), (uint32_t)uh, (uint32_t)(uh >> 32));
        const int lu = sparse_list_units(pc);
        for (int t = 1; t < lu; ++t) dst[t] = pp[t];
        if (k >= 0) {
            if ((pc & 7) == 0) dst[lu] = make_uint4(~0u, ~0u, ~0u, ~0u);
            reinterpret_cast<uint16_t *>(dst)[8 + pc] = (uint16_t)k;
        }
    }
}

// ---------------------------------------------------------------------------
// Generate: one (parent, branch) item per lane, 32 children of a warp at a
// time.  A lane writes its child straight to the row and the payload units
// reserved for it (two prefix sums, two counters); nothing waits on another
// child.  Children whose row or payload lies past the arena keep only their
// fingerprint (the level is then decided from fingerprints, or run again with
// a larger arena).
// ---------------------------------------------------------------------------
// One level by the warps worker = 0 .. nworkers-1: parents are arena rows
// (a.perm, or a.par_base on), cpw of them a warp and chunk; blk / pay_blk: rows
// and payload units a warp reserves at a time, at least a round's.  LONG: see
// NetView::long_cols.
template <int F, bool SUB, bool FK, bool LONG>
__device__ __forceinline__ void generate_range(const NetView &nv, const LevelArgs &a, int64_t n_par, int cpw, int blk,
                                               int pay_blk, bool any_result, int64_t worker, int64_t nworkers,
                                               CapScratch *cap, const BoundScratch &bound)
{
    const int lane = threadIdx.x & 31;
    const uint32_t *bl = nv.blob;
    const uint4 *scol = reinterpret_cast<const uint4 *>(bl + nv.o_scol);
    const int64_t row_cap = a.child.cap;
    const uint64_t pay_cap = a.child.pay_cap;
    unsigned n_exp = 0, n_pruned = 0, n_unwritten = 0, n_zero = 0;  // a lane's share of a launch
    bool fatal = false;
    // this warp's reserved rows and payload units (large levels: several
    // rounds' worth at a time, so that the two counters are not the limit)
    uint64_t row_next = 0, pay_next = 0;
    int row_left = 0, pay_left = 0;
    const int64_t wstride = nworkers * cpw;
    // the lane's parent of a chunk: its row, payload offset and meta word
    auto parent_at = [&](int64_t p0, uint32_t &pid, uint32_t &off, uint32_t &meta) {
        const int64_t pl = p0 + lane;
        const bool pin = lane < cpw && pl < n_par;
        pid = pin ? (uint32_t)(a.perm ? (int64_t)a.perm[pl] : a.par_base + pl) : 0u;
        off = meta = 0u;
        if (pin) {
            const uint2 h = *reinterpret_cast<const uint2 *>(a.par.hdr + pid);
            off = h.x;
            meta = h.y;
        }
    };
    uint32_t pid_n, off_n, meta_n;  // the next chunk's, read one chunk ahead
    parent_at(worker * cpw, pid_n, off_n, meta_n);
    for (int64_t p0 = worker * cpw; p0 < n_par; p0 += wstride) {
        const uint32_t pid = pid_n, mj = meta_n;
        parent_at(p0 + wstride, pid_n, off_n, meta_n);
        int dj = (int)((mj >> 10) & 0x1FFFu);
        // first-K: a parent larger than the bound has no descendant among the K smallest
        if (FK && a.fk_pc > 0 && (int)((mj >> 23) & 0x7Fu) > a.fk_pc) dj = 0;
        int incl = dj;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const int x = __shfl_up_sync(FULL, incl, off);
            if (lane >= off) incl += x;
        }
        const int prej = incl - dj;
        const int T = __shfl_sync(FULL, incl, 31);
        if (T > 32 * nv.N) {
            if (lane == 0) record_diag(a.ctr, ERR_BOUNDS, 3, T, 32 * nv.N, a.level);
            fatal = true;
        }
        uint32_t cap_for = kNoRecord;  // payload offset of the parent in s_cap
        for (int base = 0; base < T; base += 32) {
            if (__any_sync(FULL, fatal)) break;
            // pull the next chunk's payloads toward L2 (its headers
            // have arrived by the last round of this one)
            // (the second line of a payload may lie past the pool's end)
            if (base + 32 >= T && meta_n != 0u) {
                prefetch_l2(a.par.pay + off_n);
                if ((uint64_t)off_n + 6 < a.par.pay_cap) prefetch_l2(a.par.pay + off_n + 6);
            }
            // --- branch selection: one (parent, branch) item per lane ---
            const int c = base + lane;
            int j = 0;  // largest j with pre_j <= c
#pragma unroll
            for (int step = 16; step > 0; step >>= 1) {
                const int v = __shfl_sync(FULL, prej, j + step);
                if (v <= c) j += step;
            }
            const uint32_t pj = __shfl_sync(FULL, pid, j);
            const int q = c - __shfl_sync(FULL, prej, j);
            bool okl = c < T;
            int k = 0, pc = 0, np = 0, cb = 0, ce = 0;
            bool in_u = false, fits = true, opp = false;
            int32_t A = 1, C = 0;
            const uint4 *pp = a.par.pay;
            if (okl) {
                const uint4 hd = a.par.hdr[pj];
                pp += hd.x;
                pc = (int)((hd.y >> 23) & 0x7Fu);
                np = (int)(hd.z & 0x7FFu);
                const int mb = (int)((hd.z >> 11) & 0x1Fu);
                const int32_t bi = (int32_t)hd.w;
                const int piv = (int)(hd.y & 0x3FFu);
                const bool fwd = bi > 0;  // forward flow: consume the surplus
                const uint32_t abi = mag(bi);
                const int pr = piv < nv.M ? piv : 0;
                const int lptr = (fwd ? nv.o_consptr : nv.o_prodptr) + pr;
                const int lb = (int)bl[lptr], ln = (int)bl[lptr + 1] - lb;
                // subtractive variant: after the side list, the opposite list
                // (Eq. 5: less flux on a column of U that moves i the same way)
                const int optr = (fwd ? nv.o_prodptr : nv.o_consptr) + pr;
                const int on = SUB ? (int)bl[optr + 1] - (int)bl[optr] : 0;
                if (piv >= nv.M || bi == 0 || np == 0 || q >= ln + on) {
                    record_diag(a.ctr, ERR_BOUNDS, 1 + (piv >= nv.M ? 10 : 0) + (bi == 0 ? 100 : 0), (long long)q,
                                (long long)(ln + on), a.level);
                    fatal = true;
                    okl = false;
                } else {
                    opp = SUB && q >= ln;
                    const uint32_t br = opp ? bl[(fwd ? nv.o_prodent : nv.o_consent) + (int)bl[optr] + (q - ln)]
                                            : bl[(fwd ? nv.o_consent : nv.o_prodent) + lb + q];
                    k = ent_index(br);
                    const uint32_t sik = (uint32_t)ent_coef(br);  // |S_ik|
                    const uint4 s1 = scol[2 * k + 1];
                    cb = (int)s1.y;
                    ce = (int)s1.z;
                    const uint32_t tw = s1.w;  // ~0: no twin (matches no column)
                    bool twin = false;
                    if (F) {
                        const uint32_t *u = reinterpret_cast<const uint32_t *>(pp + 1);  // the bitset
                        in_u = (u[k >> 5] >> (k & 31)) & 1u;
                        twin = tw != 0xFFFFFFFFu && ((u[tw >> 5] >> (tw & 31u)) & 1u);
                    } else {
                        auto look = [&](uint32_t w) {
                            const uint32_t c0 = w & 0xFFFFu, c1 = w >> 16;
                            in_u = in_u || c0 == (uint32_t)k || c1 == (uint32_t)k;
                            twin = twin || c0 == tw || c1 == tw;
                        };
                        const int lu = sparse_list_units(pc);
                        for (int t = 1; t < lu; ++t) {
                            const uint4 u = pp[t];
                            look(u.x);
                            look(u.y);
                            look(u.z);
                            look(u.w);
                        }
                    }
                    const int sec = a.level - pc;
                    if (opp)
                        okl = in_u && sec + 1 <= a.max_sec;
                    else
                        okl = !twin && (in_u ? sec + 1 <= a.max_sec : pc + 1 <= a.max_len);
                    if (FK && okl && a.fk_pc > 0) {
                        // branch and bound: the child's descendants keep its
                        // support or grow it, so a child past the K-th result
                        // found so far cannot yield one of the K smallest
                        const int pc2 = pc + (in_u ? 0 : 1);
                        okl = pc2 < a.fk_pc || (pc2 == a.fk_pc && !after_bound<F>(bound, pp, pc, in_u ? -1 : k));
                    }
                    const uint32_t g0 = (abi == 1u || sik == 1u) ? 1u : gcd32(abi, sik);
                    A = (int32_t)(sik / g0);
                    C = (int32_t)(abi / g0);
                    // no entry of the child can leave int32
                    fits = ((uint64_t)A << mb) + (uint64_t)(uint32_t)C * s1.x < 0x80000000ull;
                    if (opp) C = -C;  // Eq. 5: flux taken away from k
                }
            }
            if (okl) ++n_exp;
            const int pc2 = pc + (in_u ? 0 : 1);
            // superset rule: the new column completes a result accepted at an
            // earlier level (counted below, once the child is known to be one)
            bool pr = false;
            if (any_result && okl && !in_u)
                pr = F ? pruned_bits(a.cells, pp, k) : pruned_list(a.cells, a.rcols, pp, pc, k);
            // first-K length-cap rules.  dead: the child cannot balance any
            // more, unless it is balanced already (it then has no one-sided
            // row); skip: nor can its update leave int32, so nothing of it
            // needs to be computed
            bool dead = false, skip = false;
            if (FK) {
                const bool at_cap = okl && !pr && a.cap_dead && pc2 >= a.max_len;
                const bool below = okl && !pr && a.cap_dead && pc2 == a.max_len - 1;
                bool stuck = false;
                unsigned need = __ballot_sync(FULL, at_cap || below);
                const uint32_t hx = (uint32_t)(pp - a.par.pay);
                while (need) {
                    const int src = __ffs((int)need) - 1;
                    need &= need - 1;
                    const uint32_t ox = __shfl_sync(FULL, hx, src);
                    const int opc = __shfl_sync(FULL, pc, src);
                    const int okc = __shfl_sync(FULL, in_u ? -1 : k, src);
                    const int room = __shfl_sync(FULL, below ? 1 : 0, src);
                    if (ox != cap_for) {
                        cap_parent<F>(nv, bl, *cap, a.par.pay + ox, opc, lane);
                        cap_for = ox;
                    }
                    const bool can = cap_child(nv, bl, *cap, okc, room, lane);
                    if (lane == src) stuck = !can;
                }
                dead = stuck || (at_cap && a.level - pc2 + 1 >= a.max_sec);
                skip = stuck && fits;
            }
            // --- rows and payload units of the children of this round ---
            const bool wr = okl && !skip;
            const int su2 = support_units<F>(pc2);
            const int units = wr ? su2 + entry_units<F>(np + ce - cb + (SUB ? 1 : 0)) : 0;
            int usum = units;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const int x = __shfl_up_sync(FULL, usum, off);
                if (lane >= off) usum += x;
            }
            const unsigned wmask = __ballot_sync(FULL, wr);
            const int utot = __shfl_sync(FULL, usum, 31);
            const int rows = __popc(wmask), rank = __popc(wmask & ((1u << lane) - 1u));
            int old_n = rows;  // rows of this round taken from the block at hand
            uint64_t fresh = 0;
            int want_r = 0;
            if (row_left < rows || pay_left < utot) {  // warp-uniform
                want_r = row_left < rows ? max(rows - row_left, blk) : 0;
                const int want_p = pay_left < utot ? max(utot, pay_blk) : 0;
                unsigned long long got = 0;
                if (lane == 0 && want_r) got = atomicAdd(&a.ctr[C_WRITTEN], (unsigned long long)want_r);
                if (lane == 1 && want_p) got = atomicAdd(&a.ctr[C_PAY], (unsigned long long)want_p);
                fresh = __shfl_sync(FULL, got, 0);
                const uint64_t units_at = __shfl_sync(FULL, got, 1);
                if (want_r) old_n = row_left;
                if (want_p) {  // a round's payloads are contiguous: the rest of the old block stays unused
                    pay_next = units_at;
                    pay_left = want_p;
                }
            }
            const uint64_t idx = rank < old_n ? row_next + (uint64_t)rank : fresh + (uint64_t)(rank - old_n);
            if (old_n < rows) {
                row_next = fresh + (uint64_t)(rows - old_n);
                row_left = want_r - (rows - old_n);
            } else {
                row_next += (uint64_t)rows;
                row_left -= rows;
            }
            const uint64_t off = pay_next + (uint64_t)(usum - units);
            pay_next += (uint64_t)utot;
            pay_left -= utot;
            const bool room = wr && (int64_t)idx < row_cap && off + (uint64_t)units <= pay_cap;
            uint4 *dst = room ? a.child.pay + off : nullptr;
            // --- the child ---
            if (wr) {
                uint4 *de = dst ? dst + su2 : nullptr;
                uint64_t fp = kOpenFp | (uint64_t)pj | ((uint64_t)k << 32) | (in_u ? kOpenInU : 0ull) |
                              (opp ? kOpenSub : 0ull) | (pr ? kOpenPruned : 0ull) | (dead ? kOpenDead : 0ull);
                uint4 hd = make_uint4((uint32_t)off, 0u, 0u, 0u);  // an open child: where its payload may go
                // (what the parent and the column hold is read again where it is
                // needed, from L1, rather than kept in registers)
                const int nc = ce - cb + (SUB ? 1 : 0);
                const bool is_long = F == 2 ? nc > kNarrowCol : (np > 64 || nc > kListCol);
                if (fits && (LONG || !is_long)) {
                    Child m;
                    NarrowMasks z;
                    if (LONG && is_long) {  // (copies: what a call takes by reference lives in local memory)
                        Child lm;
                        NarrowMasks lz;
                        if (F == 2)
                            narrow_child_long(nv, bl, pp, A, C, cb, nc, k, reinterpret_cast<int32_t *>(de), lm, lz);
                        else
                            long_child<SUB>(nv, bl, pp + support_units<F>(pc), np, A, C, cb, ce, k, de, lm);
                        m = lm;
                        if (F == 2) z = lz;
                    } else if (F == 2) {
                        narrow_child(nv, bl, pp, A, C, cb, nc, k, reinterpret_cast<int32_t *>(de), m, z);
                    } else {
                        const uint4 s0 = scol[2 * k];
                        fast_child<SUB>(nv, bl, pp + support_units<F>(pc), np, A, C, cb, ce,
                                        (uint64_t)s0.z | ((uint64_t)s0.w << 32), k, de, m);
                    }
                    if (SUB && m.zflux) {
                        ++n_zero;
                        fp = kDeadFp;
                    } else if (m.key >= kFluxKey) {
                        fp |= kOpenBal;  // all metabolites stable
                    } else if (pr || dead) {
                        if (pr) ++n_pruned;
                        fp = kDeadFp;
                    } else if (m.g == 1u) {
                        const uint64_t rh = (uint64_t)(int64_t)A * *reinterpret_cast<const uint64_t *>(pp) +
                                            (uint64_t)(int64_t)C * *reinterpret_cast<const uint64_t *>(scol + 2 * k);
                        const uint64_t uh = support_hash_of<F>(pp, in_u ? -1 : k);
                        fp = state_fp(rh, uh);
                        if (dst) {
                            write_support<F>(dst, pp, pc, in_u ? -1 : k, rh, uh, z);
                            hd.y = pack_meta(branch_key(bl, nv, m.key, SUB ? 1 : 0), pc2);
                            hd.z = (uint32_t)m.n | ((uint32_t)max_bits(m.om) << 11);
                            hd.w = (uint32_t)m.pv;
                        } else {
                            ++n_unwritten;
                        }
                    }
                }
                if ((int64_t)idx < row_cap) {
                    // an open child's z: 1 when it has a payload
                    if (fp >> 63) hd = make_uint4(hd.x, 0u, dst ? 1u : 0u, 0u);
                    a.child.hdr[idx] = hd;
                }
                if ((int64_t)idx < a.fp_cap) {
                    a.fp[idx] = fp;
                    if ((fp >> 63) && fp != kDeadFp) a.open[atomicAdd(&a.ctr[C_OPEN], 1ull)] = (uint32_t)idx;
                } else {
                    record_diag(a.ctr, ERR_BOUNDS, 7, (long long)idx, a.fp_cap, a.level);
                    fatal = true;
                }
            }
        }
        if (__any_sync(FULL, fatal)) break;
    }
    // rows reserved but not used: no fingerprint (the dedup pass skips them) and
    // no branches (the next level reads every row of the arena)
    for (int x = lane; x < row_left; x += 32) {
        const int64_t r = (int64_t)row_next + x;
        if (r < a.fp_cap) a.fp[r] = kDeadFp;
        if (r < row_cap) a.child.hdr[r] = make_uint4(0u, 0u, 0u, 0u);
    }
    // one atomic per warp and counter
    auto total = [&](unsigned v, int id) {
        const unsigned s = __reduce_add_sync(FULL, v);
        if (lane == 0 && s) atomicAdd(&a.ctr[id], (unsigned long long)s);
    };
    total(n_exp, C_EXP);
    total(n_pruned, C_PRUNED);
    total(n_unwritten, C_UNWRITTEN);
    total(n_zero, C_ZERO);
}

// ---------------------------------------------------------------------------
// Dedup: one thread per reserved row; the first row of every distinct state
// survives in place, a later copy gets a zero meta word (no branches).
// ---------------------------------------------------------------------------

// The same support and the same entries (both in any order)?  One warp; the
// payloads at px and py, |U| = pc, n entries.
template <int F>
__device__ bool same_state(const uint4 *px, const uint4 *py, int pc, int n, int lane)
{
    bool same = true;
    if (F == 2) {  // masks and values: unit by unit
        for (int i = lane; i < 3 + entry_units<F>(n); i += 32) {
            const uint4 x = __ldcg(px + i), y = __ldcg(py + i);
            same = same && x.x == y.x && x.y == y.y && x.z == y.z && x.w == y.w;
        }
        return __all_sync(FULL, same);
    }
    if (F) {
        const uint4 x = __ldcg(px + 1), y = __ldcg(py + 1);
        same = x.x == y.x && x.y == y.y && x.z == y.z && x.w == y.w;
    } else {
        const uint16_t *xl = reinterpret_cast<const uint16_t *>(px) + 8, *yl = reinterpret_cast<const uint16_t *>(py) + 8;
        for (int i = lane; i < 64; i += 32) {
            const int c = i < pc ? (int)__ldcg(xl + i) : -1;
            bool in = i >= pc;
            for (int j = 0; j < pc; ++j) in = in || (int)__ldcg(yl + j) == c;
            same = same && in;
        }
    }
    const int2 *xe = reinterpret_cast<const int2 *>(px + support_units<F>(pc));
    const int2 *ye = reinterpret_cast<const int2 *>(py + support_units<F>(pc));
    for (int i = lane; i < n; i += 32) {
        const int2 e = __ldcg(xe + i);
        bool in = false;
        for (int j = 0; j < n; ++j) {
            const int2 f = __ldcg(ye + j);
            in = in || (f.x == e.x && f.y == e.y);
        }
        same = same && in;
    }
    return __all_sync(FULL, same);
}

// An open child that balances, to the arbiter (one lane).
template <int F>
__device__ __noinline__ void finish_balanced(const NetView &nv, const LevelArgs &a, uint64_t f)
{
    const uint4 ph = a.par.hdr[(uint32_t)f];
    atomicAdd(&a.ctr[C_BAL], 1ull);
    insert_candidate<F>(a, nv.W, a.par.pay + ph.x, (int)((ph.y >> 23) & 0x7Fu),
                        (f & kOpenInU) ? -1 : (int)((f >> 32) & 0xFFFu));  // (a failure sets the error word)
}

// What any other open child needs: its parent, and A and C from the pivot's
// entry and the coefficient of k in the pivot's row.
struct OpenChild {
    const uint4 *pp;
    int pc, np, k, cb, ce;
    bool in_u;
    int32_t A, C;
};

__device__ __forceinline__ OpenChild open_child(const NetView &nv, const LevelArgs &a, uint64_t f)
{
    const uint32_t *bl = nv.blob;
    const uint4 ph = a.par.hdr[(uint32_t)f];
    OpenChild o;
    o.pp = a.par.pay + ph.x;
    o.pc = (int)((ph.y >> 23) & 0x7Fu);
    o.np = (int)(ph.z & 0x7FFu);
    o.k = (int)((f >> 32) & 0xFFFu);
    o.in_u = (f & kOpenInU) != 0;
    o.cb = (int)bl[nv.o_colptr + o.k];
    o.ce = (int)bl[nv.o_colptr + o.k + 1];
    const int piv = (int)(ph.y & 0x3FFu);
    const uint32_t sik =
        mag(reinterpret_cast<const int32_t *>(bl + nv.o_dcols)[(size_t)o.k * nv.Mpad + piv]);
    const uint32_t abi = mag((int32_t)ph.w), g0 = abi == 1u || sik == 1u ? 1u : gcd_small(abi, sik);
    o.A = (int32_t)(sik / g0);
    o.C = (f & kOpenSub) ? -(int32_t)(abi / g0) : (int32_t)(abi / g0);
    return o;
}

// Reserved row i's payload, if it has one, and its header cleared.
__device__ __forceinline__ uint4 *open_payload(const LevelArgs &a, uint64_t i, uint32_t &off)
{
    const uint4 h = i < (uint64_t)a.child.cap ? a.child.hdr[i] : make_uint4(0u, 0u, 0u, 0u);
    off = h.x;
    return h.z ? a.child.pay + h.x : nullptr;
}

template <bool SUB>
__device__ __forceinline__ uint4 child_header(const NetView &nv, uint32_t off, const Child &m, int pc)
{
    return make_uint4(off, pack_meta(branch_key(nv.blob, nv, m.key, SUB ? 1 : 0), pc),
                      (uint32_t)m.n | ((uint32_t)max_bits(m.om) << 11), (uint32_t)m.pv);
}

// Any other open child, of reserved row i, by one warp (WARP) or one lane: one
// whose update needs 64 bits, a division or more entries than the generate pass
// takes.  Returns its fingerprint (kDeadFp: none) and its
// header; live rows without a payload count as unwritten.
template <int F, bool SUB, bool WARP>
__device__ __noinline__ uint64_t finish_open(const NetView &nv, const LevelArgs &a, uint64_t f, uint64_t i, uint4 &h,
                                             int lane)
{
    const uint32_t *bl = nv.blob;
    const OpenChild o = open_child(nv, a, f);
    const int pc2 = o.pc + (o.in_u ? 0 : 1), k2 = o.in_u ? -1 : o.k;
    uint32_t off;
    uint4 *dst = open_payload(a, i, off);
    uint4 *de = dst ? dst + support_units<F>(pc2) : nullptr;
    h = make_uint4(0u, 0u, 0u, 0u);
    Child m;
    NarrowMasks z;
    const bool one = !WARP || lane == 0;
    if (!WARP && F == 2)
        slow_narrow(nv, bl, o.pp, o.A, o.C, o.cb, o.ce, o.k, reinterpret_cast<int32_t *>(de), m, z);
    else if (!WARP)
        slow_child<SUB>(nv, bl, o.pp + support_units<F>(o.pc), o.np, o.A, o.C, o.cb, o.ce, o.k, de, m);
    else if (F == 2)
        wide_narrow(nv, bl, o.pp, o.A, o.C, o.cb, o.k, reinterpret_cast<int32_t *>(de), m, z, lane);
    else
        wide_child<SUB>(nv, bl, o.pp + support_units<F>(o.pc), o.np, o.A, o.C, o.cb, o.ce, o.k, de, m, lane);
    if (SUB && m.zflux) {
        if (one) atomicAdd(&a.ctr[C_ZERO], 1ull);
        return kDeadFp;
    }
    if (m.key >= kFluxKey) {
        if (one) finish_balanced<F>(nv, a, f);
        return kDeadFp;
    }
    if (m.ovf) {
        if (one) atomicAdd(&a.ctr[C_OVF], 1ull);
        return kDeadFp;
    }
    if (f & (kOpenPruned | kOpenDead)) {
        if (one && (f & kOpenPruned)) atomicAdd(&a.ctr[C_PRUNED], 1ull);
        return kDeadFp;
    }
    const uint64_t uh = support_hash_of<F>(o.pp, k2);
    if (dst) {
        h = child_header<SUB>(nv, off, m, pc2);
        if (one) {
            write_support<F>(dst, o.pp, o.pc, k2, m.rh, uh, z);
            a.child.hdr[i] = h;
        }
    } else if (one) {
        atomicAdd(&a.ctr[C_UNWRITTEN], 1ull);
    }
    __threadfence();  // the row is complete before its slot is taken
    if (WARP) __syncwarp();
    return state_fp(m.rh, uh);
}

// Open children that a warp takes one after the other; more go to a lane each.
// With 0, 2, 4, 8, 16: the smallest query 0.684, 0.665, 0.663, 0.686, 0.731 ms,
// subtractive 5.16, 4.57, 4.56, 4.55, 4.55, a 400-row network 3.51, 3.28, 3.28,
// 3.28, 3.27, six targets of a 200-row network of even coefficients at 2^18 5.37,
// 4.81, 4.59, 4.55, 4.91; with all of them by warps a batch of 64 networks of 12
// rows took 3.5, by lanes 2.4.
constexpr uint64_t kWarpOpen = 4;

struct DedupSums {
    unsigned keep = 0, unv = 0;
    // the kept states' branches, and their payload units << 32: a lane takes at
    // most 2^32 / (1216 CTAs x 256) rows of 8191 branches, a warp's sum fits 32 bits
    unsigned long long deg_units = 0;
};

// Insert a warp's rows (lane: row i, fingerprint f, kDeadFp for none, header
// h) into the level's table.
template <int F>
__device__ __forceinline__ void dedup_insert(const LevelArgs &a, uint64_t mask, uint64_t i, uint64_t f, const uint4 &h,
                                             int lane, DedupSums &sum)
{
    const uint64_t row_cap = (uint64_t)a.child.cap;
    bool todo = f != kDeadFp;
    uint64_t pos = 0, probe = 0;
    uint32_t tag = 0;
    slot_tag_pos(f, mask, pos, tag);
    if (todo && i >= 0xFFFFFFFEull) {
        record_diag(a.ctr, ERR_BOUNDS, 10, (long long)i, 0xFFFFFFFEll, a.level);
        todo = false;
    }
    const bool written = h.y != 0u;
    while (__any_sync(FULL, todo)) {
        bool cmp = false;
        uint32_t ox = 0;
        while (todo && !cmp) {
            const unsigned long long v = atomicCAS(&a.slots[pos], kEmpty, ((unsigned long long)tag << 32) | i);
            if (v == kEmpty) {  // first of its state
                if (written) {
                    ++sum.keep;
                    const int u = support_units<F>((int)((h.y >> 23) & 0x7Fu)) + entry_units<F>((int)(h.z & 0x7FFu));
                    sum.deg_units += ((h.y >> 10) & 0x1FFFu) | (unsigned long long)u << 32;
                } else {
                    ++sum.unv;
                }
                todo = false;
                break;
            }
            if ((uint32_t)(v >> 32) == tag) {
                const uint64_t jrow = (uint32_t)v;
                // (a row that holds a slot is never cleared)
                uint4 o = make_uint4(0u, 0u, 0u, 0u);
                if (jrow < row_cap) o = __ldcg(a.child.hdr + jrow);
                // a row without its state written cannot be compared: the
                // level is then decided from the lower bound, or run again
                if (!written || o.y == 0u) {
                    if (written) a.child.hdr[i].y = 0u;
                    todo = false;
                    break;
                }
                cmp = h.y == o.y && h.z == o.z && h.w == o.w &&
                      __ldcg(reinterpret_cast<const uint64_t *>(a.child.pay + h.x)) ==
                          __ldcg(reinterpret_cast<const uint64_t *>(a.child.pay + o.x));  // row hashes
                ox = o.x;
                if (cmp) break;
            }
            pos = (pos + 1) & mask;
            if (++probe > mask) {
                record_diag(a.ctr, ERR_TABLE_FULL, 8, (long long)i, (long long)mask, a.level);
                todo = false;
            }
        }
        // the warp compares one pair at a time (a lane by itself would chain
        // n^2 loads)
        unsigned m = __ballot_sync(FULL, cmp);
        while (m) {
            const int src = __ffs((int)m) - 1;
            m &= m - 1;
            const uint32_t x = __shfl_sync(FULL, h.x, src), y = __shfl_sync(FULL, ox, src);
            const uint32_t hy = __shfl_sync(FULL, h.y, src), hz = __shfl_sync(FULL, h.z, src);
            const bool eq = same_state<F>(a.child.pay + x, a.child.pay + y, (int)((hy >> 23) & 0x7Fu),
                                          (int)(hz & 0x7FFu), lane);
            if (lane == src) {
                if (eq) {  // a later copy
                    a.child.hdr[i].y = 0u;
                    todo = false;
                } else {
                    pos = (pos + 1) & mask;
                    ++probe;
                }
            }
        }
    }
}

// The n_open open children and the rows [begin, end) by the warps whose first
// thread is number t0 of `stride` (open children: t_open).
template <int F, bool SUB>
__device__ __forceinline__ void dedup_range(const NetView &nv, const LevelArgs &a, uint64_t mask, uint64_t begin,
                                            uint64_t end, uint64_t n_open, uint64_t t0, uint64_t t_open,
                                            uint64_t stride, DedupSums &sum)
{
    const int lane = threadIdx.x & 31;
    end = end < (uint64_t)a.fp_cap ? end : (uint64_t)a.fp_cap;
    const uint64_t row_cap = (uint64_t)a.child.cap;
    // as many open children to a warp as there are for each, at most 32: the
    // balanced ones a lane each, the others by the warp, one after the other, or,
    // if they are more than a few, a lane each as well
    const uint64_t warps = stride >> 5;
    const uint64_t per = min((uint64_t)32, max((uint64_t)1, (n_open + warps - 1) / warps));
    for (uint64_t q0 = (t_open >> 5) * per; q0 < n_open; q0 += warps * per) {
        uint64_t i = 0, f = kDeadFp;
        uint4 h = make_uint4(0u, 0u, 0u, 0u);
        if ((uint64_t)lane < per && q0 + lane < n_open) {
            i = a.open[q0 + lane];
            f = a.fp[i];
            if (f & kOpenBal) {
                finish_balanced<F>(nv, a, f);
                f = kDeadFp;
                if (i < row_cap) a.child.hdr[i] = h;
            } else if (per > kWarpOpen) {
                uint4 hc;
                f = finish_open<F, SUB, false>(nv, a, f, i, hc, lane);
                h = hc;
                if (h.y == 0u && i < row_cap) a.child.hdr[i] = h;
            }
        }
        __syncwarp();
        for (unsigned m = per > kWarpOpen ? 0u : __ballot_sync(FULL, f != kDeadFp); m; m &= m - 1) {
            const int src = __ffs((int)m) - 1;
            const uint64_t row = __shfl_sync(FULL, i, src);
            uint4 hc;
            const uint64_t fc = finish_open<F, SUB, true>(nv, a, __shfl_sync(FULL, f, src), row, hc, lane);
            if (lane == src) {
                f = fc;
                h = hc;
                if (h.y == 0u && row < row_cap) a.child.hdr[row] = h;
            }
            __syncwarp();
        }
        dedup_insert<F>(a, mask, i, f, h, lane, sum);
    }
    for (uint64_t i0 = begin + t0; i0 < end; i0 += stride) {
        const uint64_t i = i0 + lane;
        uint64_t f = i < end ? a.fp[i] : kDeadFp;
        if (f >> 63) f = kDeadFp;  // nothing, or an open child
        uint4 h = make_uint4(0u, 0u, 0u, 0u);
        if (f != kDeadFp && i < row_cap) h = a.child.hdr[i];
        dedup_insert<F>(a, mask, i, f, h, lane, sum);
    }
}

// ---------------------------------------------------------------------------
// seeds (INIT) and seed sets (Prop. 1)
// ---------------------------------------------------------------------------

// Entries of a state in ascending rows, with what its header and masks need.
template <int F, bool SUB>
struct EntryWriter {
    const NetView &nv;
    const uint32_t *bl;
    uint4 *dst;
    int n = 0;
    uint32_t key = kPadKey, om = 0;
    int32_t pv = 0;
    uint64_t rh = 0;
    NarrowMasks z{0, 0, 0};
    __device__ EntryWriter(const NetView &nv_, const uint32_t *bl_, uint4 *dst_) : nv(nv_), bl(bl_), dst(dst_) {}
    __device__ void put(int row, int32_t v)
    {
        const uint32_t kk = entry_key<SUB>(nv, bl, row, v > 0);
        if (F == 2) {
            const uint32_t rk = bl[nv.o_rank + row];
            reinterpret_cast<int32_t *>(dst)[n] = v;
            z.zm |= 1ull << row;
            if (v > 0) z.pm |= 1ull << (rk & 0xFFu);
            else z.nm |= 1ull << ((rk >> 8) & 0xFFu);
        } else {
            reinterpret_cast<int2 *>(dst)[n] = make_int2((int)kk, v);
        }
        ++n;
        om |= mag(v);
        rh += (uint64_t)(int64_t)v * row_hash(row);
        if (kk < key) {
            key = kk;
            pv = v;
        }
    }
    __device__ void done()
    {
        if (F == 2)
            for (int i = n; i & 3; ++i) reinterpret_cast<int32_t *>(dst)[i] = 0;
        else if (n & 1)
            reinterpret_cast<int2 *>(dst)[n] = make_int2((int)kPadKey, 0);
    }
};

// One thread per seed column; seeds are distinct columns (no deduplication).
template <int F, bool SUB>
__device__ __forceinline__ void seed_range(const NetView &nv, const LevelArgs &a, int target, int tid, int nthreads)
{
    const uint32_t *bl = nv.blob;
    const int n_items = target >= 0 ? nv.metptr[target + 1] - nv.metptr[target] : nv.N;
    for (int it = tid; it < n_items; it += nthreads) {
        int k = it;
        if (target >= 0) {
            const uint32_t e = nv.metent[nv.metptr[target] + it];
            if (ent_coef(e) <= 0) continue;
            k = ent_index(e);
        }
        atomicAdd(&a.ctr[C_SEEDS], 1ull);
        // gcd of the column (with its flux 1 in the subtractive view)
        uint32_t g = SUB ? 1u : 0u;
        const int qb = (int)bl[nv.o_colptr + k], qe = (int)bl[nv.o_colptr + k + 1];
        for (int q = qb; q < qe; ++q) g = gcd32(g, mag(ent_coef(bl[nv.o_colent + q])));
        // the support {k}: an empty payload plus k
        const uint4 empty[2] = {make_uint4(0u, 0u, 0u, 0u), make_uint4(0u, 0u, 0u, 0u)};
        const uint64_t uh = support_hash_of<F>(empty, k);
        if (qb == qe) {
            atomicAdd(&a.ctr[C_BAL], 1ull);
            insert_candidate<F>(a, nv.W, empty, 0, k);
            continue;
        }
        const int n = qe - qb + (SUB ? 1 : 0);
        const int units = support_units<F>(1) + entry_units<F>(n);
        const uint64_t idx = atomicAdd(&a.ctr[C_NEXT], 1ull);
        const uint64_t off = atomicAdd(&a.ctr[C_PAY], (unsigned long long)units);
        if ((int64_t)idx >= a.child.cap) continue;
        if (off + (uint64_t)units > a.child.pay_cap) {
            record_diag(a.ctr, ERR_BOUNDS, 12, (long long)off, (long long)a.child.pay_cap, a.level);
            continue;
        }
        uint4 *dst = a.child.pay + off;
        if (F) {
            uint64_t u0 = 0, u1 = 0;
            add_bit(u0, u1, k);
            dst[1] = make_uint4((uint32_t)u0, (uint32_t)(u0 >> 32), (uint32_t)u1, (uint32_t)(u1 >> 32));
        } else {
            dst[1] = make_uint4((uint32_t)k | 0xFFFF0000u, ~0u, ~0u, ~0u);
        }
        EntryWriter<F, SUB> out(nv, bl, dst + support_units<F>(1));
        for (int q = 0; q < n; ++q) {
            int row;
            int32_t v;
            column_entry<SUB>(nv, bl, qb, qe, q, k, row, v);
            out.put(row, v / (int32_t)g);
        }
        out.done();
        const uint64_t s0 = F == 2 ? out.z.zm : (F ? 0ull : uh);
        dst[0] = make_uint4((uint32_t)out.rh, (uint32_t)(out.rh >> 32), (uint32_t)s0, (uint32_t)(s0 >> 32));
        if (F == 2)
            dst[2] = make_uint4((uint32_t)out.z.pm, (uint32_t)(out.z.pm >> 32), (uint32_t)out.z.nm, (uint32_t)(out.z.nm >> 32));
        const uint32_t key = out.key, om = out.om;
        const int32_t pv = out.pv;
        const uint32_t bkey = branch_key(bl, nv, key, SUB ? 1 : 0);
        a.child.hdr[idx] =
            make_uint4((uint32_t)off, pack_meta(bkey, 1), (uint32_t)n | ((uint32_t)max_bits(om) << 11), (uint32_t)pv);
        atomicAdd(&a.ctr[C_DEGSUM], (unsigned long long)(bkey >> 16));
    }
}

// one of a kernel's instances: form, subtractive view
#define EFM_FORM(KERNEL, CALL)                                                    \
    do {                                                                          \
        if (nv.form == 2) CALL((KERNEL<2, false>));                               \
        else if (nv.form == 1 && a.sub) CALL((KERNEL<1, true>));                  \
        else if (nv.form == 1) CALL((KERNEL<1, false>));                          \
        else if (a.sub) CALL((KERNEL<0, true>));                                  \
        else CALL((KERNEL<0, false>));                                            \
    } while (0)

}  // namespace
}  // namespace efm
