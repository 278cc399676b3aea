// efm_sparse.cu -- the traversal's level pass on sparse states.
//
// A state keeps only what it holds: the columns of its support and the
// unbalanced entries of its extra-flux row.  Most entries of a row are zero
// (a state of the 850-row genome-shaped network holds 8 to 19 unbalanced
// rows, one of the 58-row core-shaped network about 10), so the AND update
// EF' = A EF + C S_int[:, k] is a merge of two short sorted lists, and a
// state takes about 100 bytes instead of a support bitset and a full row.
//
// Measured against the dense rows it replaces (a group of 32 lanes per child,
// the whole row in registers: 1817 warp instructions a child, 3.5 KB written),
// one GB300, event to event: four genome-shaped targets at a 2^22 budget 362
// -> 45 ms, six targets of a 400-row network at 2^17 23.9 -> 5.3 ms, first-K
// = 1000 on three genome targets 103 -> 51 ms, the subtractive variant on the
// core-shaped network 12.1 -> 8.1 ms.  Networks of at most 64 rows keep their
// dense rows (efm_kernels.cu): there this pass is level with theirs at 2^21
// children and slower beyond (785 against 540 ms on the core-shaped network
// at a 2^26 budget).
//
// Layout (Arena::hdr and Arena::pay): one 16-byte header per row of the
// arena, and a payload in 16-byte units somewhere in the arena's pool:
//   header  x = payload offset in units, y = meta (0: the row carries no
//           state), z = entries | bits of max|EF| << 11, w = EF of the pivot
//   payload 8 bytes: sum of the columns' hash constants (mod 2^64);
//           the columns of U, ascending, 16 bits each, padded with 0xFFFF to
//           a unit; then the entries (row, value), ascending rows, 8 bytes
//           each, padded with zeros to a unit.
// Equal states have equal payloads, so two states are compared unit by unit.
// In the subtractive variant (Eq. 5) the entries go on with the flux of every
// column k of U at row M + k.
#include "efm_device.cuh"

namespace efm {
namespace {

constexpr int kGenWarps = 8;      // warps per CTA
constexpr int kNoRow = 0x7FFFFFFF;  // past the last entry of a list
constexpr uint32_t kPadCol = 0xFFFFu;

__device__ __forceinline__ uint64_t column_hash(int k) { return mix64(0x51ed27f3a5b1c3d9ull * (uint64_t)(k + 1)); }

__device__ __forceinline__ uint64_t state_fp(uint64_t rows, uint64_t cols)
{
    const uint64_t f = rows ^ mix64(cols + 0x632BE59BD9B4E019ull);
    return f == kDeadFp ? kDeadFp - 1 : f;
}

__device__ __forceinline__ uint64_t entry_hash(int row, int32_t v)
{
    uint64_t x = (((uint64_t)(uint32_t)row << 32) | (uint32_t)v) * 0x9E3779B97F4A7C15ull;
    x ^= x >> 32;
    return x * 0xD6E8FEB86659FD93ull;
}

// 16-bit column i of a payload's list
__device__ __forceinline__ int list_col(const uint4 *pay, int i)
{
    return reinterpret_cast<const uint16_t *>(pay)[4 + i];
}

__device__ __forceinline__ uint64_t list_hash(const uint4 *pay)
{
    return *reinterpret_cast<const uint64_t *>(pay);
}

__device__ __forceinline__ const int2 *entries_of(const uint4 *pay, int pc)
{
    return reinterpret_cast<const int2 *>(pay + sparse_list_units(pc));
}

__device__ __forceinline__ int max_bits(uint32_t om) { return om ? 32 - __clz((int)om) : 0; }

// ---------------------------------------------------------------------------
// balanced supports: the columns of a list (or none) plus column k (or none,
// k < 0) as the bitset words the arbiter reads
// ---------------------------------------------------------------------------

// word w of the bitset; pos walks the list (call with w = 0, 1, ...)
__device__ __forceinline__ uint64_t list_word(const uint4 *pay, int pc, int k, int w, int &pos)
{
    uint64_t x = 0;
    while (pos < pc) {
        const int c = list_col(pay, pos);
        if ((c >> 6) != w) break;
        x |= 1ull << (c & 63);
        ++pos;
    }
    if (k >= 0 && (k >> 6) == w) x |= 1ull << (k & 63);
    return x;
}

// Insert the support into the set of supports judged in this traversal (one
// thread); h: the sum of its columns' hash constants.
__device__ __noinline__ int insert_list(const LevelArgs &a, int W, const uint4 *pay, int pc, int k, uint64_t h)
{
    uint64_t p;
    uint32_t tag;
    slot_tag_pos(h, a.cslot_mask, p, tag);
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
            int pos = 0;
            for (int w = 0; w < W; ++w) dst[w] = list_word(pay, pc, k, w, pos);
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
            int pos = 0;
            for (int w = 0; w < W && eq; ++w) eq = __ldcg(src + w) == list_word(pay, pc, k, w, pos);
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

__device__ __forceinline__ uint64_t col_bit(int c) { return 1ull << ((uint32_t)(c * 0x9E3779B1u) >> 26); }

__device__ __forceinline__ uint32_t cell_slot(uint32_t key, uint32_t mask)
{
    uint32_t x = key * 0x85EBCA6Bu;
    x ^= x >> 15;
    x *= 0xC2B2AE35u;
    return (x ^ (x >> 13)) & mask;
}

// Does a result E with k in E lie inside U + {k}?  One lane.  The cells
// (k, s) of the sentinels s in U are looked up; a cell's results are tested
// by signature, then column by column.
__device__ __noinline__ bool pruned_cells(const CellIndex &ix, const uint16_t *rcols, const uint4 *pay, int pc, int k)
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
        // a list holds each result at most once: n_res bounds it
        for (int64_t n = 0; head != kNoRecord && n < ix.n_res; ++n) {
            const uint4 e = ix.ent[head];
            const uint64_t sig = (uint64_t)e.x | ((uint64_t)e.y << 32);
            if ((sig & ~su) == 0) {
                const uint16_t *lst = rcols + (size_t)e.w * kRcolStride;
                const int m = lst[0];
                bool sub = true;
                int q = 0;  // both lists ascend
                for (int j = 1; j <= m && sub; ++j) {
                    const int c = lst[j];
                    if (c == k) continue;
                    while (q < pc && list_col(pay, q) < c) ++q;
                    sub = q < pc && list_col(pay, q) == c;
                }
                if (sub) return true;
            }
            head = e.z;
        }
    }
    return false;
}

// ---------------------------------------------------------------------------
// the AND update as a merge of two ascending lists
// ---------------------------------------------------------------------------

// The entries of column k: S_int[:, k] and, in the subtractive view, flux 1
// on k at row M + k.
template <bool SUB>
struct ColumnIter {
    const uint32_t *ent;
    int q, end, row;
    int32_t val;
    int flux_row;
    __device__ __forceinline__ ColumnIter(const NetView &nv, const uint32_t *bl, int k)
        : ent(bl + nv.o_colent), q((int)bl[nv.o_colptr + k]), end((int)bl[nv.o_colptr + k + 1]), flux_row(nv.M + k)
    {
        load();
    }
    __device__ __forceinline__ void load()
    {
        if (q < end) {
            const uint32_t f = ent[q];
            row = ent_index(f);
            val = ent_coef(f);
        } else if (SUB && q == end) {
            row = flux_row;
            val = 1;
        } else {
            row = kNoRow;
            val = 0;
        }
    }
    __device__ __forceinline__ void next()
    {
        ++q;
        load();
    }
};

// What one pass over the child's entries finds.
struct Merged {
    int nnz, nbal;     // entries; entries of balance rows
    uint32_t key;      // pivot key of the balance rows
    int32_t pv;        // the pivot's entry
    uint64_t hash;
    uint32_t g, om;    // gcd and OR of the magnitudes (entries that fit int32)
    bool big, zflux;   // an entry left int32; a flux entry is not positive (Prop. 3)
};

// dst (null: nothing is written): where the entries go.
template <bool SUB>
__device__ __forceinline__ void merge_child(const NetView &nv, const uint32_t *bl, const int2 *pe, int np, int k,
                                            int32_t A, int32_t C, uint4 *dst, Merged &r)
{
    r.nnz = r.nbal = 0;
    r.key = 0xFFFFFFFFu;
    r.pv = 0;
    r.hash = 0;
    r.g = r.om = 0;
    r.big = r.zflux = false;
    ColumnIter<SUB> col(nv, bl, k);
    int2 e = pe[0];  // a state has at least one entry
    int pi = 1;
    int sx = 0, sy = 0;  // an entry waiting for its pair (16-byte stores)
    for (;;) {
        const int row = e.x < col.row ? e.x : col.row;
        if (row == kNoRow) break;
        int64_t t = 0;
        if (e.x == row) {
            t = (int64_t)A * e.y;
            e = pi < np ? pe[pi] : make_int2(kNoRow, 0);
            ++pi;
        }
        if (col.row == row) {
            t += (int64_t)C * col.val;
            col.next();
        }
        if (SUB && row >= nv.M && t <= 0) r.zflux = true;
        if (t == 0) continue;
        const int32_t v = (int32_t)t;
        const uint32_t av = (uint32_t)(v < 0 ? -v : v);
        if (t != (int64_t)v || v == INT32_MIN) {
            r.big = true;
        } else {
            r.om |= av;
            if (r.g != 1u) r.g = gcd32(r.g, av);
        }
        r.hash += entry_hash(row, v);
        if (!SUB || row < nv.M) {
            if (SUB) ++r.nbal;
            const uint32_t kk = bl[(t > 0 ? nv.o_keypos : nv.o_keyneg) + row];
            if (kk < r.key) {
                r.key = kk;
                r.pv = v;
            }
        }
        if (r.nnz & 1) {
            if (dst) dst[r.nnz >> 1] = make_uint4((uint32_t)sx, (uint32_t)sy, (uint32_t)row, (uint32_t)v);
        } else {
            sx = row;
            sy = v;
        }
        ++r.nnz;
    }
    if (dst && (r.nnz & 1)) dst[r.nnz >> 1] = make_uint4((uint32_t)sx, (uint32_t)sy, 0u, 0u);
    if (!SUB) r.nbal = r.nnz;
}

// The rare child whose entries share a divisor or leave int32 before the
// division: the gcd and the range in 64 bits, then the divided entries.
// Returns true when some entry stays outside int32 (the child is dropped).
template <bool SUB>
__device__ __noinline__ bool settle_child(const NetView &nv, const uint32_t *bl, const int2 *pe, int np, int k,
                                          int32_t A, int32_t C, uint4 *dst, Merged &r)
{
    uint64_t g = 0, mx = 0;
    for (int pass = 0; pass < 2; ++pass) {
        ColumnIter<SUB> col(nv, bl, k);
        int2 e = pe[0];
        int pi = 1, n = 0;
        int sx = 0, sy = 0;
        if (pass == 1) {
            if (g == 0 || mx / g > 2147483647ull) return true;
            r.hash = 0;
            r.om = 0;
        }
        for (;;) {
            const int row = e.x < col.row ? e.x : col.row;
            if (row == kNoRow) break;
            int64_t t = 0;
            if (e.x == row) {
                t = (int64_t)A * e.y;
                e = pi < np ? pe[pi] : make_int2(kNoRow, 0);
                ++pi;
            }
            if (col.row == row) {
                t += (int64_t)C * col.val;
                col.next();
            }
            if (t == 0) continue;
            if (pass == 0) {
                const uint64_t at = abs64(t);
                g = gcd64(g, at);
                mx = at > mx ? at : mx;
                continue;
            }
            const int32_t v = (int32_t)(t / (int64_t)g);
            r.om |= (uint32_t)(v < 0 ? -v : v);
            r.hash += entry_hash(row, v);
            if (row == (int)(r.key & 0xFFFFu)) r.pv = v;
            if (n & 1) {
                if (dst) dst[n >> 1] = make_uint4((uint32_t)sx, (uint32_t)sy, (uint32_t)row, (uint32_t)v);
            } else {
                sx = row;
                sy = v;
            }
            ++n;
        }
        if (pass == 1 && dst && (n & 1)) dst[n >> 1] = make_uint4((uint32_t)sx, (uint32_t)sy, 0u, 0u);
    }
    return false;
}

// The child's column list: the parent's, with k inserted at position ins
// (ins < 0: a secondary step, the same columns).
__device__ __forceinline__ void write_list(uint4 *dst, const uint4 *pp, int pc, int k, int ins, uint64_t uh)
{
    const int lu0 = sparse_list_units(pc);
    const int lu1 = sparse_list_units(pc + (ins >= 0 ? 1 : 0));
    const uint32_t *pw = reinterpret_cast<const uint32_t *>(pp) + 2;  // words of two columns
    const int nw0 = 4 * lu0 - 2;
    uint32_t prev = 0;
    auto word = [&](int w) -> uint32_t {
        const uint32_t x = w < nw0 ? pw[w] : 0xFFFFFFFFu;
        uint32_t y = x;
        if (ins >= 0) {
            if (2 * w > ins) y = __funnelshift_l(prev, x, 16);
            else if (2 * w == ins) y = (uint32_t)k | (x << 16);
            else if (2 * w + 1 == ins) y = (x & 0xFFFFu) | ((uint32_t)k << 16);
        }
        prev = x;
        return y;
    };
    {
        const uint32_t a = word(0), b = word(1);
        dst[0] = make_uint4((uint32_t)uh, (uint32_t)(uh >> 32), a, b);
    }
    for (int t = 1; t < lu1; ++t) {
        const int w = 4 * t - 2;
        const uint32_t a = word(w), b = word(w + 1), c = word(w + 2), d = word(w + 3);
        dst[t] = make_uint4(a, b, c, d);
    }
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

__device__ void cap_parent(const NetView &nv, const uint32_t *bl, CapScratch &s, const uint4 *pay, int pc, int lane)
{
    __syncwarp();
    s.pc[lane] = 0;
    s.pp[lane] = 0;
    for (int i = lane; i < EFM_MAX_COLUMNS / 32; i += 32) s.u[i] = 0;
    __syncwarp();
    for (int i = lane; i < pc; i += 32) {
        const int c = list_col(pay, i);
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
// list.  Sets *one_sided to the number of such rows; returns false when the
// child can never balance.
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
    uint32_t x = c ^ p;  // one-sided rows of this lane's word
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

// ---------------------------------------------------------------------------
// Generate: one (parent, branch) item per lane, 32 children of a warp at a
// time; a lane merges its parent's entries with column k's and writes its
// child straight to the place reserved for it (rows and payload units of the
// 32 children by one atomic each).  Nothing waits on another child.
// ---------------------------------------------------------------------------
template <bool SUB, bool FK>
__global__ void __launch_bounds__(kGenWarps * 32, 4) generate_sparse_kernel(NetView nv, LevelArgs a)
{
    __shared__ CapScratch s_cap[FK ? kGenWarps : 1];
    __shared__ uint16_t s_bound[FK ? 64 : 1];
    const int lane = threadIdx.x & 31;
    const int wid = threadIdx.x >> 5;
    const uint32_t *bl = nv.blob;
    const int64_t row_cap = a.child.cap;
    const uint64_t pay_cap = a.child.pay_cap;
    unsigned long long n_exp = 0, n_ovf = 0, n_bal = 0, n_pruned = 0, n_unwritten = 0, n_zero = 0;
    bool fatal = false;
    if (FK) {
        if (a.fk_pc > 0) {  // the bound's columns, ascending (warp 0, word by word)
            if (threadIdx.x == 0) {
                int n = 0;
                for (int w = 0; w < nv.W; ++w)
                    for (uint64_t x = a.fk_sup[w]; x && n < 64; x &= x - 1)
                        s_bound[n++] = (uint16_t)(w * 64 + __ffsll((long long)x) - 1);
            }
        }
        __syncthreads();
    }
    // this warp's reserved rows and payload units (large levels: several
    // rounds' worth at a time, so that the two counters are not the limit)
    uint64_t row_next = 0, pay_next = 0;
    int row_left = 0, pay_left = 0;
    const int cpw = a.cpw;
    const int64_t worker = (int64_t)blockIdx.x * kGenWarps + wid;
    const int64_t wstride = (int64_t)gridDim.x * kGenWarps * cpw;
    for (int64_t p0 = worker * cpw; p0 < a.n_par; p0 += wstride) {
        const int64_t pl = p0 + lane;
        const bool pin = lane < cpw && pl < a.n_par;
        uint4 hd = make_uint4(0u, 0u, 0u, 0u);
        if (pin) hd = a.par.hdr[a.perm ? (int64_t)a.perm[pl] : a.par_base + pl];
        int dj = (int)((hd.y >> 10) & 0x1FFFu);
        // first-K: a parent larger than the bound has no descendant among the K smallest
        if (FK && a.fk_pc > 0 && (int)((hd.y >> 23) & 0x7Fu) > a.fk_pc) dj = 0;
        int incl = dj;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const int x = __shfl_up_sync(FULL, incl, off);
            if (lane >= off) incl += x;
        }
        const int prej = incl - dj;
        const int T = __shfl_sync(FULL, incl, 31);
        if (T > 64 * nv.N) {
            if (lane == 0) record_diag(a.ctr, ERR_BOUNDS, 3, T, 64 * nv.N, a.level);
            fatal = true;
        }
        uint32_t cap_for = kNoRecord;  // payload offset of the parent in s_cap
        for (int base = 0; base < T; base += 32) {
            if (__any_sync(FULL, fatal)) break;
            // --- branch selection: one (parent, branch) item per lane ---
            const int c = base + lane;
            int j = 0;  // largest j with pre_j <= c
#pragma unroll
            for (int step = 16; step > 0; step >>= 1) {
                const int v = __shfl_sync(FULL, prej, j + step);
                if (v <= c) j += step;
            }
            const uint32_t hx = __shfl_sync(FULL, hd.x, j), hy = __shfl_sync(FULL, hd.y, j);
            const uint32_t hz = __shfl_sync(FULL, hd.z, j);
            const int32_t bi = (int32_t)__shfl_sync(FULL, hd.w, j);
            const int q = c - __shfl_sync(FULL, prej, j);
            const uint4 *pp = a.par.pay + hx;
            const int pc = (int)((hy >> 23) & 0x7Fu), np = (int)(hz & 0x7FFu);
            bool okl = c < T;
            int k = 0, ins = 0;
            bool in_u = false;
            int32_t A = 1, C = 0;
            if (okl) {
                const int piv = (int)(hy & 0x3FFu);
                const bool fwd = bi > 0;  // forward flow: consume the surplus
                const uint32_t abi = (uint32_t)(bi < 0 ? -bi : bi);
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
                    const bool opp = SUB && q >= ln;
                    const uint32_t br = opp ? bl[(fwd ? nv.o_prodent : nv.o_consent) + (int)bl[optr] + (q - ln)]
                                            : bl[(fwd ? nv.o_consent : nv.o_prodent) + lb + q];
                    k = ent_index(br);
                    const uint32_t sik = (uint32_t)ent_coef(br);  // |S_ik|
                    const uint32_t tw = bl[nv.o_twin + k];        // -1: no twin (matches no column)
                    bool twin = false;
                    auto look = [&](uint32_t w) {
                        const uint32_t c0 = w & 0xFFFFu, c1 = w >> 16;
                        in_u = in_u || c0 == (uint32_t)k || c1 == (uint32_t)k;
                        twin = twin || c0 == tw || c1 == tw;
                        ins += (c0 < (uint32_t)k ? 1 : 0) + (c1 < (uint32_t)k ? 1 : 0);
                    };
                    const int lu = sparse_list_units(pc);
                    {
                        const uint4 u = pp[0];
                        look(u.z);
                        look(u.w);
                    }
                    for (int t = 1; t < lu; ++t) {
                        const uint4 u = pp[t];
                        look(u.x);
                        look(u.y);
                        look(u.z);
                        look(u.w);
                    }
                    const int sec = a.level - pc;
                    if (opp)
                        okl = in_u && sec + 1 <= a.max_sec;
                    else
                        okl = !twin && (in_u ? sec + 1 <= a.max_sec : pc + 1 <= a.max_len);
                    if (FK && okl && a.fk_pc > 0) {
                        // branch and bound: the child's descendants keep its
                        // support or grow it, so a child past the K-th result
                        // found so far cannot yield one of the K smallest.  Of
                        // two supports of equal size, the one whose ascending
                        // list is smaller at the first difference comes first.
                        const int pc2 = pc + (in_u ? 0 : 1);
                        if (pc2 > a.fk_pc) {
                            okl = false;
                        } else if (pc2 == a.fk_pc) {
                            for (int i = 0; i < pc2; ++i) {
                                const int own = in_u || i < ins ? list_col(pp, i) : (i == ins ? k : list_col(pp, i - 1));
                                const int b = (int)s_bound[i];
                                if (own != b) {
                                    okl = own < b;
                                    break;
                                }
                            }
                        }
                    }
                    const uint32_t g0 = (abi == 1u || sik == 1u) ? 1u : gcd32(abi, sik);
                    A = (int32_t)(sik / g0);
                    C = (int32_t)(abi / g0);
                    if (opp) C = -C;  // Eq. 5: flux taken away from k
                }
            }
            if (okl) ++n_exp;
            const int pc2 = pc + (in_u ? 0 : 1);
            // superset rule: the new column completes a result accepted at an
            // earlier level (counted below, once the child is known to be one)
            bool pr = false;
            if (okl && !in_u && a.cells.n_res > 0) pr = pruned_cells(a.cells, a.rcols, pp, pc, k);
            // first-K length-cap rules.  dead: the child cannot balance any
            // more, unless it is balanced already (it then has no one-sided
            // row); skip: nor can its update leave int32, so nothing of it
            // needs to be computed
            bool dead = false, skip = false;
            if (FK) {
                const bool at_cap = okl && !pr && a.cap_dead && pc2 >= a.max_len;
                const bool below = okl && !pr && a.cap_dead && pc2 == a.max_len - 1;
                bool one_sided = false;
                unsigned need = __ballot_sync(FULL, at_cap || below);
                while (need) {
                    const int src = __ffs((int)need) - 1;
                    need &= need - 1;
                    const uint32_t ox = __shfl_sync(FULL, hx, src);
                    const int opc = __shfl_sync(FULL, pc, src);
                    const int ok_ = __shfl_sync(FULL, in_u ? -1 : k, src);
                    const int room = __shfl_sync(FULL, below ? 1 : 0, src);
                    if (ox != cap_for) {
                        cap_parent(nv, bl, s_cap[FK ? wid : 0], a.par.pay + ox, opc, lane);
                        cap_for = ox;
                    }
                    const bool can = cap_child(nv, bl, s_cap[FK ? wid : 0], ok_, room, lane);
                    if (lane == src) one_sided = !can;
                }
                dead = one_sided || (at_cap && a.level - pc2 + 1 >= a.max_sec);
                // |A| max|EF| + |C| max|S| below 2^31: no entry can overflow
                skip = one_sided && ((uint64_t)A << ((hz >> 11) & 0x1Fu)) + (uint64_t)(uint32_t)C * EFM_MAX_COEF <
                                        0x80000000ull;
            }
            // --- rows and payload units of the children of this round ---
            const bool wr = okl && !pr && !dead;
            const int cb = okl ? (int)bl[nv.o_colptr + k + 1] - (int)bl[nv.o_colptr + k] : 0;
            const int units = wr ? sparse_list_units(pc2) + ((np + cb + (SUB ? 1 : 0) + 1) >> 1) : 0;
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
                want_r = row_left < rows ? max(rows - row_left, a.blk) : 0;
                const int want_p = pay_left < utot ? max(utot, a.pay_blk) : 0;
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
            if (okl && !skip) {
                const int2 *pe = entries_of(pp, pc);
                const int lu2 = sparse_list_units(pc2);
                Merged m;
                merge_child<SUB>(nv, bl, pe, np, k, A, C, dst ? dst + lu2 : nullptr, m);
                bool live = false;
                const uint64_t uh = list_hash(pp) + (in_u ? 0ull : column_hash(k));
                if (SUB && m.zflux) {
                    ++n_zero;
                } else if (m.nbal == 0) {
                    ++n_bal;  // all metabolites stable: to the arbiter
                    if (insert_list(a, nv.W, pp, pc, in_u ? -1 : k, uh) < INS_DUP) fatal = true;
                } else if ((m.big || m.g != 1u) &&
                           settle_child<SUB>(nv, bl, pe, np, k, A, C, dst ? dst + lu2 : nullptr, m)) {
                    ++n_ovf;
                } else if (pr) {
                    ++n_pruned;
                } else {
                    live = !dead;
                }
                if (wr) {
                    const bool written = live && dst != nullptr;
                    if (written) write_list(dst, pp, pc, k, in_u ? -1 : ins, uh);
                    if ((int64_t)idx < row_cap)
                        a.child.hdr[idx] =
                            written ? make_uint4((uint32_t)off, pack_meta(branch_key(bl, nv, m.key, SUB ? 1 : 0), pc2),
                                                 (uint32_t)m.nnz | ((uint32_t)max_bits(m.om) << 11), (uint32_t)m.pv)
                                    : make_uint4(0u, 0u, 0u, 0u);
                    if (live && !written) ++n_unwritten;
                    if ((int64_t)idx < a.fp_cap) {
                        a.fp[idx] = live ? state_fp(m.hash, uh) : kDeadFp;
                    } else {
                        record_diag(a.ctr, ERR_BOUNDS, 7, (long long)idx, a.fp_cap, a.level);
                        fatal = true;
                    }
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
    auto total = [&](unsigned long long v, int id) {
        const unsigned s = __reduce_add_sync(FULL, (unsigned)v);  // a lane counts far below 2^27 items a launch
        if (lane == 0 && s) atomicAdd(&a.ctr[id], (unsigned long long)s);
    };
    total(n_exp, C_EXP);
    total(n_ovf, C_OVF);
    total(n_bal, C_BAL);
    total(n_pruned, C_PRUNED);
    total(n_unwritten, C_UNWRITTEN);
    total(n_zero, C_ZERO);
}

// ---------------------------------------------------------------------------
// Dedup: one thread per reserved row; the first row of every distinct state
// survives in place, a later copy gets a zero meta word (no branches).
// ---------------------------------------------------------------------------

__device__ __forceinline__ bool same_sparse(const Arena &ar, const uint4 &x, const uint4 &y)
{
    if (x.y != y.y || x.z != y.z || x.w != y.w) return false;
    const int n = sparse_list_units((int)((x.y >> 23) & 0x7Fu)) + (((int)(x.z & 0x7FFu) + 1) >> 1);
    const uint4 *p = ar.pay + x.x, *r = ar.pay + y.x;
    bool eq = true;
    for (int i = 0; i < n && eq; ++i) {
        const uint4 u = __ldcg(p + i), v = __ldcg(r + i);
        eq = u.x == v.x && u.y == v.y && u.z == v.z && u.w == v.w;
    }
    return eq;
}

__global__ void __launch_bounds__(256) dedup_sparse_kernel(LevelArgs a)
{
    __shared__ unsigned long long s_keep[8], s_deg[8], s_unv[8];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const uint64_t begin = a.ctr[C_DEDUP_BEGIN];
    uint64_t end = a.ctr[C_WRITTEN];
    end = end < (uint64_t)a.fp_cap ? end : (uint64_t)a.fp_cap;
    const uint64_t row_cap = (uint64_t)a.child.cap;
    unsigned long long deg = 0, n_unv = 0, n_keep = 0;
    bool fatal = false;
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t i = begin + (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < end && !fatal; i += stride) {
        const uint64_t f = a.fp[i];
        if (f == kDeadFp) continue;
        uint64_t pos;
        uint32_t tag;
        slot_tag_pos(f, a.slot_mask, pos, tag);
        if (i >= 0xFFFFFFFEull) {
            record_diag(a.ctr, ERR_BOUNDS, 10, (long long)i, 0xFFFFFFFEll, a.level);
            fatal = true;
            break;
        }
        uint4 h = make_uint4(0u, 0u, 0u, 0u);
        if (i < row_cap) h = a.child.hdr[i];
        const bool written = h.y != 0u;
        for (uint64_t probe = 0;; ++probe) {
            if (probe > a.slot_mask) {
                record_diag(a.ctr, ERR_TABLE_FULL, 8, (long long)i, (long long)a.slot_mask, a.level);
                fatal = true;
                break;
            }
            const unsigned long long v = atomicCAS(&a.slots[pos], kEmpty, ((unsigned long long)tag << 32) | i);
            if (v == kEmpty) {  // first of its state
                if (written) {
                    ++n_keep;
                    deg += (h.y >> 10) & 0x1FFFu;
                } else {
                    ++n_unv;
                }
                break;
            }
            if ((uint32_t)(v >> 32) == tag) {
                const uint64_t jrow = (uint32_t)v;
                // (the other row's header may be cleared meanwhile only if it
                // is a later copy itself, and a later copy holds no slot)
                uint4 o = make_uint4(0u, 0u, 0u, 0u);
                if (jrow < row_cap) o = __ldcg(a.child.hdr + jrow);
                // a row without its state written cannot be compared: the
                // level is then decided from the lower bound, or run again
                if (!written || o.y == 0u) {
                    if (written) a.child.hdr[i].y = 0u;
                    break;
                }
                if (same_sparse(a.child, h, o)) {  // a later copy
                    a.child.hdr[i].y = 0u;
                    break;
                }
            }
            pos = (pos + 1) & a.slot_mask;
        }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        deg += __shfl_xor_sync(FULL, deg, off);
        n_unv += __shfl_xor_sync(FULL, n_unv, off);
        n_keep += __shfl_xor_sync(FULL, n_keep, off);
    }
    if (lane == 0) {
        s_keep[wid] = n_keep;
        s_deg[wid] = deg;
        s_unv[wid] = n_unv;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long k = 0, d = 0, u = 0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
            k += s_keep[w];
            d += s_deg[w];
            u += s_unv[w];
        }
        if (k) atomicAdd(&a.ctr[C_NEXT], k);
        if (d) atomicAdd(&a.ctr[C_DEGSUM], d);
        if (u) atomicAdd(&a.ctr[C_UNV], u);
    }
}

__global__ void dedup_advance_sparse_kernel(unsigned long long *ctr) { ctr[C_DEDUP_BEGIN] = ctr[C_WRITTEN]; }

// ---------------------------------------------------------------------------
// seeds (INIT) and seed sets (Prop. 1)
// ---------------------------------------------------------------------------

// One thread per seed column; seeds are distinct columns (no deduplication).
template <bool SUB>
__global__ void __launch_bounds__(256) seed_sparse_kernel(NetView nv, LevelArgs a, int target)
{
    const uint32_t *bl = nv.blob;
    const int n_items = target >= 0 ? nv.metptr[target + 1] - nv.metptr[target] : nv.N;
    for (int it = blockIdx.x * blockDim.x + threadIdx.x; it < n_items; it += gridDim.x * blockDim.x) {
        int k = it;
        if (target >= 0) {
            const uint32_t e = nv.metent[nv.metptr[target] + it];
            if (ent_coef(e) <= 0) continue;
            k = ent_index(e);
        }
        atomicAdd(&a.ctr[C_SEEDS], 1ull);
        // gcd of the column (with its flux 1 in the subtractive view)
        uint32_t g = SUB ? 1u : 0u;
        int n = 0;
        const int qb = (int)bl[nv.o_colptr + k], qe = (int)bl[nv.o_colptr + k + 1];
        for (int q = qb; q < qe; ++q) {
            const int32_t v = ent_coef(bl[nv.o_colent + q]);
            if (v == 0) continue;
            g = gcd32(g, (uint32_t)(v < 0 ? -v : v));
            ++n;
        }
        const uint64_t uh = column_hash(k);
        if (n == 0) {
            atomicAdd(&a.ctr[C_BAL], 1ull);
            insert_list(a, nv.W, nullptr, 0, k, uh);
            continue;
        }
        const int nnz = n + (SUB ? 1 : 0);
        const int units = sparse_list_units(1) + ((nnz + 1) >> 1);
        const uint64_t idx = atomicAdd(&a.ctr[C_NEXT], 1ull);
        const uint64_t off = atomicAdd(&a.ctr[C_PAY], (unsigned long long)units);
        if ((int64_t)idx >= a.child.cap) continue;
        if (off + (uint64_t)units > a.child.pay_cap) {
            record_diag(a.ctr, ERR_BOUNDS, 12, (long long)off, (long long)a.child.pay_cap, a.level);
            continue;
        }
        uint4 *dst = a.child.pay + off;
        dst[0] = make_uint4((uint32_t)uh, (uint32_t)(uh >> 32), (uint32_t)k | (kPadCol << 16), 0xFFFFFFFFu);
        int2 *pe = reinterpret_cast<int2 *>(dst + sparse_list_units(1));
        int w = 0;
        uint32_t key = 0xFFFFFFFFu, om = 0;
        int32_t pv = 0;
        for (int q = qb; q < qe; ++q) {
            const uint32_t f = bl[nv.o_colent + q];
            const int row = ent_index(f);
            const int32_t v = ent_coef(f) / (int32_t)g;
            if (v == 0) continue;
            pe[w++] = make_int2(row, v);
            om |= (uint32_t)(v < 0 ? -v : v);
            const uint32_t kk = bl[(v > 0 ? nv.o_keypos : nv.o_keyneg) + row];
            if (kk < key) {
                key = kk;
                pv = v;
            }
        }
        if (SUB) {
            pe[w++] = make_int2(nv.M + k, 1);
            om |= 1u;
        }
        if (w & 1) pe[w] = make_int2(0, 0);
        const uint32_t bkey = branch_key(bl, nv, key, SUB ? 1 : 0);
        a.child.hdr[idx] = make_uint4((uint32_t)off, pack_meta(bkey, 1),
                                      (uint32_t)w | ((uint32_t)max_bits(om) << 11), (uint32_t)pv);
        atomicAdd(&a.ctr[C_DEGSUM], (unsigned long long)(bkey >> 16));
    }
}

// One state with flux 1 on each column of R_in: EF = the sum of their S_int
// columns, normalised.  One warp; the sums in shared memory.
template <bool SUB>
__global__ void __launch_bounds__(32) seedset_sparse_kernel(NetView nv, LevelArgs a, const int32_t *cols, int n_cols)
{
    __shared__ long long acc[EFM_MAX_INTERNAL];
    __shared__ uint16_t sorted[64];
    const int lane = threadIdx.x;
    const uint32_t *bl = nv.blob;
    const int rows = nv.M + (SUB ? nv.N : 0);  // at most EFM_MAX_INTERNAL
    for (int r = lane; r < EFM_MAX_INTERNAL; r += 32) acc[r] = 0;
    __syncwarp();
    uint64_t uh = 0;
    for (int i = 0; i < n_cols; ++i) {
        const int k = cols[i];
        uh += column_hash(k);
        for (int q = (int)bl[nv.o_colptr + k] + lane; q < (int)bl[nv.o_colptr + k + 1]; q += 32) {
            const uint32_t f = bl[nv.o_colent + q];
            acc[ent_index(f)] += ent_coef(f);  // a column's rows are distinct
        }
        if (SUB && lane == 0) acc[nv.M + k] += 1;
        __syncwarp();
    }
    // ascending columns: a column's place is the number of smaller ones
    for (int i = lane; i < n_cols; i += 32) {
        int pos = 0;
        for (int j = 0; j < n_cols; ++j) pos += cols[j] < cols[i] ? 1 : 0;
        sorted[pos] = (uint16_t)cols[i];
    }
    uint64_t g = 0;
    int n = 0, nb = 0;
    for (int r = lane; r < rows; r += 32) {
        if (acc[r] != 0) {
            g = gcd64(g, abs64(acc[r]));
            ++n;
            if (r < nv.M) ++nb;
        }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        g = gcd64(g, __shfl_xor_sync(FULL, g, off));
        n += __shfl_xor_sync(FULL, n, off);
        nb += __shfl_xor_sync(FULL, nb, off);
    }
    if (g == 0) g = 1;
    bool bad = false;
    for (int r = lane; r < rows; r += 32) bad = bad || abs64(acc[r]) / g > 2147483647ull;
    bad = __any_sync(FULL, bad);
    __syncwarp();
    if (lane == 0) atomicAdd(&a.ctr[C_SEEDS], 1ull);
    if (bad) {
        if (lane == 0) atomicAdd(&a.ctr[C_OVF], 1ull);
        return;
    }
    if (lane != 0) return;
    // the payload, by one lane: at most 64 columns and 1024 entries
    const int lu = sparse_list_units(n_cols);
    const int units = lu + ((n + 1) >> 1);
    if (a.child.cap < 1 || (uint64_t)units > a.child.pay_cap) {
        record_diag(a.ctr, ERR_BOUNDS, 13, units, (long long)a.child.pay_cap, a.level);
        return;
    }
    uint16_t *lst = reinterpret_cast<uint16_t *>(a.child.pay);
    *reinterpret_cast<uint64_t *>(a.child.pay) = uh;
    for (int i = 0; i < 8 * lu - 4; ++i) lst[4 + i] = i < n_cols ? sorted[i] : (uint16_t)kPadCol;
    if (nb == 0) {
        atomicAdd(&a.ctr[C_BAL], 1ull);
        insert_list(a, nv.W, a.child.pay, n_cols, -1, uh);
        return;
    }
    int2 *pe = reinterpret_cast<int2 *>(a.child.pay + lu);
    int w = 0;
    uint32_t key = 0xFFFFFFFFu, om = 0;
    int32_t pv = 0;
    for (int r = 0; r < rows; ++r) {
        if (acc[r] == 0) continue;
        const int32_t v = (int32_t)(acc[r] / (long long)g);
        pe[w++] = make_int2(r, v);
        om |= (uint32_t)(v < 0 ? -v : v);
        if (r < nv.M) {
            const uint32_t kk = bl[(v > 0 ? nv.o_keypos : nv.o_keyneg) + r];
            if (kk < key) {
                key = kk;
                pv = v;
            }
        }
    }
    if (w & 1) pe[w] = make_int2(0, 0);
    const uint32_t bkey = branch_key(bl, nv, key, SUB ? 1 : 0);
    a.child.hdr[0] = make_uint4(0u, pack_meta(bkey, n_cols), (uint32_t)w | ((uint32_t)max_bits(om) << 11),
                                (uint32_t)pv);
    atomicAdd(&a.ctr[C_NEXT], 1ull);
    atomicAdd(&a.ctr[C_PAY], (unsigned long long)units);
    atomicAdd(&a.ctr[C_DEGSUM], (unsigned long long)(bkey >> 16));
}

// ---------------------------------------------------------------------------
// the superset rule's index over the accepted results
// ---------------------------------------------------------------------------

__global__ void cell_count_kernel(const uint16_t *rcols, int64_t n, int32_t *cnt)
{
    const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= n) return;
    const uint16_t *lst = rcols + (size_t)r * kRcolStride;
    for (int j = 1; j <= (int)lst[0]; ++j) atomicAdd(&cnt[lst[j]], 1);
}

__global__ void cell_insert_kernel(const uint16_t *rcols, int64_t n, const int32_t *cnt, uint2 *cells, uint32_t mask,
                                   uint4 *ent, int ent_stride, unsigned long long *ksig, uint32_t *single)
{
    const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= n) return;
    const uint16_t *lst = rcols + (size_t)r * kRcolStride;
    const int m = lst[0];
    if (m == 1) {  // a one-column result: every child adding that column contains it
        single[lst[1]] = 1u;
        return;
    }
    // the two columns with the fewest results (ties by column)
    int m1 = -1, m2 = -1;
    long long k1 = 0x7FFFFFFFFFFFFFFFll, k2 = 0x7FFFFFFFFFFFFFFFll;
    uint64_t sig = 0;
    for (int j = 1; j <= m; ++j) {
        const int c = lst[j];
        sig |= col_bit(c);
        const long long key = ((long long)cnt[c] << 16) | c;
        if (key < k1) {
            k2 = k1;
            m2 = m1;
            k1 = key;
            m1 = c;
        } else if (key < k2) {
            k2 = key;
            m2 = c;
        }
    }
    for (int j = 1; j <= m; ++j) {
        const int k = lst[j];
        const int s = k == m1 ? m2 : m1;
        atomicOr(&ksig[k], (unsigned long long)col_bit(s));
        const uint32_t key = ((uint32_t)k << 12) | (uint32_t)s;
        const int64_t id = r * ent_stride + (j - 1);
        uint32_t p = cell_slot(key, mask);
        for (uint32_t probe = 0; probe <= mask; ++probe) {
            const uint32_t v = atomicCAS(&cells[p].x, kNoRecord, key);
            if (v == kNoRecord || v == key) {
                const uint32_t next = atomicExch(&cells[p].y, (uint32_t)id);
                ent[id] = make_uint4((uint32_t)sig, (uint32_t)(sig >> 32), next, (uint32_t)r);
                break;
            }
            p = (p + 1) & mask;
        }
    }
}

__global__ void live_sparse_kernel(const uint4 *hdr, int64_t n, uint32_t *live, unsigned long long *count)
{
    const int lane = threadIdx.x & 31;
    for (int64_t i0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) & ~31ll; i0 < n;
         i0 += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = i0 + lane;
        const bool keep = i < n && hdr[i].y != 0u;
        const unsigned m = __ballot_sync(FULL, keep);
        unsigned long long base = 0;
        if (lane == 0 && m) base = atomicAdd(count, (unsigned long long)__popc(m));
        base = __shfl_sync(FULL, base, 0);
        if (keep) live[base + __popc(m & ((1u << lane) - 1u))] = (uint32_t)i;
    }
}

template <bool SUB, bool FK>
int grid_of(int sm_count)
{
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, generate_sparse_kernel<SUB, FK>, kGenWarps * 32, 0) !=
            cudaSuccess ||
        per_sm < 1) {
        cudaGetLastError();
        per_sm = 1;
    }
    return sm_count * per_sm;
}

}  // namespace

int sparse_grid(bool sub, bool first_k, int sm_count)
{
    if (sub) return grid_of<true, false>(sm_count);
    return first_k ? grid_of<false, true>(sm_count) : grid_of<false, false>(sm_count);
}

cudaError_t launch_generate_sparse(const NetView &nv, const LevelArgs &a, int grid, cudaStream_t s)
{
    if (a.sub)
        generate_sparse_kernel<true, false><<<grid, kGenWarps * 32, 0, s>>>(nv, a);
    else if (a.cap_dead || a.fk_pc > 0)
        generate_sparse_kernel<false, true><<<grid, kGenWarps * 32, 0, s>>>(nv, a);
    else
        generate_sparse_kernel<false, false><<<grid, kGenWarps * 32, 0, s>>>(nv, a);
    return cudaGetLastError();
}

cudaError_t launch_dedup_sparse(const LevelArgs &a, int sm_count, cudaStream_t s)
{
    dedup_sparse_kernel<<<sm_count * 8, 256, 0, s>>>(a);
    dedup_advance_sparse_kernel<<<1, 1, 0, s>>>(a.ctr);
    return cudaGetLastError();
}

cudaError_t launch_seed_sparse(const NetView &nv, const LevelArgs &a, int target, cudaStream_t s)
{
    const int blocks = 4;
    if (a.sub)
        seed_sparse_kernel<true><<<blocks, 256, 0, s>>>(nv, a, target);
    else
        seed_sparse_kernel<false><<<blocks, 256, 0, s>>>(nv, a, target);
    return cudaGetLastError();
}

cudaError_t launch_seedset_sparse(const NetView &nv, const LevelArgs &a, const int32_t *cols, int n_cols,
                                  cudaStream_t s)
{
    if (a.sub)
        seedset_sparse_kernel<true><<<1, 32, 0, s>>>(nv, a, cols, n_cols);
    else
        seedset_sparse_kernel<false><<<1, 32, 0, s>>>(nv, a, cols, n_cols);
    return cudaGetLastError();
}

cudaError_t launch_cells(const NetView &nv, const uint16_t *rcols, int64_t n_res, int32_t *cnt, const CellIndex &ix,
                         int ent_stride, cudaStream_t s)
{
    cudaError_t e;
    if ((e = cudaMemsetAsync(cnt, 0, sizeof(int32_t) * (size_t)nv.N, s)) != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(ix.ksig, 0, 8 * (size_t)nv.N, s)) != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(ix.single, 0, 4 * (size_t)nv.N, s)) != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(ix.cells, 0xFF, 8 * ((size_t)ix.mask + 1), s)) != cudaSuccess) return e;
    if (n_res <= 0) return cudaSuccess;
    const int tb = 128;
    const unsigned blocks = (unsigned)((n_res + tb - 1) / tb);
    cell_count_kernel<<<blocks, tb, 0, s>>>(rcols, n_res, cnt);
    cell_insert_kernel<<<blocks, tb, 0, s>>>(rcols, n_res, cnt, ix.cells, ix.mask, ix.ent, ent_stride,
                                            (unsigned long long *)ix.ksig, ix.single);
    return cudaGetLastError();
}

cudaError_t launch_live_sparse(const uint4 *hdr, int64_t n, uint32_t *live, unsigned long long *count, int sm_count,
                               cudaStream_t s)
{
    if (n <= 0) return cudaSuccess;
    const int64_t blocks = std::min<int64_t>((n + 255) / 256, (int64_t)sm_count * 8);
    live_sparse_kernel<<<(unsigned)blocks, 256, 0, s>>>(hdr, n, live, count);
    return cudaGetLastError();
}

}  // namespace efm
