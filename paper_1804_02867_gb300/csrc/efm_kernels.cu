// efm_kernels.cu -- sm_103a kernels of the pathway traversal.
//
// One traversal level (expansion of the frontier F_{l-1} into F_l) is the
// METAx step of Alg. 3 restated exhaustively and in exact integers:
//   * the acting metabolite of a pathway is its unbalanced internal
//     metabolite with the fewest reactions able to fix it (ties by index);
//     extra flux EF_i > 0 is a forward flow and all outputs of i are tried,
//     EF_i < 0 a backward flow and all inputs are tried (Def. 9, Eq. 3);
//   * the AND update gives the new reaction the flux that zeroes EF_i,
//     EF' = a*EF + c*S_int[:,k] with a = |S_ik|/g, c = |EF_i|/g,
//     g = gcd(|EF_i|, |S_ik|), then divides EF' by the gcd of its entries;
//     adding flux to a reaction already in the pathway is a secondary step
//     (Def. 10, Eq. 4) bounded by max_secondary (MAX_LOOP, Sec. 3.2);
//   * a balanced child (all metabolites Stable) goes to the arbiter
//     (Sec. 3.2.2) through a support hash set; an unbalanced child whose
//     support contains an accepted result is pruned (Def. 3 minimality);
//     the rest is deduplicated on (support, EF) in a hash table and the
//     new states are compacted into the next frontier.
// The arbiter decides minimality exactly: nullity(S_int[:,U]) == 1 is
// tested by Gaussian elimination modulo primes p = 2^31 - c, with enough
// primes that their product exceeds the Hadamard bound of the columns.
//
// This file holds the minimality test, the walks, the batch and the sorting of
// results; the level pass itself (states, expansion, merging of duplicates) is
// efm_level.cuh, launched over the grid by efm_sparse.cu.
#include "efm_level.cuh"

namespace efm {
namespace {

constexpr int kSpinLimit = 1 << 20;  // x ~1 us sleep: about one second

// primes p = 2^31 - c (c < 2^10), the 24 largest below 2^31
__constant__ uint32_t c_prime_c[kNumPrimes] = {1,   19,  61,  69,  85,  99,  105, 151, 159, 171, 225, 249,
                                              295, 325, 379, 399, 411, 469, 477, 511, 525, 571, 579, 589};

// ---------------------------------------------------------------------------
// hash sets (publish-after-write slots)
//
// A slot is one 64-bit word: (tag << 32) | index.  An inserter claims an
// empty slot with CAS as (tag, PENDING), writes the record, fences, then
// publishes the index.  A prober whose tag matches waits (bounded) for the
// index and compares the full record; records are never compared by tag
// alone, so the set is exact.
// ---------------------------------------------------------------------------

// word w of the support U' = U (pu, or empty if null) plus column k
__device__ __forceinline__ uint64_t child_word(const uint64_t *pu, int w, int k)
{
    uint64_t x = pu ? pu[w] : 0ull;
    if (w == (k >> 6)) x |= 1ull << (k & 63);
    return x;
}

// Insert the support U' = U + {k} of a balanced pathway into the set of
// supports judged in this traversal (one thread).
__device__ __noinline__ int insert_support(const LevelArgs &a, int W, const uint64_t *pu, int k)
{
    uint64_t h = 0;
    for (int w = 0; w < W; ++w) h += mix64(child_word(pu, w, k) ^ (0x51ed27f3a5b1c3d9ull * (uint64_t)(w + 1)));
    uint64_t pos;
    uint32_t tag;
    slot_tag_pos(h, a.cslot_mask, pos, tag);
    for (uint64_t probe = 0; probe <= a.cslot_mask; ++probe) {
        unsigned long long v = atomicCAS(&a.cslots[pos], kEmpty, ((unsigned long long)tag << 32) | kPending);
        if (v == kEmpty) {
            const unsigned long long idx = atomicAdd(&a.ctr[C_CAND_N], 1ull);
            if ((int64_t)idx >= a.cand_cap) {
                atomicOr(&a.ctr[C_ERR], (unsigned long long)ERR_CAND_CAP);
                atomicExch(&a.cslots[pos], ((unsigned long long)tag << 32) | kOverflowIdx);
                return INS_ARENA_FULL;
            }
            uint64_t *dst = a.cand + (size_t)idx * W;
            for (int w = 0; w < W; ++w) dst[w] = child_word(pu, w, k);
            __threadfence();
            atomicExch(&a.cslots[pos], ((unsigned long long)tag << 32) | idx);
            return INS_NEW;
        }
        if ((uint32_t)(v >> 32) == tag) {
            int spins = 0;
            while ((uint32_t)v == kPending) {
                if (++spins > kSpinLimit) {
                    atomicOr(&a.ctr[C_ERR], (unsigned long long)ERR_TIMEOUT);
                    return INS_TIMEOUT;
                }
                __nanosleep(64);
                v = load_volatile(&a.cslots[pos]);
            }
            const uint32_t idx = (uint32_t)v;
            if (idx == kOverflowIdx) return INS_ARENA_FULL;
            const uint64_t *src = a.cand + (size_t)idx * W;
            bool eq = true;
            for (int w = 0; w < W && eq; ++w) eq = __ldcg(src + w) == child_word(pu, w, k);
            if (eq) return INS_DUP;
        }
        pos = (pos + 1) & a.cslot_mask;
    }
    atomicOr(&a.ctr[C_ERR], (unsigned long long)ERR_TABLE_FULL);
    return INS_TABLE_FULL;
}

// Pivot key of a state: min over unbalanced rows of (degree << 16 | row)
// (warp-cooperative; lane l holds rows l + 32 e).
template <int EPL>
__device__ __forceinline__ uint32_t pivot_key(const uint32_t *bl, const NetView &nv, const int32_t (&t)[EPL], int lane)
{
    uint32_t kmin = 0xFFFFFFFFu;
#pragma unroll
    for (int e = 0; e < EPL; ++e) {
        const int m = lane + 32 * e;
        if (t[e] != 0 && m < nv.M) {  // rows past M hold flux (subtractive variant) or padding
            const uint32_t k = t[e] > 0 ? bl[nv.o_keypos + m] : bl[nv.o_keyneg + m];
            kmin = k < kmin ? k : kmin;
        }
    }
    return __reduce_min_sync(FULL, kmin);
}

// ---------------------------------------------------------------------------
// Monte-Carlo mode: the paper's own random walks (Alg. 3 with one random OR
// branch per step), in the exact integer form of the traversal.  One warp
// per walk; entry m of the extra-flux row sits in lane m % 32.  Walk w draws
// its numbers from counters 128 w + s (s = 0 picks the seed column, s >= 1
// the branch of step s): the first output of SplitMix64 (Steele, Lea and
// Flood, 2014) started from state seed + counter * 0x9E3779B97F4A7C15.
// ---------------------------------------------------------------------------

__device__ __forceinline__ uint64_t splitmix_at(uint64_t seed, uint64_t c)
{
    uint64_t z = seed + (c + 1) * 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

// gcd normalisation of a row held across the warp, with the int32 range test
template <int EPL>
__device__ __forceinline__ void walk_normalise(const int64_t (&t64)[EPL], int32_t (&t)[EPL], bool &zero, bool &ovf)
{
    uint64_t g = 0;
#pragma unroll
    for (int e = 0; e < EPL; ++e) g = gcd64(g, abs64(t64[e]));
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) g = gcd64(g, __shfl_xor_sync(FULL, g, off));
    zero = g == 0;
    bool bad = false;
#pragma unroll
    for (int e = 0; e < EPL; ++e) {
        const int64_t v = g > 1 ? t64[e] / (int64_t)g : t64[e];
        bad = bad || v > 2147483647ll || v < -2147483647ll;
        t[e] = (int32_t)v;
    }
    ovf = __any_sync(FULL, bad);
}

// --- narrow networks (at most 64 internal rows and 128 columns): a walk per
// lane.  A lane's row sits in shared memory, entry m of lane l at 32 m + l (no
// bank conflicts whatever rows the lanes touch); which entries are nonzero,
// their signs at the pivot keys' ranks and the +-1 rows are masks in
// registers, so a step touches the rows of column k alone unless A > 1 or no
// +-1 entry proves the gcd to be 1.  A lane takes its next walk as soon as one
// ends.  Bound by issue: one GB300, core-shaped network, 2^20 walks of at most
// 30 columns: 27.0 ms with a warp per walk and 64-bit rows in registers, 4.2
// ms this way (the whole call 28.9 -> 4.5). ---

constexpr int kWalkWarps = 4;

__device__ __forceinline__ int walk_pick(uint64_t x, int n)  // x mod n, n <= EFM_MAX_COLUMNS
{
    const uint32_t c = (uint32_t)n;
    const uint32_t p = (0xFFFFFFFFu % c + 1u) % c;  // 2^32 mod n
    return (int)((((uint32_t)(x >> 32) % c) * p + (uint32_t)x % c) % c);
}

struct WalkState {
    uint64_t zm, pm, nm, um;  // nonzero rows; positive / negative entries by key rank; +-1 rows
    uint32_t pmax;            // at least the largest magnitude
};

// The row divided by g, or rebuilt by f(row, old value) in 64 bits first (the
// rows of rows); exact masks and magnitude.  False: an entry outside int32.
template <typename Value>
__device__ __noinline__ bool walk_rebuild(const NetView &nv, const uint32_t *bl, int32_t *row, uint64_t rows, WalkState &z,
                                          Value f)
{
    uint64_t g = 0, mx = 0;
    for (uint64_t x = rows; x; x &= x - 1) {
        const int m = __ffsll((long long)x) - 1;
        const uint64_t at = abs64(f(m));
        if (at) g = gcd64(g, at);
        mx = at > mx ? at : mx;
    }
    if (g == 0) {
        z = WalkState{0, 0, 0, 0, 0};
        return true;
    }
    if (mx / g > 2147483647ull) return false;
    WalkState y{0, 0, 0, 0, (uint32_t)(mx / g)};
    for (uint64_t x = rows; x; x &= x - 1) {
        const int m = __ffsll((long long)x) - 1;
        const int32_t v = (int32_t)(f(m) / (int64_t)g);
        row[32 * m] = v;
        if (v == 0) continue;
        const uint32_t rk = bl[nv.o_rank + m];
        y.zm |= 1ull << m;
        if (v > 0) y.pm |= 1ull << (rk & 0xFFu);
        else y.nm |= 1ull << ((rk >> 8) & 0xFFu);
        if (v == 1 || v == -1) y.um |= 1ull << m;
    }
    z = y;
    return true;
}

__global__ void __launch_bounds__(kWalkWarps * 32) walk_narrow_kernel(const __grid_constant__ NetView nv,
                                                                      const __grid_constant__ LevelArgs a, int target,
                                                                      uint64_t seed, int64_t n_walks)
{
    extern __shared__ int32_t s_rows[];  // per warp: M x 32 entries
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int32_t *row = s_rows + (size_t)wid * 32 * nv.M + lane;
    const uint32_t *bl = nv.blob;
    const uint4 *scol = reinterpret_cast<const uint4 *>(bl + nv.o_scol);
    const uint2 *nent = reinterpret_cast<const uint2 *>(bl + nv.o_nent);
    const int tb = target >= 0 ? nv.metptr[target] : 0, te = target >= 0 ? nv.metptr[target + 1] : 0;
    int n_seeds = target >= 0 ? 0 : nv.N;
    for (int q = tb; q < te; ++q) n_seeds += ent_coef(nv.metent[q]) > 0 ? 1 : 0;
    // (64-bit counters in the lanes cost 1.6 %: a lane adds 32-bit ones up before they wrap)
    unsigned n_walk = 0, n_exp = 0, n_ovf = 0, n_bal = 0, n_dead = 0, max_steps = 0;
    const int64_t total = (int64_t)gridDim.x * blockDim.x;
    int64_t w = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    bool running = false;
    WalkState z{0, 0, 0, 0, 0};
    uint64_t U[2] = {0, 0};
    int j = 0, pc = 0, sec = 0, s = 0;
    if (n_seeds == 0) w = n_walks;
    while (w < n_walks) {
        bool ended = false;
        if (!running) {
            // the seed: the pick-th positive entry of the target's row
            int pick = walk_pick(splitmix_at(seed, (uint64_t)w * 128u), n_seeds);
            j = pick;
            if (target >= 0)
                for (int q = tb; q < te; ++q) {
                    const uint32_t e = nv.metent[q];
                    if (ent_coef(e) <= 0) continue;
                    if (pick-- == 0) {
                        j = ent_index(e);
                        break;
                    }
                }
            ++n_walk;
            U[0] = j < 64 ? 1ull << j : 0ull;
            U[1] = j < 64 ? 0ull : 1ull << (j - 64);
            pc = 1;
            sec = 0;
            s = 0;
            running = true;
            const uint4 s1 = scol[2 * j + 1];
            uint64_t rows = 0;
            for (int q = (int)s1.y; q < (int)s1.z; ++q) {
                const uint2 e = nent[q];
                row[32 * (e.x & 63u)] = (int32_t)e.y;
                rows |= 1ull << (e.x & 63u);
            }
            walk_rebuild(nv, bl, row, rows, z, [&](int m) { return (int64_t)row[32 * m]; });
        }
        ++s;  // this step's number
        if (z.zm == 0) {
            ++n_bal;
            insert_support(a, nv.W, U, j);  // (a failure sets the error word)
            ended = true;
        } else if (s > 127) {  // every step adds a column or a secondary step: unreachable
            record_diag(a.ctr, ERR_BOUNDS, 5, s, 127, 0);
            ended = true;
        } else {
            const uint32_t key = mask_key(bl, nv, z.pm, z.nm);
            const int piv = (int)(key & 0xFFFFu);
            const int32_t bi = row[32 * piv];
            const bool fwd = bi > 0;
            const int lptr = (fwd ? nv.o_consptr : nv.o_prodptr) + piv;
            const int lb = (int)bl[lptr], le = (int)bl[lptr + 1];
            const uint32_t *list = bl + (fwd ? nv.o_consent : nv.o_prodent);
            auto valid = [&](int q) -> bool {
                const int k = ent_index(list[q]);
                const uint32_t tw = bl[nv.o_twin + k];
                if (tw != 0xFFFFFFFFu && (((tw < 64u ? U[0] : U[1]) >> (tw & 63u)) & 1ull)) return false;
                return (((k < 64 ? U[0] : U[1]) >> (k & 63)) & 1ull) ? sec + 1 <= a.max_sec : pc + 1 <= a.max_len;
            };
            int cnt = 0;
            for (int q = lb; q < le; ++q) cnt += valid(q) ? 1 : 0;
            if (cnt == 0) {
                ++n_dead;
                ended = true;
            } else {
                int r = walk_pick(splitmix_at(seed, (uint64_t)w * 128u + (uint64_t)s), cnt);
                int qs = lb;
                for (int q = lb; q < le; ++q)
                    if (valid(q) && r-- == 0) {
                        qs = q;
                        break;
                    }
                const uint32_t br = list[qs];
                const int k = ent_index(br);
                const uint32_t sik = (uint32_t)ent_coef(br), abi = mag(bi);
                const uint32_t g0 = (abi == 1u || sik == 1u) ? 1u : gcd32(abi, sik);
                const int32_t A = (int32_t)(sik / g0), C = (int32_t)(abi / g0);
                ++n_exp;
                if (((k < 64 ? U[0] : U[1]) >> (k & 63)) & 1ull) {
                    ++sec;
                } else {
                    if (k < 64) U[0] |= 1ull << k;
                    else U[1] |= 1ull << (k - 64);
                    ++pc;
                }
                j = k;
                const uint4 s1 = scol[2 * k + 1];
                const int cb = (int)s1.y, ce = (int)s1.z;
                const int ox = nv.o_colx + 10 * k;
                const uint64_t mask = blob_u64(bl, ox + 4);
                if ((uint64_t)A * z.pmax + (uint64_t)C * s1.x < 0x80000000ull) {
                    uint64_t newz = 0, newp = 0, newn = 0, newu = 0;
                    uint32_t mx = (uint32_t)A * z.pmax;
                    for (int q = cb; q < ce; ++q) {
                        const uint2 e = nent[q];
                        const int m = (int)(e.x & 63u);
                        const int32_t v = (z.zm >> m) & 1ull ? row[32 * m] : 0;
                        const int32_t t = A * v + C * (int32_t)e.y;
                        row[32 * m] = t;
                        newz |= (uint64_t)(t != 0) << m;
                        newp |= (uint64_t)(t > 0) << ((e.x >> 8) & 63u);
                        newn |= (uint64_t)(t < 0) << ((e.x >> 16) & 63u);
                        newu |= (uint64_t)(t == 1 || t == -1) << m;
                        mx = max(mx, mag(t));
                    }
                    const uint64_t keep = z.zm & ~mask;
                    if (A != 1)
                        for (uint64_t x = keep; x; x &= x - 1) row[32 * (__ffsll((long long)x) - 1)] *= A;
                    z.zm = keep | newz;
                    z.pm = (z.pm & ~blob_u64(bl, ox)) | newp;
                    z.nm = (z.nm & ~blob_u64(bl, ox + 2)) | newn;
                    z.um = (A == 1 ? z.um & ~mask : 0ull) | newu;
                    z.pmax = mx;
                    if (z.um == 0 && z.zm != 0) {
                        uint32_t g = 0;
                        for (uint64_t x = z.zm; x && g != 1u; x &= x - 1)
                            g = gcd_small(g, mag(row[32 * (__ffsll((long long)x) - 1)]));
                        if (g != 1u)
                            walk_rebuild(nv, bl, row, z.zm, z, [&](int m) { return (int64_t)row[32 * m]; });
                    }
                } else {
                    // an entry may leave int32 before the division: in 64 bits
                    const uint64_t zm = z.zm;
                    const bool fit = walk_rebuild(nv, bl, row, zm | mask, z, [&](int m) {
                        int64_t t = (zm >> m) & 1ull ? (int64_t)A * row[32 * m] : 0;
                        if ((mask >> m) & 1ull)
                            for (int q = cb; q < ce; ++q) {
                                const uint2 e = nent[q];
                                if ((int)(e.x & 63u) == m) t += (int64_t)C * (int32_t)e.y;
                            }
                        return t;
                    });
                    if (!fit) {
                        ++n_ovf;
                        ended = true;
                    }
                }
                max_steps = max(max_steps, (unsigned)s);
            }
        }
        if (ended) {
            running = false;
            w += total;
            if ((n_walk | n_exp) >> 31) {
                atomicAdd(&a.ctr[C_SEEDS], (unsigned long long)n_walk);
                atomicAdd(&a.ctr[C_EXP], (unsigned long long)n_exp);
                atomicAdd(&a.ctr[C_OVF], (unsigned long long)n_ovf);
                atomicAdd(&a.ctr[C_BAL], (unsigned long long)n_bal);
                atomicAdd(&a.ctr[C_PRUNED], (unsigned long long)n_dead);
                n_walk = n_exp = n_ovf = n_bal = n_dead = 0;
            }
        }
    }
    auto total_of = [&](unsigned long long v, int id) {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(FULL, v, off);
        if (lane == 0 && v) atomicAdd(&a.ctr[id], v);
    };
    total_of(n_walk, C_SEEDS);
    total_of(n_exp, C_EXP);
    total_of(n_ovf, C_OVF);
    total_of(n_bal, C_BAL);
    total_of(n_dead, C_PRUNED);
    const unsigned most = __reduce_max_sync(FULL, max_steps);
    if (lane == 0 && most) atomicMax(&a.ctr[C_LEVELS], (unsigned long long)most);
}

// the output rows of a batch's jobs, job i's words [off[i], off[i + 1]) of dst
__global__ void __launch_bounds__(128) batch_gather_kernel(const BatchJob *jobs, const int64_t *off, int n_jobs,
                                                           uint64_t *dst)
{
    for (int i = blockIdx.x; i < n_jobs; i += gridDim.x) {
        const uint64_t *src = jobs[i].out;
        const int64_t b = off[i], n = off[i + 1] - b;
        for (int64_t q = threadIdx.x; q < n; q += blockDim.x) dst[b + q] = src[q];
    }
}

template <int EPL>
__global__ void __launch_bounds__(kExpandWarps * 32) walk_kernel(NetView nv, LevelArgs a, int target, uint64_t seed,
                                                                 int64_t n_walks)
{
    __shared__ uint64_t sU[kExpandWarps][kMaxW];
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    uint64_t *U = sU[wid];
    const uint32_t *bl = nv.blob;
    const int W = nv.W, Mpad = nv.Mpad;
    const int32_t *dcol = reinterpret_cast<const int32_t *>(bl + nv.o_dcols);
    unsigned long long n_walk = 0, n_exp = 0, n_ovf = 0, n_bal = 0, n_dead = 0, max_steps = 0;
    bool fatal = false;
    // the target's seed columns: its row's positive entries, ascending columns
    const int tb = target >= 0 ? nv.metptr[target] : 0;
    const int te = target >= 0 ? nv.metptr[target + 1] : 0;
    int n_seeds = target >= 0 ? 0 : nv.N;
    for (int q0 = tb; q0 < te; q0 += 32) {
        const int q = q0 + lane;
        n_seeds += __popc(__ballot_sync(FULL, q < te && ent_coef(nv.metent[q]) > 0));
    }
    const int64_t gw = (int64_t)blockIdx.x * kExpandWarps + wid, nw = (int64_t)gridDim.x * kExpandWarps;
    for (int64_t w = gw; w < n_walks && n_seeds > 0 && !fatal; w += nw) {
        const uint64_t c0 = (uint64_t)w * 128u;
        int pick = (int)(splitmix_at(seed, c0) % (uint64_t)n_seeds);
        int j = pick;
        if (target >= 0) {
            for (int q0 = tb; q0 < te; q0 += 32) {
                const int q = q0 + lane;
                const unsigned m = __ballot_sync(FULL, q < te && ent_coef(nv.metent[q]) > 0);
                const int c = __popc(m);
                if (pick < c) {
                    j = ent_index(nv.metent[q0 + (int)__fns(m, 0, pick + 1)]);
                    break;
                }
                pick -= c;
            }
        }
        ++n_walk;
        for (int x = lane; x < W; x += 32) U[x] = x == (j >> 6) ? 1ull << (j & 63) : 0ull;
        __syncwarp();
        int64_t t64[EPL];
#pragma unroll
        for (int e = 0; e < EPL; ++e) t64[e] = dcol[(size_t)j * Mpad + lane + 32 * e];
        int32_t t[EPL];
        bool zero, ovf;
        walk_normalise<EPL>(t64, t, zero, ovf);
        if (ovf) {
            ++n_ovf;
            continue;
        }
        int pc = 1, sec = 0;
        unsigned long long steps = 0;
        for (int s = 1;; ++s) {
            if (zero) {
                ++n_bal;
                if (lane == 0 && insert_support(a, W, U, j) < INS_DUP) fatal = true;
                fatal = __any_sync(FULL, fatal);
                break;
            }
            if (s > 127) {  // every step adds a column or a secondary step: unreachable
                if (lane == 0) record_diag(a.ctr, ERR_BOUNDS, 5, s, 127, 0);
                fatal = true;
                break;
            }
            const uint32_t key = pivot_key<EPL>(bl, nv, t, lane);
            const int piv = (int)(key & 0xFFFFu);
            int32_t mine = 0;
#pragma unroll
            for (int e = 0; e < EPL; ++e)
                if (e == (piv >> 5)) mine = t[e];
            const int32_t bi = __shfl_sync(FULL, mine, piv & 31);
            const bool fwd = bi > 0;
            const int lptr = (fwd ? nv.o_consptr : nv.o_prodptr) + piv;
            const int lb = (int)bl[lptr], le = (int)bl[lptr + 1];
            const int lent = fwd ? nv.o_consent : nv.o_prodent;
            auto valid_at = [&](int q) -> bool {
                if (q >= le) return false;
                const int k = ent_index(bl[lent + q]);
                const int tw = (int)bl[nv.o_twin + k];
                if (tw >= 0 && bit_of(U, tw)) return false;
                return bit_of(U, k) ? sec + 1 <= a.max_sec : pc + 1 <= a.max_len;
            };
            int cnt = 0;
            for (int q0 = lb; q0 < le; q0 += 32) cnt += __popc(__ballot_sync(FULL, valid_at(q0 + lane)));
            if (cnt == 0) {
                ++n_dead;
                break;
            }
            int r = (int)(splitmix_at(seed, c0 + (uint64_t)s) % (uint64_t)cnt);
            int qs = lb;
            for (int q0 = lb; q0 < le; q0 += 32) {
                const unsigned m = __ballot_sync(FULL, valid_at(q0 + lane));
                const int c = __popc(m);
                if (r < c) {
                    qs = q0 + (int)__fns(m, 0, r + 1);
                    break;
                }
                r -= c;
            }
            const uint32_t br = bl[lent + qs];
            const int k = ent_index(br);
            const uint32_t sik = (uint32_t)ent_coef(br);  // |S_ik|
            const uint32_t abi = (uint32_t)(bi < 0 ? -bi : bi);
            const uint32_t g0 = gcd32(abi, sik);
            const int64_t A = (int64_t)(sik / g0), C = (int64_t)(abi / g0);
#pragma unroll
            for (int e = 0; e < EPL; ++e) t64[e] = A * t[e] + C * dcol[(size_t)k * Mpad + lane + 32 * e];
            ++n_exp;
            ++steps;
            const bool in_u = bit_of(U, k);
            __syncwarp();
            if (in_u) {
                ++sec;
            } else {
                if (lane == 0) U[k >> 6] |= 1ull << (k & 63);
                ++pc;
            }
            __syncwarp();
            j = k;
            walk_normalise<EPL>(t64, t, zero, ovf);
            if (ovf) {
                ++n_ovf;
                break;
            }
        }
        max_steps = steps > max_steps ? steps : max_steps;
    }
    if (lane == 0) {
        if (n_walk) atomicAdd(&a.ctr[C_SEEDS], n_walk);
        if (n_exp) atomicAdd(&a.ctr[C_EXP], n_exp);
        if (n_ovf) atomicAdd(&a.ctr[C_OVF], n_ovf);
        if (n_bal) atomicAdd(&a.ctr[C_BAL], n_bal);
        if (n_dead) atomicAdd(&a.ctr[C_PRUNED], n_dead);
        if (max_steps) atomicMax(&a.ctr[C_LEVELS], max_steps);
    }
}

// ---------------------------------------------------------------------------
// a7/a8: exact minimality test by elimination modulo primes, then append.
// ---------------------------------------------------------------------------

__device__ __forceinline__ uint32_t mulmod(uint32_t x, uint32_t y, uint32_t p, uint32_t c)
{
    // p = 2^31 - c: 2^31 == c (mod p)
    const uint64_t z = (uint64_t)x * y;
    const uint64_t r1 = (z & 0x7FFFFFFFull) + (z >> 31) * c;
    uint32_t r2 = (uint32_t)((r1 & 0x7FFFFFFFull) + (r1 >> 31) * c);
    if (r2 >= p) r2 -= p;
    return r2;
}

__device__ __forceinline__ uint32_t submod(uint32_t x, uint32_t y, uint32_t p) { return x >= y ? x - y : x + p - y; }

__device__ __forceinline__ uint32_t to_mod(int32_t s, uint32_t p)
{
    return s >= 0 ? (uint32_t)s : p - (uint32_t)(-s);
}

// coefficient S_int[row, col] from the column CSR (0 if absent)
__device__ __forceinline__ int32_t coef_at(const uint32_t *bl, const NetView &nv, int col, int row)
{
    for (int q = (int)bl[nv.o_colptr + col]; q < (int)bl[nv.o_colptr + col + 1]; ++q) {
        const uint32_t e = bl[nv.o_colent + q];
        if (ent_index(e) == row) return ent_coef(e);
    }
    return 0;
}

// Do the columns cols[0..nn) of S_int have full column rank modulo p?
// Rows touched by the columns are streamed; each is reduced against the
// echelon basis held in shared memory (lane l owns columns l and l + 32).
__device__ bool full_rank_mod_p(const uint32_t *bl, const NetView &nv, const int *cols, int nn, uint32_t p, uint32_t c,
                                uint32_t *basis /* [64][64] */, int *pivcol /* [64] */, uint32_t *rowmap /* M bits */,
                                int lane)
{
    const int mwords = (nv.M + 31) >> 5;
    for (int w = lane; w < mwords; w += 32) rowmap[w] = 0;
    __syncwarp();
    const int c0 = lane < nn ? cols[lane] : -1;
    const int c1 = lane + 32 < nn ? cols[lane + 32] : -1;
    int rank = 0;
    for (int j = 0; j < nn; ++j) {
        const int col = cols[j];
        for (int q = (int)bl[nv.o_colptr + col]; q < (int)bl[nv.o_colptr + col + 1]; ++q) {
            const int row = ent_index(bl[nv.o_colent + q]);
            const uint32_t word = rowmap[row >> 5];
            if ((word >> (row & 31)) & 1u) continue;
            __syncwarp();
            if (lane == 0) rowmap[row >> 5] = word | (1u << (row & 31));
            __syncwarp();
            uint32_t y0 = c0 >= 0 ? to_mod(coef_at(bl, nv, c0, row), p) : 0u;
            uint32_t y1 = c1 >= 0 ? to_mod(coef_at(bl, nv, c1, row), p) : 0u;
            // (cross-multiplied: scaling a row by a nonzero pivot keeps the rank,
            // and no inverse, a chain of 60 products, has to be taken)
            for (int i = 0; i < rank; ++i) {
                const int pc = pivcol[i];
                const uint32_t f = __shfl_sync(FULL, pc < 32 ? y0 : y1, pc & 31);
                if (f != 0) {
                    const uint32_t b = basis[i * 64 + pc];
                    y0 = submod(mulmod(y0, b, p, c), mulmod(f, basis[i * 64 + lane], p, c), p);
                    y1 = submod(mulmod(y1, b, p, c), mulmod(f, basis[i * 64 + lane + 32], p, c), p);
                }
            }
            const unsigned m0 = __ballot_sync(FULL, y0 != 0);
            const unsigned m1 = __ballot_sync(FULL, y1 != 0);
            if (m0 == 0 && m1 == 0) continue;
            const int pv = m0 ? __ffs((int)m0) - 1 : 32 + __ffs((int)m1) - 1;
            basis[rank * 64 + lane] = y0;
            basis[rank * 64 + lane + 32] = y1;
            if (lane == 0) pivcol[rank] = pv;
            __syncwarp();
            ++rank;
            if (rank == nn) return true;
        }
    }
    return false;
}

// The same test with the rows in the lanes, for columns that touch at most 64
// rows.  The submatrix stands in shared memory, a column of kRankStride words
// after the other (a lane's row and a column's entry in one row are both free
// of bank conflicts); a step finds a pivot for one column by ballot and only
// the rows with an entry in it change, and there only the columns of the pivot
// row's entries if the pivot is +-1.  A column without a pivot is a
// combination of those before it, which ends the test.
//
// One candidate is one warp's serial chain and most levels have fewer
// candidates than the chip has warps, so the chain's length is what counts: a
// row of 20 columns against a basis of 20 takes 20 dependent steps of 64-bit
// products in the streaming form above, a column here takes one.  One GB300, a
// core query: 22.4 -> 14.6 us a launch of the test (7 us of it the launch and
// the level state); calls: eight core targets at 2^17 9.46 -> 8.85 ms, a set of
// seeds 3.37 -> 3.09, one core query 2.39 -> 2.27, the genome-shaped network
// 24.3 -> 23.1.  Columns that touch more rows than that keep the streaming form.
constexpr int kRankStride = 65;

// row map of the columns and its prefix counts; returns the number of rows
__device__ int rank_rows(const uint32_t *bl, const NetView &nv, const int *cols, int nn, uint32_t *rowmap, int *prefix,
                         int lane)
{
    rowmap[lane] = 0;
    __syncwarp();
    for (int j = lane; j < nn; j += 32) {
        const int col = cols[j];
        for (int q = (int)bl[nv.o_colptr + col]; q < (int)bl[nv.o_colptr + col + 1]; ++q) {
            const int row = ent_index(bl[nv.o_colent + q]);
            atomicOr(&rowmap[row >> 5], 1u << (row & 31));
        }
    }
    __syncwarp();
    const int n = __popc(rowmap[lane]);
    int sum = n;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const int x = __shfl_up_sync(FULL, sum, off);
        if (lane >= off) sum += x;
    }
    prefix[lane] = sum - n;
    __syncwarp();
    return __shfl_sync(FULL, sum, 31);
}

__device__ bool full_rank_rows(const uint32_t *bl, const NetView &nv, const int *cols, int nn, uint32_t p, uint32_t c,
                               uint32_t *A /* [nn][kRankStride] */, const uint32_t *rowmap, const int *prefix, int lane)
{
    uint4 *z = reinterpret_cast<uint4 *>(A);
    for (int i = lane; i < (nn * kRankStride + 3) / 4; i += 32) z[i] = make_uint4(0u, 0u, 0u, 0u);
    __syncwarp();
    for (int j = lane; j < nn; j += 32) {
        const int col = cols[j];
        for (int q = (int)bl[nv.o_colptr + col]; q < (int)bl[nv.o_colptr + col + 1]; ++q) {
            const uint32_t e = bl[nv.o_colent + q];
            const int row = ent_index(e);
            const int at = prefix[row >> 5] + __popc(rowmap[row >> 5] & ((1u << (row & 31)) - 1u));
            A[j * kRankStride + at] = to_mod(ent_coef(e), p);
        }
    }
    __syncwarp();
    unsigned free0 = FULL, free1 = FULL;  // rows that are no pivot yet
    for (int j = 0; j < nn; ++j) {
        const uint32_t y0 = A[j * kRankStride + lane], y1 = A[j * kRankStride + 32 + lane];
        unsigned m0 = __ballot_sync(FULL, y0 != 0) & free0, m1 = __ballot_sync(FULL, y1 != 0) & free1;
        if ((m0 | m1) == 0) return false;
        const unsigned e0 = __ballot_sync(FULL, y0 == 1u || y0 == p - 1u) & m0;
        const unsigned e1 = __ballot_sync(FULL, y1 == 1u || y1 == p - 1u) & m1;
        const int r = e0 ? __ffs((int)e0) - 1 : e1 ? 31 + __ffs((int)e1) : m0 ? __ffs((int)m0) - 1 : 31 + __ffs((int)m1);
        const unsigned r0 = r < 32 ? 1u << r : 0u, r1 = r < 32 ? 0u : 1u << (r - 32);
        free0 &= ~r0;
        free1 &= ~r1;
        m0 &= ~r0;
        m1 &= ~r1;
        if ((m0 | m1) == 0) continue;
        const uint32_t b = A[j * kRankStride + r];
        const bool unit = b == 1u || b == p - 1u;
        // columns to change: the pivot row's entries, or all if rows are scaled
        // (cross-multiplied: no inverse, a chain of 60 products, is taken)
        unsigned long long todo;
        {
            const bool t0 = lane > j && lane < nn && (!unit || A[lane * kRankStride + r] != 0u);
            const bool t1 = lane + 32 > j && lane + 32 < nn && (!unit || A[(lane + 32) * kRankStride + r] != 0u);
            todo = (unsigned long long)__ballot_sync(FULL, t0) | (unsigned long long)__ballot_sync(FULL, t1) << 32;
        }
        const bool a0 = (m0 >> lane) & 1u, a1 = (m1 >> lane) & 1u;
        const uint32_t f0 = b == 1u || !unit ? y0 : p - y0, f1 = b == 1u || !unit ? y1 : p - y1;  // (y > 0 where used)
        while (todo) {
            uint32_t *x = A + (__ffsll((long long)todo) - 1) * kRankStride;
            todo &= todo - 1ull;
            const uint32_t t = x[r];
            if (a0) x[lane] = submod(unit ? x[lane] : mulmod(x[lane], b, p, c), mulmod(f0, t, p, c), p);
            if (a1) x[lane + 32] = submod(unit ? x[lane + 32] : mulmod(x[lane + 32], b, p, c), mulmod(f1, t, p, c), p);
        }
        __syncwarp();
    }
    return true;
}

// shared memory of one minimality warp: matrix, columns 64, pivots or prefix counts 64, row map 32
constexpr int kAcceptWarpWords = 64 * kRankStride + 64 + 64 + 32;

// Minimality test of the candidates [cand_begin, cand_end) by the warps
// gw = 0 .. nw-1; ws: this warp's shared-memory scratch (kAcceptWarpWords).
__device__ void accept_range(const NetView &nv, const AcceptArgs &a, uint32_t *ws, int64_t gw, int64_t nw)
{
    const int lane = threadIdx.x & 31;
    const int W = nv.W;
    uint32_t *basis = ws;
    int *cols = reinterpret_cast<int *>(ws + 64 * kRankStride);
    int *pivcol = cols + 64;
    uint32_t *rowmap = reinterpret_cast<uint32_t *>(pivcol + 64);
    const uint32_t *bl = nv.blob;
    unsigned long long n_acc = 0;
    for (int64_t ci = a.cand_begin + gw; ci < a.cand_end; ci += nw) {
        const uint64_t *U = a.cand + (size_t)ci * W;
        const uint64_t u0 = lane < W ? U[lane] : 0ull;
        const uint64_t u1 = lane + 32 < W ? U[lane + 32] : 0ull;
        const int n = support_columns(u0, u1, cols);
        if (n > 64) {
            if (lane == 0) atomicOr(&a.ctr[C_ERR], (unsigned long long)ERR_LEN);
            continue;
        }
        // Drop one column: the kept nn = n - 1 columns must be independent.
        // (The balanced flux ray is positive on every column of U, so the
        // dropped column is a combination of the others.)
        const int nn = n - 1;
        uint32_t hb = 0;
        if (lane < nn) hb += bl[nv.o_hbits + cols[lane]];
        if (lane + 32 < nn) hb += bl[nv.o_hbits + cols[lane + 32]];
        hb = __reduce_add_sync(FULL, hb);  // log2 of the squared Hadamard bound
        const int kp = (int)(hb / 61u) + 1;  // each prime gives > 2^30.5 = 2^(61/2)
        if (kp > kNumPrimes) {
            if (lane == 0) atomicOr(&a.ctr[C_ERR], (unsigned long long)ERR_PRIMES);
            continue;
        }
        bool ok = nn == 0;
        __syncwarp();
        const int rows = rank_rows(bl, nv, cols, nn, rowmap, pivcol, lane);
        for (int pi = 0; pi < kp && !ok && rows >= nn; ++pi) {
            const uint32_t cc = c_prime_c[pi];
            if (rows <= 64)
                ok = full_rank_rows(bl, nv, cols, nn, 0x80000000u - cc, cc, basis, rowmap, pivcol, lane);
            else
                ok = full_rank_mod_p(bl, nv, cols, nn, 0x80000000u - cc, cc, basis, pivcol, rowmap, lane);
            __syncwarp();
        }
        if (ok) {
            unsigned long long idx = 0;
            if (lane == 0) idx = atomicAdd(&a.ctr[C_RES_N], 1ull);
            idx = __shfl_sync(FULL, idx, 0);
            if ((int64_t)idx < a.res_cap) {
                uint64_t *dst = a.res + (size_t)idx * W;
                if (lane < W) dst[lane] = u0;
                if (lane + 32 < W) dst[lane + 32] = u1;
                if (a.rcols) {
                    uint16_t *lst = a.rcols + (size_t)idx * kRcolStride;
                    for (int j = lane; j < n; j += 32) lst[1 + j] = (uint16_t)cols[j];
                    if (lane == 0) lst[0] = (uint16_t)n;
                }
                if ((int64_t)idx < a.ix.room)
                    file_result(a.ix, W, (int64_t)idx, cols, n, __shfl_sync(FULL, u0, 0), __shfl_sync(FULL, u0, 1));
            } else if (lane == 0) {
                atomicOr(&a.ctr[C_ERR], (unsigned long long)ERR_RES_CAP);
            }
            ++n_acc;
        }
        __syncwarp();
    }
    if (lane == 0 && n_acc) atomicAdd(&a.ctr[C_RES], n_acc);
}

__device__ __forceinline__ uint64_t next_pow2_dev(uint64_t x)
{
    uint64_t p = 1;
    while (p < x) p <<= 1;
    return p;
}

// Levels without a host round trip.  With one launch list and one counter copy
// per level (15 calls, 60-90 us a level at small frontiers) the small searches
// waited on the host: the last CTA of the minimality test now decides the
// level and sets the next one's parameters, and the host launches up to four
// levels (three kernels each) ahead.  One GB300, calls through the library:
// the smallest query 1.28 -> 0.87 ms, one core query 3.1 -> 2.4, eight core
// targets at 2^17 13.6 -> 9.3, a 400-row network 5.4 -> 4.1.

// The end of a level (one thread, after every CTA of its last launch is done):
// the decisions on it, and the next level's parameters.  v: the counters and
// the state as they stand.
__device__ void advance_level(const AcceptArgs &a, const unsigned long long *v)
{
    unsigned long long *c = a.ctr, *st = a.st;
    const unsigned long long *sv = v + C_COUNT;
    auto get = [&](int i) { return v[i]; };
    const bool seeds = a.advance == 3;
    st[S_PENDING] = 0ull;
    if (!seeds) st[S_EXPANDS] = sv[S_EXPANDS] + 1;
    if (a.advance == 1) return;
    const uint64_t next = get(C_NEXT), unv = get(C_UNV), written = seeds ? next : get(C_WRITTEN);
    const uint64_t deg = get(C_DEGSUM), units = get(C_PAY), unwritten = get(C_UNWRITTEN);
    const uint64_t front = next + (unwritten ? unv : 0ull);
    const uint64_t kept = seeds ? units : get(C_KEPT);  // (seeds take what they reserve)
    // algorithmic bytes: the header and payload of every distinct parent and
    // new state, 16 bytes of slot traffic per child
    if (!seeds)
        st[S_BYTES] = sv[S_BYTES] + 16 * (sv[S_NFRONT] + sv[S_UNITS] + next + kept + (get(C_EXP) - sv[S_SNAP]));
    unsigned long long stop = STOP_NONE;
    if (get(C_ERR)) {
        stop = STOP_ERROR;
    } else if (a.max_frontier > 0 && (int64_t)front > a.max_frontier) {
        stop = STOP_TRUNCATED;
    } else if (seeds && (int64_t)next > a.child_rows) {  // more seeds than rows
        atomicOr(&c[C_ERR], (unsigned long long)ERR_TABLE_FULL);
        stop = STOP_ERROR;
    } else if (unwritten) {
        st[S_STOP] = STOP_RERUN;  // the counters stay as they are for the host
        return;
    }
    st[S_LEVEL] = (unsigned long long)a.level;
    st[S_NROWS] = written < (uint64_t)a.child_rows ? written : (uint64_t)a.child_rows;
    st[S_NFRONT] = front;
    st[S_DEG] = deg;
    st[S_UNITS] = kept;
    if (stop == STOP_NONE) {
        st[S_FRONTIER] = sv[S_FRONTIER] + front;
        if (front > sv[S_FRONTIER_MAX]) st[S_FRONTIER_MAX] = front;
        if (a.max_results > 0 && (int64_t)get(C_RES) >= a.max_results) stop = STOP_CAPPED;
        else if (front == 0) stop = STOP_DONE;
        else if (a.level + 1 > a.max_level) {  // every step adds a column or a secondary step: unreachable
            atomicOr(&c[C_ERR], (unsigned long long)ERR_WATCHDOG);
            stop = STOP_ERROR;
        }
    }
    // rows and payload units one warp reserves at a time: at large levels about
    // a 16th of what it writes (what stays unused is dead weight in the arena),
    // else exactly what a round needs
    uint64_t blk = deg / (16ull * (uint64_t)a.warps);
    blk = blk > 512 ? 512 : (blk < 32 ? 0 : blk);
    const uint64_t avg = written ? units / written : 8;
    const uint64_t reserved = deg + blk * (uint64_t)a.warps + 64;
    const uint64_t slots = next_pow2_dev(2 * reserved + 64);
    st[S_BLK] = blk;
    st[S_PAY_BLK] = blk * (avg + 2);
    st[S_RESERVED] = reserved;
    st[S_SLOTS] = slots;
    const int snap[] = {C_EXP, C_OVF, C_BAL, C_PRUNED, C_ZERO};
    for (int i = 0; i < 5; ++i) st[S_SNAP + i] = get(snap[i]);
    if (stop == STOP_NONE && (int64_t)get(C_RES_N) > a.ix.room) stop = STOP_INDEX;
    if (stop == STOP_NONE && ((int64_t)reserved > a.fp_cap || slots > a.slot_cap)) stop = STOP_TABLES;
    const int clear[] = {C_NEXT, C_DEGSUM, C_WRITTEN, C_UNWRITTEN, C_UNV, C_PAY, C_KEPT, C_DEDUP_BEGIN};
    if (stop == STOP_NONE || stop == STOP_INDEX || stop == STOP_TABLES)
        for (int i = 0; i < 8; ++i) c[clear[i]] = 0ull;
    st[S_STOP] = stop;
}

__global__ void __launch_bounds__(kAcceptWarps * 32) accept_kernel(NetView nv, AcceptArgs a)
{
    extern __shared__ __align__(16) uint32_t smem[];
    const int wid = threadIdx.x >> 5;
    if (a.advance) {
        if (a.st[S_STOP] != STOP_NONE) return;
        // a level that will run again is judged then: nothing may be filed before
        const uint64_t front = a.ctr[C_NEXT] + a.ctr[C_UNV];
        const bool rerun = a.advance == 2 && a.ctr[C_UNWRITTEN] != 0ull &&
                           !(a.max_frontier > 0 && (int64_t)front > a.max_frontier);
        // the expansion launches before this one have finished: the range is stable
        a.cand_begin = (int64_t)a.ctr[C_ACC_BEGIN];
        const int64_t n = (int64_t)a.ctr[C_CAND_N];
        a.cand_end = rerun ? a.cand_begin : (n < a.cand_cap ? n : a.cand_cap);
    }
    const int64_t cand_end = a.cand_end;
    accept_range(nv, a, smem + wid * kAcceptWarpWords, (int64_t)blockIdx.x * kAcceptWarps + wid,
                 (int64_t)gridDim.x * kAcceptWarps);
    if (!a.advance) return;
    // the last CTA moves the level state on
    __shared__ int s_last;
    __shared__ unsigned long long s_ctr[C_COUNT + S_COUNT];
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(&a.st[S_TICKET], 1ull) == (unsigned long long)gridDim.x - 1;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    for (int i = threadIdx.x; i < C_COUNT + S_COUNT; i += blockDim.x) s_ctr[i] = __ldcg(&a.ctr[i]);  // (the state follows)
    __syncthreads();
    if (threadIdx.x == 0) {
        a.st[S_TICKET] = 0ull;
        a.ctr[C_ACC_BEGIN] = (unsigned long long)cand_end;
        a.ctr[C_DEDUP_BEGIN] = s_ctr[C_WRITTEN];  // (a chunk; a level clears it)
        a.ctr[C_OPEN] = 0ull;
        advance_level(a, s_ctr);
    }
}

// ---------------------------------------------------------------------------
// output order: (|U|, ascending column list), bitonic sort of indices
// ---------------------------------------------------------------------------

__device__ bool support_greater(const uint64_t *res, int W, uint32_t x, uint32_t y)
{
    if (x == 0xFFFFFFFFu) return y != 0xFFFFFFFFu;
    if (y == 0xFFFFFFFFu) return false;
    const uint64_t *a = res + (size_t)x * W, *b = res + (size_t)y * W;
    int ca = 0, cb = 0;
    for (int w = 0; w < W; ++w) {
        ca += __popcll(a[w]);
        cb += __popcll(b[w]);
    }
    if (ca != cb) return ca > cb;
    for (int w = 0; w < W; ++w) {
        const uint64_t d = a[w] ^ b[w];
        if (d) {
            const uint64_t low = d & (~d + 1);
            return (a[w] & low) == 0;  // the set holding the smaller column is smaller
        }
    }
    return false;
}

// Sort record of a support: |U| and its nine lowest columns, 12 bits each --
// the order of the records is the order of the supports but for ties, which
// the words decide -- and the support's index.  Padding sorts last.  (With a
// record of four columns, 2^14 genome-shaped results took 2.0 ms, most of it
// in the ties.)
struct SortRec {
    unsigned long long key, key2;
    uint32_t idx, pad;
};

constexpr int kSortBlock = 512;            // threads
constexpr int kSortTile = 2 * kSortBlock;  // records a block sorts in shared memory

__global__ void sort_init_kernel(const uint64_t *res, int W, SortRec *rec, int64_t n, int64_t n2)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n2) return;
    SortRec r{~0ull, ~0ull, 0xFFFFFFFFu, 0u};
    if (i < n) {
        const uint64_t *U = res + (size_t)i * W;
        int pc = 0, got = 0;
        unsigned long long low = 0, low2 = 0;
        for (int w = 0; w < W; ++w) {
            uint64_t x = U[w];
            pc += __popcll(x);
            for (; x && got < 9; x &= x - 1, ++got) {
                const unsigned long long c = (unsigned)(w * 64 + __ffsll((long long)x) - 1);
                if (got < 4) low |= c << (36 - 12 * got);
                else low2 |= c << (48 - 12 * (got - 4));
            }
        }
        // (a support with fewer columns than another differs in |U|)
        r.key = ((unsigned long long)pc << 48) | low;
        r.key2 = low2;
        r.idx = (uint32_t)i;
    }
    rec[i] = r;
}

__device__ __forceinline__ bool rec_greater(const uint64_t *res, int W, const SortRec &x, const SortRec &y)
{
    if (x.key != y.key) return x.key > y.key;
    if (x.key2 != y.key2) return x.key2 > y.key2;
    return support_greater(res, W, x.idx, y.idx);
}

// the sort without keys, for callers whose scratch holds 4 bytes a support
__device__ __forceinline__ bool rec_greater(const uint64_t *res, int W, uint32_t x, uint32_t y)
{
    return support_greater(res, W, x, y);
}
__device__ __forceinline__ uint32_t rec_index(uint32_t r) { return r; }
__device__ __forceinline__ uint32_t rec_index(const SortRec &r) { return r.idx; }

__global__ void sort_init_kernel(const uint64_t *, int, uint32_t *idx, int64_t n, int64_t n2)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n2) idx[i] = i < n ? (uint32_t)i : 0xFFFFFFFFu;
}

template <typename Rec>
__global__ void bitonic_step_kernel(const uint64_t *res, int W, Rec *rec, int64_t n2, int64_t k, int64_t j)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n2) return;
    const int64_t l = i ^ j;
    if (l <= i) return;
    const Rec x = rec[i], y = rec[l];
    const bool up = (i & k) == 0;
    if (rec_greater(res, W, x, y) == up) {
        rec[i] = y;
        rec[l] = x;
    }
}

// The steps with partners inside a tile, in shared memory: the merges
// k = k0, 2 k0, ... k1, each from j = min(k, tile) / 2 down.
template <typename Rec>
__global__ void __launch_bounds__(kSortBlock) bitonic_tile_kernel(const uint64_t *res, int W, Rec *rec, int64_t n2,
                                                                  int64_t k0, int64_t k1)
{
    __shared__ Rec t[kSortTile];
    const int64_t base = (int64_t)blockIdx.x * kSortTile;
    const int n = (int)(n2 - base < kSortTile ? n2 - base : kSortTile);  // a power of two
    for (int i = threadIdx.x; i < n; i += kSortBlock) t[i] = rec[base + i];
    for (int64_t k = k0; k <= k1; k <<= 1)
        for (int j = (int)(k < n ? k : n) >> 1; j > 0; j >>= 1) {
            __syncthreads();
            for (int q = threadIdx.x; q < n / 2; q += kSortBlock) {
                const int i = ((q & ~(j - 1)) << 1) | (q & (j - 1)), l = i | j;
                const bool up = ((base + i) & k) == 0;
                const Rec x = t[i], y = t[l];
                if (rec_greater(res, W, x, y) == up) {
                    t[i] = y;
                    t[l] = x;
                }
            }
        }
    __syncthreads();
    for (int i = threadIdx.x; i < n; i += kSortBlock) rec[base + i] = t[i];
}

template <typename Rec>
__global__ void gather_kernel(const uint64_t *res, int W, const Rec *rec, int64_t n_keep, uint64_t *out)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n_keep * W) return;
    const int64_t r = i / W;
    const int w = (int)(i % W);
    out[i] = res[(size_t)rec_index(rec[r]) * W + w];
}

// ---------------------------------------------------------------------------
// Batched traversal: one persistent launch over many (network, target) jobs.
// Each CTA pulls jobs from a device queue and runs the whole level loop of a
// job (seed, generate, dedup, minimality test, sorted output) with CTA
// barriers between the steps, in its own slice of a scratch pool.  The steps
// are the grid-wide level pass's device code and the level decisions
// (truncation, cap, counters) those of the single-job path.  A job whose
// levels do not fit the slice (its rows before deduplication, or more results
// than the superset index holds) is left to the host, which runs it by itself.
// ---------------------------------------------------------------------------

// CTA-level sort of results [0, n) into out (first n_keep rows)
__device__ void cta_sort(const uint64_t *res, int64_t n, int W, uint32_t *idx, uint64_t *out, int64_t n_keep)
{
    if (n <= 0 || n_keep <= 0) return;
    const int64_t n2 = (int64_t)next_pow2_dev((uint64_t)n);
    for (int64_t i = threadIdx.x; i < n2; i += blockDim.x) idx[i] = i < n ? (uint32_t)i : 0xFFFFFFFFu;
    __syncthreads();
    for (int64_t k = 2; k <= n2; k <<= 1)
        for (int64_t j = k >> 1; j > 0; j >>= 1) {
            for (int64_t i = threadIdx.x; i < n2; i += blockDim.x) {
                const int64_t l = i ^ j;
                if (l <= i) continue;
                const uint32_t x = idx[i], y = idx[l];
                const bool up = (i & k) == 0;
                if (support_greater(res, W, x, y) == up) {
                    idx[i] = y;
                    idx[l] = x;
                }
            }
            __syncthreads();
        }
    for (int64_t i = threadIdx.x; i < n_keep * W; i += blockDim.x) out[i] = res[(size_t)idx[i / W] * W + i % W];
    __syncthreads();
}

constexpr int kBatchAcceptWarps = 2;

// 16-byte stores of ~0 (the regions are multiples of 16 bytes)
__device__ __forceinline__ void cta_fill(void *p, size_t bytes)
{
    uint4 *t = reinterpret_cast<uint4 *>(p);
    for (size_t i = threadIdx.x; i < bytes / 16; i += blockDim.x) t[i] = make_uint4(~0u, ~0u, ~0u, ~0u);
}

template <int F>
__device__ void run_job(const BatchArgs &ba, const BatchJob &job, char *slice, uint32_t *sm, const NetView &nv,
                        LevelArgs &a, AcceptArgs &acc, unsigned long long *sh)
{
    unsigned long long *ctr = job.ctr;
    const int tid = threadIdx.x, nthreads = blockDim.x, nwarps = blockDim.x >> 5;
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const BatchLayout &L = ba.layout;
    const BoundScratch no_bound{};
    auto arena = [&](int i) {
        Arena r{};
        r.hdr = reinterpret_cast<uint4 *>(slice + L.o_hdr[i]);
        r.pay = reinterpret_cast<uint4 *>(slice + L.o_pay[i]);
        r.cap = L.cap;
        r.pay_cap = L.pay_cap;
        return r;
    };
    if (tid == 0) {
        a = LevelArgs{};
        a.slots = reinterpret_cast<unsigned long long *>(slice + L.o_slots);
        a.cslots = reinterpret_cast<unsigned long long *>(slice + L.o_cslots);
        a.cslot_mask = L.cslot_cap - 1;
        a.cand = reinterpret_cast<uint64_t *>(slice + L.o_cand);
        a.cand_cap = L.cand_cap;
        a.res = reinterpret_cast<const uint64_t *>(slice + L.o_res);
        a.rcols = reinterpret_cast<const uint16_t *>(slice + L.o_rcols);
        a.fp = reinterpret_cast<uint64_t *>(slice + L.o_fp);
        a.fp_cap = L.fp_cap;
        a.open = reinterpret_cast<uint32_t *>(slice + L.o_open);
        a.max_len = job.max_len;
        a.max_sec = ba.max_sec;
        a.ctr = ctr;
        a.child = arena(0);
        CellIndex &ix = a.cells;
        ix.cells = reinterpret_cast<uint2 *>(slice + L.o_cells);
        ix.mask = L.cell_mask;
        ix.ent = reinterpret_cast<uint4 *>(slice + L.o_ent);
        ix.ksig = reinterpret_cast<uint64_t *>(slice + L.o_ksig);
        ix.single = reinterpret_cast<uint32_t *>(slice + L.o_single);
        ix.cnt = reinterpret_cast<int32_t *>(slice + L.o_cnt);
        ix.ent_stride = L.ent_stride;
        ix.room = L.index_room;
        acc = AcceptArgs{};
        acc.cand = a.cand;
        acc.res = reinterpret_cast<uint64_t *>(slice + L.o_res);
        acc.res_cap = L.res_cap;
        acc.rcols = F == 0 ? reinterpret_cast<uint16_t *>(slice + L.o_rcols) : nullptr;
        acc.ctr = ctr;
        acc.ix = ix;
    }
    cta_fill(slice + L.o_cslots, L.cslot_cap * 8);
    __syncthreads();
    auto read_ctr = [&]() {
        __syncthreads();
        for (int i = tid; i < C_COUNT; i += nthreads) sh[i] = __ldcg(&ctr[i]);
        __syncthreads();
    };
    auto set_ctr = [&](int i, unsigned long long v) {
        if (tid == 0) ctr[i] = v;
    };
    const unsigned ERRMASK = ERR_TIMEOUT | ERR_CAND_CAP | ERR_RES_CAP | ERR_TABLE_FULL | ERR_PRIMES | ERR_LEN |
                             ERR_WATCHDOG | ERR_BOUNDS;
    bool index_ready = false;
    int64_t cand_done = 0;
    // the minimality test of the candidates since the last one (sh is current)
    auto accept_new = [&]() {
        const int64_t end = (int64_t)min(sh[C_CAND_N], (unsigned long long)L.cand_cap);
        if (end > cand_done) {
            if (!index_ready) {  // (most jobs' first levels accept nothing)
                for (int i = tid; i < nv.N; i += nthreads) {
                    a.cells.cnt[i] = 0;
                    a.cells.single[i] = 0u;
                    a.cells.ksig[2 * i] = a.cells.ksig[2 * i + 1] = 0ull;
                }
                cta_fill(a.cells.cells, F ? (size_t)128 * 4 * nv.N : 8 * ((size_t)L.cell_mask + 1));
                index_ready = true;
            }
            if (tid == 0) {
                acc.cand_begin = cand_done;
                acc.cand_end = end;
            }
            __syncthreads();
            if (wid < kBatchAcceptWarps) accept_range(nv, acc, sm + wid * kAcceptWarpWords, wid, kBatchAcceptWarps);
        }
        cand_done = end;
        read_ctr();
    };

    // level 0: seeds, then the minimality test of balanced seeds
    int cur = 0;
    seed_range<F, false>(nv, a, job.target, tid, nthreads);
    read_ctr();
    if (sh[C_ERR] & ERRMASK) return;
    accept_new();
    if (sh[C_ERR] & ERRMASK) return;
    int64_t res_n = (int64_t)min(sh[C_RES_N], (unsigned long long)L.res_cap);
    int64_t n_front = (int64_t)sh[C_NEXT], n_rows = n_front;
    uint64_t deg_sum = sh[C_DEGSUM];
    unsigned long long status = 0, frontier = 0, frontier_max = 0, levels = 1;
    bool stop = false;
    if (n_front > ba.max_frontier) {
        status |= EFM_TRUNCATED;
        stop = true;
    } else {
        frontier += n_front;
        frontier_max = max(frontier_max, (unsigned long long)n_front);
        if (ba.max_results > 0 && (int64_t)sh[C_RES] >= ba.max_results) {
            status |= EFM_CAPPED;
            stop = true;
        }
    }
    for (int level = 1; !stop && n_front > 0; ++level) {
        if (level > a.max_len + a.max_sec + 1) {
            if (tid == 0) atomicOr(&ctr[C_ERR], (unsigned long long)ERR_WATCHDOG);
            return;
        }
        const uint64_t reserved = deg_sum + 64;
        const uint64_t nslots = next_pow2_dev(2 * reserved + 64);
        if ((int64_t)reserved > L.fp_cap || nslots > L.slot_cap || res_n > L.index_room) {
            set_ctr(C_DONE, 2ull);  // to the host
            return;
        }
        cta_fill(slice + L.o_slots, nslots * 8);
        const int clear[] = {C_NEXT, C_DEGSUM, C_WRITTEN, C_UNWRITTEN, C_UNV, C_PAY, C_OPEN, C_DEDUP_BEGIN};
        if (tid == 0) {
            for (int i = 0; i < 8; ++i) ctr[clear[i]] = 0ull;
            a.par = arena(cur);
            a.child = arena(cur ^ 1);
            a.level = level;
        }
        __syncthreads();
        const int cpw = (int)min((int64_t)ba.tile, max((int64_t)1, (n_rows + nwarps - 1) / nwarps));
        generate_range<F, false, false, true>(nv, a, n_rows, cpw, 0, 0, res_n > 0, wid, nwarps, nullptr, no_bound);
        __syncthreads();
        DedupSums sum;
        // (counters past L1: this SM may hold older ones)
        dedup_range<F, false>(nv, a, nslots - 1, __ldcg(&ctr[C_DEDUP_BEGIN]), __ldcg(&ctr[C_WRITTEN]),
                              __ldcg(&ctr[C_OPEN]), tid & ~31, tid & ~31, nthreads, sum);
        unsigned keep = __reduce_add_sync(FULL, sum.keep), unv = __reduce_add_sync(FULL, sum.unv);
        unsigned deg = __reduce_add_sync(FULL, (unsigned)sum.deg_units);  // (far below 2^32 in a slice)
        if (lane == 0) {
            if (keep) atomicAdd(&ctr[C_NEXT], (unsigned long long)keep);
            if (unv) atomicAdd(&ctr[C_UNV], (unsigned long long)unv);
            if (deg) atomicAdd(&ctr[C_DEGSUM], (unsigned long long)deg);
        }
        read_ctr();
        if (sh[C_ERR] & ERRMASK) return;
        const bool unwritten = sh[C_UNWRITTEN] != 0ull;
        n_front = (int64_t)(sh[C_NEXT] + (unwritten ? sh[C_UNV] : 0ull));
        if (unwritten && n_front <= ba.max_frontier) {
            set_ctr(C_DONE, 2ull);  // not decided: to the host
            return;
        }
        n_rows = (int64_t)min(sh[C_WRITTEN], (unsigned long long)L.cap);
        deg_sum = sh[C_DEGSUM];
        accept_new();
        if (sh[C_ERR] & ERRMASK) return;
        res_n = (int64_t)min(sh[C_RES_N], (unsigned long long)L.res_cap);
        levels = level + 1;
        cur ^= 1;
        if (n_front > ba.max_frontier) {
            status |= EFM_TRUNCATED;
            break;
        }
        frontier += n_front;
        frontier_max = max(frontier_max, (unsigned long long)n_front);
        if (ba.max_results > 0 && (int64_t)sh[C_RES] >= ba.max_results) {
            status |= EFM_CAPPED;
            break;
        }
    }
    if ((int64_t)sh[C_RES_N] > L.res_cap) {
        if (tid == 0) atomicOr(&ctr[C_ERR], (unsigned long long)ERR_RES_CAP);
        return;
    }
    const int64_t n_keep = ba.max_results > 0 ? min(res_n, ba.max_results) : res_n;
    cta_sort(acc.res, res_n, nv.W, reinterpret_cast<uint32_t *>(slice + L.o_sort), job.out, n_keep);
    if (sh[C_OVF]) status |= EFM_OVERFLOW_DROPPED;
    set_ctr(C_LEVELS, levels);
    set_ctr(C_FRONTIER, frontier);
    set_ctr(C_FRONTIER_MAX, frontier_max);
    set_ctr(C_STATUS, status);
    set_ctr(C_OUT_N, (unsigned long long)n_keep);
    set_ctr(C_DONE, 1ull);
}

// The levels of one search while they are small, by one CTA: from the state's
// level on, until the search stops, a level has more than `limit` branches, or
// one has more new balanced supports than a few warps should judge (S_PENDING:
// the grid then ends that level).
// Latency bounds such a level: three launches of chains of dependent reads,
// each on a cold L1.  Here a barrier ends a phase, and the network's tables and
// the rows just written are in the SM's L1.  One GB300, with three launches for
// every level and this way: the smallest query 0.835 -> 0.739 ms, eight core
// targets at 2^17 8.86 -> 8.06, a 400-row network 4.13 -> 3.92, the subtractive
// variant 6.07 -> 5.83, a set of seeds 3.09 -> 2.95.
constexpr int kSmallWarps = 16;
constexpr int kSmallAcceptWarps = 8;

template <int F, bool SUB>
__global__ void __launch_bounds__(kSmallWarps * 32, 1) small_kernel(const __grid_constant__ NetView nv,
                                                                    const __grid_constant__ LevelArgs a0,
                                                                    const __grid_constant__ AcceptArgs acc0,
                                                                    const __grid_constant__ Arena first,
                                                                    const __grid_constant__ Arena second, int limit)
{
    extern __shared__ __align__(16) uint32_t smem[];
    __shared__ LevelArgs a;
    __shared__ AcceptArgs acc;
    __shared__ unsigned long long v[C_COUNT + S_COUNT];
    const int tid = threadIdx.x, nthreads = kSmallWarps * 32, wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const unsigned long long *sv = v + C_COUNT;
    const BoundScratch no_bound{};
    auto read_state = [&]() {
        __syncthreads();
        for (int i = tid; i < C_COUNT + S_COUNT; i += nthreads) v[i] = __ldcg(&a0.ctr[i]);
        __syncthreads();
    };
    if (tid == 0) {
        a = a0;
        acc = acc0;
    }
    for (bool odd = false;; odd = !odd) {
        read_state();
        if (sv[S_STOP] != STOP_NONE || sv[S_DEG] > (unsigned long long)limit || sv[S_NROWS] > (unsigned long long)limit)
            return;
        const uint64_t slots = sv[S_SLOTS];
        const int64_t n_par = (int64_t)sv[S_NROWS];
        const bool any_result = v[C_RES_N] != 0ull;
        cta_fill(a0.slots, slots * 8);
        if (tid == 0) {
            a.par = odd ? second : first;
            a.child = odd ? first : second;
            a.level = acc.level = (int)sv[S_LEVEL] + 1;
            acc.child_rows = a.child.cap;
        }
        __syncthreads();
        const int cpw = (int)min((int64_t)32, max((int64_t)1, (n_par + kSmallWarps - 1) / kSmallWarps));
        generate_range<F, SUB, false, true>(nv, a, n_par, cpw, 0, 0, any_result, wid, kSmallWarps, nullptr, no_bound);
        read_state();
        DedupSums sum;
        dedup_range<F, SUB>(nv, a, slots - 1, v[C_DEDUP_BEGIN], v[C_WRITTEN], v[C_OPEN], tid & ~31, tid & ~31, nthreads,
                            sum);
        const unsigned keep = __reduce_add_sync(FULL, sum.keep), unv = __reduce_add_sync(FULL, sum.unv);
        const unsigned units = __reduce_add_sync(FULL, (unsigned)(sum.deg_units >> 32));
        const unsigned deg = __reduce_add_sync(FULL, (unsigned)sum.deg_units);  // (limit children of at most 2^13 branches)
        if (lane == 0) {
            if (keep) atomicAdd(&a.ctr[C_NEXT], (unsigned long long)keep);
            if (unv) atomicAdd(&a.ctr[C_UNV], (unsigned long long)unv);
            if (units) atomicAdd(&a.ctr[C_KEPT], (unsigned long long)units);
            if (deg) atomicAdd(&a.ctr[C_DEGSUM], (unsigned long long)deg);
        }
        read_state();
        // (as in the launch for one level: one that will run again is judged then)
        const bool rerun = v[C_UNWRITTEN] != 0ull &&
                           !(acc.max_frontier > 0 && (int64_t)(v[C_NEXT] + v[C_UNV]) > acc.max_frontier);
        const int64_t begin = (int64_t)v[C_ACC_BEGIN], n = (int64_t)v[C_CAND_N];
        const int64_t end = rerun ? begin : (n < acc.cand_cap ? n : acc.cand_cap);
        if (end - begin > kSmallCandidates) {
            if (tid == 0) a0.st[S_PENDING] = 1ull;
            return;
        }
        if (end > begin) {
            if (tid == 0) {
                acc.cand_begin = begin;
                acc.cand_end = end;
            }
            __syncthreads();
            if (wid < kSmallAcceptWarps)
                accept_range(nv, acc, smem + wid * kAcceptWarpWords, wid, kSmallAcceptWarps);
            read_state();
        }
        if (tid == 0) {
            a.ctr[C_ACC_BEGIN] = (unsigned long long)end;
            a.ctr[C_DEDUP_BEGIN] = v[C_WRITTEN];
            a.ctr[C_OPEN] = 0ull;
            advance_level(acc, v);
        }
    }
}

// A CTA takes jobs off a queue and runs each through the same level pass, its
// states, tables and index in the CTA's slice of the pool.  Latency bounds it:
// a level of a small job is a chain of short phases with barriers between, so
// what counts is how fast one CTA goes through its job.  With 128 registers
// (two CTAs of 8 warps on an SM) 512 uneven networks take 5.4 ms, with 85 and
// three CTAs 5.6 to 6.0, with 64 and four 6.0 to 6.2 (spills); on rows of every
// metabolite, with 255 registers and one CTA, the call took 15.8 before its
// fetches and takes 6.2 now.
__global__ void __launch_bounds__(kBatchThreads, 2) batch_kernel(const __grid_constant__ BatchArgs ba)
{
    extern __shared__ __align__(16) uint32_t smem[];
    __shared__ int s_job;
    __shared__ NetView s_nv;
    __shared__ LevelArgs s_a;
    __shared__ AcceptArgs s_acc;
    __shared__ unsigned long long s_ctr[C_COUNT];
    char *slice = ba.pool + (size_t)blockIdx.x * ba.layout.slice_bytes;
    const int chunk = ba.chunk > 0 ? ba.chunk : 1;
    for (;;) {
        if (threadIdx.x == 0) s_job = (int)atomicAdd(ba.queue, (unsigned)chunk);
        __syncthreads();
        const int q0 = s_job;
        __syncthreads();
        if (q0 >= ba.n_jobs) break;
        for (int qi = q0; qi < q0 + chunk && qi < ba.n_jobs; ++qi) {
            const BatchJob &job = ba.jobs[ba.order[qi]];
            if (threadIdx.x == 0) s_nv = job.nv;
            __syncthreads();
            if (s_nv.form == 2) run_job<2>(ba, job, slice, smem, s_nv, s_a, s_acc, s_ctr);
            else if (s_nv.form == 1) run_job<1>(ba, job, slice, smem, s_nv, s_a, s_acc, s_ctr);
            else run_job<0>(ba, job, slice, smem, s_nv, s_a, s_acc, s_ctr);
            __syncthreads();
        }
    }
}

}  // namespace

cudaError_t launch_accept_new(const NetView &nv, const AcceptArgs &a, int sm_count, cudaStream_t s)
{
    const size_t sm = (size_t)kAcceptWarps * kAcceptWarpWords * 4;
    const cudaError_t e = cudaFuncSetAttribute(accept_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    accept_kernel<<<sm_count, kAcceptWarps * 32, sm, s>>>(nv, a);
    return cudaGetLastError();
}

cudaError_t launch_accept(const NetView &nv, const AcceptArgs &a, cudaStream_t s)
{
    const int64_t n = a.cand_end - a.cand_begin;
    if (n <= 0) return cudaSuccess;
    const size_t sm = (size_t)kAcceptWarps * kAcceptWarpWords * 4;
    // (each time: the attribute belongs to the device, and to its context)
    const cudaError_t e = cudaFuncSetAttribute(accept_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return e;
    int64_t blocks = (n + kAcceptWarps - 1) / kAcceptWarps;
    if (blocks > 4096) blocks = 4096;
    accept_kernel<<<(int)blocks, kAcceptWarps * 32, sm, s>>>(nv, a);
    return cudaGetLastError();
}

cudaError_t launch_walks(const NetView &nv, const LevelArgs &a, int target, uint64_t seed, int64_t n_walks, int sm_count,
                         cudaStream_t s)
{
    if (n_walks <= 0) return cudaSuccess;
    // A lane takes a walk in several times the time of a warp, so few walks go to
    // a warp each.  Kernel times of n walks by warps grow with n, by lanes they
    // are level until the chip is full: they meet at 68 walks an SM on the
    // smallest network (one row a lane of the warp; 0.046 against 0.124 ms at
    // 1000 walks, 0.173 / 0.130 at 16000), at half of that on the core-shaped one
    // (two rows; 0.103 / 0.193 at 1000, 0.259 / 0.193 at 8000), and where
    // reactions are long, whose rows a lane takes one by one, at 110 (0.148 /
    // 0.916 at 1000, 0.828 / 0.943 at 16000, 1.63 / 0.99 at 32000).
    const int64_t few = (int64_t)sm_count * (nv.long_cols ? 220 : 68) / nv.EPL;
    if (nv.form == 2 && n_walks >= few) {
        const size_t sm = (size_t)kWalkWarps * 32 * 4 * (size_t)std::max(nv.M, 1);
        int per_sm = 1;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, walk_narrow_kernel, kWalkWarps * 32, sm) != cudaSuccess ||
            per_sm < 1) {
            cudaGetLastError();
            per_sm = 1;
        }
        const int64_t blocks = (n_walks + kWalkWarps * 32 - 1) / (kWalkWarps * 32);
        walk_narrow_kernel<<<(int)std::min<int64_t>(blocks, (int64_t)sm_count * per_sm), kWalkWarps * 32, sm, s>>>(
            nv, a, target, seed, n_walks);
        return cudaGetLastError();
    }
    const int64_t want = (n_walks + kExpandWarps - 1) / kExpandWarps;
    const int grid = (int)std::min<int64_t>(want, (int64_t)sm_count * 8);
    switch (nv.EPL) {
#define EFM_WALK(E)                                                                       \
    case E:                                                                               \
        walk_kernel<E><<<grid, kExpandWarps * 32, 0, s>>>(nv, a, target, seed, n_walks); \
        break;
        EFM_WALK(1) EFM_WALK(2) EFM_WALK(4) EFM_WALK(8) EFM_WALK(16) EFM_WALK(28) EFM_WALK(32)
#undef EFM_WALK
    default:
        return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

size_t sort_scratch_bytes(int64_t n2) { return (size_t)n2 * sizeof(SortRec); }

// kernels a sort of n2 (a power of two) records launches
int sort_launches(int64_t n2)
{
    int n = 3;
    for (int64_t k = 2 * kSortTile; k <= n2; k <<= 1) {
        ++n;
        for (int64_t j = k >> 1; j >= kSortTile; j >>= 1) ++n;
    }
    return n;
}

template <typename Rec>
static cudaError_t sort_with(const uint64_t *res, int64_t n, int W, Rec *rec, int64_t n2, uint64_t *out, int64_t n_keep,
                             cudaStream_t s)
{
    if (n <= 0 || n_keep <= 0) return cudaSuccess;
    const int tb = 256;
    const int blocks = (int)((n2 + tb - 1) / tb);
    const int tiles = (int)((n2 + kSortTile - 1) / kSortTile);
    sort_init_kernel<<<blocks, tb, 0, s>>>(res, W, rec, n, n2);
    bitonic_tile_kernel<<<tiles, kSortBlock, 0, s>>>(res, W, rec, n2, 2, std::min<int64_t>(n2, kSortTile));
    for (int64_t k = 2 * kSortTile; k <= n2; k <<= 1) {
        for (int64_t j = k >> 1; j >= kSortTile; j >>= 1) bitonic_step_kernel<<<blocks, tb, 0, s>>>(res, W, rec, n2, k, j);
        bitonic_tile_kernel<<<tiles, kSortBlock, 0, s>>>(res, W, rec, n2, k, k);
    }
    const int64_t items = n_keep * W;
    gather_kernel<<<(int)((items + tb - 1) / tb), tb, 0, s>>>(res, W, rec, n_keep, out);
    return cudaGetLastError();
}

cudaError_t launch_sort_results(const uint64_t *res, int64_t n, int W, void *scratch, int64_t n2, uint64_t *out,
                                int64_t n_keep, cudaStream_t s)
{
    return sort_with(res, n, W, reinterpret_cast<SortRec *>(scratch), n2, out, n_keep, s);
}

cudaError_t launch_sort_index(const uint64_t *res, int64_t n, int W, uint32_t *idx, int64_t n2, uint64_t *out,
                              int64_t n_keep, cudaStream_t s)
{
    return sort_with(res, n, W, idx, n2, out, n_keep, s);
}

cudaError_t launch_small(const NetView &nv, const LevelArgs &a, const AcceptArgs &acc, const Arena &first,
                         const Arena &second, int limit, cudaStream_t s)
{
    const size_t sm = (size_t)kSmallAcceptWarps * kAcceptWarpWords * 4;
#define EFM_LAUNCH(K)                                                                                   \
    do {                                                                                                \
        cudaError_t e = cudaFuncSetAttribute(K, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);  \
        if (e != cudaSuccess) return e;                                                                 \
        K<<<1, kSmallWarps * 32, sm, s>>>(nv, a, acc, first, second, limit);                            \
    } while (0)
    EFM_FORM(small_kernel, EFM_LAUNCH);
#undef EFM_LAUNCH
    return cudaGetLastError();
}

cudaError_t launch_batch_gather(const BatchJob *jobs, const int64_t *off, int n_jobs, uint64_t *dst, cudaStream_t s)
{
    batch_gather_kernel<<<std::min(n_jobs, 4096), 128, 0, s>>>(jobs, off, n_jobs, dst);
    return cudaGetLastError();
}

int batch_blocks_per_sm(int warps)
{
    int per_sm = 0;
    const size_t sm = batch_smem_bytes(warps);
    cudaFuncSetAttribute(batch_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)batch_smem_bytes(kBatchThreads / 32));
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, batch_kernel, warps * 32, sm) != cudaSuccess ||
        per_sm < 1) {
        cudaGetLastError();
        per_sm = 1;
    }
    return per_sm;
}

size_t batch_smem_bytes(int)
{
    return (size_t)kBatchAcceptWarps * kAcceptWarpWords * 4;
}

cudaError_t launch_batch(const BatchArgs &ba, int grid, int warps, cudaStream_t s)
{
    if (warps < kAcceptWarps || warps > kBatchThreads / 32) return cudaErrorInvalidValue;
    const size_t sm = batch_smem_bytes(warps);
    cudaFuncSetAttribute(batch_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)batch_smem_bytes(kBatchThreads / 32));
    batch_kernel<<<grid, warps * 32, sm, s>>>(ba);
    return cudaGetLastError();
}

}  // namespace efm
