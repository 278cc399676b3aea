// efm_sparse.cu -- kernels and launches of the level pass over the whole grid.
#include "efm_level.cuh"

namespace efm {
namespace {

constexpr int kGenWarps = 8;      // warps per CTA
// CTAs per SM of the generate pass.  It waits on memory more than it computes
// (long-scoreboard stalls lead), so 48 registers and 40 warps per SM beat 64
// registers and 32 although they spill: 485 against 501 ms on the core-shaped
// network at a 2^26 budget; 24 warps 537.
constexpr int kGenBlocks = 5;

template <int F, bool SUB, bool FK, bool LONG>
__global__ void __launch_bounds__(kGenWarps * 32, kGenBlocks) generate_kernel(const __grid_constant__ NetView nv,
                                                                              const __grid_constant__ LevelArgs a)
{
    __shared__ CapScratch s_cap[FK ? kGenWarps : 1];
    __shared__ BoundScratch s_bound;
    if (a.st[S_STOP] != STOP_NONE) return;
    const int wid = threadIdx.x >> 5;
    if (a.first) {  // the level's state table, cleared for the dedup pass
        const uint64_t n = a.st[S_SLOTS] / 2;  // (at least 64 slots, two a store)
        uint4 *t = reinterpret_cast<uint4 *>(a.slots);
        for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x)
            t[i] = make_uint4(~0u, ~0u, ~0u, ~0u);
    }
    const int64_t n_par = a.manual ? a.n_par : (int64_t)a.st[S_NROWS];
    // (a level in several launches reserves exactly what a round needs: the
    // tables have room for one launch's unused rows)
    const int blk = a.manual ? 0 : (int)a.st[S_BLK], pay_blk = a.manual ? 0 : (int)a.st[S_PAY_BLK];
    const bool any_result = a.ctr[C_RES_N] != 0ull;  // (none is accepted while this kernel runs)
    if (FK) {
        if (a.fk_pc > 0) {
            for (int i = threadIdx.x; i < EFM_MAX_COLUMNS / 32; i += blockDim.x)
                s_bound.bits[i] = i < 2 * nv.W ? (uint32_t)(a.fk_sup[i >> 1] >> (32 * (i & 1))) : 0u;
            if (threadIdx.x == 0) {
                int n = 0;
                for (int w = 0; w < nv.W; ++w)
                    for (uint64_t x = a.fk_sup[w]; x && n < 64; x &= x - 1)
                        s_bound.cols[n++] = (uint16_t)(w * 64 + __ffsll((long long)x) - 1);
                s_bound.n = n;
            }
        }
        __syncthreads();
    }
    // parents per warp and chunk: fewer at small levels, so that their items
    // spread over all warps
    const int cpw = (int)min((int64_t)32, max((int64_t)1, (n_par + a.warps - 1) / a.warps));
    generate_range<F, SUB, FK, LONG>(nv, a, n_par, cpw, blk, pay_blk, any_result, (int64_t)blockIdx.x * kGenWarps + wid,
                               (int64_t)gridDim.x * kGenWarps, s_cap + (FK ? wid : 0), s_bound);
}

template <int F, bool SUB>
__global__ void __launch_bounds__(256, 6) dedup_kernel(const __grid_constant__ NetView nv,
                                                       const __grid_constant__ LevelArgs a)
{
    __shared__ unsigned long long s_keep[8], s_deg[8], s_unv[8];
    if (a.st[S_STOP] != STOP_NONE) return;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    DedupSums sum;
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    const uint64_t in_cta = threadIdx.x & ~31u;
    // (the open children from the grid's end: at a small level other CTAs than
    // those with its rows)
    // (counters through L1: a read of every warp from L2 costs 20 us a level)
    dedup_range<F, SUB>(nv, a, a.st[S_SLOTS] - 1, a.ctr[C_DEDUP_BEGIN], a.ctr[C_WRITTEN], a.ctr[C_OPEN],
                        (uint64_t)blockIdx.x * blockDim.x + in_cta,
                        stride - blockDim.x - (uint64_t)blockIdx.x * blockDim.x + in_cta, stride, sum);
    unsigned long long deg = sum.deg_units, n_unv = sum.unv, n_keep = sum.keep;
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
        unsigned long long k = 0, d = 0, u = 0, p = 0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
            k += s_keep[w];
            d += (uint32_t)s_deg[w];
            p += s_deg[w] >> 32;
            u += s_unv[w];
        }
        if (k) atomicAdd(&a.ctr[C_NEXT], k);
        if (d) atomicAdd(&a.ctr[C_DEGSUM], d);
        if (p) atomicAdd(&a.ctr[C_KEPT], p);
        if (u) atomicAdd(&a.ctr[C_UNV], u);
    }
}

template <int F, bool SUB>
__global__ void __launch_bounds__(256) seed_kernel(NetView nv, LevelArgs a, int target)
{
    seed_range<F, SUB>(nv, a, target, blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x);
}

// One state with flux 1 on each column of R_in: EF = the sum of their S_int
// columns, normalised.  One warp; the sums in shared memory.
template <int F, bool SUB>
__global__ void __launch_bounds__(32) seedset_kernel(NetView nv, LevelArgs a, const int32_t *cols, int n_cols)
{
    __shared__ long long acc[EFM_MAX_INTERNAL];
    const int lane = threadIdx.x;
    const uint32_t *bl = nv.blob;
    const int rows = nv.M + (SUB ? nv.N : 0);  // at most EFM_MAX_INTERNAL
    for (int r = lane; r < EFM_MAX_INTERNAL; r += 32) acc[r] = 0;
    __syncwarp();
    for (int i = 0; i < n_cols; ++i) {
        const int k = cols[i];
        for (int q = (int)bl[nv.o_colptr + k] + lane; q < (int)bl[nv.o_colptr + k + 1]; q += 32) {
            const uint32_t f = bl[nv.o_colent + q];
            acc[ent_index(f)] += ent_coef(f);  // a column's rows are distinct
        }
        if (SUB && lane == 0) acc[nv.M + k] += 1;
        __syncwarp();
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
    if (lane != 0) return;
    // the rest by one lane: at most 64 columns and 1024 entries
    atomicAdd(&a.ctr[C_SEEDS], 1ull);
    if (bad) {
        atomicAdd(&a.ctr[C_OVF], 1ull);
        return;
    }
    const int su = support_units<F>(n_cols);
    const int units = su + entry_units<F>(n);
    if (a.child.cap < 1 || (uint64_t)units > a.child.pay_cap) {
        record_diag(a.ctr, ERR_BOUNDS, 13, units, (long long)a.child.pay_cap, a.level);
        return;
    }
    uint4 *dst = a.child.pay;
    uint64_t uh = 0;
    if (F) {
        uint64_t u0 = 0, u1 = 0;
        for (int i = 0; i < n_cols; ++i) add_bit(u0, u1, cols[i]);
        dst[1] = make_uint4((uint32_t)u0, (uint32_t)(u0 >> 32), (uint32_t)u1, (uint32_t)(u1 >> 32));
    } else {
        uint16_t *lst = reinterpret_cast<uint16_t *>(dst) + 8;
        for (int i = 0; i < 8 * su - 8; ++i) {
            lst[i] = i < n_cols ? (uint16_t)cols[i] : (uint16_t)0xFFFFu;
            if (i < n_cols) uh += column_hash(cols[i]);
        }
        reinterpret_cast<uint64_t *>(dst)[1] = uh;
    }
    if (nb == 0) {
        atomicAdd(&a.ctr[C_BAL], 1ull);
        insert_candidate<F>(a, nv.W, dst, n_cols, -1);
        return;
    }
    EntryWriter<F, SUB> out(nv, bl, dst + su);
    for (int r = 0; r < rows; ++r)
        if (acc[r] != 0) out.put(r, (int32_t)(acc[r] / (long long)g));
    out.done();
    const uint64_t s0 = F == 2 ? out.z.zm : uh;
    dst[0] = make_uint4((uint32_t)out.rh, (uint32_t)(out.rh >> 32), (uint32_t)s0, (uint32_t)(s0 >> 32));
    if (F == 2)
        dst[2] = make_uint4((uint32_t)out.z.pm, (uint32_t)(out.z.pm >> 32), (uint32_t)out.z.nm, (uint32_t)(out.z.nm >> 32));
    const uint32_t key = out.key, om = out.om;
    const int32_t pv = out.pv;
    const int w = out.n;
    const uint32_t bkey = branch_key(bl, nv, key, SUB ? 1 : 0);
    a.child.hdr[0] = make_uint4(0u, pack_meta(bkey, n_cols), (uint32_t)w | ((uint32_t)max_bits(om) << 11), (uint32_t)pv);
    atomicAdd(&a.ctr[C_NEXT], 1ull);
    atomicAdd(&a.ctr[C_PAY], (unsigned long long)units);
    atomicAdd(&a.ctr[C_DEGSUM], (unsigned long long)(bkey >> 16));
}

// results [0, n) into an empty index, a warp each (the minimality test files
// what it accepts; this is for an index that has to grow)
__global__ void __launch_bounds__(128) index_kernel(CellIndex ix, const uint64_t *res, int W, int64_t n)
{
    __shared__ int cols[4][64];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int64_t r = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; r < n;
         r += ((int64_t)gridDim.x * blockDim.x) >> 5) {
        const uint64_t u0 = lane < W ? res[(size_t)r * W + lane] : 0ull;
        const uint64_t u1 = lane + 32 < W ? res[(size_t)r * W + lane + 32] : 0ull;
        const int m = support_columns(u0, u1, cols[wid]);
        file_result(ix, W, r, cols[wid], m, __shfl_sync(FULL, u0, 0), __shfl_sync(FULL, u0, 1));
        __syncwarp();
    }
}

// Surviving rows [0, n) of an arena appended to a list, for the passes that
// sample a frontier.
__global__ void live_list_kernel(const uint4 *hdr, int64_t n, uint32_t *live, unsigned long long *count)
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

template <typename K>
int grid_of(K kernel, int sm_count)
{
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, kGenWarps * 32, 0) != cudaSuccess || per_sm < 1) {
        cudaGetLastError();
        per_sm = 1;
    }
    return sm_count * per_sm;
}

// one of the kernel's instances: form, subtractive view, first-K rules, long columns
#define EFM_GENERATE_OF(CALL, F, SUB, FK)                                         \
    do {                                                                          \
        if (nv.long_cols) CALL((generate_kernel<F, SUB, FK, true>));              \
        else CALL((generate_kernel<F, SUB, FK, false>));                          \
    } while (0)
#define EFM_GENERATE(CALL)                                                        \
    do {                                                                          \
        if (nv.form == 2 && first_k) EFM_GENERATE_OF(CALL, 2, false, true);       \
        else if (nv.form == 2) EFM_GENERATE_OF(CALL, 2, false, false);            \
        else if (nv.form == 1 && sub) EFM_GENERATE_OF(CALL, 1, true, false);      \
        else if (nv.form == 1 && first_k) EFM_GENERATE_OF(CALL, 1, false, true);  \
        else if (nv.form == 1) EFM_GENERATE_OF(CALL, 1, false, false);            \
        else if (sub) EFM_GENERATE_OF(CALL, 0, true, false);                      \
        else if (first_k) EFM_GENERATE_OF(CALL, 0, false, true);                  \
        else EFM_GENERATE_OF(CALL, 0, false, false);                              \
    } while (0)

}  // namespace

int generate_grid(const NetView &nv, bool sub, bool first_k, int sm_count)
{
    int grid = sm_count;
#define EFM_GRID(K) grid = grid_of(K, sm_count)
    EFM_GENERATE(EFM_GRID);
#undef EFM_GRID
    return grid;
}

cudaError_t launch_generate(const NetView &nv, const LevelArgs &a, int grid, cudaStream_t s)
{
    const bool sub = a.sub != 0, first_k = a.cap_dead || a.fk_pc > 0;
#define EFM_LAUNCH(K) K<<<grid, kGenWarps * 32, 0, s>>>(nv, a)
    EFM_GENERATE(EFM_LAUNCH);
#undef EFM_LAUNCH
    return cudaGetLastError();
}

cudaError_t launch_dedup(const NetView &nv, const LevelArgs &a, int sm_count, cudaStream_t s)
{
#define EFM_LAUNCH(K) K<<<sm_count * 8, 256, 0, s>>>(nv, a)
    EFM_FORM(dedup_kernel, EFM_LAUNCH);
#undef EFM_LAUNCH
    return cudaGetLastError();
}

cudaError_t launch_seed(const NetView &nv, const LevelArgs &a, int target, cudaStream_t s)
{
#define EFM_LAUNCH(K) K<<<4, 256, 0, s>>>(nv, a, target)
    EFM_FORM(seed_kernel, EFM_LAUNCH);
#undef EFM_LAUNCH
    return cudaGetLastError();
}

cudaError_t launch_seedset(const NetView &nv, const LevelArgs &a, const int32_t *cols, int n_cols, cudaStream_t s)
{
#define EFM_LAUNCH(K) K<<<1, 32, 0, s>>>(nv, a, cols, n_cols)
    EFM_FORM(seedset_kernel, EFM_LAUNCH);
#undef EFM_LAUNCH
    return cudaGetLastError();
}

size_t cell_table_bytes(const NetView &nv, uint64_t entries)
{
    if (nv.W <= 2) return (size_t)128 * 128 * 4;
    uint64_t p = 64;
    while (p < 2 * entries) p <<= 1;
    return (size_t)p * 8;
}

cudaError_t launch_index(const NetView &nv, const CellIndex &ix, const uint64_t *res, int64_t n, cudaStream_t s)
{
    cudaError_t e;
    const int W = nv.W;
    const size_t table = W <= 2 ? (size_t)128 * nv.N * 4 : 8 * ((size_t)ix.mask + 1);
    if ((e = cudaMemsetAsync(ix.cnt, 0, sizeof(int32_t) * (size_t)nv.N, s)) != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(ix.ksig, 0, 16 * (size_t)nv.N, s)) != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(ix.single, 0, 4 * (size_t)nv.N, s)) != cudaSuccess) return e;
    if ((e = cudaMemsetAsync(ix.cells, 0xFF, table, s)) != cudaSuccess) return e;
    if (n <= 0) return cudaSuccess;
    index_kernel<<<(unsigned)std::min<int64_t>((n + 3) / 4, 4096), 128, 0, s>>>(ix, res, W, n);
    return cudaGetLastError();
}

cudaError_t launch_live_list(const uint4 *hdr, int64_t n, uint32_t *live, unsigned long long *count, int sm_count,
                             cudaStream_t s)
{
    if (n <= 0) return cudaSuccess;
    const int64_t blocks = std::min<int64_t>((n + 255) / 256, (int64_t)sm_count * 8);
    live_list_kernel<<<(unsigned)blocks, 256, 0, s>>>(hdr, n, live, count);
    return cudaGetLastError();
}

}  // namespace efm
