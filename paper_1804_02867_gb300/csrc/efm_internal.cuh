// efm_internal.cuh -- shared declarations of the CUDA path (not part of the ABI).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "../../include/efmgraph.h"

namespace efm {

constexpr int kMaxW = 64;           // support words (EFM_MAX_COLUMNS / 64)
constexpr int kExpandWarps = 8;     // warps per CTA of the expansion kernel
constexpr int kAcceptWarps = 4;     // warps per CTA of the minimality kernel
constexpr unsigned long long kEmpty = ~0ull;
constexpr uint32_t kPending = 0xFFFFFFFFu;
constexpr uint32_t kOverflowIdx = 0xFFFFFFFEu;
constexpr int kNumPrimes = 24;
constexpr int64_t kFirstKChunkMin = 8192;     // first-K search: fewest parents per expansion launch
constexpr int64_t kFirstKChunks = 32;         // first-K search: launches per level, at most
constexpr int64_t kResultWindow = 256;        // first-K search: new results fetched with the counters
// Most branches of a level that one CTA runs (launch_small).  Up to there a
// level by one CTA takes less than three launches; with 512, 1024, 2048, 4096:
// the smallest query 0.80, 0.80, 0.84, 0.90 ms (three launches for every level:
// 0.84), eight core targets at 2^17 8.05, 8.10, 8.20, 8.78 (8.86), a 400-row
// network 3.93, 3.90, 4.07, 4.20 (4.13), the subtractive variant 5.85, 5.83,
// 5.95, 6.6 (6.07).
constexpr int kSmallBranches = 1024;
// Most new balanced supports that its eight warps judge; more are left to the
// grid: 1000 supports of 61 columns 7.9 ms by one CTA and 1.3 by the grid, 900
// of 31 columns 2.0 and 0.9, 60 of 61 columns 1.1 either way.
constexpr int kSmallCandidates = 64;
constexpr int kWaitSpinLimit = 1 << 20;       // polls of a bounded device-side wait (with ~0.25 us sleeps)

// device error bits (ctr[C_ERR])
enum : unsigned { ERR_TIMEOUT = 1u, ERR_CAND_CAP = 2u, ERR_RES_CAP = 4u, ERR_TABLE_FULL = 8u,
                  ERR_PRIMES = 16u, ERR_LEN = 32u, ERR_WATCHDOG = 64u, ERR_BOUNDS = 128u };

// device counter block (unsigned long long each)
enum {
    C_LEVELS = 0, C_SEEDS, C_EXP, C_OVF, C_BAL, C_CAND, C_RES, C_PRUNED, C_FRONTIER, C_FRONTIER_MAX, C_STATUS,
    C_NEXT = 12,  // states allocated in the arena being written
    C_DEGSUM,     // sum of pivot degrees of the states written (children bound of the next level)
    C_CAND_N,     // candidate list length (cumulative)
    C_RES_N,      // result list length (cumulative)
    C_ERR,        // ERR_* bits
    C_WRITTEN,    // generate/dedup split: child rows reserved so far in the level
    C_UNWRITTEN,  // children whose row did not fit the child arena
    C_UNV,        // distinct fingerprints among the children without a row
    C_OUT_N = 20, // batched traversal: rows written to the job's output
    C_DONE,       // batched traversal: 1 = job finished, 2 = left to the host
    C_ACC_BEGIN,  // first candidate the next device-range minimality launch judges
    C_DEDUP_BEGIN,  // first reserved row the next dedup launch examines
    C_DIAG = 24,  // first bounds/watchdog record: code, value, limit, level
    C_ZERO = 28,  // subtractive steps discarded: no positive flux left on the reaction (Prop. 3)
    C_OPEN,       // open children listed by the generate pass, not yet finished
    C_LIVE,       // surviving rows counted by the live-list pass
    C_PAY = 32,   // payload units reserved so far in the level
    C_KEPT,       // payload units that its distinct states take
    C_COUNT = 40
};

// Level state of a traversal, kept on the device behind its counter block
// (unsigned long long each): the last CTA of a level's minimality test decides
// whether the search goes on and sets the next level's parameters, so that
// the host can launch several levels without a round trip between them.
enum {
    S_STOP = 0,   // STOP_*: later launches return at once
    S_LEVEL,      // last completed level
    S_NROWS,      // its arena rows (the next level's parents)
    S_NFRONT,     // its distinct states
    S_DEG,        // sum of their branch counts
    S_UNITS,      // payload units of its distinct states
    S_SLOTS,      // next level: slots of the state table (a power of two)
    S_RESERVED,   // next level: rows that may be reserved
    S_BLK,        // next level: rows a warp reserves at a time
    S_PAY_BLK,    // next level: payload units a warp reserves at a time
    S_FRONTIER,   // sum and largest of the levels' distinct states
    S_FRONTIER_MAX,
    S_BYTES,      // algorithmic bytes of the expansions so far
    S_EXPANDS,    // expansion launches: levels, chunks of a first-K level and levels run again
    S_TICKET,     // CTAs of the running minimality launch that are done
    S_PENDING,    // 1: launch_small left the minimality test of a level to the grid
    S_SNAP,       // C_EXP, C_OVF, C_BAL, C_PRUNED, C_ZERO when the running level began
    S_COUNT = S_SNAP + 8
};
enum : unsigned long long {
    STOP_NONE = 0,
    STOP_DONE,       // the frontier is empty
    STOP_TRUNCATED,  // it exceeds the budget
    STOP_CAPPED,     // max_results reached
    STOP_RERUN,      // children without a row: the level again, with a larger arena
    STOP_TABLES,     // the next level needs larger tables
    STOP_INDEX,      // the superset rule's index is full
    STOP_ERROR       // an error bit, or too many levels
};

// Static network, packed into one 16-byte aligned word array (the "blob").
// Packed entry: (index << 20) | (coefficient & 0xFFFFF), index < 4096,
// coefficient a signed 20-bit value.
struct NetView {
    const uint32_t *blob;  // device
    int M, N, W, Mpad, EPL;
    int o_colptr, o_colent;    // S_int by column: rows with coefficients
    int o_consptr, o_consent;  // per internal row: consuming columns, |coef|
    int o_prodptr, o_prodent;  // per internal row: producing columns, |coef|
    int o_twin;                // per column: twin column or -1 (as int32)
    int o_keypos, o_keyneg;    // per internal row: (degree << 16) | row
    int o_hbits;               // per column: ceil(log2(|S_int[:,k]|^2))
    int o_dcols;               // dense S_int by column: N rows of Mpad int32 (16-byte aligned)
    // per column, 8 words (16-byte aligned): HC = sum_m S_int[m][k] R[m] (2 words, R: the row
    // hash constants), mask of its rows modulo 64 (2), max |S_int[m][k]|, its range of words
    // in colent (2), its twin column or ~0
    int o_scol;
    // how the level pass keeps a state: 2 = narrow (at most 64 internal rows and 128 columns:
    // masks and the values in row order), 1 = bitset support and a list of entries (at most 128
    // columns), 0 = column list and a list of entries
    int form;
    int long_cols;  // long children are common: see has_long_columns
    int o_rank, o_keyr, o_colx, o_nent;  // narrow: see efm_netprep.h
    const int32_t *metptr;     // full S rows over split columns (seeds), [n_met + 1]
    const uint32_t *metent;    // packed (column, coefficient)
    int n_met;
};

// Entries that a lane of the generate pass takes at most: of a column (kept in
// registers on narrow networks), and 64 of a list.  Longer children are left to
// the dedup pass, a warp each, or, in the instances of the kernels for networks
// where they are common (any column past the line; or, lists, columns so long
// that states pass 64 entries within a few levels), taken by a lane all the same.
// One GB300, dense rows (before sparse states), a lane each in the dedup pass, a
// warp each there, a lane each in the generate pass: 90 reactions of 10 to 20
// metabolites on 60 rows at 2^18 3.0, 5.5, 7.5 and 2.4 ms; 500 of 30 to 80 on 300
// rows 23, 40, 53 and 12; 100 of 20 to 60 on 100 rows 4.6, 11.7, 15.9 and 4.5 (at
// 2^14, where a level has few children, 1.5, 3.7, 3.2 and 2.1).  On the core-shaped
// network, whose columns are short, the code for them costs 14 % (spills: 467 and
// 533 ms at 2^26).  A warp each is right for the few of other networks (see
// kWarpOpen): a small level waits for one lane's chain (eight core targets at 2^17 7.8 -> 6.7 ms,
// subtractive 5.8 -> 4.6, a 400-row network 3.8 -> 3.4).
constexpr int kNarrowCol = 8, kListCol = 32, kListMean = 8;

__host__ __device__ inline int ent_index(uint32_t e) { return (int)(e >> 20); }
__host__ __device__ inline int32_t ent_coef(uint32_t e) { return ((int32_t)(e << 12)) >> 12; }

// One arena of pathway states (layout in efm_level.cuh).
struct Arena {
    uint4 *hdr;         // [cap]
    uint4 *pay;         // [pay_cap] 16-byte units
    uint64_t pay_cap;
    int64_t cap;
};

// Payload units of a state's hashes and column list
__host__ __device__ inline int sparse_list_units(int pc) { return 1 + ((pc + 7) >> 3); }

// The superset rule's index.  A result E is filed, for each of its columns k,
// in cell (k, s) where s is E's other column with the fewest results (its
// sentinel): a child adding k contains E only if it holds s, so it looks up
// the cells (k, s) of its own columns s and no others.  A cell is the head of
// a list of entries.
//   at most 128 columns: cells is a table of heads, [N][128]; ksig holds two
//     words a column, bit s set when cell (k, s) is not empty; an entry is two
//     units: E's words; (next, result)
//   else: cells is a hash table of (k << 12 | s, head); ksig holds one word a
//     column, a signature of its sentinels; an entry is one unit: a signature
//     of E's columns, next, result
// Empty keys, heads and ends of lists are ~0.
struct CellIndex {
    uint2 *cells;
    uint32_t mask;      // hash table: slots - 1
    uint4 *ent;
    uint64_t *ksig;
    uint32_t *single;   // [N]: 1 if {k} itself is a result
    int64_t room;       // results it has room for (0: no index)
    int32_t *cnt;       // [N]: filed results per column
    int ent_stride;     // entries of result r start at r * ent_stride
};

struct LevelArgs {
    unsigned long long *st;     // level state
    int manual;                 // 1: the parents are n_par, par_base and perm below; 0: all rows of the last level
    int first;                  // first launch of its level: clear the state table
    int warps;                  // warps of the generate launch
    Arena par;
    int64_t n_par;
    Arena child;
    unsigned long long *slots;  // state hash table
    unsigned long long *cslots; // balanced-support hash table
    uint64_t cslot_mask;
    uint64_t *cand;             // [cand_cap][W]
    int64_t cand_cap;
    const uint64_t *res;        // [res_cap][W]
    const uint16_t *rcols;      // per result: column count, then its columns (stride kRcolStride)
    CellIndex cells;            // the level pass
    int level, max_len, max_sec;
    unsigned long long *ctr;
    // first-K search (zero / null otherwise)
    const uint32_t *perm;       // parent order: position -> arena index (null: arena rows par_base + position)
    int64_t par_base;
    int fk_pc;                  // bound: |U| of the K-th smallest result found so far (0 = no bound)
    const uint64_t *fk_sup;     // bound: its support (W words)
    // first-K: drop an unbalanced child at the length cap that no sequence of
    // secondary steps can balance (0 = keep every child)
    int cap_dead;
    // generate/dedup split (single-job traversal): every surviving child gets
    // a reserved row and a fingerprint; the dedup pass keeps one per state
    uint64_t *fp;               // [fp_cap] fingerprint per reserved row (kDeadFp: unused)
    int64_t fp_cap;
    uint32_t *open;             // [fp_cap] rows of the open children
    // subtractive variant (Eq. 5): states also hold the flux of their columns,
    // a state's branches also take flux away from a column in U, and its meta
    // degree counts both lists of the pivot
    int sub;
};

constexpr uint32_t kNoRecord = 0xFFFFFFFFu;

constexpr unsigned long long kDeadFp = ~0ull;  // fingerprint of a reserved row left unused

constexpr int kRcolStride = 65;  // column count + up to 64 columns per result

struct AcceptArgs {
    const uint64_t *cand;
    int64_t cand_begin, cand_end;  // ignored with advance: [ctr[C_ACC_BEGIN], ctr[C_CAND_N]) instead
    int64_t cand_cap;
    uint64_t *res;
    uint16_t *rcols;            // written on accept when non-null
    int64_t res_cap;
    unsigned long long *ctr;
    // single-job traversal
    CellIndex ix;               // accepted results are filed here
    unsigned long long *st;
    int advance;                // what the last CTA does: 0 nothing, 1 a chunk of a level ends, 2 a level, 3 the seeds
    int level, max_level;
    int64_t max_frontier, max_results;
    int64_t fp_cap, child_rows;
    uint64_t slot_cap;
    int warps;                  // warps of the next generate launch
};

// Batched traversal: per-CTA scratch slice layout (byte offsets)
constexpr int kBatchThreads = 256;
struct BatchLayout {
    size_t slice_bytes;
    size_t o_hdr[2], o_pay[2];
    size_t o_slots, o_fp, o_open, o_cslots, o_cand, o_res, o_cnt, o_ksig, o_single, o_cells, o_ent, o_sort, o_rcols;
    int64_t cap, fp_cap, cand_cap, res_cap, index_room;
    uint64_t pay_cap, slot_cap, cslot_cap;
    uint32_t cell_mask;
    int ent_stride;
};

struct BatchJob {
    NetView nv;
    int target, max_len;
    uint64_t *out;            // [res_cap][W] sorted supports
    unsigned long long *ctr;  // [C_COUNT] counters of this job (zeroed by the host)
};

struct BatchArgs {
    const BatchJob *jobs;
    const int *order;         // queue schedule: job index per queue position
    int n_jobs;
    unsigned int *queue;      // next queue position (zeroed by the host)
    char *pool;               // gridDim.x slices of layout.slice_bytes
    BatchLayout layout;
    int max_sec;
    int64_t max_frontier, max_results;
    int tile;                 // most parents a warp takes per pass (1..32)
    int chunk;                // queue positions a CTA claims at a time (>= 1)
};

// Learned proposal: MLP 128 -> 256 (ReLU) -> 1.  FP32 parameters in one
// buffer: W1 [256][128] (hidden unit, feature; the bias of the hidden layer
// is the weight of the constant feature), w2 [256], b2.
constexpr int kMlpFeatures = 128;
constexpr int kMlpHidden = 256;
constexpr int kMlpTileRows = 128;
constexpr int kMlpW1 = 0;
constexpr int kMlpW2 = kMlpHidden * kMlpFeatures;
constexpr int kMlpB2 = kMlpW2 + kMlpHidden;
constexpr int kMlpParams = kMlpB2 + 1;

// Byte offset of element (row, k) in a 128-column BF16 tile laid out as the
// K-major operand of tcgen05 without swizzling: 8 x 8 core matrices (8 rows
// of 16 bytes), 16 of them along K per group of 8 rows.
__host__ __device__ inline uint32_t mlp_blk_off(int row, int k)
{
    return (uint32_t)((((row >> 3) * 16 + (k >> 3)) * 128) + (row & 7) * 16 + (k & 7) * 2);
}

// kernels (efm_mlp.cu)
// map: frontier position -> arena row (null: identity); rows r take positions first + r * stride
cudaError_t launch_features(const NetView &nv, const Arena &par, const uint32_t *map, int64_t first, int64_t stride,
                            int64_t n, int level, int max_len, int max_sec, const uint64_t *dep, void *X, int64_t row0,
                            cudaStream_t s);
cudaError_t launch_labels(const Arena &par, int W, const uint32_t *map, int64_t first, int64_t stride, int64_t n,
                          const uint64_t *ans, int64_t n_ans, float *y, int64_t row0, cudaStream_t s);
cudaError_t launch_mlp_score(const void *X, int64_t n_rows, const void *wb, const float *params, float *score,
                             unsigned *err, cudaStream_t s);
cudaError_t launch_mlp_train(const void *X, const float *y, int64_t n_rows, const int32_t *tiles, int n_tiles,
                             const void *wb, const float *params, float pos_weight, float inv_n, float *grad,
                             float *loss, unsigned *err, cudaStream_t s);
cudaError_t launch_adam(float *params, float *grad, float *mom, float lr, int step, void *wb, cudaStream_t s);
cudaError_t launch_pack_w(const float *params, void *wb, cudaStream_t s);
// perm[i] = map[position of the i-th highest score] (map null: the position itself)
cudaError_t launch_score_order(const float *score, int64_t n, const uint32_t *map, unsigned *hist, uint32_t *perm,
                               cudaStream_t s);
cudaError_t launch_pack_rows(const float *x, int64_t n, void *X, int64_t row0, cudaStream_t s);
size_t mlp_score_smem();
size_t mlp_train_smem();

// kernels (efm_sparse.cu): the level pass
cudaError_t launch_seed(const NetView &nv, const LevelArgs &a, int target, cudaStream_t s);
cudaError_t launch_seedset(const NetView &nv, const LevelArgs &a, const int32_t *cols, int n_cols, cudaStream_t s);
// one expansion: children with rows, payloads and fingerprints, then one pass
// that keeps the first row of every distinct state
int generate_grid(const NetView &nv, bool sub, bool first_k, int sm_count);
cudaError_t launch_generate(const NetView &nv, const LevelArgs &a, int grid, cudaStream_t s);
cudaError_t launch_dedup(const NetView &nv, const LevelArgs &a, int sm_count, cudaStream_t s);
// an empty superset index, then the results [0, n) filed in it
size_t cell_table_bytes(const NetView &nv, uint64_t entries);
cudaError_t launch_index(const NetView &nv, const CellIndex &ix, const uint64_t *res, int64_t n, cudaStream_t s);
// the surviving rows (meta != 0) of [0, n) appended to live; *count must be 0
cudaError_t launch_live_list(const uint4 *hdr, int64_t n, uint32_t *live, unsigned long long *count, int sm_count,
                             cudaStream_t s);
// kernels (efm_kernels.cu)
cudaError_t launch_accept(const NetView &nv, const AcceptArgs &a, cudaStream_t s);
// minimality test of the candidates appended since the last such launch (range read on the
// device); accepted results are filed in the index; then the level state moves on
cudaError_t launch_accept_new(const NetView &nv, const AcceptArgs &a, int sm_count, cudaStream_t s);
// the levels from the state's on while they have at most `limit` branches, by one CTA; the
// parents of the first are in `first`, of the next in `second`, and so on
cudaError_t launch_small(const NetView &nv, const LevelArgs &a, const AcceptArgs &acc, const Arena &first,
                         const Arena &second, int limit, cudaStream_t s);
// sort by (|U|, ascending columns); n2: n rounded up to a power of two; scratch: sort_scratch_bytes(n2)
size_t sort_scratch_bytes(int64_t n2);
int sort_launches(int64_t n2);
cudaError_t launch_sort_results(const uint64_t *res, int64_t n, int W, void *scratch, int64_t n2, uint64_t *out,
                                int64_t n_keep, cudaStream_t s);
// the same with n2 indices (4 bytes each) as the only scratch
cudaError_t launch_sort_index(const uint64_t *res, int64_t n, int W, uint32_t *idx, int64_t n2, uint64_t *out,
                              int64_t n_keep, cudaStream_t s);
cudaError_t launch_step_count(const NetView &nv, unsigned *r, cudaStream_t s);
cudaError_t launch_or_words(uint64_t *a, const uint64_t *b, int64_t n, cudaStream_t s);
cudaError_t launch_depthy(const NetView &nv, int L, unsigned r, unsigned long long n_paths, unsigned long long *dep_out,
                          unsigned long long *dep_in, int sm_count, cudaStream_t s);
// one thread waits on `flag` for kWaitSpinLimit polls; ERR_TIMEOUT in *err if it stays 0
cudaError_t launch_stalled_wait(const uint32_t *flag, unsigned long long *err, unsigned long long *polls,
                                cudaStream_t s);
cudaError_t launch_flux(const NetView &nv, const uint64_t *sup, int64_t n, int64_t *flux, int8_t *status, int sm_count,
                        cudaStream_t s);
cudaError_t launch_walks(const NetView &nv, const LevelArgs &a, int target, uint64_t seed, int64_t n_walks, int sm_count,
                         cudaStream_t s);
// the batched traversal runs `warps` warps per CTA (4 or 8), one job at a time
cudaError_t launch_batch(const BatchArgs &ba, int grid, int warps, cudaStream_t s);
// the output rows of every job (words off[i] .. off[i + 1]) into one array
cudaError_t launch_batch_gather(const BatchJob *jobs, const int64_t *off, int n_jobs, uint64_t *dst, cudaStream_t s);
int batch_blocks_per_sm(int warps);
size_t batch_smem_bytes(int warps);

}  // namespace efm
