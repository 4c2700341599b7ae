// Internal declarations shared by the translation units of libcp_gb300.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <memory>
#include <string>
#include <vector>

#include "cp_tm.h"

namespace cp {

// ------------------------------------------------------------------ errors
void set_error(const std::string &msg);
int fail(int code, const std::string &msg);
// Distinct primes in [2, 2^31), 1..CP_MAX_PRIMES of them (Miller-Rabin on the host).
int check_primes(const uint32_t *primes, int n);

#define CP_CUDA_TRY(expr)                                                                \
    do {                                                                                 \
        cudaError_t _e = (expr);                                                         \
        if (_e != cudaSuccess)                                                           \
            return ::cp::fail(CP_ECUDA, std::string(#expr) + ": " + cudaGetErrorString(_e)); \
    } while (0)

// Device allocation helpers (library-owned memory).
int dev_alloc(void **p, size_t bytes);
void dev_free(void *p);

// Device memory handed out in pieces of 256-byte multiples and given back as a whole.
// Small pieces come from common blocks, which grow from 64 KB to 1 MB; one of kPoolPiece
// bytes or more has an allocation of its own.
constexpr size_t kPoolPiece = 256 << 10;
class DevPool {
    std::vector<void *> blocks_;
    char *at_ = nullptr;
    size_t left_ = 0, next_ = 64 << 10;

  public:
    DevPool() = default;
    DevPool(const DevPool &) = delete;
    DevPool &operator=(const DevPool &) = delete;
    ~DevPool();
    int alloc(void **p, size_t bytes);
};

// ------------------------------------------------------------------ state spaces
// Point counts go up to CP_MAXN in the rank tables (contracted spaces use L-1).
constexpr int kMaxN = 24;
constexpr int kTblStride = kMaxN + 1;

// cnt[n] = number of NCNNN partitions of n points (cnt[0] = 1, cnt[n] = M_{n-1});
// off[n*kTblStride + k] = rank of the first n-point partition whose first point
// has its smallest partner at relative position 2+k (eq. (M_recurs)).
// cntc[n] = Catalan C_n (non-crossing partitions of n points), offc[n*kTblStride + k]
// = rank of the first n-point non-crossing partition whose first point has its
// smallest partner at relative position 1+k.
struct RankTables {
    uint64_t cnt[kTblStride];
    uint64_t off[kTblStride * kTblStride];
    uint64_t cntc[kTblStride];
    uint64_t offc[kTblStride * kTblStride];
};

// A state space of one per-site factor.
//  SPACE_B: NCNNN partitions in the paper's order (first `size` ranks).
//  SPACE_X: partitions NCNNN except that e ~ e+1 is allowed (square lattice,
//           Sec. 3.4).  Ordered by interleaving: the NCNNN partitions in B
//           order, each NCNNN partition t in which e is alone and e-1 !~ e+1
//           immediately followed by J_{e,e+1} t.  prefix[b] = number of such t
//           with B-rank < b, so rank(t) = b + prefix[b] and rank(J t) = that + 1.
//  SPACE_C: all non-crossing partitions (the any-v Potts model, Sec. 3.2), in
//           the order: first point alone first, then by its smallest partner.
enum SpaceKind : int32_t { SPACE_B = 0, SPACE_X = 1, SPACE_C = 2 };
struct Space {
    int32_t kind;
    int32_t m;      // number of sites
    int32_t e;      // excepted pair (SPACE_X)
    int32_t pad;
    uint64_t size;  // number of ranks used
    const uint32_t *prefix;  // SPACE_X: [M_{m-1} + 1] on the device
};

// Kind of per-site factor.
enum OpKind : int32_t {
    OP_SQUARE = 0, OP_TRIANGULAR = 1, OP_LAST = 2, OP_IDENTITY = 3,  // chromatic (v = -1, projected)
    OP_POTTS_SQUARE = 4, OP_POTTS_TRIANGULAR = 5, OP_POTTS_LAST = 6  // any v, no projectors
};

struct OpDesc {
    int32_t kind;
    int32_t m;
    int32_t i;       // 0-based site
    int32_t max_terms;
    Space in, out;
    int32_t v;         // Potts coupling (OP_POTTS_*)
    int32_t src_bits;  // edge format of the table
    int32_t fused;     // 1: two-site table, factor (kind_b, i_b) applied after (kind, i)
    int32_t kind_b;
    int32_t i_b;
    int32_t pad2;
};

// Packed CSR edge: src (src_bits) | shift << src_bits (2 bits) | coef << (src_bits + 2)
// (two's complement in the remaining bits).  Chromatic tables: 27 / 2 / 3 bits
// (coefficients +1, -1, -2, -3).  Potts tables take as few source bits as the
// space needs (at least 16), leaving 30 - src_bits bits for the coefficient.
constexpr uint32_t kSrcBits = 27;
constexpr uint32_t kSrcMask = (1u << kSrcBits) - 1u;
constexpr uint32_t kPottsMinSrcBits = 16;
inline int potts_src_bits(uint64_t n_states) {
    int b = (int)kPottsMinSrcBits;
    while (b < (int)kSrcBits && (1ull << b) - 1 < n_states) ++b;
    return b;
}

// Degree windows.  P~ counts w^(vertices - components) (a horizontal or vertical
// edge that joins two components costs one factor w), so the polynomial of a
// state s of a strip with V vertices so far has terms only in the degrees
//   lo_s <= d <= V - blocks_s:
// V - d components, of which the state's own blocks are a part, and at least
// lo_s joins to have built its blocks at all (lo_s: shortest path from e_0 in the
// factors' tables, with each transition's shift as its length, over any number
// of rows).  A window word packs lo (low byte; 254: at least 254; 255: never
// reached) and the number of blocks (high byte).  On truncated vectors, d <= D,
// most states of a wide strip have a short window or none.
//
// CSR-by-destination table of one per-site factor, on the device.
struct SiteTable {
    OpDesc op;
    uint64_t n_src = 0, n_dst = 0, nnz = 0;
    uint64_t n_site_out = 0;  // output states of the per-site factors it stands for (n_dst, or mid + n_dst)
    uint32_t *row_ptr = nullptr;  // [n_dst + 1]
    uint32_t *edges = nullptr;    // [nnz] while the table is built (of its own from kBigTable edges on)
    uint2 *wedges = nullptr;      // [nnz] the edges as the gathers read them (GatherTask::edges)
    uint4 *units = nullptr;           // [n_units] units of work of the chunk kernel (GatherTask::units)
    uint32_t n_units = 0;
    const uint16_t *win_in = nullptr, *win_out = nullptr;  // window words of the source and destination states
    int sites = 1;                    // per-site factors it stands for (vertices added)
    uint32_t max_coef_sum = 0;        // largest sum of |coefficient| into one destination (an upper bound)
    uint32_t max_abs_coef = 0;        // largest |coefficient|
};

// A wide strip's tables take gigabytes: edges of such a table are freed as soon as its
// wedges are there, so that there is no second copy of more than one of them.
constexpr uint64_t kBigTable = 1u << 24;

// All tables of one (lattice, L) on one device; shared between strips.
struct TableSet {
    int device = 0, lattice = 0, L = 0, potts = 0, v = -1, src_bits = (int)kSrcBits, paired = 0;
    uint64_t S_b = 0, S_max = 0;
    // T_1..T_L and T_1^last..T_{L-1}^last (identity for L = 1), one table per
    // factor, or (paired) one two-site table per consecutive pair of factors
    // (T_2 T_1, T_4 T_3, ...; an odd one out stays single)
    std::vector<SiteTable> row;
    std::vector<SiteTable> last;
    std::vector<uint32_t *> x_prefix;  // square lattice: prefix table of X_e, e = 0..L-2
    DevPool pool;                      // what the tables, prefixes and windows lie in
    size_t bytes = 0;
    ~TableSet();
};

// Rank tables on the current device (built once per device by a kernel).
int device_rank_tables(const RankTables **out_dev, RankTables *host_copy);

// Build or fetch from the cache the tables of (lattice, L) on the current device
// (chromatic polynomial: the projected factorisation of Sec. 3.2-3.3), paired
// or not according to factor_pairing() and the row size.
// row_bytes = bytes of one state's row, (D+1) * padded_primes(n_primes) * 4, of the caller's vectors.
int get_tables(int lattice, int L, size_t row_bytes, cudaStream_t stream, std::shared_ptr<TableSet> *out);
// Library-wide choice for tables built from now on: 0 = one table per factor, 1 = two-site
// tables for rows of at least kPairRowBytes (kPairWideRowBytes on the square lattice from
// width kPairWide on; default), 2 = every square table, 3 = every table.
constexpr size_t kPairRowBytes = 352, kPairWideRowBytes = 1536;
constexpr int kPairWide = 16;
int factor_pairing();
int set_factor_pairing(int mode);
// Tables of the any-v Potts transfer matrix T_i = V_i H_{i,i+1} (square) or
// V_i H_{i-1,i} H_{i,i+1} (triangular) on non-crossing partitions.
int get_potts_tables(int lattice, int L, int v, cudaStream_t stream, std::shared_ptr<TableSet> *out);

// ------------------------------------------------------------------ gather
// One per-site factor application: out[dst] = sum_e coef_e * w^{shift_e} in[src_e]  (mod p),
// on the degree windows of the source and destination states: words outside a
// state's window are never read nor written.  Words are signed representatives
// in [-p, p) as 32-bit two's complement.
struct GatherTask {
    const uint32_t *in;
    uint32_t *out;
    const uint32_t *row_ptr;
    const uint2 *edges;       // x: packed edge; y: window word of its source, row within its unit << 16, first edge of
                              // the row << 21
    const uint32_t *primes;   // prime block (fill_prime_block) on the device
    const uint16_t *win_out;  // window words (lo | blocks << 8) of the destination states
    const uint4 *units;       // chunk kernel: the table's units of work
    uint32_t n_units;
    uint32_t rows;            // destination rows of this task
    uint32_t C;               // chunks per row (16-byte chunks if vec4, else words)
    uint32_t cpd;             // chunks per degree (= n_primes / VEC)
    uint32_t vec4;            // 1: 16-byte chunks, 0: 4-byte chunks
    uint32_t block_begin;     // first block (chunk kernel: unit) of this task in the launch
    uint32_t magic_cpd;       // x / cpd = umulhi(x, magic_cpd) for x * cpd < 2^32 (0: cpd == 1)
    uint32_t n_primes;
    uint32_t src_bits;        // edge format of the table
    uint32_t seg;             // chunk kernel: degrees of one pass over a row
    uint32_t r32;             // 32 modulo cpd
    uint32_t chunk;           // 1: rows and coefficients suit the chunk kernel
    uint32_t fast;            // 1: the coefficients and primes suit its 32-bit reduction (fast_ok, modred.cuh)
    uint32_t fast_k0;         // their offset
    int32_t v_in, v_out;      // vertices of the input and of the output vector (window bound V - blocks)
    int32_t cap;              // highest degree kept, D
    uint32_t first;           // 1: the input vector is e_0 at height 1 (degree 0: nothing else is read)
};

// Units of work of the chunk kernel, in row order: consecutive destination rows with
// at most unit_edges(nnz) edges together and at most 32 rows, one row of up to
// split_edges, or a part of one row with more.  {first row; rows | heavy << 6 | part << 8;
// first edge; one past the last edge}.  Rows differ a hundredfold in edges (the
// states of many single sites collect most) and the heavy ones lie together, so
// work is dealt out by edges and not by rows, and a heavy row's degrees are split
// over kSplitParts warps.  A warp walks its edges one after another, 32 listed at a time.
// Large tables have units of 64 edges (start-up and draining per unit: square k = 33 sweep
// 82.2 ms, triangular 29.9, width 17 on 5 primes 5.98, against 83.0, 31.8, 6.43 with 32 and
// 85.8, 30.1, 5.74 with 128, whose last wave is long); tables of fewer than 8192 units
// (two waves of resident warps) halve them, down to 4 edges (triangular 13 x 14 on 8
// primes 2.80 ms, served mix 5.39, square sweep 86.4; the line at 4096 units 3.00, 5.56,
// 85.9, at 16384 2.76, 5.39, 87.7: the last three with rows split from 24 or 32 edges).  Rows of
// more than two units' edges are split (from one unit's on: square sweep 86.4, triangular
// 34.0 ms, against 83.0 and 31.8), from 24 edges in the smallest units (16: triangular
// 13 x 14 2.89), into four parts (two or eight: 1-3% slower solves).
constexpr uint32_t kSplitParts = 4;
inline uint32_t unit_edges(uint64_t nnz) {
    uint32_t u = 64;
    while (u > 4 && nnz < 8192ull * u) u /= 2;
    return u;
}
inline uint32_t split_edges(uint32_t unit) { return unit < 12 ? 24 : 2 * unit; }
constexpr uint32_t kPackRows = 32;   // rows packed into units together

// What a vector's primes are to the gathers: the prime lanes, then each lane's
// multiplier of the chunk kernel's reductions (256 bytes).
constexpr int kPrimeWords = 2 * CP_MAX_PRIMES;
void fill_prime_block(const uint32_t *primes, int n_primes, int lanes, uint32_t *block);

constexpr int kGatherThreads = 256;  // 8 warps; one warp per destination row at a time
constexpr int kGatherItems = 4;      // default rows per warp (the tile: 8 * rows per block)

// Append the task of one per-site factor applied to a vector of v_in vertices.
// final: the output is the read-out's result, whose row is written whole.
constexpr int kFinalVertices = 1 << 29;
void append_gather_task(std::vector<GatherTask> *tasks, const SiteTable &tab, const uint32_t *in, uint32_t *out,
                        const uint32_t *primes_dev, int D1, int P, int v_in, uint32_t min_prime, bool final = false);
// Prime lanes of a vector's rows: padded to a multiple of four (repeats of the
// last prime), so that rows are 16-byte chunked and take the chunk kernel.
inline int padded_primes(int P) { return (P + 3) & ~3; }
// Gather tile (low 12 bits): 1, 2, 4, 8 = register kernel with that many rows
// per warp (8 warps per block); 16, 32, 64, 128 = chunk kernel.  The other bits are
// accepted as cp_tm.h lists them and choose nothing.  A batch with rows that are
// not 16-byte chunked or with large coefficients uses the register kernel.
constexpr int kTileChunk = 32;
constexpr int kChunkWarps = 2;         // warps of a block of the chunk kernel
constexpr int kChunkBlocksPerSM = 14;   // its launch bound
constexpr int kChunkSteps = 4;         // 32-chunk steps of a row held in registers
// The encodings cp_strip_set_tile and cp_sweep_create accept (besides 0).
bool tile_valid(int tile);
bool tile_is_chunk(int items);
bool chunk_usable(const GatherTask &t);
// Blocks (chunk kernel: units) of one task and of a whole launch (fills block_begin; returns the total).
uint32_t task_blocks(const GatherTask &t, int items);
uint32_t assign_blocks(std::vector<GatherTask> &tasks, int items);
// Effective tile for a batch (falls back to the register kernel when needed).
int effective_tile(const std::vector<GatherTask> &tasks, int items);
// The chunk kernel takes coefficients as signed bytes, with sums below kChunkMaxSum; of
// which fast_ok (modred.cuh) says for which primes the 32-bit reduction is exact.
constexpr uint32_t kChunkMaxCoef = 127;
bool table_fast(const SiteTable &tab, uint32_t min_prime);
// Launch a batch of tasks (block_begin assigned for `items`), by value in the
// kernel's parameters.  dv is added to the tasks' vertex counts (a strip's row h
// uses the tasks of row 1 with dv = L (h - 1)); first: as if GatherTask::first were
// set in each task.
int launch_gather(const GatherTask *tasks, int n_tasks, uint32_t total_blocks, int items, cudaStream_t st, int dv = 0,
                  bool first = false);
constexpr int kMaxLaunchTasks = 128;  // tasks of one launch; larger batches take several
template <int N>
struct TaskPack {
    GatherTask t[N];
};
// The pack's task whose blocks (units) hold id.
template <int N>
__device__ __forceinline__ int find_task(const TaskPack<N> &pack, int n_tasks, uint32_t id) {
    int lo = 0, hi = n_tasks - 1;
    while (N > 1 && lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (pack.t[mid].block_begin <= id) lo = mid; else hi = mid - 1;
    }
    return lo;
}
// Calls f with the tasks copied into the smallest pack that holds them, in runs of
// at most kMaxLaunchTasks with block_begin counted from the run's first task;
// f(pack, n_tasks, blocks).
template <class F>
inline int for_packs(const GatherTask *tasks, int n_tasks, uint32_t total_blocks, F f) {
    for (int i = 0; i < n_tasks; i += kMaxLaunchTasks) {
        const int n = n_tasks - i < kMaxLaunchTasks ? n_tasks - i : kMaxLaunchTasks;
        const uint32_t begin = tasks[i].block_begin, end = i + n < n_tasks ? tasks[i + n].block_begin : total_blocks;
        auto fill = [&](auto &pack) {
            for (int k = 0; k < n; ++k) {
                pack.t[k] = tasks[i + k];
                pack.t[k].block_begin -= begin;
            }
            return f(pack, n, end - begin);
        };
        int rc;
        if (n == 1) {
            TaskPack<1> p;
            rc = fill(p);
        } else if (n <= 32) {
            TaskPack<32> p;
            rc = fill(p);
        } else {
            TaskPack<kMaxLaunchTasks> p;
            rc = fill(p);
        }
        if (rc) return rc;
    }
    return CP_OK;
}
// Create what the gathers and their checks need on the device (its error word; call
// outside stream capture).
int prepare_gather_kernels();
// Error words that kernels set: pinned host memory mapped on the device.
struct ErrorWord {
    int *host = nullptr, *dev = nullptr;
};
int error_word_alloc(ErrorWord *w);
void error_word_free(ErrorWord *w);
int error_word_take(const ErrorWord &w);  // its value, cleared (after a synchronisation)
// The device's word, set by a bounded wait that ran out (of the kernels only
// cp_debug_wait_timeout's waits); check_device_error syncs `st`, returns CP_ETIMEOUT (and
// clears the word) if it was set.
int *device_error_flag();
int check_device_error(cudaStream_t st);

// Extract the e0 row laid out [D1][Pp] (signed representatives) into [P][D1]
// residues in [0, p).
int launch_transpose_row(const uint32_t *row, uint32_t *out, const uint32_t *primes_dev, int D1, int P, int Pp,
                         cudaStream_t st);

// Adds to *sum_dev the degrees in the windows of n states of a vector of v vertices
// capped at degree cap (first: of e_0 at height 1).
int add_window_degrees(const uint16_t *win, uint64_t n, int v, int cap, unsigned long long *sum_dev, cudaStream_t st);

// ------------------------------------------------------------------ CRT (crt.cu)
// Device CRT of residues [P][n_coeffs] into limbs [n_coeffs][limbs]; with
// flags_dev, per-coefficient flags (bit 0: bound_dev[j] + 2 > bit length of the
// prime product; bit 1: the first P-1 primes give another value).
int launch_crt(const uint32_t *res_dev, const uint32_t *primes_host, int P, int n_coeffs, uint32_t *limbs_dev,
               int limbs, const uint32_t *bound_dev, uint32_t *flags_dev, cudaStream_t st, int arrays = 1);
int primes_product_bits(const uint32_t *primes, int P);
// Bit lengths of C(n_edges, j), j < n_coeffs (Whitney's bound |c_j| <= C(|E|, j)).
void binomial_bits(uint64_t n_edges, int n_coeffs, uint32_t *bits_out);
uint64_t rectangle_edges(int lattice, int L, int N);
// CP_OK if no flag is set, else CP_EPRIMES with a message counting them.
int crt_outcome(const uint32_t *flags, int n_coeffs);
// Load the CRT module (and the static array of cp_crt_static) on the current device.
int crt_static_touch();

// What an object's padding lanes take beyond the rows of its primes alone.  The lanes of
// all objects on a device together get at most 1 / kPadFraction of its memory, so that
// strips of one prime, four times as large with them, still leave room for the next ones;
// an object whose lanes do not fit in that has rows of its primes alone (the register
// kernel; results are the same).  Given back with the object.
constexpr size_t kPadFraction = 8;
class PadShare {
    int dev_ = -1;
    size_t bytes_ = 0;

  public:
    PadShare() = default;
    PadShare(const PadShare &) = delete;
    PadShare &operator=(const PadShare &) = delete;
    ~PadShare();
    bool take(size_t bytes);  // on the current device, in addition to what it holds
};

}  // namespace cp
