// Transition tables of the per-site factors, built on the GPU.
//
// For every source state of a factor's input space: unrank it, apply the
// factor's single-edge operators (Sec. 3.1-3.3), drop the terms the
// projectors kill, rank each surviving partition in the output space, and
// emit (dst, src, shift, coef) terms.  The terms are then counting-sorted by
// destination into a CSR table, so that the per-site kernel is a gather.
// Tables depend only on (lattice, L, site): they are built once per device
// and shared by every strip, row, height and prime.
#include <cuda_runtime.h>

#include <algorithm>
#include <map>
#include <mutex>
#include <string>
#include <tuple>
#include <utility>

#include "cp_internal.h"
#include "modred.cuh"
#include "ncnnn.cuh"

namespace cp {

// ------------------------------------------------------------------ rank tables

// cnt and off from the recursion M_p = M_{p-1} + sum_{k=0}^{p-2} M_k M_{p-k-2}, eq. (M_recurs).
__global__ void rank_tables_kernel(RankTables *T) {
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    uint64_t M[kTblStride];
    M[0] = 1;
    M[1] = 1;
    for (int p = 2; p < kTblStride; ++p) {
        uint64_t s = M[p - 1];
        for (int k = 0; k <= p - 2; ++k) s += M[k] * M[p - k - 2];
        M[p] = s;
    }
    T->cnt[0] = 1;
    for (int n = 1; n < kTblStride; ++n) T->cnt[n] = M[n - 1];
    for (int k = 0; k < kTblStride * kTblStride; ++k) T->off[k] = 0;
    for (int n = 3; n < kTblStride; ++n) {
        uint64_t o = T->cnt[n - 1];
        for (int k = 0; k <= n - 3; ++k) {
            T->off[n * kTblStride + k] = o;
            o += T->cnt[k + 1] * T->cnt[n - k - 2];
        }
    }
    // Catalan numbers and the offsets of the non-crossing order (partner at 1+k)
    T->cntc[0] = 1;
    for (int n = 1; n < kTblStride; ++n) {
        uint64_t c = 0;
        for (int k = 0; k < n; ++k) c += T->cntc[k] * T->cntc[n - 1 - k];
        T->cntc[n] = c;
    }
    for (int k = 0; k < kTblStride * kTblStride; ++k) T->offc[k] = 0;
    for (int n = 2; n < kTblStride; ++n) {
        uint64_t o = T->cntc[n - 1];
        for (int k = 0; k <= n - 2; ++k) {
            T->offc[n * kTblStride + k] = o;
            o += T->cntc[k] * T->cntc[n - 1 - k];
        }
    }
}

// ------------------------------------------------------------------ term generation

struct Term {
    Labels s;
    int32_t coef;
    int32_t shift;
};

constexpr int kMaxTerms = 8;   // terms of one factor applied to one partition

// H_{a,b} = 1 - J_{a,b} at v = -1: a term with a ~ b is killed (H s = s - s), otherwise
// it splits into itself and the joined partition with -w.
__device__ int op_h(Term *t, int n, int m, int a, int b) {
    int k = n;
    for (int j = 0; j < n; ++j) {
        if (t[j].s.v[a] == t[j].s.v[b]) { t[j].coef = 0; continue; }
        Term u = t[j];
        join_blocks(u.s, m, a, b);
        u.coef = -u.coef;
        u.shift += 1;
        t[k++] = u;
    }
    int w = 0;
    for (int j = 0; j < k; ++j)
        if (t[j].coef != 0) t[w++] = t[j];
    return w;
}

// V_i = D_i - w.
__device__ int op_v(Term *t, int n, int m, int i) {
    for (int j = 0; j < n; ++j) {
        Term u = t[j];
        u.coef = -u.coef;
        u.shift += 1;
        t[n + j] = u;
        detach_site(t[j].s, m, i);
    }
    return 2 * n;
}

__device__ int op_d(Term *t, int n, int m, int i) {
    for (int j = 0; j < n; ++j) detach_site(t[j].s, m, i);
    return n;
}

// P_{j,j+1} for j in [lo, hi) except `skip`.
__device__ int op_p(Term *t, int n, int m, int lo, int hi, int skip) {
    if (lo >= hi) return n;
    const uint32_t pairs = ((1u << hi) - 1u) & ~((1u << lo) - 1u) & ~(skip >= 0 ? 1u << skip : 0u);
    int w = 0;
    for (int j = 0; j < n; ++j)
        if ((adjacent_pairs(t[j].s, m) & pairs) == 0) t[w++] = t[j];
    return w;
}

// Any-v operators (Sec. 3.1): H_{a,b} = 1 + v J_{a,b}, where J is the identity
// (no w) when a ~ b and joins with a factor w otherwise; V_i = v w + D_i.
__device__ int op_hv(Term *t, int n, int m, int a, int b, int v) {
    int k = n;
    for (int j = 0; j < n; ++j) {
        if (t[j].s.v[a] == t[j].s.v[b]) {
            t[j].coef *= (1 + v);
            continue;
        }
        Term u = t[j];
        join_blocks(u.s, m, a, b);
        u.coef *= v;
        u.shift += 1;
        t[k++] = u;
    }
    int w = 0;
    for (int j = 0; j < k; ++j)
        if (t[j].coef != 0) t[w++] = t[j];
    return w;
}

__device__ int op_vv(Term *t, int n, int m, int i, int v) {
    for (int j = 0; j < n; ++j) {
        Term u = t[j];
        u.coef *= v;
        u.shift += 1;
        t[n + j] = u;
        detach_site(t[j].s, m, i);
    }
    int w = 0;
    for (int j = 0; j < 2 * n; ++j)
        if (t[j].coef != 0) t[w++] = t[j];
    return w;
}

// Terms of one factor applied to one partition.
__device__ __noinline__ int factor_terms(const OpDesc &op, const Labels &s, Term *t) {
    int m = op.m, i = op.i, n = 1;
    t[0].s = s;
    t[0].coef = 1;
    t[0].shift = 0;
    switch (op.kind) {
        case OP_SQUARE:  // (prod_{j!=i} P) V_i H_{i,i+1};  T_m = (prod P) V_m      eq. (T_sq_proj)
            if (i < m - 1) n = op_h(t, n, m, i, i + 1);
            n = op_v(t, n, m, i);
            n = op_p(t, n, m, 0, m - 1, i < m - 1 ? i : -1);
            break;
        case OP_TRIANGULAR:  // (prod P) V_i H_{i-1,i} H_{i,i+1}                    Sec. 3.3
            if (i < m - 1) n = op_h(t, n, m, i, i + 1);
            if (i > 0) n = op_h(t, n, m, i - 1, i);
            n = op_v(t, n, m, i);
            n = op_p(t, n, m, 0, m - 1, -1);
            break;
        case OP_LAST:  // (prod_{j>i} P) D_i H_{i,i+1}                                eq. (T_last_i)
            if (i < m - 1) n = op_h(t, n, m, i, i + 1);
            n = op_d(t, n, m, i);
            n = op_p(t, n, m, i + 1, m - 1, -1);
            break;
        case OP_POTTS_SQUARE:  // V_i H_{i,i+1}: the rows of T = (prod V)(prod H), Sec. 3.2
            if (i < m - 1) n = op_hv(t, n, m, i, i + 1, op.v);
            n = op_vv(t, n, m, i, op.v);
            break;
        case OP_POTTS_TRIANGULAR:  // V_i H_{i-1,i} H_{i,i+1} (H_{i-1,i}: the diagonal, Sec. 3.3)
            if (i < m - 1) n = op_hv(t, n, m, i, i + 1, op.v);
            if (i > 0) n = op_hv(t, n, m, i - 1, i, op.v);
            n = op_vv(t, n, m, i, op.v);
            break;
        case OP_POTTS_LAST:  // D_i H_{i,i+1}: last horizontal edges; every state ends at e_0
            if (i < m - 1) n = op_hv(t, n, m, i, i + 1, op.v);
            n = op_d(t, n, m, i);
            break;
        default:  // identity
            break;
    }
    return n;
}

// Rank of a term's state in the output space, or ~0u with the error bit set.
__device__ __forceinline__ uint32_t term_dst(const Labels &s, const Space &out, const RankTables &T, int *bad) {
    if (!space_contains(s, out)) {
        *bad |= 1;
        return ~0u;
    }
    const uint64_t r = space_rank(s, out, T);
    if (r >= out.size) {
        *bad |= 1;
        return ~0u;
    }
    return (uint32_t)r;
}

// One packed edge into slot w of its source, if it fits (err bits below).
__device__ __forceinline__ void put_term(const OpDesc &op, uint64_t src, uint32_t dst, int coef, int shift, int w, int K,
                                         uint32_t *slot_dst, uint32_t *slot_edge, int *bad) {
    const int sb = op.src_bits, cb = 30 - sb;  // coefficient bits
    if (w >= K) {
        *bad |= 2;
        return;
    }
    if (coef < -(1 << (cb - 1)) || coef > (1 << (cb - 1)) - 1 || shift > 3) {
        *bad |= 4;
        slot_dst[src * K + w] = ~0u;
        return;
    }
    slot_dst[src * K + w] = dst;
    slot_edge[src * K + w] =
        (uint32_t)src | ((uint32_t)shift << sb) | (((uint32_t)coef & ((1u << cb) - 1u)) << (sb + 2));
}

// One thread per source state.  slot_dst[src*K + t] = destination rank or ~0u,
// slot_edge[...] = packed edge.  err bits: 1 bad rank / membership, 2 too many
// terms, 4 coefficient out of range, 8 unrank/rank mismatch of the source.
__global__ void build_terms_kernel(OpDesc op, const RankTables *Tg, uint32_t *slot_dst, uint32_t *slot_edge, int K,
                                   int *err) {
    __shared__ RankTables T;
    stage_tables(T, Tg);
    uint64_t src = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (src >= op.in.size) return;
    Labels s;
    space_unrank(src, op.in, s, T);
    int bad = 0;
    if (!space_contains(s, op.in) || space_rank(s, op.in, T) != src) bad |= 8;
    Term t[kMaxTerms];
    const int n = factor_terms(op, s, t);
    uint32_t dst[kMaxTerms];
    for (int j = 0; j < n; ++j) dst[j] = term_dst(t[j].s, op.out, T, &bad);
    // merge equal (dst, shift)
    for (int j = 0; j < n; ++j) {
        if (t[j].coef == 0 || dst[j] == ~0u) continue;
        for (int q = j + 1; q < n; ++q)
            if (dst[q] == dst[j] && t[q].shift == t[j].shift && t[q].coef != 0) {
                t[j].coef += t[q].coef;
                t[q].coef = 0;
            }
    }
    int w = 0;
    for (int j = 0; j < n; ++j)
        if (t[j].coef != 0 && dst[j] != ~0u) put_term(op, src, dst[j], t[j].coef, t[j].shift, w++, K, slot_dst, slot_edge, &bad);
    for (; w < K; ++w) slot_dst[src * K + w] = ~0u;
    if (bad) atomicOr(err, bad);
}

// A two-site table, the second factor applied to every term of the first: LANES threads
// per source state, each for every LANES-th term of the first factor, which meet in
// shared memory to merge equal (dst, shift).  A source has at most 14 terms before that
// on the square lattice (8 a lane of two) and 23 on the triangular one (15 a lane of
// two), at every width, as a factor changes little beyond the sites beside its own; a
// lane has room for kLane, and the build fails if one needs more.  Bound by unranking,
// relabelling and ranking in local memory: one thread per source took 170 us a table at
// width 12 (5 798 states), eight 95 us, and with the labels as words 85 us (four lanes or
// a warp per source: the cold tables of that width 2.91 or 2.71 ms against 2.55).  Tables
// that fill the SMs anyway take fewer lanes, as each repeats the first factor, and live
// on the L1 that the shared slots leave to local memory: cold tables (without padding
// slots to 64 a source, and with small stacks in the ranking), square width 17 two lanes
// 56.1 ms (64 slots 61.6, one lane 60.2), triangular width 14 two lanes 5.6 (one 6.1),
// width 16 one 15.9 (two 17.3), width 18 one 107.8 (two 130.9, 64 slots 175).
template <int LANES, int kLane>
__global__ void __launch_bounds__(128)
    build_fused_terms_kernel(OpDesc op, const RankTables *Tg, uint32_t *slot_dst, uint32_t *slot_edge, int K, int *err) {
    constexpr int kSources = 128 / LANES, kAll = LANES * kLane;
    __shared__ RankTables T;
    __shared__ uint32_t s_key[kSources][kAll + 1];  // destination << 3 | shift
    __shared__ int s_coef[kSources][kAll + 1];
    stage_tables(T, Tg);
    const int grp = threadIdx.x / LANES, lane = threadIdx.x % LANES;
    const uint64_t src = (uint64_t)blockIdx.x * kSources + grp;
    const bool have = src < op.in.size;
    uint32_t *key = s_key[grp];
    int *coef = s_coef[grp];
    int bad = 0, mine = 0;  // mine: this lane's terms, the first of its kLane slots
    if (have) {
        Labels s;
        space_unrank(src, op.in, s, T);
        if (lane == 0 && (!space_contains(s, op.in) || space_rank(s, op.in, T) != src)) bad |= 8;
        Term a[kMaxTerms], t[kMaxTerms];
        const int na = factor_terms(op, s, a);
        OpDesc ob = op;
        ob.kind = op.kind_b;
        ob.i = op.i_b;
        for (int j = lane; j < na; j += LANES) {
            const int n = factor_terms(ob, a[j].s, t);
            for (int q = 0; q < n; ++q) {
                const uint32_t d = term_dst(t[q].s, op.out, T, &bad);
                if (d == ~0u) continue;
                if (mine == kLane) {
                    bad |= 2;
                    break;
                }
                const int k = lane * kLane + mine++;
                key[k] = d << 3 | (uint32_t)(t[q].shift + a[j].shift);
                coef[k] = t[q].coef * a[j].coef;
            }
        }
    }
    int end[LANES];  // end of each lane's terms
#pragma unroll
    for (int l = 0; l < LANES; ++l) end[l] = l * kLane + __shfl_sync(0xffffffffu, mine, l, LANES);
    __syncwarp();
    // of equal (dst, shift) the first stands for them all with the sum of their
    // coefficients; the slots are the lanes' terms one after another, counted, then written
    int w = 0;
    uint32_t keep = ~0u;  // of this lane's terms, one bit each
    static_assert(kLane <= 32, "a bit per slot of a lane");
    for (int round = 0; round < 2; ++round) {
        int c = 0;
        for (int i = 0; i < mine; ++i) {
            if (!(keep >> i & 1u)) continue;
            const int k = lane * kLane + i;
            const uint32_t x = key[k];
            int sum = 0;
            bool first = true;
#pragma unroll
            for (int l = 0; l < LANES; ++l)
                for (int m = l * kLane; m < end[l]; ++m)
                    if (key[m] == x) {
                        sum += coef[m];
                        first = first && m >= k;
                    }
            if (!first || sum == 0) {
                keep &= ~(1u << i);
                continue;
            }
            if (round) put_term(op, src, x >> 3, sum, (int)(x & 7u), w + c, K, slot_dst, slot_edge, &bad);
            ++c;
        }
        if (round) break;
        w = c;
        for (int o = 1; o < LANES; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, w, o, LANES);
            if (lane >= o) w += y;
        }
        const int total = __shfl_sync(0xffffffffu, w, LANES - 1, LANES);
        w -= c;
        if (have)
            for (int r = total + lane; r < K; r += LANES) slot_dst[src * K + r] = ~0u;
    }
    if (bad) atomicOr(err, bad);
}

// ------------------------------------------------------------------ CSR by destination

// Edges per destination, and sum of |coef| per destination into csum.
__global__ void count_kernel(const uint32_t *slot_dst, const uint32_t *slot_edge, uint64_t n_slots, int src_bits,
                             uint32_t *cnt, uint32_t *csum, int *max_coef) {
    uint32_t m = 0;  // largest |coefficient| seen by this thread
    for (uint64_t k = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n_slots;
         k += (uint64_t)gridDim.x * blockDim.x) {
        uint32_t d = slot_dst[k];
        if (d == ~0u) continue;
        atomicAdd(&cnt[d], 1u);
        const int c = (int)slot_edge[k] >> (src_bits + 2);
        const uint32_t a = (uint32_t)(c < 0 ? -c : c);
        atomicAdd(&csum[d], a);
        m = max(m, a);
    }
    for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) atomicMax(max_coef, (int)m);
}

constexpr int kScanThreads = 1024;

// Exclusive scan, three launches: per-block sums, scan of the block sums, per-block
// scan + offset.  Up to kScanAlone blocks the last launch does it alone, each block
// adding up the words before its own: at most 31 loads a thread, all in flight at
// once, against two launches more (a table of width 12 has 16 blocks; a launch there
// is 2.3 us, and two scans a table make them a tenth of its build).
constexpr uint64_t kScanAlone = 32;
__device__ __forceinline__ uint32_t block_inclusive_scan(uint32_t v, uint32_t *warp_sums) {
    int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        uint32_t y = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += y;
    }
    if (lane == 31) warp_sums[wid] = v;
    __syncthreads();
    if (wid == 0) {
        uint32_t x = lane < (int)(blockDim.x >> 5) ? warp_sums[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        warp_sums[lane] = x;
    }
    __syncthreads();
    if (wid > 0) v += warp_sums[wid - 1];
    return v;
}

__global__ void scan_block_sums(const uint32_t *in, uint64_t n, uint32_t *block_sums) {
    __shared__ uint32_t ws[32];
    uint64_t k = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    uint32_t v = k < n ? in[k] : 0;
    uint32_t s = block_inclusive_scan(v, ws);
    if (threadIdx.x == blockDim.x - 1) block_sums[blockIdx.x] = s;
}

__global__ void scan_sums_serial(uint32_t *sums, uint32_t n_blocks) {
    // single block: exclusive scan of the block sums in chunks of blockDim
    __shared__ uint32_t ws[32];
    __shared__ uint32_t carry;
    if (threadIdx.x == 0) carry = 0;
    __syncthreads();
    for (uint32_t base = 0; base < n_blocks; base += blockDim.x) {
        uint32_t k = base + threadIdx.x;
        uint32_t v = k < n_blocks ? sums[k] : 0;
        uint32_t inc = block_inclusive_scan(v, ws);
        uint32_t c = carry;
        if (k < n_blocks) sums[k] = c + inc - v;
        __syncthreads();
        if (threadIdx.x == blockDim.x - 1) carry = c + inc;
        __syncthreads();
    }
}

// With `of`, also the largest of of[0..n) into *largest (a warp maximum, one atomic
// per warp; on its own that was one more launch of 4.6 us a table); with `total`, the sum there too.
__global__ void scan_finish(const uint32_t *in, uint64_t n, const uint32_t *block_off, uint32_t *out, const uint32_t *of,
                            int *largest, uint32_t *total) {
    __shared__ uint32_t ws[32], before;
    const uint64_t k = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    uint32_t off = 0;
    if (block_off) {
        off = block_off[blockIdx.x];
    } else {
        if (threadIdx.x == 0) before = 0;
        __syncthreads();
#pragma unroll 8
        for (uint32_t b = 0; b < blockIdx.x; ++b) off += in[b * blockDim.x + threadIdx.x];
        off = __reduce_add_sync(0xffffffffu, off);
        if ((threadIdx.x & 31) == 0) atomicAdd(&before, off);
        __syncthreads();
        off = before;
    }
    const uint32_t v = k < n ? in[k] : 0;
    const uint32_t inc = block_inclusive_scan(v, ws);
    const uint32_t exc = off + inc - v;
    if (k < n) out[k] = exc;
    if (k == n - 1) {
        out[n] = exc + v;
        if (total) *total = exc + v;
    }
    if (of) {
        const uint32_t m = __reduce_max_sync(0xffffffffu, k < n ? of[k] : 0u);
        if ((threadIdx.x & 31) == 0) atomicMax(largest, (int)m);
    }
}

__global__ void fill_kernel(const uint32_t *slot_dst, const uint32_t *slot_edge, uint64_t n_slots,
                            const uint32_t *row_ptr, uint32_t *cursor, uint32_t *edges) {
    for (uint64_t k = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n_slots;
         k += (uint64_t)gridDim.x * blockDim.x) {
        uint32_t d = slot_dst[k];
        if (d == ~0u) continue;
        uint32_t pos = row_ptr[d] + atomicAdd(&cursor[d], 1u);
        edges[pos] = slot_edge[k];
    }
}

// Deterministic order inside each destination: by packed value (src, then shift/coef;
// all different).  One warp per destination: every entry's place is the number of
// smaller ones, up to kSortRegs entries a lane.  (An insertion sort by one thread per
// destination took 62 us a table at width 12, for the few rows of a hundred entries.)
constexpr int kSortRegs = 8;
__global__ void sort_segments_kernel(const uint32_t *row_ptr, uint64_t n_dst, uint32_t *edges) {
    const uint64_t d = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const uint32_t lane = threadIdx.x & 31;
    if (d >= n_dst) return;
    const uint32_t b = row_ptr[d], n = row_ptr[d + 1] - b;
    if (n <= 32) {
        const uint32_t x = lane < n ? edges[b + lane] : 0xffffffffu;
        uint32_t at = 0;
        for (uint32_t i = 0; i < n; ++i) at += __shfl_sync(0xffffffffu, x, i) < x ? 1u : 0u;
        if (lane < n) edges[b + at] = x;
    } else if (n <= 32 * kSortRegs) {
        uint32_t x[kSortRegs], at[kSortRegs] = {};
#pragma unroll
        for (int m = 0; m < kSortRegs; ++m) x[m] = lane + 32 * m < n ? edges[b + lane + 32 * m] : 0xffffffffu;
        for (uint32_t i = 0; i < n; ++i) {
            const uint32_t y = edges[b + i];
#pragma unroll
            for (int m = 0; m < kSortRegs; ++m) at[m] += y < x[m] ? 1u : 0u;
        }
        __syncwarp();
#pragma unroll
        for (int m = 0; m < kSortRegs; ++m)
            if (lane + 32 * m < n) edges[b + at[m]] = x[m];
    } else if (lane == 0) {
        for (uint32_t i = 1; i < n; ++i) {
            const uint32_t x = edges[b + i];
            uint32_t j = i;
            for (; j > 0 && edges[b + j - 1] > x; --j) edges[b + j] = edges[b + j - 1];
            edges[b + j] = x;
        }
    }
}

// flag[b] = 1 if the NCNNN partition of rank b has e alone and e-1 !~ e+1, so that
// J_{e,e+1} of it lies in X_e (every partition of X_e with e ~ e+1 arises once).
__global__ void x_partner_kernel(int m, int e, const RankTables *Tg, uint32_t *flag) {
    __shared__ RankTables T;
    stage_tables(T, Tg);
    uint64_t b = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= T.cnt[m]) return;
    Labels s;
    ncnnn_unrank(b, 0, m, s, T);
    bool alone = true;
    for (int i = 0; i < m; ++i)
        if (i != e && s.v[i] == s.v[e]) alone = false;
    flag[b] = (alone && (e == 0 || s.v[e - 1] != s.v[e + 1])) ? 1u : 0u;
}

// ------------------------------------------------------------------ degree windows

// Window words of a space before the shortest paths are known: lo = 255 (not
// reached), the number of blocks in the high byte; e0 != 0: rank 0 is e_0, lo = 0.
__global__ void init_win_kernel(Space sp, const RankTables *Tg, uint16_t *win, int e0) {
    __shared__ RankTables T;
    stage_tables(T, Tg);
    const uint64_t r = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= sp.size) return;
    Labels s;
    space_unrank(r, sp, s, T);
    int blocks = 0;
    for (int i = 0; i < sp.m; ++i) blocks = max(blocks, (int)s.v[i] + 1);
    win[r] = (uint16_t)((blocks << 8) | (e0 && r == 0 ? 0 : 255));
}

// The same for a read-out space: its states are the first ranks of the row space.
__global__ void copy_blocks_kernel(const uint16_t *win_row, uint16_t *win, uint64_t n) {
    const uint64_t r = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (r < n) win[r] = win_row[r] | 255;
}

// One relaxation of the shortest paths over a table: lo_dst = min(lo_dst, lo_src + shift).
// Skipped when *prev is given and zero (the pass before changed nothing); *changed
// is set where a value fell.  A small table's launch lasts as long as its longest
// row's chain of dependent loads (rows of a hundred edges come up), so eight lanes
// share a row there; a large one is bound by its instructions and takes a thread per
// row (cold tables of square strips with rows of 336 bytes, one lane and eight: width 14,
// 57 346 rows, 6.7 and 7.6 ms, width 16 18.1 and 27.6; width 13, 21 309 rows, 4.9 and 4.8).
constexpr uint64_t kWinManyLanes = 32768;  // rows up to which a row takes eight lanes
template <uint32_t kLanes>
__global__ void relax_win_kernel(const uint32_t *row_ptr, const uint32_t *edges, uint64_t n_dst, int src_bits,
                                 const uint16_t *win_in, uint16_t *win_out, const int *prev, int *changed) {
    if (prev && *prev == 0) return;
    const uint64_t k = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x, d = k / kLanes;
    const uint32_t mask = (1u << src_bits) - 1u, lane = k % kLanes;
    uint32_t m = 255;
    if (d < n_dst)
        for (uint32_t e = row_ptr[d] + lane, e1 = row_ptr[d + 1]; e < e1; e += kLanes) {
            const uint32_t q = edges[e], lo = win_in[q & mask] & 0xffu;
            if (lo != 255) m = min(m, min(lo + ((q >> src_bits) & 3u), 254u));
        }
    for (uint32_t o = kLanes / 2; o > 0; o >>= 1) m = min(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (d >= n_dst || lane) return;
    const uint32_t w = win_out[d];
    if (m < (w & 0xffu)) {
        win_out[d] = (uint16_t)((w & 0xff00u) | m);
        *changed = 1;
    }
}

// Every transition keeps its source's window inside its destination's: lo_dst <=
// lo_src + shift, and V_src - blocks_src + shift <= V_dst - blocks_dst.  With e0 (a row's
// last table), no state but e_0 (rank 0) has degree 0.  (Lanes as above.)
template <uint32_t kLanes>
__global__ void check_win_kernel(const uint32_t *row_ptr, const uint32_t *edges, uint64_t n_dst, int src_bits, int sites,
                                 const uint16_t *win_in, const uint16_t *win_out, int e0, int *bad) {
    const uint64_t k = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x, d = k / kLanes;
    if (d >= n_dst) return;
    const uint32_t mask = (1u << src_bits) - 1u, w = win_out[d];
    bool ok = !e0 || ((w & 0xffu) == 0) == (d == 0);
    for (uint32_t e = row_ptr[d] + (uint32_t)(k % kLanes), e1 = row_ptr[d + 1]; e < e1; e += kLanes) {
        const uint32_t q = edges[e], sh = (q >> src_bits) & 3u, x = win_in[q & mask];
        if ((x & 0xffu) == 255) continue;
        ok = ok && (w & 0xffu) <= min((x & 0xffu) + sh, 254u) && (w >> 8) + sh <= (x >> 8) + (uint32_t)sites;
    }
    if (!ok) *bad = 1;
}

// ------------------------------------------------------------------ host side

// Working memory of one table set's build: one device allocation, handed out from
// the start for each table (the build's kernels run on one stream, in order) and
// freed with the object, instead of a dozen allocations and frees, each a
// synchronisation, per table.  What stays of a set and its plain edges lie in pools for
// the same reason, and a table stops the host once (for its edges' number): with four
// allocations and two stops a table, small sets of one table per factor took longer
// than without degree windows (cold, square Potts width 7 1.97 ms, 1.66 without, now 1.44;
// square width 9, 336-byte rows, 2.94, 2.72 and 2.20).
struct Scratch {
    char *base = nullptr;
    size_t cap = 0, used = 0;
    cudaStream_t st;
    DevPool edges;                // plain edges of the set's tables, below kBigTable of them
    uint32_t *counts = nullptr;   // units of each table (kMaxTables words), then the windows' flags (kWinFlags)
    int n_counts = 0;
    bool idle = false;            // nothing of the build is in flight any more
    explicit Scratch(cudaStream_t s) : st(s) {}
    Scratch(const Scratch &) = delete;
    ~Scratch() {
        if (!idle) cudaStreamSynchronize(st);
        dev_free(base);
    }
    // Start over with at least `bytes` bytes.
    int reset(size_t bytes) {
        used = 0;
        if (bytes <= cap) return CP_OK;
        if (base) cudaStreamSynchronize(st);
        dev_free(base);
        base = nullptr;
        cap = 0;
        const int rc = dev_alloc((void **)&base, bytes);
        if (!rc) cap = bytes;
        return rc;
    }
    static size_t span(size_t bytes) { return (bytes + 255) & ~(size_t)255; }
    template <class T>
    T *take(size_t n) {  // (reset() made room)
        T *p = reinterpret_cast<T *>(base + used);
        used += span(n * sizeof(T));
        return p;
    }
};

static size_t scan_bytes(uint64_t n) { return Scratch::span(((n + kScanThreads - 1) / kScanThreads + 1) * 4); }

// out[0..n]: exclusive scan of cnt, with the total at the end, and the largest of
// of[0..n) into *largest (asynchronous on sc->st).
static int scan_exclusive(const uint32_t *cnt, uint64_t n, uint32_t *out, Scratch *sc, const uint32_t *of = nullptr,
                          int *largest = nullptr, uint32_t *total = nullptr) {
    uint64_t nb = (n + kScanThreads - 1) / kScanThreads;
    if (nb > (1u << 31)) return fail(CP_EINVAL, "scan too large");
    uint32_t *sums = nullptr;
    if (nb > kScanAlone) {
        sums = sc->take<uint32_t>(nb + 1);
        scan_block_sums<<<(unsigned)nb, kScanThreads, 0, sc->st>>>(cnt, n, sums);
        scan_sums_serial<<<1, kScanThreads, 0, sc->st>>>(sums, (uint32_t)nb);
    }
    scan_finish<<<(unsigned)nb, kScanThreads, 0, sc->st>>>(cnt, n, sums, out, of, largest, total);
    CP_CUDA_TRY(cudaGetLastError());
    return CP_OK;
}

static int build_x_prefix(int m, int e, Scratch *sc, DevPool *pool, uint32_t **out) {
    const RankTables *T_dev = nullptr;
    RankTables T;
    int rc = device_rank_tables(&T_dev, &T);
    if (rc) return rc;
    const uint64_t Sb = T.cnt[m];
    if ((rc = sc->reset(Scratch::span(Sb * 4) + scan_bytes(Sb)))) return rc;
    uint32_t *flag = sc->take<uint32_t>(Sb), *pre = nullptr;
    if ((rc = pool->alloc((void **)&pre, (Sb + 1) * 4))) return rc;
    x_partner_kernel<<<(unsigned)((Sb + 127) / 128), 128, 0, sc->st>>>(m, e, T_dev, flag);
    rc = scan_exclusive(flag, Sb, pre, sc);
    uint32_t total = 0;
    cudaError_t ce = cudaMemcpyAsync(&total, pre + Sb, 4, cudaMemcpyDeviceToHost, sc->st);
    if (ce == cudaSuccess) ce = cudaStreamSynchronize(sc->st);
    if (!rc && ce != cudaSuccess) rc = fail(CP_ECUDA, std::string("x_partner: ") + cudaGetErrorString(ce));
    if (!rc && total != T.cnt[m - 1]) rc = fail(CP_ESTATE, "excepted space has the wrong size");
    if (!rc) *out = pre;
    return rc;
}

// Packs the rows of one run of kPackRows into units (cp_internal.h), in order: one
// thread per run.  Without `units` it only counts them.
__global__ void pack_units_kernel(const uint32_t *row_ptr, uint64_t n, uint32_t most, uint32_t split, uint32_t *cnt,
                                  const uint32_t *pos, uint4 *units, uint32_t *total) {
    const uint64_t c = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x, r0 = c * kPackRows;
    if (r0 >= n) return;
    const uint64_t r1 = min(n, r0 + kPackRows);
    uint32_t k = units ? pos[c] : 0;
    uint64_t u0 = r0;  // first row of the open unit
    uint32_t ub = row_ptr[r0], b = ub;
    for (uint64_t r = r0; r <= r1; ++r) {
        const uint32_t e = r < r1 ? row_ptr[r + 1] : b;  // the row's edges are [b, e)
        const bool heavy = e - b > split;
        if (r > u0 && (r == r1 || heavy || e - ub > most || r - u0 == 32)) {  // close the open unit
            if (units) units[k] = make_uint4((uint32_t)u0, (uint32_t)(r - u0), ub, b);
            ++k;
            u0 = r;
            ub = b;
        }
        if (heavy) {
            for (uint32_t i = 0; i < kSplitParts; ++i) {
                if (units) units[k] = make_uint4((uint32_t)r, 1u | (1u << 6) | (i << 8), b, e);
                ++k;
            }
            u0 = r + 1;
            ub = e;
        }
        b = e;
    }
    if (!units) cnt[c] = k;
    else if (r1 == n) *total = k;
}

// Source states up to which a two-site table takes eight lanes each, and a triangular one two.
constexpr uint64_t kFusedManyLanes = 16384, kFusedTwoLanes = 65536;

constexpr int kMaxTables = 2 * CP_MAX_L;  // of a set: a row's and the read-out's
// Of the windows: changed, one per pass; the checks' flag; what the read-out's tables changed (not used).
constexpr int kMaxPasses = 64, kWinFlags = kMaxPasses + 2;

static uint64_t unit_runs(uint64_t n_dst) { return (n_dst + kPackRows - 1) / kPackRows; }

// Units of a table, in the room that build_table reserved; n_units is read back with the
// windows' flags (build_windows), so a small table has room for the most there can be: a
// unit is closed by a run's end, by the next row's edges (two neighbours then have more
// than `most` between them) or by a heavy row, which is kSplitParts itself.
static int build_units(SiteTable *tab, Scratch *sc, DevPool *pool) {
    const uint64_t n = tab->n_dst, runs = unit_runs(n);
    uint32_t *cnt = sc->take<uint32_t>(runs), *pos = sc->take<uint32_t>(runs + 1);
    const unsigned grid = (unsigned)((runs + 63) / 64);
    const uint32_t most = unit_edges(tab->nnz), split = split_edges(most);
    pack_units_kernel<<<grid, 64, 0, sc->st>>>(tab->row_ptr, n, most, split, cnt, nullptr, nullptr, nullptr);
    int rc = scan_exclusive(cnt, runs, pos, sc);
    if (rc) return rc;
    uint64_t room = std::min<uint64_t>(n, runs + 2 * tab->nnz / most + 1 + tab->nnz / split) + kSplitParts * (tab->nnz / split);
    if (room * sizeof(uint4) >= kPoolPiece) {
        uint32_t units = 0;
        CP_CUDA_TRY(cudaMemcpyAsync(&units, pos + runs, 4, cudaMemcpyDeviceToHost, sc->st));
        CP_CUDA_TRY(cudaStreamSynchronize(sc->st));
        room = units;
    }
    if ((rc = pool->alloc((void **)&tab->units, room * sizeof(uint4)))) return rc;
    if (!sc->counts && (rc = sc->edges.alloc((void **)&sc->counts, (kMaxTables + kWinFlags) * 4))) return rc;
    pack_units_kernel<<<grid, 64, 0, sc->st>>>(tab->row_ptr, n, most, split, nullptr, pos, tab->units,
                                               sc->counts + sc->n_counts++);
    CP_CUDA_TRY(cudaGetLastError());
    return CP_OK;
}

// The edges as the gathers read them, one warp per unit: each with its source's
// window word, its row within the unit and whether it is the row's first.  (A heavy
// row's parts write the same words.)
__global__ void fill_wedges_kernel(const uint4 *units, uint32_t n_units, const uint32_t *row_ptr, const uint32_t *edges,
                                   int src_bits, const uint16_t *win_in, uint2 *out) {
    const uint32_t k = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (k >= n_units) return;
    const uint4 u = units[k];
    const uint32_t nrows = u.y & 63u;
    for (uint32_t r = 0; r < nrows; ++r) {
        const uint32_t b = row_ptr[u.x + r], e1 = row_ptr[u.x + r + 1];
        for (uint32_t e = b + lane; e < e1; e += 32) {
            const uint32_t q = edges[e];
            out[e] = make_uint2(q, (uint32_t)win_in[q & ((1u << src_bits) - 1u)] | (r << 16) | (e == b ? 1u << 21 : 0u));
        }
    }
}

static int build_table(const OpDesc &op, const RankTables *T_dev, Scratch *sc, DevPool *pool, SiteTable *tab) {
    tab->op = op;
    tab->n_src = op.in.size;
    tab->n_dst = op.out.size;
    tab->n_site_out = op.out.size;
    if (op.in.size > ((1ull << op.src_bits) - 1) || op.out.size >= 0xFFFFFFFFull)
        return fail(CP_EINVAL, "state space too large for the edge format");
    const int K = op.max_terms;
    const uint64_t n_slots = op.in.size * (uint64_t)K, n_dst = op.out.size, runs = unit_runs(n_dst);
    const cudaStream_t st = sc->st;
    int rc = sc->reset(2 * Scratch::span(n_slots * 4) + Scratch::span((3 * n_dst + 4) * 4) + scan_bytes(n_dst) +
                       2 * Scratch::span((runs + 1) * 4) + scan_bytes(runs));
    if (rc) return rc;
    uint32_t *slot_dst = sc->take<uint32_t>(n_slots), *slot_edge = sc->take<uint32_t>(n_slots);
    uint32_t *cnt = sc->take<uint32_t>(3 * n_dst + 4), *cursor = cnt + n_dst, *csum = cursor + n_dst;
    int *err = reinterpret_cast<int *>(csum + n_dst);  // error bits, largest sum, largest coefficient, edges
    if ((rc = pool->alloc((void **)&tab->row_ptr, (n_dst + 1) * 4))) return rc;
    CP_CUDA_TRY(cudaMemsetAsync(cnt, 0, (3 * n_dst + 4) * 4, st));
    const int bt = 128;
    if (op.fused) {
        auto go = [&](auto kernel, int lanes) {
            kernel<<<(unsigned)((op.in.size * lanes + bt - 1) / bt), bt, 0, st>>>(op, T_dev, slot_dst, slot_edge, K, err);
        };
        if (op.in.size <= kFusedManyLanes) go(build_fused_terms_kernel<8, kMaxTerms>, 8);
        else if (op.kind != OP_TRIANGULAR) go(build_fused_terms_kernel<2, 8>, 2);
        else if (op.in.size <= kFusedTwoLanes) go(build_fused_terms_kernel<2, 16>, 2);
        else go(build_fused_terms_kernel<1, 24>, 1);
    } else
        build_terms_kernel<<<(unsigned)((op.in.size + bt - 1) / bt), bt, 0, st>>>(op, T_dev, slot_dst, slot_edge, K, err);
    count_kernel<<<1216, 256, 0, st>>>(slot_dst, slot_edge, n_slots, op.src_bits, cnt, csum, err + 2);
    CP_CUDA_TRY(cudaGetLastError());
    if ((rc = scan_exclusive(cnt, n_dst, tab->row_ptr, sc, csum, err + 1, reinterpret_cast<uint32_t *>(err + 3))))
        return rc;
    int herr[4] = {0, 0, 0, 0};
    CP_CUDA_TRY(cudaMemcpyAsync(herr, err, sizeof(herr), cudaMemcpyDeviceToHost, st));
    const cudaError_t e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return fail(CP_ECUDA, std::string("table build: ") + cudaGetErrorString(e));
    // The gathers reduce p 2^21 + sum_e coef_e x_e (x_e < p) exactly while
    // sum_e |coef_e| into every state stays below 2^20 (modred.cuh).
    if (herr[0] == 0 && herr[1] >= (int)kReduceMaxCoefSum)
        return fail(CP_EINVAL, "too many transitions into one state for the exact modular reduction");
    if (herr[0] == 4)
        return fail(CP_EINVAL, "a transition coefficient does not fit the " + std::to_string(30 - op.src_bits) +
                                   "-bit field of this width's edge format (|v| too large)");
    if (herr[0])
        return fail(CP_ESTATE, "transition table check failed (flags " + std::to_string(herr[0]) + ") for op kind " +
                                   std::to_string(op.kind) + " m=" + std::to_string(op.m) + " i=" +
                                   std::to_string(op.i));
    const uint32_t nnz = (uint32_t)herr[3];
    tab->nnz = nnz;
    tab->max_coef_sum = (uint32_t)herr[1];
    tab->max_abs_coef = (uint32_t)herr[2];
    rc = nnz >= kBigTable ? dev_alloc((void **)&tab->edges, (size_t)nnz * 4)
                          : sc->edges.alloc((void **)&tab->edges, (size_t)nnz * 4);
    if (rc) return rc;
    fill_kernel<<<1216, 256, 0, st>>>(slot_dst, slot_edge, n_slots, tab->row_ptr, cursor, tab->edges);
    sort_segments_kernel<<<(unsigned)((n_dst + 7) / 8), 256, 0, st>>>(tab->row_ptr, n_dst, tab->edges);
    CP_CUDA_TRY(cudaGetLastError());
    return build_units(tab, sc, pool);
}

TableSet::~TableSet() {
    for (auto *chain : {&row, &last})  // (only of a build that failed)
        for (auto &t : *chain)
            if (t.nnz >= kBigTable) dev_free(t.edges);
}

// Window words of every space of the two chains (cp_internal.h): the blocks by
// unranking, lo by relaxing the row's tables from e_0 until a whole row changes
// nothing (values only fall, a row per pass; a state needs about as many rows as
// its blocks are nested: up to width 17 the last change came in pass (L + 1) / 2, of
// Potts strips L / 2 + 1, so one more does in a round, each a no-op once nothing
// changes), then the read-out's tables once.
static int build_windows(TableSet *ts, const RankTables *T_dev, Scratch *sc) {
    const cudaStream_t st = sc->st;
    auto grid = [](uint64_t n) { return (unsigned)((n + 127) / 128); };
    int rc;
    auto new_win = [&](uint64_t n, uint16_t **w) -> int {
        if ((rc = ts->pool.alloc((void **)w, n * 2))) return rc;
        ts->bytes += n * 2;
        return CP_OK;
    };
    const size_t nf = ts->row.size();
    std::vector<uint16_t *> win(nf);
    for (size_t i = 0; i < nf; ++i) {
        if ((rc = new_win(ts->row[i].n_src, &win[i]))) return rc;
        init_win_kernel<<<grid(ts->row[i].n_src), 128, 0, st>>>(ts->row[i].op.in, T_dev, win[i], i == 0 ? 1 : 0);
    }
    for (size_t i = 0; i < nf; ++i) {
        ts->row[i].win_in = win[i];
        ts->row[i].win_out = win[i + 1 < nf ? i + 1 : 0];
    }
    const uint16_t *w = win[0];
    for (auto &t : ts->last) {
        uint16_t *o = nullptr;
        if ((rc = new_win(t.n_dst, &o))) return rc;
        copy_blocks_kernel<<<grid(t.n_dst), 128, 0, st>>>(win[0], o, t.n_dst);
        t.win_in = w;
        t.win_out = o;
        w = o;
    }
    const int per_round = ts->potts ? ts->L / 2 + 2 : (ts->L + 1) / 2 + 1;
    int *flags = reinterpret_cast<int *>(sc->counts + kMaxTables);
    cudaError_t e = cudaMemsetAsync(flags, 0, kWinFlags * sizeof(int), st);
    auto relax = [&](const SiteTable &t, const int *prev, int *changed) {
        const bool many = t.n_dst <= kWinManyLanes;
        (many ? relax_win_kernel<8> : relax_win_kernel<1>)<<<grid(t.n_dst * (many ? 8 : 1)), 128, 0, st>>>(
            t.row_ptr, t.edges, t.n_dst, t.op.src_bits, t.win_in, const_cast<uint16_t *>(t.win_out), prev, changed);
    };
    int back[kMaxTables + kWinFlags] = {}, pass = 0;  // counts and flags
    const int *host = back + kMaxTables;
    bool done = false;
    while (e == cudaSuccess && !done && pass < kMaxPasses) {
        const int to = std::min(kMaxPasses, pass + per_round);
        for (; pass < to; ++pass)
            for (auto &t : ts->row) relax(t, pass ? flags + pass - 1 : nullptr, flags + pass);
        // (the row's part is complete when the last pass changed nothing; the rest is redone otherwise)
        for (auto &t : ts->last) relax(t, nullptr, flags + kMaxPasses + 1);
        if (pass > per_round) e = cudaMemsetAsync(flags + kMaxPasses, 0, sizeof(int), st);
        for (auto *chain : {&ts->row, &ts->last})
            for (auto &t : *chain) {
                const bool many = t.n_dst <= kWinManyLanes;
                (many ? check_win_kernel<8> : check_win_kernel<1>)<<<grid(t.n_dst * (many ? 8 : 1)), 128, 0, st>>>(
                    t.row_ptr, t.edges, t.n_dst, t.op.src_bits, t.sites, t.win_in, t.win_out, t.win_out == win[0] ? 1 : 0,
                    flags + kMaxPasses);
            }
        if (e == cudaSuccess) e = cudaGetLastError();
        if (e == cudaSuccess) e = cudaMemcpyAsync(back, sc->counts, sizeof(back), cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        done = host[pass - 1] == 0;
    }
    if (e != cudaSuccess) return fail(CP_ECUDA, std::string("degree windows: ") + cudaGetErrorString(e));
    if (!done || host[kMaxPasses]) return fail(CP_ESTATE, "degree windows of the state spaces are inconsistent");
    int k = 0;
    for (auto *chain : {&ts->row, &ts->last})
        for (auto &t : *chain) t.n_units = (uint32_t)back[k++];
    // the edges as the gathers read them replace the plain ones
    for (auto *chain : {&ts->row, &ts->last})
        for (auto &t : *chain) {
            if ((rc = ts->pool.alloc((void **)&t.wedges, t.nnz * sizeof(uint2)))) return rc;
            if (t.n_units)
                fill_wedges_kernel<<<(t.n_units + 7) / 8, 256, 0, st>>>(t.units, t.n_units, t.row_ptr, t.edges,
                                                                       t.op.src_bits, t.win_in, t.wedges);
            CP_CUDA_TRY(cudaGetLastError());
            if (t.nnz >= kBigTable) {
                CP_CUDA_TRY(cudaStreamSynchronize(st));
                dev_free(t.edges);
            }
            t.edges = nullptr;  // (the others go with the build's working memory)
        }
    CP_CUDA_TRY(cudaStreamSynchronize(st));
    sc->idle = true;
    return CP_OK;
}

__global__ void window_degrees_kernel(const uint16_t *win, uint64_t n, int v, int cap, unsigned long long *sum) {
    unsigned long long s = 0;
    for (uint64_t k = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (uint64_t)gridDim.x * blockDim.x) {
        const int lo = win[k] & 0xff, hi = min(cap, v - (win[k] >> 8));
        if (lo != 0xff && hi >= lo) s += hi - lo + 1;
    }
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) atomicAdd(sum, s);
}

int add_window_degrees(const uint16_t *win, uint64_t n, int v, int cap, unsigned long long *sum_dev, cudaStream_t st) {
    window_degrees_kernel<<<304, 256, 0, st>>>(win, n, v, cap, sum_dev);
    CP_CUDA_TRY(cudaGetLastError());
    return CP_OK;
}

// Identity factor on a 1-state space (T_1^last = D_1 on the width-1 strip).
static int identity_table(int m, Scratch *sc, DevPool *pool, SiteTable *tab) {
    OpDesc op{};
    op.kind = OP_IDENTITY;
    op.m = m;
    op.src_bits = (int)kSrcBits;
    op.in = Space{SPACE_B, m, 0, 0, 1, nullptr};
    op.out = op.in;
    tab->op = op;
    tab->n_src = tab->n_dst = tab->nnz = tab->n_site_out = 1;
    tab->max_coef_sum = tab->max_abs_coef = 1;
    int rc = pool->alloc((void **)&tab->row_ptr, 12);  // row_ptr and its edge
    if (rc) return rc;
    tab->edges = tab->row_ptr + 2;
    const uint32_t words[3] = {0, 1, 0u | (1u << (kSrcBits + 2))};
    CP_CUDA_TRY(cudaMemcpyAsync(tab->row_ptr, words, sizeof(words), cudaMemcpyHostToDevice, sc->st));
    if ((rc = sc->reset(4096))) return rc;
    return build_units(tab, sc, pool);
}

// Tables of a chain of per-site factors: one per factor, or (paired) one
// two-site table per consecutive pair, the second factor composed after the
// first on every term (an odd one out stays single).  Two chromatic factors
// compose to shifts of at most 3 and coefficients of magnitude at most 5
// (square) or 10 (triangular), so the edges keep a 2-bit shift and take 26 or
// 25 source bits; the build checks both bounds.
static int build_chain(const std::vector<OpDesc> &ops, int paired, int lattice, const RankTables *T_dev,
                       Scratch *sc, TableSet *ts, std::vector<SiteTable> *out) {
    int rc;
    for (size_t i = 0; i < ops.size();) {
        SiteTable tab;
        if (paired && i + 1 < ops.size()) {
            OpDesc f = ops[i];
            f.fused = 1;
            f.kind_b = ops[i + 1].kind;
            f.i_b = ops[i + 1].i;
            f.out = ops[i + 1].out;
            f.max_terms = ops[i].kind == OP_LAST ? 4 : (lattice == CP_SQUARE ? 16 : 24);
            f.src_bits = lattice == CP_SQUARE ? 26 : 25;
            rc = build_table(f, T_dev, sc, &ts->pool, &tab);
            tab.n_site_out = ops[i].out.size + ops[i + 1].out.size;
            tab.sites = 2;
            i += 2;
        } else {
            rc = build_table(ops[i], T_dev, sc, &ts->pool, &tab);
            i += 1;
        }
        if (rc) {
            out->push_back(tab);  // the set frees what there is of it
            return rc;
        }
        ts->bytes += (tab.n_dst + 1 + 2 * tab.nnz) * 4;
        out->push_back(tab);
    }
    return CP_OK;
}

static int build_tableset(int lattice, int L, int paired, cudaStream_t st, std::shared_ptr<TableSet> *out) {
    const RankTables *T_dev = nullptr;
    RankTables T;
    int rc = device_rank_tables(&T_dev, &T);
    if (rc) return rc;
    auto ts = std::make_shared<TableSet>();
    Scratch sc(st);
    cudaGetDevice(&ts->device);
    ts->lattice = lattice;
    ts->L = L;
    ts->paired = paired;
    const uint64_t Sb = T.cnt[L];
    const uint64_t Sx = L >= 2 ? T.cnt[L] + T.cnt[L - 1] : Sb;
    ts->S_b = Sb;
    ts->S_max = lattice == CP_SQUARE ? Sx : Sb;
    if (lattice == CP_SQUARE) {
        for (int e = 0; e + 1 < L; ++e) {
            uint32_t *pre = nullptr;
            if ((rc = build_x_prefix(L, e, &sc, &ts->pool, &pre))) return rc;
            ts->x_prefix.push_back(pre);
            ts->bytes += (Sb + 1) * 4;
        }
    }
    std::vector<OpDesc> row_ops, last_ops;
    for (int i = 0; i < L; ++i) {
        OpDesc op{};
        op.m = L;
        op.i = i;
        op.src_bits = (int)kSrcBits;
        if (lattice == CP_SQUARE) {
            op.kind = OP_SQUARE;
            op.max_terms = 4;
            op.in = i == 0 ? Space{SPACE_B, L, 0, 0, Sb, nullptr} : Space{SPACE_X, L, i - 1, 0, Sx, ts->x_prefix[i - 1]};
            op.out = i == L - 1 ? Space{SPACE_B, L, 0, 0, Sb, nullptr} : Space{SPACE_X, L, i, 0, Sx, ts->x_prefix[i]};
        } else {
            op.kind = OP_TRIANGULAR;
            op.max_terms = 8;
            op.in = Space{SPACE_B, L, 0, 0, Sb, nullptr};
            op.out = op.in;
        }
        row_ops.push_back(op);
    }
    for (int i = 0; i + 1 < L; ++i) {  // T_L^last = D_L is the identity on e_0
        OpDesc op{};
        op.kind = OP_LAST;
        op.m = L;
        op.i = i;
        op.src_bits = (int)kSrcBits;
        op.max_terms = 2;
        op.in = Space{SPACE_B, L, 0, 0, T.cnt[L - i], nullptr};
        op.out = Space{SPACE_B, L, 0, 0, T.cnt[L - i - 1], nullptr};
        last_ops.push_back(op);
    }
    if ((rc = build_chain(row_ops, paired, lattice, T_dev, &sc, ts.get(), &ts->row))) return rc;
    if (L == 1) {
        SiteTable tab;
        if ((rc = identity_table(1, &sc, &ts->pool, &tab))) return rc;
        ts->last.push_back(tab);
    } else if ((rc = build_chain(last_ops, paired, lattice, T_dev, &sc, ts.get(), &ts->last))) {
        return rc;
    }
    if ((rc = build_windows(ts.get(), T_dev, &sc))) return rc;
    *out = ts;
    return CP_OK;
}

// Any-v Potts tables on the non-crossing partitions (Catalan space), no projectors.
static int build_potts_tableset(int lattice, int L, int v, cudaStream_t st, std::shared_ptr<TableSet> *out) {
    const RankTables *T_dev = nullptr;
    RankTables T;
    int rc = device_rank_tables(&T_dev, &T);
    if (rc) return rc;
    auto ts = std::make_shared<TableSet>();
    Scratch sc(st);
    cudaGetDevice(&ts->device);
    ts->lattice = lattice;
    ts->L = L;
    ts->potts = 1;
    ts->v = v;
    const uint64_t S = T.cntc[L];
    ts->src_bits = potts_src_bits(S);
    ts->S_b = ts->S_max = S;
    for (int i = 0; i < L; ++i) {
        OpDesc op{};
        op.kind = lattice == CP_SQUARE ? OP_POTTS_SQUARE : OP_POTTS_TRIANGULAR;
        op.m = L;
        op.i = i;
        op.v = v;
        op.src_bits = ts->src_bits;
        op.max_terms = lattice == CP_SQUARE ? 4 : 8;
        op.in = Space{SPACE_C, L, 0, 0, S, nullptr};
        op.out = op.in;
        SiteTable tab;
        rc = build_table(op, T_dev, &sc, &ts->pool, &tab);
        ts->bytes += (tab.n_dst + 1 + 2 * tab.nnz) * 4;
        ts->row.push_back(tab);
        if (rc) return rc;
    }
    if (L == 1) {
        SiteTable tab;
        if ((rc = identity_table(1, &sc, &ts->pool, &tab))) return rc;
        ts->last.push_back(tab);
    } else {
        for (int i = 0; i + 1 < L; ++i) {  // D_L is the identity on e_0
            OpDesc op{};
            op.kind = OP_POTTS_LAST;
            op.m = L;
            op.i = i;
            op.v = v;
            op.src_bits = ts->src_bits;
            op.max_terms = 2;
            op.in = Space{SPACE_C, L, 0, 0, T.cntc[L - i], nullptr};
            op.out = Space{SPACE_C, L, 0, 0, T.cntc[L - i - 1], nullptr};
            SiteTable tab;
            rc = build_table(op, T_dev, &sc, &ts->pool, &tab);
            ts->bytes += (tab.n_dst + 1 + 2 * tab.nnz) * 4;
            ts->last.push_back(tab);
            if (rc) return rc;
        }
    }
    if ((rc = build_windows(ts.get(), T_dev, &sc))) return rc;
    *out = ts;
    return CP_OK;
}

static std::mutex g_cache_mu;
static std::map<std::tuple<int, int, int>, std::shared_ptr<TableSet>> g_cache[64];  // per device
static int g_pairing = 1;  // 0 never, 1 rows of >= kPairRowBytes, 2 every square table, 3 every table

int factor_pairing() {
    std::lock_guard<std::mutex> lk(g_cache_mu);
    return g_pairing;
}

int set_factor_pairing(int mode) {
    std::lock_guard<std::mutex> lk(g_cache_mu);
    const int old = g_pairing;
    g_pairing = mode < 0 ? 0 : (mode > 3 ? 3 : mode);
    return old;
}
static std::map<std::tuple<int, int, int>, std::shared_ptr<TableSet>> g_potts_cache[64];

int get_tables(int lattice, int L, size_t row_bytes, cudaStream_t st, std::shared_ptr<TableSet> *out) {
    int dev = 0;
    CP_CUDA_TRY(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) return fail(CP_EINVAL, "device index");
    std::lock_guard<std::mutex> lk(g_cache_mu);
    // Two-site tables halve the launches, the vector traffic and the rows to begin and
    // reduce, with as many edges in all.  Per row, one table per factor and two-site:
    // square width 16 D 63 on 16 primes 4.81 and 3.96 ms, width 14 on 4 primes 0.467 and
    // 0.327 ms, width 8 D 71 on 8 primes 62 and 35 us; triangular width 16 D 32 on 16
    // primes 1.42 and 1.36 ms, width 13 D 181 on 4 primes 0.274 and 0.247 ms, width 9
    // D 80 on 8 primes 77 and 45 us; and half the tables to build: a first square 11 x 10
    // solve with D 30 on 4 primes (496-byte rows) 5.5 and 3.9 ms.  Four or eight rows and the
    // read-out, time with one table per factor over time with two-site tables:
    //   row bytes            176        352        496        1312       2624
    //   width 4 to 8       1.1-1.7    1.2-1.7    1.2-1.7    1.3-1.7    1.5-1.6
    //   width 10 square      1.06       1.10       1.10       1.21       1.38
    //   width 12 square      0.94       0.93       0.98       1.05       1.11
    //   width 12 triangular  1.03       1.00       1.09       1.18       1.23
    //   width 14, 15       1.4-2.1    1.3-1.5    1.25-1.4   1.2-1.3    1.2-1.3
    //   width 16 square      0.97       1.30       1.27       1.28       1.27
    //   width 16 triangular  1.00       1.24       1.18       1.18       1.18
    //   width 17, 18       0.8-0.9    0.9-1.0    1.04-1.1   1.07-1.15  1.08-1.15
    // so at 352 bytes the widest strips break even.  Wide square strips wait for rows of 1536
    // bytes: with units of 32 edges shorter rows lost there (width 17 D 40 on 5 primes, four
    // rows and the read-out, 6.76 and 7.08 ms); with units of 64 they gain (8 primes 5.95 and
    // 5.19 ms), but two-site tables take longer to build (width 17 44 and 56 ms, width 19
    // 277 and 433), which takes some sixty such rows to pay back.
    const bool wide_short = lattice == CP_SQUARE && L >= kPairWide && row_bytes < kPairWideRowBytes;
    const int paired = g_pairing == 3 || (lattice == CP_SQUARE && g_pairing == 2) ||
                       (g_pairing == 1 && row_bytes >= kPairRowBytes && !wide_short);
    auto key = std::make_tuple(lattice, L, paired);
    auto it = g_cache[dev].find(key);
    if (it != g_cache[dev].end()) {
        *out = it->second;
        return CP_OK;
    }
    std::shared_ptr<TableSet> ts;
    int rc = build_tableset(lattice, L, paired, st, &ts);
    if (rc) return rc;
    g_cache[dev][key] = ts;
    *out = ts;
    return CP_OK;
}

int get_potts_tables(int lattice, int L, int v, cudaStream_t st, std::shared_ptr<TableSet> *out) {
    int dev = 0;
    CP_CUDA_TRY(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) return fail(CP_EINVAL, "device index");
    std::lock_guard<std::mutex> lk(g_cache_mu);
    auto key = std::make_tuple(lattice, L, v);
    auto it = g_potts_cache[dev].find(key);
    if (it != g_potts_cache[dev].end()) {
        *out = it->second;
        return CP_OK;
    }
    std::shared_ptr<TableSet> ts;
    int rc = build_potts_tableset(lattice, L, v, st, &ts);
    if (rc) return rc;
    g_potts_cache[dev][key] = ts;
    *out = ts;
    return CP_OK;
}

// Copy one cached (or freshly built) chromatic table to the host.
int debug_table(int lattice, int L, int paired, int which, int index, uint32_t *row_ptr_host, uint64_t max_rows,
                uint32_t *edges_host, uint64_t max_edges, uint64_t info[4]) {
    const int old = set_factor_pairing(paired ? 3 : 0);
    std::shared_ptr<TableSet> ts;
    int rc = get_tables(lattice, L, 0, 0, &ts);
    set_factor_pairing(old);
    if (rc) return rc;
    const std::vector<SiteTable> &v = which ? ts->last : ts->row;
    if (index < 0 || index >= (int)v.size()) return fail(CP_EINVAL, "table index out of range");
    const SiteTable &t = v[index];
    if (info) {
        info[0] = t.n_src;
        info[1] = t.n_dst;
        info[2] = t.nnz;
        info[3] = (uint64_t)t.op.src_bits;
    }
    if (row_ptr_host) {
        if (max_rows < t.n_dst + 1) return fail(CP_EINVAL, "max_rows < n_dst + 1");
        CP_CUDA_TRY(cudaMemcpy(row_ptr_host, t.row_ptr, 4 * (t.n_dst + 1), cudaMemcpyDeviceToHost));
    }
    if (edges_host) {
        if (max_edges < t.nnz) return fail(CP_EINVAL, "max_edges < nnz");
        CP_CUDA_TRY(cudaMemcpy2D(edges_host, 4, t.wedges, sizeof(uint2), 4, t.nnz, cudaMemcpyDeviceToHost));
    }
    return CP_OK;
}

void clear_table_cache() {
    std::lock_guard<std::mutex> lk(g_cache_mu);
    for (auto &c : g_cache) c.clear();  // strips keep their own shared_ptr alive
    for (auto &c : g_potts_cache) c.clear();
}

static std::mutex g_rt_mu;
static RankTables *g_rt_dev[64];
static RankTables g_rt_host[64];

int device_rank_tables(const RankTables **out_dev, RankTables *host_copy) {
    int dev = 0;
    CP_CUDA_TRY(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) return fail(CP_EINVAL, "device index");
    std::lock_guard<std::mutex> lk(g_rt_mu);
    if (!g_rt_dev[dev]) {
        RankTables *p = nullptr;
        int rc = dev_alloc((void **)&p, sizeof(RankTables));
        if (rc) return rc;
        rank_tables_kernel<<<1, 32>>>(p);
        CP_CUDA_TRY(cudaGetLastError());
        CP_CUDA_TRY(cudaMemcpy(&g_rt_host[dev], p, sizeof(RankTables), cudaMemcpyDeviceToHost));
        g_rt_dev[dev] = p;
    }
    *out_dev = g_rt_dev[dev];
    if (host_copy) *host_copy = g_rt_host[dev];
    return CP_OK;
}

// ------------------------------------------------------------------ debug: rank/unrank sweep

__global__ void check_space_kernel(Space sp, const RankTables *Tg, unsigned long long *bad) {
    __shared__ RankTables T;
    stage_tables(T, Tg);
    uint64_t r = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= sp.size) return;
    Labels s;
    space_unrank(r, sp, s, T);
    Labels c = s;
    canonicalise(c, sp.m);
    bool ok = space_contains(s, sp) && space_rank(s, sp, T) == r;
    for (int i = 0; i < sp.m; ++i) ok = ok && c.v[i] == s.v[i];
    if (!ok) atomicAdd(bad, 1ull);
}

int check_space(int kind, int m, int e, uint64_t *n_bad, uint64_t *size) {
    const RankTables *T_dev = nullptr;
    RankTables T;
    int rc = device_rank_tables(&T_dev, &T);
    if (rc) return rc;
    Space sp{kind, m, e, 0, kind == SPACE_X ? T.cnt[m] + T.cnt[m - 1] : (kind == SPACE_C ? T.cntc[m] : T.cnt[m]),
             nullptr};
    uint32_t *pre = nullptr;
    DevPool pool;
    Scratch sc(nullptr);
    if (kind == SPACE_X && (rc = build_x_prefix(m, e, &sc, &pool, &pre))) return rc;
    sp.prefix = pre;
    unsigned long long *bad = nullptr;
    if ((rc = pool.alloc((void **)&bad, 8))) return rc;
    CP_CUDA_TRY(cudaMemset(bad, 0, 8));
    check_space_kernel<<<(unsigned)((sp.size + 127) / 128), 128>>>(sp, T_dev, bad);
    CP_CUDA_TRY(cudaGetLastError());
    unsigned long long h = 0;
    CP_CUDA_TRY(cudaMemcpy(&h, bad, 8, cudaMemcpyDeviceToHost));
    *n_bad = h;
    *size = sp.size;
    return CP_OK;
}

// Copy the ranked partitions of a space to the host (labels, m bytes each).
__global__ void enumerate_kernel(Space sp, const RankTables *Tg, uint8_t *out) {
    __shared__ RankTables T;
    stage_tables(T, Tg);
    uint64_t r = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= sp.size) return;
    Labels s;
    space_unrank(r, sp, s, T);
    for (int i = 0; i < sp.m; ++i) out[r * sp.m + i] = s.v[i];
}

int enumerate_space(int kind, int m, int e, uint8_t *out_host, uint64_t max_states, uint64_t *size) {
    const RankTables *T_dev = nullptr;
    RankTables T;
    int rc = device_rank_tables(&T_dev, &T);
    if (rc) return rc;
    Space sp{kind, m, e, 0, kind == SPACE_X ? T.cnt[m] + T.cnt[m - 1] : (kind == SPACE_C ? T.cntc[m] : T.cnt[m]),
             nullptr};
    *size = sp.size;
    if (sp.size > max_states) return fail(CP_EINVAL, "output buffer too small");
    uint32_t *pre = nullptr;
    DevPool pool;
    Scratch sc(nullptr);
    if (kind == SPACE_X && (rc = build_x_prefix(m, e, &sc, &pool, &pre))) return rc;
    sp.prefix = pre;
    uint8_t *d = nullptr;
    if ((rc = pool.alloc((void **)&d, sp.size * m))) return rc;
    enumerate_kernel<<<(unsigned)((sp.size + 127) / 128), 128>>>(sp, T_dev, d);
    CP_CUDA_TRY(cudaGetLastError());
    CP_CUDA_TRY(cudaMemcpy(out_host, d, sp.size * m, cudaMemcpyDeviceToHost));
    return CP_OK;
}

}  // namespace cp
