// Device code for the connectivity states of the top row (Sec. 3.1-3.4):
// label arrays, the single-edge operators, and the rank/unrank bijection of
// the NCNNN partitions and of the square lattice's excepted spaces.
#pragma once

#include <stdint.h>

#include "cp_internal.h"

namespace cp {

constexpr int kMaxL = CP_MAX_L;
// A partition of the sites 0..m-1: block labels in first-occurrence order.  Also as
// words of four labels: the arrays live in local memory, where a byte at a time was a
// chain of dependent accesses per operator (relabelling through a 32-entry map, about a
// thousand cycles), so the operators below treat four labels at once and keep the
// order of first occurrence without a map.  Bytes past the m-th mean nothing.
struct Labels {
    union {
        uint8_t v[kMaxL];
        uint32_t w[kMaxL / 4];
    };
};
static_assert(kMaxL % 4 == 0 && kMaxL <= 32, "whole words; a bit per site or label");

// Labels in first-occurrence order, from any (validation).
__device__ __forceinline__ void canonicalise(Labels &s, int m) {
    uint8_t map[32];
#pragma unroll
    for (int k = 0; k < 32; ++k) map[k] = 0xFF;
    uint8_t next = 0;
    for (int i = 0; i < m; ++i) {
        uint8_t x = s.v[i];
        if (map[x] == 0xFF) map[x] = next++;
        s.v[i] = map[x];
    }
}

// Number of blocks among the sites before i.
__device__ __forceinline__ uint32_t blocks_before(const Labels &s, int i) {
    uint32_t x = 0;  // largest label, byte by byte
    for (int k = 0; k < i >> 2; ++k) x = __vmaxu4(x, s.w[k]);
    if (i & 3) x = __vmaxu4(x, s.w[i >> 2] & ((1u << 8 * (i & 3)) - 1u));
    x = __vmaxu4(x, x >> 16);
    return i ? (max(x & 0xffu, (x >> 8) & 0xffu)) + 1 : 0;
}

// The smallest site t in (a, b) of site a's block, or -1.
__device__ __forceinline__ int next_in_block(const Labels &s, int a, int b) {
    if (a + 1 >= b) return -1;
    const uint32_t x = s.v[a] * 0x01010101u;
    int k = (a + 1) >> 2;
    uint32_t eq = __vcmpeq4(s.w[k], x) & (~0u << 8 * ((a + 1) & 3));
    while (eq == 0) {
        if (4 * ++k >= b) return -1;
        eq = __vcmpeq4(s.w[k], x);
    }
    const int t = 4 * k + (__ffs((int)eq) - 1) / 8;
    return t < b ? t : -1;
}

// J_{a,b} for a !~ b: merge the two blocks (the factor w is the caller's shift).  The
// later label goes, and the ones above it move down by one.
__device__ __forceinline__ void join_blocks(Labels &s, int m, int a, int b) {
    const uint32_t la = min(s.v[a], s.v[b]) * 0x01010101u, lb = max(s.v[a], s.v[b]) * 0x01010101u;
    for (int k = 0; 4 * k < m; ++k) {
        const uint32_t x = s.w[k], eq = __vcmpeq4(x, lb);
        s.w[k] = (eq & la) | (~eq & __vadd4(x, __vcmpgtu4(x, lb)));
    }
}

// D_i: site i becomes a singleton.  If its block x began before i, the singleton takes
// the first label not seen before i; if it begins at i, the singleton keeps x and the rest
// of the block takes the first label not seen before its next site.  The labels from
// there on move up by one.
__device__ __forceinline__ void detach_site(Labels &s, int m, int i) {
    const uint32_t x = s.v[i], c = blocks_before(s, i);
    uint32_t from = c;
    if (x == c) {
        const int f = next_in_block(s, i, m);
        if (f < 0) return;
        from = blocks_before(s, f);
    }
    const uint32_t x4 = x * 0x01010101u, from4 = from * 0x01010101u;
    for (int k = i >> 2; 4 * k < m; ++k) {
        const uint32_t y = s.w[k], eq = x == c ? __vcmpeq4(y, x4) : 0u;
        s.w[k] = (eq & from4) | (~eq & __vsub4(y, __vcmpgeu4(y, from4)));
    }
    s.v[i] = (uint8_t)c;
}

// Non-crossing test in O(m): the blocks that may go on are open, a bit each; a block
// that reappears must be one of them and closes the later ones (labels grow in the
// order of first occurrence).
__device__ __forceinline__ bool is_noncrossing(const Labels &s, int m) {
    uint32_t open = 0, next = 0;
    bool ok = true;
    for (int i = 0; i < m; ++i) {
        const uint32_t x = s.v[i];
        if (x == next) {
            open |= 1u << next++;
        } else {
            ok = ok && x < next && (open >> x & 1u);
            open &= (2u << (x & 31u)) - 1u;
        }
    }
    return ok;
}

// Bit j: the sites j and j + 1 are in one block.
__device__ __forceinline__ uint32_t adjacent_pairs(const Labels &s, int m) {
    uint32_t bits = 0;
    for (int k = 0; 4 * k < m - 1; ++k) {
        const uint32_t x = s.w[k], y = k + 1 < kMaxL / 4 ? s.w[k + 1] : 0u;
        const uint32_t eq = __vcmpeq4(x, __funnelshift_r(x, y, 8)) & 0x01010101u;
        bits |= (eq * 0x01020408u >> 24 & 15u) << 4 * k;
    }
    return bits & ((1u << (m - 1)) - 1u);
}

// Neighbour rule: no (j, j+1) in one block, except the pair j == skip.
__device__ __forceinline__ bool nn_ok(const Labels &s, int m, int skip) {
    return (adjacent_pairs(s, m) & ~(skip >= 0 ? 1u << skip : 0u)) == 0;
}

// The parts of a partition that a ranking (unranking) puts off are disjoint, with a point
// of a block before each, so kMaxL / 2 entries hold those of an NCNNN partition, whose
// parts have a point at least; ranks are below 2^32 (M_19, Catalan(16)).

// Rank of an NCNNN partition of the points lo..hi-1 in the paper's order
// (Sec. 3.4): a point alone first (rank of the rest), then by the smallest
// partner lo+2+k of point lo, inner points as the most significant digit and
// the right part (from the partner on) as the least significant one.
// Returns ~0ull if the partition violates the neighbour rule at the first point.
__device__ __forceinline__ uint64_t ncnnn_rank(const Labels &s, int lo, int hi, const RankTables &T) {
    uint8_t sa[kMaxL / 2], sb[kMaxL / 2];
    uint32_t smul[kMaxL / 2];
    int sp = 0;
    uint64_t r = 0;
    int a = lo, b = hi;
    uint64_t mu = 1;
    for (;;) {
        while (b - a > 2) {
            int n = b - a;
            if (s.v[a + 1] == s.v[a]) return ~0ull;
            const int j = next_in_block(s, a, b);
            if (j < 0) { ++a; continue; }
            int k = j - a - 2;
            uint64_t cr = T.cnt[b - j];
            r += mu * T.off[n * kTblStride + k];
            sa[sp] = (uint8_t)(a + 1); sb[sp] = (uint8_t)j; smul[sp] = (uint32_t)(mu * cr); ++sp;   // inner part, later
            a = j;                                                   // right part, now
        }
        if (b - a == 2 && s.v[a] == s.v[a + 1]) return ~0ull;
        if (sp == 0) break;
        --sp;
        a = sa[sp]; b = sb[sp]; mu = smul[sp];
    }
    return r;
}

// Inverse of ncnnn_rank on points lo..hi-1; labels are assigned in
// first-occurrence order, so the result is canonical when lo == 0.
__device__ __forceinline__ void ncnnn_unrank(uint64_t r, int lo, int hi, Labels &s, const RankTables &T) {
#pragma unroll
    for (int k = 0; k < kMaxL / 4; ++k) s.w[k] = ~0u;
    uint8_t next = 0;
    uint8_t sa[kMaxL / 2], sb[kMaxL / 2];
    uint32_t sr[kMaxL / 2];
    int sp = 0;
    int a = lo, b = hi;
    for (;;) {
        while (b - a >= 1) {
            if (s.v[a] == 0xFF) s.v[a] = next++;
            int n = b - a;
            if (n <= 2) {
                if (n == 2) s.v[a + 1] = next++;
                break;
            }
            if (r < T.cnt[n - 1]) { ++a; continue; }   // point a alone
            int k = 0;
            while (k + 1 <= n - 3 && T.off[n * kTblStride + k + 1] <= r) ++k;
            r -= T.off[n * kTblStride + k];
            uint64_t cr = T.cnt[n - k - 2];
            uint64_t inner = r / cr, right = r - inner * cr;
            int j = a + 2 + k;
            s.v[j] = s.v[a];
            sa[sp] = (uint8_t)j; sb[sp] = (uint8_t)b; sr[sp] = (uint32_t)right; ++sp;   // right part after the inner one
            a = a + 1; b = j; r = inner;
        }
        if (sp == 0) break;
        --sp;
        a = sa[sp]; b = sb[sp]; r = sr[sp];
    }
}

// Rank of a non-crossing partition of points lo..hi-1: the first point alone
// first (rank of the rest), then by its smallest partner lo+1+k, inner points
// as the most significant digit and the right part (from the partner on) as
// the least significant one.  The count recursion is Catalan's.
__device__ __forceinline__ uint64_t nc_rank(const Labels &s, int lo, int hi, const RankTables &T) {
    uint8_t sa[kMaxL + 1], sb[kMaxL + 1];
    uint32_t smul[kMaxL + 1];
    int sp = 0;
    uint64_t r = 0;
    int a = lo, b = hi;
    uint64_t mu = 1;
    for (;;) {
        while (b - a > 1) {
            const int n = b - a, j = next_in_block(s, a, b);
            if (j < 0) { ++a; continue; }
            int k = j - a - 1;
            r += mu * T.offc[n * kTblStride + k];
            sa[sp] = (uint8_t)(a + 1); sb[sp] = (uint8_t)j; smul[sp] = (uint32_t)(mu * T.cntc[b - j]); ++sp;  // inner part, later
            a = j;                                                              // right part, now
        }
        if (sp == 0) break;
        --sp;
        a = sa[sp]; b = sb[sp]; mu = smul[sp];
    }
    return r;
}

__device__ __forceinline__ void nc_unrank(uint64_t r, int lo, int hi, Labels &s, const RankTables &T) {
#pragma unroll
    for (int k = 0; k < kMaxL / 4; ++k) s.w[k] = ~0u;
    uint8_t next = 0;
    uint8_t sa[kMaxL + 1], sb[kMaxL + 1];
    uint32_t sr[kMaxL + 1];
    int sp = 0;
    int a = lo, b = hi;
    for (;;) {
        while (b - a >= 1) {
            if (s.v[a] == 0xFF) s.v[a] = next++;
            int n = b - a;
            if (n == 1) break;
            if (r < T.cntc[n - 1]) { ++a; continue; }  // point a alone
            int k = 0;
            while (k + 1 <= n - 2 && T.offc[n * kTblStride + k + 1] <= r) ++k;
            r -= T.offc[n * kTblStride + k];
            uint64_t cr = T.cntc[n - 1 - k];
            uint64_t inner = r / cr, right = r - inner * cr;
            int j = a + 1 + k;
            s.v[j] = s.v[a];
            sa[sp] = (uint8_t)j; sb[sp] = (uint8_t)b; sr[sp] = (uint32_t)right; ++sp;  // right part after the inner one
            a = a + 1; b = j; r = inner;
        }
        if (sp == 0) break;
        --sp;
        a = sa[sp]; b = sb[sp]; r = sr[sp];
    }
}

// Rank in a space (SPACE_B: the paper's order; SPACE_X: the interleaved order,
// see Space).  Returns ~0ull for a partition outside the space's rule.
__device__ __forceinline__ uint64_t space_rank(const Labels &s, const Space &sp, const RankTables &T) {
    const int m = sp.m;
    if (sp.kind == SPACE_X) {
        const int e = sp.e;
        if (s.v[e] == s.v[e + 1]) {
            Labels t = s;
            detach_site(t, m, e);
            uint64_t b = ncnnn_rank(t, 0, m, T);
            return b == ~0ull ? b : b + sp.prefix[b] + 1;
        }
        uint64_t b = ncnnn_rank(s, 0, m, T);
        return b == ~0ull ? b : b + sp.prefix[b];
    }
    if (sp.kind == SPACE_C) return nc_rank(s, 0, m, T);
    return ncnnn_rank(s, 0, m, T);
}

__device__ __forceinline__ void space_unrank(uint64_t r, const Space &sp, Labels &s, const RankTables &T) {
    const int m = sp.m;
    if (sp.kind == SPACE_X) {
        // largest b with b + prefix[b] <= r (strictly increasing in b)
        uint64_t lo = 0, hi = T.cnt[m] - 1;
        while (lo < hi) {
            uint64_t mid = (lo + hi + 1) >> 1;
            if (mid + sp.prefix[mid] <= r) lo = mid; else hi = mid - 1;
        }
        ncnnn_unrank(lo, 0, m, s, T);
        if (r != lo + sp.prefix[lo]) join_blocks(s, m, sp.e, sp.e + 1);
        return;
    }
    if (sp.kind == SPACE_C) {
        nc_unrank(r, 0, m, s, T);
        return;
    }
    ncnnn_unrank(r, 0, m, s, T);
}

// Membership test of a canonical partition in a space (debug/validation).
__device__ __forceinline__ bool space_contains(const Labels &s, const Space &sp) {
    if (sp.kind == SPACE_C) return is_noncrossing(s, sp.m);
    return is_noncrossing(s, sp.m) && nn_ok(s, sp.m, sp.kind == SPACE_X ? sp.e : -1);
}

// Stage the rank tables into shared memory (all threads of the block call).
__device__ __forceinline__ void stage_tables(RankTables &dst, const RankTables *src) {
    const uint64_t *a = reinterpret_cast<const uint64_t *>(src);
    uint64_t *b = reinterpret_cast<uint64_t *>(&dst);
    for (int k = threadIdx.x; k < (int)(sizeof(RankTables) / 8); k += blockDim.x) b[k] = a[k];
    __syncthreads();
}

}  // namespace cp
