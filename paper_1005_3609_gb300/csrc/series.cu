// Finite-lattice combination of the rectangles into the bulk, surface and
// corner series, modulo each prime (Sec. 4.1-4.3).
//
// f_x = sum_{(r,s) in B(k)} weight_x(r,s) log P~_{r,s}, eqs. (fb)-(fc), with
// P~ written in z (w = z/(1+z), eq. (def_z)) on the square lattice and in x
// (w = -x/(1-x)^2, q = 2 - x - 1/x) on the triangular one.  Each P~ has
// constant term 1, so log and exp are power series with denominators up to
// n < p: everything is exact modulo p.  Output per prime:
//   series 0: square sum alpha_k z^k = (1+z)^2 exp(f_b - log q)   (Table 1)
//             triangular (1-x)^2 exp(f_b - log q)   (= Baxter's product, eq. (efb))
//   series 1: exp(f_s);  series 2: exp(f_c).
// For the square lattice at odd k the extra term mu_{2m} z^{4m-1}, m = (k-1)/2,
// is added to f_b and -m mu_{2m} z^{4m-1} to f_s (Sec. 4.2), which extends the
// bulk and surface series by one term.
#include <cuda_runtime.h>

#include "cp_internal.h"
#include "modarith.cuh"
#include "series.h"

namespace cp {

// Finite-lattice weights (Sec. 4.1); beta with (r+s+2)/2 on delta_{r+s,k-3}
// (the printed (r+s-2)/2 violates the sum rules), all integers.
__device__ long long flm_weight(int which, int k, int r, int s) {
    const int t = r + s;
    const long long f = (r == s) ? 1 : 2;
    if (which == 0) {
        int c = t == k ? 1 : t == k - 1 ? -3 : t == k - 2 ? 3 : t == k - 3 ? -1 : 0;
        return f * c;
    }
    if (which == 1) {  // (2 - delta) * num / 2, num even whenever r == s
        long long num = t == k ? (2 - t) : t == k - 1 ? (3 * t - 2) : t == k - 2 ? -(3 * t + 2) : t == k - 3 ? (t + 2) : 0;
        return f * num / 2;
    }
    long long rs = (long long)r * s;
    long long c = t == k ? (long long)(r - 1) * (s - 1) : t == k - 1 ? (1 + t - 3 * rs)
                : t == k - 2 ? (3 * rs + t - 1) : t == k - 3 ? -(long long)(r + 1) * (s + 1) : 0;
    return f * c;
}

// The value of `v` (one of M registers a lane, entry i in lane i % 32, register i / 32) at index i.
template <int M>
__device__ __forceinline__ uint32_t lane_value(const uint32_t (&v)[M], int i) {
    uint32_t x = 0;
#pragma unroll
    for (int m = 0; m < M; ++m) {
        const uint32_t y = __shfl_sync(0xffffffffu, v[m], i & 31);
        x = (i >> 5) == m ? y : x;
    }
    return x;
}

constexpr int kSeriesWarps = 8;           // rectangles per block
constexpr int kSeriesRegs = kMaxSeries / 32;

// mu_{2m} mod p from sum_{p>=4} mu_p y^p = y^4 (2-2y-y sqrt(1-4y)) / ((1-4y)(2+y))
//                                        + y^6 (3-4y-4 sqrt(1-4y)) / (1-4y)^2      (y = x^2)
// by one warp; tmp: six rows of kMaxSeries words.
__device__ uint32_t mu_mod(int idx, const Mod &M, const uint32_t *inv, uint32_t (*tmp)[kMaxSeries], int lane) {
    const uint32_t p = M.p;
    const int n = idx + 1;
    uint32_t *sq = tmp[0], *g1 = tmp[1], *q1 = tmp[2], *a = tmp[3], *b = tmp[4], *t = tmp[5];
    // sqrt(1-4y) = 1 - 2 sum_{j>=1} C_{j-1} y^j, Catalan C_j = C_{j-1} 2(2j-1)/(j+1)
    const uint32_t inv2 = (p + 1) / 2;
    uint32_t cat = 1, pow4 = 1, half = inv2;
    for (int j = 0; j < n; ++j) {
        if (lane == 0) {
            sq[j] = j ? sb(0, mm(2, cat, M), p) : 1;
            g1[j] = pow4;                             // 1/(1-4y)
            q1[j] = j & 1 ? sb(0, half, p) : half;    // 1/(2+y)
        }
        if (j) cat = mm(mm(cat, from_int(2 * (2 * j - 1), p), M), inv[j + 1], M);
        pow4 = mm(pow4, 4, M);
        half = mm(half, inv2, M);
    }
    __syncwarp();
    for (int j = lane; j < n; j += 32) {  // numerators
        uint32_t x = j == 0 ? 2 : 0, y = j == 0 ? 3 : 0;
        if (j == 1) x = sb(x, 2, p);
        if (j >= 1) x = sb(x, sq[j - 1], p);
        if (j == 1) y = sb(y, 4, p);
        a[j] = x;
        b[j] = sb(y, mm(4, sq[j], M), p);
    }
    __syncwarp();
    // idx-th coefficients: y^4 (a g1) q1 and y^6 b (g1 g1)
    for (int j = lane; j < n; j += 32) {
        uint32_t x = 0;
        for (int i = 0; i <= j; ++i) x = ad(x, mm(a[i], g1[j - i], M), p);
        t[j] = x;
    }
    __syncwarp();
    uint32_t u = 0;
    for (int i = lane; i <= idx - 4; i += 32) u = ad(u, mm(t[i], q1[idx - 4 - i], M), p);
    __syncwarp();
    for (int j = lane; j < n; j += 32) {
        uint32_t y = 0;
        for (int i = 0; i <= j; ++i) y = ad(y, mm(g1[i], g1[j - i], M), p);
        t[j] = y;
    }
    __syncwarp();
    for (int i = lane; i <= idx - 6; i += 32) u = ad(u, mm(b[i], t[idx - 6 - i], M), p);
    for (int o = 16; o > 0; o >>= 1) u = ad(u, __shfl_xor_sync(0xffffffffu, u, o), p);
    return u;
}

// One block per prime and kSeriesWarps rectangles, one warp per rectangle for its
// substitution and logarithm; the block that finishes a prime's last rectangle
// combines the prime's logarithms and takes the exponentials, one warp per series.
// What bounds it: chains of dependent modular products.  Every recurrence is run
// outward -- an entry that is final is sent to all lanes, which add its products to
// the entries still open -- so a step costs one exchange and one product instead of
// a sum over the entries before it: k = 17 on 8 primes 178 -> 39 us (one thread per
// rectangle and one block per prime before), k = 33 on 16 primes 73 us.
__global__ void __launch_bounds__(32 * kSeriesWarps)
    flm_series_kernel(uint32_t *__restrict__ ptilde, const int2 *__restrict__ rects, const uint32_t *__restrict__ primes,
                      SeriesParams sp, uint32_t *__restrict__ logs, uint32_t *__restrict__ finished,
                      uint32_t *__restrict__ out, int *err) {
    extern __shared__ uint32_t B[];  // [n][n + 1]: coefficient of t^i in w(t)^d
    __shared__ uint32_t inv[kMaxSeries];
    __shared__ uint32_t work[kSeriesWarps][kMaxSeries];
    __shared__ uint32_t tmp[6][kMaxSeries];
    __shared__ uint32_t wgt[3][kMaxSeriesRects];
    __shared__ uint32_t last;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int pi = blockIdx.y, grp = pi / sp.Pg, pk = pi - grp * sp.Pg;
    const uint32_t p = primes[grp * kPrimeWords + pk];
    const Mod M = make_mod(p);
    const int n = sp.n, ld = n + 1;
    for (int i = tid; i < n; i += blockDim.x) inv[i] = i ? pw((uint32_t)i, p - 2, M) : 0u;
    // w = z/(1+z): (1+z) w^d = z w^(d-1);  w = -x/(1-x)^2: (1-x)^2 w^d = -x w^(d-1)
    for (int i = 0; i < n; ++i) {
        if (tid < n) {
            const int d = tid;
            const uint32_t up = i >= 1 ? B[(i - 1) * ld + d] : 0u, left = i >= 1 && d >= 1 ? B[(i - 1) * ld + d - 1] : 0u;
            uint32_t x = i == 0 && d == 0 ? 1u : 0u;
            if (d >= 1 && i >= 1) {
                if (sp.lattice == CP_SQUARE) x = sb(left, up, p);
                else x = sb(sb(ad(up, up, p), i >= 2 ? B[(i - 2) * ld + d] : 0u, p), left, p);
            }
            B[i * ld + d] = x;
        }
        __syncthreads();
    }
    const int j = blockIdx.x * kSeriesWarps + warp;
    uint32_t *mine = work[warp];
    if (j < sp.n_rects) {
        uint32_t *src = ptilde + ((size_t)grp * sp.n_rects + j) * sp.D1 * sp.Pp + pk;
        for (int d = lane; d < n; d += 32) {
            uint32_t c = 0;
            if (d < sp.D1) {
                c = src[(size_t)d * sp.Pp];  // a signed representative: its residue stays in its place
                c = (int)c < 0 ? c + p : c;
                src[(size_t)d * sp.Pp] = c;
            }
            mine[d] = c;
        }
        __syncwarp();
        uint32_t f[kSeriesRegs], s[kSeriesRegs];
#pragma unroll
        for (int m = 0; m < kSeriesRegs; ++m) {
            const int i = lane + 32 * m;
            uint32_t x = 0;
            if (i < n)
                for (int d = 0; d <= i; ++d) x = ad(x, mm(mine[d], B[i * ld + d], M), p);
            f[m] = x;
        }
        __syncwarp();
#pragma unroll
        for (int m = 0; m < kSeriesRegs; ++m)
            if (lane + 32 * m < n) mine[lane + 32 * m] = f[m];
        __syncwarp();
        if (lane == 0 && f[0] != 1) atomicOr_system(err, 1);
        // log f: h = f'/f with h_i = (i+1) f_{i+1} - sum_{q=1..i} f_q h_{i-q}; g_i = h_{i-1}/i
#pragma unroll
        for (int m = 0; m < kSeriesRegs; ++m) {
            const int i = lane + 32 * m;
            s[m] = i + 1 < n ? mm(mine[i + 1], (uint32_t)(i + 1), M) : 0u;
        }
        for (int q = 0; q + 2 < n; ++q) {
            const uint32_t h = lane_value(s, q);
#pragma unroll
            for (int m = 0; m < kSeriesRegs; ++m) {
                const int i = lane + 32 * m;
                if (32 * m < n && i > q && i + 1 < n) s[m] = sb(s[m], mm(mine[i - q], h, M), p);
            }
        }
        uint32_t *g = logs + ((size_t)pi * sp.n_rects + j) * n;
        if (lane == 0) g[0] = 0;
#pragma unroll
        for (int m = 0; m < kSeriesRegs; ++m) {
            const int i = lane + 32 * m;
            if (i + 1 < n) g[i + 1] = mm(s[m], inv[i + 1], M);
        }
    }
    // the prime's last block goes on
    __threadfence();
    __syncthreads();
    if (tid == 0) last = atomicInc(finished + pi, gridDim.x - 1) == gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    for (int r = tid; r < 3 * sp.n_rects; r += blockDim.x) {
        const int x = r / sp.n_rects, k = r - x * sp.n_rects;
        wgt[x][k] = from_int(flm_weight(x, sp.k, rects[k].x, rects[k].y), p);
    }
    __syncthreads();
    for (int r = tid; r < 3 * n; r += blockDim.x) {  // work[x][q] = q a_q of series x
        const int x = r / n, i = r - x * n;
        uint32_t a = 0;
        for (int k = 0; k < sp.n_rects; ++k)
            a = ad(a, mm(wgt[x][k], __ldcg(logs + ((size_t)pi * sp.n_rects + k) * n + i), M), p);
        work[x][i] = mm(a, (uint32_t)i, M);
    }
    __syncthreads();
    const int x = warp;
    if (x == 3 && sp.add_mu) {
        const uint32_t mu = mu_mod(2 * sp.mmax, M, inv, tmp, lane);
        if (lane == 0) work[3][0] = mu;
    }
    if (x < 3) {
        // E = exp(a): E_0 = 1, i E_i = sum_{q=1..i} q a_q E_{i-q}
        uint32_t s[kSeriesRegs];
#pragma unroll
        for (int m = 0; m < kSeriesRegs; ++m) s[m] = lane + 32 * m < n ? mine[lane + 32 * m] : 0u;  // E_0's part of i E_i
        if (lane == 0) s[0] = 1;  // E_0 itself
        for (int q = 1; q < n; ++q) {
            const uint32_t e = mm(lane_value(s, q), inv[q], M);
#pragma unroll
            for (int m = 0; m < kSeriesRegs; ++m) {
                const int i = lane + 32 * m;
                if (i == q) s[m] = e;
                else if (32 * m < n && i > q && i < n) s[m] = ad(s[m], mm(mine[i - q], e, M), p);
            }
        }
        __syncwarp();
#pragma unroll
        for (int m = 0; m < kSeriesRegs; ++m)
            if (lane + 32 * m < n) mine[lane + 32 * m] = s[m];
    }
    __syncthreads();
    if (x < 3) {
        uint32_t *o = out + ((size_t)x * sp.P + pi) * n;
        const bool sq = sp.lattice == CP_SQUARE;
        for (int i = lane; i < n; i += 32) {
            uint32_t v = mine[i];
            if (x == 0) {  // (1 +- t)^2 E
                if (i >= 1) v = sq ? ad(v, mm(2, mine[i - 1], M), p) : sb(v, mm(2, mine[i - 1], M), p);
                if (i >= 2) v = ad(v, mine[i - 2], p);
            }
            // first-order: exp(f + c t^{n-1}) = exp(f) (1 + c t^{n-1}) mod t^n; series 0 and 1 start with 1
            if (i == n - 1 && sp.add_mu && x < 2)
                v = ad(v, x == 0 ? work[3][0] : sb(0, mm((uint32_t)sp.mmax, work[3][0], M), p), p);
            o[i] = v;
        }
    }
}

size_t series_scratch_words(const SeriesParams &sp) { return (size_t)sp.P * sp.n_rects * sp.n + sp.P; }

int launch_flm_series(uint32_t *ptilde, const int2 *rects, const uint32_t *primes, const SeriesParams &sp,
                      uint32_t *scratch, uint32_t *out, int *err, cudaStream_t st) {
    if (sp.n_rects > kMaxSeriesRects) return fail(CP_EINVAL, "too many rectangles for the series kernel");
    const size_t shm = (size_t)sp.n * (sp.n + 1) * 4;
    CP_CUDA_TRY(cudaFuncSetAttribute(flm_series_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     kMaxSeries * (kMaxSeries + 1) * 4));
    const dim3 grid((sp.n_rects + kSeriesWarps - 1) / kSeriesWarps, sp.P);
    uint32_t *finished = scratch + (size_t)sp.P * sp.n_rects * sp.n;
    flm_series_kernel<<<grid, 32 * kSeriesWarps, shm, st>>>(ptilde, rects, primes, sp, scratch, finished, out, err);
    CP_CUDA_TRY(cudaGetLastError());
    return CP_OK;
}

}  // namespace cp
