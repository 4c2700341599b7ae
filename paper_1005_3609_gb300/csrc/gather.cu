// The per-site operator kernel: one sparse factor T_i (or T_i^last) applied to
// a state vector, as a gather over the factor's CSR-by-destination table.
//
//   out[dst][d][p] = sum_{e in CSR(dst)} coef_e * in[src_e][d - shift_e][p]   (mod p)
//
// with in[..][d < 0] = 0 and degrees above D dropped: multiplying by w = 1/q
// is a shift of the coefficient index (Sec. 3.1, 3.5).  Rows are laid out
// [state][degree][prime], so a shift by one degree is a shift by n_primes
// words and, for n_primes % 4 == 0, every access is an aligned 16-byte load
// that reads four primes of one degree.  The coefficients are exact integers:
// each term coef * x (|x| <= p < 2^31: inputs are residues or the signed
// representatives in [-p, p) that intermediate launches store) is added to a
// signed 64-bit accumulator and
// the sum is reduced modulo p once per word (Sec. 3.5), in integer arithmetic
// only (modred.cuh).  Only the degrees in the states' windows (cp_internal.h)
// are read, computed and written.
//
// One launch processes a batch of independent tasks (factors of different
// strips); each block belongs to one task and covers 8 * rpw consecutive
// destination rows of it, one warp per row at a time.
#include <cuda_runtime.h>

#include <algorithm>
#include <mutex>
#include <string>

#include "cp_internal.h"
#include "modred.cuh"

namespace cp {

__device__ __forceinline__ uint32_t reduce(long long acc, const ModRed &mr) {
    return modred_reduce(acc, mr.p, mr.m, mr.s);
}

__device__ __forceinline__ int edge_coef(uint32_t e, uint32_t sb) { return (int)e >> (sb + 2); }
__device__ __forceinline__ uint32_t edge_shift(uint32_t e, uint32_t sb) { return (e >> sb) & 3u; }
__device__ __forceinline__ uint32_t edge_src(uint32_t e, uint32_t sb) { return e & ((1u << sb) - 1u); }
__device__ __forceinline__ uint32_t fast_div(uint32_t x, uint32_t magic) { return magic ? __umulhi(x, magic) : x; }

constexpr int kWarps = kGatherThreads / 32;
constexpr unsigned kFull = 0xffffffffu;

// The degrees [lo, hi) that an edge contributes to its destination.
struct EdgeWin {
    int lo, hi;
};
__device__ __forceinline__ EdgeWin edge_window(const GatherTask &t, const uint2 &q, int dcap_in, int dv) {
    const int sh = (int)edge_shift(q.x, t.src_bits), lo = (int)(q.y & 0xffu);
    const int hi = min(dcap_in, t.v_in + dv - (int)((q.y >> 8) & 0xffu)) + 1;
    return lo == 0xff ? EdgeWin{0, 0} : EdgeWin{lo + sh, hi + sh};
}

// 16 (4) bytes from global memory where pred != 0, else zero, without a branch.
template <bool V4>
__device__ __forceinline__ uint4 load_if(const uint32_t *in, size_t off, uint32_t pred) {
    uint4 v = make_uint4(0, 0, 0, 0);
    if (V4)
        asm("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %5, 0;\n\t@p ld.global.nc.v4.u32 {%0, %1, %2, %3}, [%4];\n\t}"
            : "+r"(v.x), "+r"(v.y), "+r"(v.z), "+r"(v.w)
            : "l"(reinterpret_cast<const uint4 *>(in) + off), "r"(pred));
    else
        asm("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %2, 0;\n\t@p ld.global.nc.u32 %0, [%1];\n\t}"
            : "+r"(v.x)
            : "l"(in + off), "r"(pred));
    return v;
}

// acc += coef * in[src][chunk c - shift*cpd], for the edges held one per lane
// in `my` and `win` (edge j in lane j), kFlight loads in flight per lane.
// deg0, deg1: the lowest and the highest degree of the warp's chunks; edges that
// reach none of them are passed over.  A launch lasts as long as its heaviest row, a
// chain of dependent steps of kFlight edges: with a branch per load instead of a
// predicate and every edge walked, square 12 x 13 on 8 primes with one and eight rows a
// warp took 7.3 and 18.9 ms (on whole rows, before degree windows, 6.0 and 12.3), now 3.8
// and 8.9.
template <int kFlight, bool V4>
__device__ __forceinline__ void gather_edges(const GatherTask &t, uint32_t my, const EdgeWin &win, int n, uint32_t c,
                                             int deg, int deg0, int deg1, bool active, long long *acc) {
    uint32_t left = __ballot_sync(kFull, (int)(threadIdx.x & 31) < n && win.lo <= deg1 && win.hi > deg0);
    while (left) {
        uint32_t q[kFlight];
        uint4 x[kFlight];
#pragma unroll
        for (int j = 0; j < kFlight; ++j) {
            const int e = left ? __ffs((int)left) - 1 : 0;
            q[j] = __shfl_sync(kFull, my, e);
            const int lo = __shfl_sync(kFull, win.lo, e), hi = __shfl_sync(kFull, win.hi, e);
            const uint32_t sh = edge_shift(q[j], t.src_bits);
            const size_t off = (size_t)edge_src(q[j], t.src_bits) * t.C + (c - sh * t.cpd);
            x[j] = load_if<V4>(t.in, off, left && active && deg >= lo && deg < hi ? 1u : 0u);
            left &= left - 1;
        }
#pragma unroll
        for (int j = 0; j < kFlight; ++j) {
            const long long cf = edge_coef(q[j], t.src_bits);  // absent edges loaded zero
            acc[0] += (long long)(int)x[j].x * cf;
            if (V4) {
                acc[1] += (long long)(int)x[j].y * cf;
                acc[2] += (long long)(int)x[j].z * cf;
                acc[3] += (long long)(int)x[j].w * cf;
            }
        }
    }
}

// One warp per destination row: the row's CSR entries are read once (two
// row_ptr words, then the edge list one edge per lane, each with its source's
// window) and broadcast with shuffles; the lanes sweep the chunks of the row's
// window 32 at a time.  The next row's CSR is fetched while the current row is
// computed.
template <int kFlight, bool V4>
__device__ __forceinline__ void gather_rows(const GatherTask &t, uint32_t row0, int rpw, const ModRed *s_mr, int dv,
                                            int first) {
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int dcap_in = first || t.first ? 0 : t.cap;
    uint32_t row = row0 + warp;
    uint32_t rp = (row < t.rows && lane < 2) ? __ldg(t.row_ptr + row + lane) : 0;
    uint32_t e0 = __shfl_sync(kFull, rp, 0), ne = __shfl_sync(kFull, rp, 1) - e0;
    uint2 my = (row < t.rows && lane < ne) ? __ldg(t.edges + e0 + lane) : make_uint2(0, 0);
#pragma unroll 1
    for (int k = 0; k < rpw; ++k) {
        if (row >= t.rows) return;
        const uint32_t nrow = row + kWarps;
        uint32_t nrp = (k + 1 < rpw && nrow < t.rows && lane < 2) ? __ldg(t.row_ptr + nrow + lane) : 0;
        const uint32_t w = __ldg(t.win_out + row);
        const int lo = (int)(w & 0xffu);
        const int end = lo == 0xff ? 0 : min(t.cap, t.v_out + dv - (int)(w >> 8)) + 1;
        const EdgeWin win = (lo < end && lane < ne) ? edge_window(t, my, dcap_in, dv) : EdgeWin{0, 0};
        const uint32_t c_end = (uint32_t)max(end, 0) * t.cpd;
#pragma unroll 1
        for (uint32_t j = (uint32_t)lo * t.cpd; j < c_end; j += 32) {
            const uint32_t c = j + lane;
            const bool active = c < c_end;
            const uint32_t deg = fast_div(c, t.magic_cpd);
            const int deg0 = (int)fast_div(j, t.magic_cpd), deg1 = (int)fast_div(min(j + 32, c_end) - 1, t.magic_cpd);
            const uint32_t pc = (c - deg * t.cpd) * (V4 ? 4 : 1);  // prime of the first word
            long long acc[4] = {modred_bias(s_mr[pc].p), V4 ? modred_bias(s_mr[pc + 1].p) : 0,
                                V4 ? modred_bias(s_mr[pc + 2].p) : 0, V4 ? modred_bias(s_mr[pc + 3].p) : 0};
            gather_edges<kFlight, V4>(t, my.x, win, (int)min(ne, 32u), c, (int)deg, deg0, deg1, active, acc);
            for (uint32_t eb = 32; eb < ne; eb += 32) {  // rows with more than 32 edges
                const uint2 mb = (eb + lane < ne) ? __ldg(t.edges + e0 + eb + lane) : make_uint2(0, 0);
                const EdgeWin wb = (eb + lane < ne) ? edge_window(t, mb, dcap_in, dv) : EdgeWin{0, 0};
                gather_edges<kFlight, V4>(t, mb.x, wb, (int)min(ne - eb, 32u), c, (int)deg, deg0, deg1, active, acc);
            }
            if (active) {
                const size_t o = (size_t)row * t.C + c;
                if (V4) {
                    const uint4 r = make_uint4(reduce(acc[0], s_mr[pc]), reduce(acc[1], s_mr[pc + 1]),
                                               reduce(acc[2], s_mr[pc + 2]), reduce(acc[3], s_mr[pc + 3]));
                    __stcs(reinterpret_cast<uint4 *>(t.out) + o, r);
                } else {
                    __stcs(t.out + o, reduce(acc[0], s_mr[pc]));
                }
            }
        }
        row = nrow;
        e0 = __shfl_sync(kFull, nrp, 0);
        ne = __shfl_sync(kFull, nrp, 1) - e0;
        my = (row < t.rows && lane < ne) ? __ldg(t.edges + e0 + lane) : make_uint2(0, 0);
    }
}

template <int kFlight, int N>
__global__ void __launch_bounds__(kGatherThreads)
    gather_kernel(const __grid_constant__ TaskPack<N> pack, int n_tasks, int rpw, int dv, int first) {
    __shared__ ModRed s_mr[CP_MAX_PRIMES];
    const GatherTask &t = pack.t[find_task(pack, n_tasks, blockIdx.x)];
    if (threadIdx.x < t.n_primes) {
        s_mr[threadIdx.x] = modred_make(__ldg(t.primes + threadIdx.x));
    }
    __syncthreads();
    // rows of the block: row0 + warp + 8 k, k < rpw
    const uint32_t row0 = (blockIdx.x - t.block_begin) * (uint32_t)(kWarps * rpw);
    if (t.vec4) gather_rows<kFlight, true>(t, row0, rpw, s_mr, dv, first);
    else gather_rows<kFlight, false>(t, row0, rpw, s_mr, dv, first);
}

bool tile_is_chunk(int items) { return (items & 0xFFF) >= 16; }

uint32_t task_blocks(const GatherTask &t, int items) {
    if (tile_is_chunk(items)) return t.n_units;
    const uint32_t per = (uint32_t)(kWarps * items);
    return (t.rows + per - 1) / per;
}

// A batch the chunk kernel cannot take uses the register kernel.
int effective_tile(const std::vector<GatherTask> &tasks, int items) {
    if (!tile_is_chunk(items)) return items & 0xFFF;
    for (auto &t : tasks)
        if (!chunk_usable(t)) return kGatherItems;
    return items;
}

bool tile_valid(int tile) {
    const int rows = tile & 0xFFF, ring = (tile >> 12) & 0xFF, edges = (tile >> 20) & 15, cpt = (tile >> 24) & 15;
    if (rows == 1 || rows == 2 || rows == 4 || rows == 8) return (tile >> 12) == 0;
    return (rows == 16 || rows == 32 || rows == 64 || rows == 128) && (tile >> 30) == 0 && ((tile >> 28) & 3) != 3 &&
           (ring == 0 || (ring >= 16 && ring <= 192)) && (edges <= 2 || edges == 4 || edges == 8) &&
           (cpt <= 2 || cpt == 4);
}

uint32_t assign_blocks(std::vector<GatherTask> &tasks, int items) {
    uint32_t blk = 0;
    for (auto &t : tasks) {
        t.block_begin = blk;
        blk += task_blocks(t, items);
    }
    return blk;
}

// ceil(2^32 / d) for d >= 2 (0 encodes d == 1).
static uint32_t magic_for(uint32_t d) { return d <= 1 ? 0u : (uint32_t)(((1ull << 32) + d - 1) / d); }

void fill_prime_block(const uint32_t *primes, int n_primes, int lanes, uint32_t *block) {
    for (int k = 0; k < lanes; ++k) {
        block[k] = primes[std::min(k, n_primes - 1)];
        block[CP_MAX_PRIMES + k] = chunk_magic(block[k]);
    }
}

bool table_fast(const SiteTable &tab, uint32_t min_prime) {
    return tab.max_abs_coef <= kChunkMaxCoef && fast_ok(tab.max_coef_sum, min_prime);
}

void append_gather_task(std::vector<GatherTask> *tasks, const SiteTable &tab, const uint32_t *in, uint32_t *out,
                        const uint32_t *primes_dev, int D1, int P, int v_in, uint32_t min_prime, bool final) {
    const bool v4 = (P % 4) == 0;
    const uint32_t vec = v4 ? 4 : 1;
    GatherTask t{};
    t.in = in;
    t.out = out;
    t.row_ptr = tab.row_ptr;
    t.edges = tab.wedges;
    t.primes = primes_dev;
    t.win_out = tab.win_out;
    t.units = tab.units;
    t.n_units = tab.n_units;
    t.rows = (uint32_t)tab.n_dst;
    t.C = (uint32_t)((uint64_t)D1 * P / vec);
    t.cpd = (uint32_t)P / vec;
    t.vec4 = v4 ? 1 : 0;
    t.magic_cpd = magic_for(t.cpd);
    t.seg = 32u * kChunkSteps / std::min(t.cpd, 32u * kChunkSteps);
    t.r32 = 32u % t.cpd;
    t.n_primes = (uint32_t)P;
    t.src_bits = (uint32_t)tab.op.src_bits;
    t.chunk = v4 && tab.max_abs_coef <= kChunkMaxCoef && tab.max_coef_sum < kChunkMaxSum ? 1u : 0u;
    t.fast = table_fast(tab, min_prime) ? 1u : 0u;
    t.fast_k0 = fast_offset(tab.max_coef_sum);
    t.v_in = v_in;
    t.v_out = final ? kFinalVertices : v_in + tab.sites;
    t.cap = D1 - 1;
    tasks->push_back(t);
}

int launch_gather_chunk(const GatherTask *tasks, int n_tasks, uint32_t n_units, cudaStream_t st, int dv, bool first);

// Launches of up to three waves of resident blocks (two of them per SM with 98 registers,
// 152 SMs) keep eight loads in flight instead of four: there the heaviest row's chain is
// what they last.  Four and eight: square 12 x 12 on 8 primes, two rows a warp (499 blocks)
// 4.60 and 3.87 ms, width 13, two rows (1332 blocks) 1.64 and 1.67, one row (2664) 1.35 and
// 1.71; short rows of one-factor tables lose 3 to 10% below the line.
constexpr uint32_t kFewBlocks = 3 * 2 * 152;

static int launch_gather_rows(const GatherTask *tasks, int n_tasks, uint32_t total_blocks, int rpw, cudaStream_t st, int dv,
                              bool first) {
    return for_packs(tasks, n_tasks, total_blocks, [&](const auto &pack, int n, uint32_t blocks) -> int {
        constexpr int N = sizeof(pack.t) / sizeof(GatherTask);
        if (!blocks) return CP_OK;
        if (blocks <= kFewBlocks) gather_kernel<8, N><<<blocks, kGatherThreads, 0, st>>>(pack, n, rpw, dv, first ? 1 : 0);
        else gather_kernel<4, N><<<blocks, kGatherThreads, 0, st>>>(pack, n, rpw, dv, first ? 1 : 0);
        CP_CUDA_TRY(cudaGetLastError());
        return CP_OK;
    });
}

int launch_gather(const GatherTask *tasks, int n_tasks, uint32_t total_blocks, int items, cudaStream_t st, int dv,
                  bool first) {
    if (n_tasks <= 0 || total_blocks == 0) return CP_OK;
    if (tile_is_chunk(items)) return launch_gather_chunk(tasks, n_tasks, total_blocks, st, dv, first);
    const int rpw = items & 0xFFF;
    if (rpw != 1 && rpw != 2 && rpw != 4 && rpw != 8)
        return fail(CP_EINVAL, "gather tile must be 1, 2, 4, 8, 16, 32, 64 or 128");
    return launch_gather_rows(tasks, n_tasks, total_blocks, rpw, st, dv, first);
}

int prepare_gather_kernels() {
    return device_error_flag() ? CP_OK : CP_ECUDA;
}

// An error word in pinned host memory, mapped on the device: the host reads it after a
// synchronisation without a copy of its own (a blocking 4-byte copy took about 8 us of
// every read-out and of every server step).
int error_word_alloc(ErrorWord *w) {
    CP_CUDA_TRY(cudaHostAlloc((void **)&w->host, sizeof(int), cudaHostAllocMapped | cudaHostAllocPortable));
    *w->host = 0;
    const cudaError_t e = cudaHostGetDevicePointer((void **)&w->dev, w->host, 0);
    if (e != cudaSuccess) {
        error_word_free(w);
        return fail(CP_ECUDA, std::string("error word: ") + cudaGetErrorString(e));
    }
    return CP_OK;
}

void error_word_free(ErrorWord *w) {
    if (w->host) cudaFreeHost(w->host);
    *w = ErrorWord{};
}

int error_word_take(const ErrorWord &w) { return __atomic_exchange_n(w.host, 0, __ATOMIC_ACQ_REL); }

static std::mutex g_err_mu;
static ErrorWord *device_error_word() {
    static ErrorWord words[64];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return nullptr;
    std::lock_guard<std::mutex> lk(g_err_mu);
    if (!words[dev].host && error_word_alloc(&words[dev])) return nullptr;
    return &words[dev];
}

int *device_error_flag() {
    ErrorWord *w = device_error_word();
    return w ? w->dev : nullptr;
}

int check_device_error(cudaStream_t st) {
    ErrorWord *w = device_error_word();
    if (!w) return fail(CP_ECUDA, "device error word unavailable");
    CP_CUDA_TRY(cudaStreamSynchronize(st));
    const int h = error_word_take(*w);
    if (h) return fail(CP_ETIMEOUT, "a bounded wait on the device ran out (flags " + std::to_string(h) + ")");
    return CP_OK;
}

// [D1][Pp] signed representatives -> [P][D1] residues
__global__ void transpose_row_kernel(const uint32_t *row, uint32_t *out, const uint32_t *primes, int D1, int P, int Pp) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= D1 * P) return;
    const int p = k / D1, d = k - p * D1;
    const uint32_t x = row[(size_t)d * Pp + p];
    out[k] = (int)x < 0 ? x + primes[p] : x;
}

int launch_transpose_row(const uint32_t *row, uint32_t *out, const uint32_t *primes_dev, int D1, int P, int Pp,
                         cudaStream_t st) {
    const int n = D1 * P;
    transpose_row_kernel<<<(n + 255) / 256, 256, 0, st>>>(row, out, primes_dev, D1, P, Pp);
    CP_CUDA_TRY(cudaGetLastError());
    return CP_OK;
}

// Diagnostic: the gathers' reduction applied to given accumulator values.
__global__ void debug_reduce_kernel(const long long *v, const uint32_t *p, int n, uint32_t *out) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    const ModRed mr = modred_make(p[k]);
    out[k] = reduce(modred_bias(mr.p) + v[k], mr);
}

}  // namespace cp

extern "C" int cp_debug_reduce(const int64_t *v_host, const uint32_t *p_host, int n, uint32_t *out_host) {
    using namespace cp;
    if (n < 0 || (n > 0 && (!v_host || !p_host || !out_host))) return fail(CP_EINVAL, "bad arguments");
    for (int k = 0; k < n; ++k) {
        const uint32_t p = p_host[k];
        if (p < 2 || p >= (1u << 31)) return fail(CP_EINVAL, "p must be in [2, 2^31)");
        const long long lim = (long long)p * (long long)kReduceMaxCoefSum;
        if (v_host[k] <= -lim || v_host[k] >= lim) return fail(CP_EINVAL, "|v| must be below p * 2^20");
    }
    if (n == 0) return CP_OK;
    long long *v_d = nullptr;
    uint32_t *p_d = nullptr, *o_d = nullptr;
    int rc = dev_alloc((void **)&v_d, 8ull * n);
    if (!rc) rc = dev_alloc((void **)&p_d, 4ull * n);
    if (!rc) rc = dev_alloc((void **)&o_d, 4ull * n);
    cudaError_t e = cudaSuccess;
    if (!rc) {
        e = cudaMemcpy(v_d, v_host, 8ull * n, cudaMemcpyHostToDevice);
        if (e == cudaSuccess) e = cudaMemcpy(p_d, p_host, 4ull * n, cudaMemcpyHostToDevice);
        if (e == cudaSuccess) {
            debug_reduce_kernel<<<(n + 255) / 256, 256>>>(v_d, p_d, n, o_d);
            e = cudaGetLastError();
        }
        if (e == cudaSuccess) e = cudaMemcpy(out_host, o_d, 4ull * n, cudaMemcpyDeviceToHost);
    }
    dev_free(v_d);
    dev_free(p_d);
    dev_free(o_d);
    if (rc) return rc;
    if (e != cudaSuccess) return fail(CP_ECUDA, std::string("cp_debug_reduce: ") + cudaGetErrorString(e));
    return CP_OK;
}
